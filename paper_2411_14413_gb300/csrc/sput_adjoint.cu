// sput_adjoint.cu -- likelihood-ratio backward pass and the arrival-count ->
// composition map with its backward pass (sm_103a).
//
// Pressure enters the transport only through the free flights (Eq. for
// lambda: lambda_m = v / (n_g <sigma g>), n_g = p / (k_B T)).  The forward
// kernel accumulates for every landing atom the score
//   S = sum over collisions (1 - l_k/lambda_k) - t_land/lambda_land
//     = d ln p(path) / d ln n_g,
// per tally cell.  Hence d E[count_c] / d ln p = E[sum_{atoms in c} S]; the
// backward kernel contracts dL/dcount with that score tally.
//
// Composition (Methods paragraph after Table 1: arrival fractions weighted
// with the sputter rates, then with bulk density and atomic mass, in at.%):
//   a_j(m) = R_j(P_j) * N_j(m) / N_j(ref) * rho_j / M_j,   c_j(m) = 100 a_j(m) / sum_k a_k(m),
// N_j(m) the arrivals of cathode j summed over measurement patch m, ref the
// central patch, R_j linear in power through two calibration points.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>

#include "sput.h"
#include "sput_internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCath = 16;

// Blocks of the cluster that reduces one instance (or the composition backward): one block per
// instance left 148 of 152 SMs idle on a four-cathode map and waited on its own loads.  The
// partial sums meet in the first block's shared memory and are added in block order, so the
// result does not depend on timing.
constexpr int kCluster = 8;
constexpr int kReduceThreads = 512;

struct CompParams {
    int n_cath, n_cells, n_points, ref;
    double R[kMaxCath];      // R_j(P_j)
    double dRdP[kMaxCath];   // slope of the rate line
    double w[kMaxCath];      // rho_j / M_j
};

__device__ double warp_sum(double x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
}

// Another block's shared memory may be touched only once that block has started: every thread
// arrives at the cluster's barrier when its kernel starts, and waits there for the others just
// before the stores to the first block, behind the kernel's own loads.
__device__ void cluster_started() { cg::cluster_group::barrier_arrive(); }
__device__ void cluster_wait() { cg::cluster_group::barrier_wait(); }

// Sum of x over the threads of the cluster, in thread 0 of its first block; part: shared memory of
// kCluster + 32 doubles; the kernel called cluster_started() first.  The last step is a cluster barrier: no block ends before the stores to it.
__device__ double cluster_sum(double x, double* part)
{
    cg::cluster_group cl = cg::this_cluster();
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) part[kCluster + (threadIdx.x >> 5)] = x;
    __syncthreads();
    cluster_wait();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x >> 5) ? part[kCluster + threadIdx.x] : 0.0;
        t = warp_sum(t);
        if (threadIdx.x == 0) cl.map_shared_rank(part, 0)[cl.block_rank()] = t;
    }
    cl.sync();
    double s = 0.0;
    if (threadIdx.x == 0 && cl.block_rank() == 0)
        for (int b = 0; b < kCluster; ++b) s += part[b];
    return s;
}

// grad[i] = sum_c g[i][c] * score[i][c], one cluster per instance.  16 bytes per cell; at 4 x 40000
// cells bound by latency: 31 us with one block of 256 threads per instance, 7.5 us so (under ncu).
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kReduceThreads)
    lr_backward_kernel(const double* g, const double* score, double* grad, long long n_cells)
{
    __shared__ double part[kCluster + 32];
    cluster_started();
    const int inst = blockIdx.x / kCluster;
    const long long base = (long long)inst * n_cells;
    double s = 0.0;
#pragma unroll 4
    for (long long c = (long long)(blockIdx.x % kCluster) * blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)kCluster * blockDim.x)
        s += g[base + c] * score[base + c];
    s = cluster_sum(s, part);
    if (threadIdx.x == 0 && blockIdx.x % kCluster == 0) grad[inst] = s;
}

// Derivative with respect to the Thompson cut-off.  The launch energy has the
// density p(E) = E/(E+U)^3 / Z(E_max) on (0, E_max], Z = E_max^2 / (2U (E_max+U)^2),
// so d ln p(E)/dE_max = -p(E_max) for every E inside the support, and the moving
// end of the support adds p(E_max) E[f | E = E_max]:
//   d E[f]/dE_max = p(E_max) (E[f | E = E_max] - E[f]),  p(E_max) = 2U / (E_max (E_max + U)).
// With a boundary run of the same particles launched at E_max (counts_cut) and
// dE_max/dE_i = k Lambda, one cluster per instance forms
//   grad[i] = k Lambda p(E_max) sum_c g[i][c] (counts_cut[i][c] - counts[i][c]).
// Voltage lines V_i(P) = V_a + (V_b - V_a)(P - P_a)/(P_b - P_a) (Table S1), with
// E_i = e V for singly charged ions: dE_i/dP_i in eV/W per instance.
struct VoltParams {
    double dEdP[kMaxCath];
};

// grad_power (optional) gets grad[i] * dE_i/dP_i added: the path from the cathode
// power through the discharge voltage to the cut-off.
template <typename CountT>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kReduceThreads)
    emax_backward_kernel(const double* g, const CountT* counts, const CountT* counts_cut, const sput::DevInstance* inst,
                         double* grad, long long n_cells, double* grad_power, VoltParams vp)
{
    __shared__ double part[kCluster + 32];
    cluster_started();
    const int i = blockIdx.x / kCluster;
    const long long base = (long long)i * n_cells;
    double s = 0.0;
#pragma unroll 4
    for (long long c = (long long)(blockIdx.x % kCluster) * blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)kCluster * blockDim.x)
        s += g[base + c] * ((double)counts_cut[base + c] - (double)counts[base + c]);
    const double t = cluster_sum(s, part);
    if (threadIdx.x == 0 && blockIdx.x % kCluster == 0) {
        const sput::DevInstance I = inst[i];
        const double q = I.thompson_q, U = I.U_s;
        const double Em = U * q / (1.0 - q);
        const double gE = (double)I.kLambda * 2.0 * U / (Em * (Em + U)) * t;
        grad[i] = gE;
        if (grad_power) grad_power[i] += gE * vp.dEdP[i];
    }
}

// N[j][m] = sum of counts of cathode j over the cells of patch m; blockIdx.y = j
__global__ void patch_sum_kernel(const long long* counts, const int32_t* patch, double* N, int n_cells, int n_points)
{
    const int j = blockIdx.y;
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)n_cells; c += gridDim.x * blockDim.x) {
        const int m = patch[c];
        const long long n = counts[(size_t)j * n_cells + c];
        if (m >= 0 && m < n_points && n) atomicAdd(N + (size_t)j * n_points + m, (double)n);
    }
}

// a_j(m) = W_j N_j(m) with W_j = R_j w_j / N_j(ref), 0 where the reference point is empty
__device__ double arrival_weight(const double* N, const CompParams& cp, int j)
{
    const double nref = N[(size_t)j * cp.n_points + cp.ref];
    return nref > 0.0 ? cp.R[j] * cp.w[j] / nref : 0.0;
}

// One thread per point, 32 to a block: FP64 runs at two FMAs per clock on an SM, so the points are
// spread over SMs and each divides once (the weights are divided once per block).
__global__ void composition_kernel(const double* N, double* comp, CompParams cp)
{
    __shared__ double W[kMaxCath];
    if (threadIdx.x < cp.n_cath) W[threadIdx.x] = arrival_weight(N, cp, threadIdx.x);
    __syncwarp();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= cp.n_points) return;
    double a[kMaxCath], A = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxCath; ++j)
        if (j < cp.n_cath) {
            a[j] = W[j] * N[(size_t)j * cp.n_points + m];
            A += a[j];
        }
    const double scale = A > 0.0 ? 100.0 / A : 0.0;
#pragma unroll
    for (int j = 0; j < kMaxCath; ++j)
        if (j < cp.n_cath) comp[(size_t)m * cp.n_cath + j] = scale * a[j];
}

// dL/dN[j][m] and dL/dP_j from dL/dc[m][j]; one cluster of 32-thread blocks.
//   dL/da_j(m) = (100/A) (g_j - sum_k g_k c_k / 100)
// a_j(m) depends on N_j(m), on N_j(ref) through 1/N_j(ref) and on R_j linearly, so with
// S_j = sum_m a_j dL/da_j: dL/dN_j(ref) gets -S_j / N_j(ref) and dL/dR_j = S_j / R_j.
// One block added 2 n_cath values per point with FP64 atomics on a handful of shared-memory
// words: 95 us for 342 points and four cathodes; so 15 us (under ncu).
__global__ void __cluster_dims__(kCluster, 1, 1)
    composition_backward_kernel(const double* N, const double* gc, double* gN, double* gP, CompParams cp)
{
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double W[kMaxCath];
    __shared__ bool on[kMaxCath];  // atoms at the reference point
    __shared__ double part[kCluster][kMaxCath];
    cluster_started();
    if (threadIdx.x < cp.n_cath) {
        W[threadIdx.x] = arrival_weight(N, cp, threadIdx.x);
        on[threadIdx.x] = N[(size_t)threadIdx.x * cp.n_points + cp.ref] > 0.0;
    }
    __syncwarp();
    double S[kMaxCath];
#pragma unroll
    for (int j = 0; j < kMaxCath; ++j) S[j] = 0.0;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < cp.n_points; m += gridDim.x * blockDim.x) {
        double a[kMaxCath], A = 0.0, gdota = 0.0;
#pragma unroll
        for (int j = 0; j < kMaxCath; ++j)
            if (j < cp.n_cath) {
                a[j] = W[j] * N[(size_t)j * cp.n_points + m];
                A += a[j];
                gdota += gc[(size_t)m * cp.n_cath + j] * a[j];
            }
        const bool off = A <= 0.0;
        const double scale = 100.0 / A;
        gdota /= A;
#pragma unroll
        for (int j = 0; j < kMaxCath; ++j)
            if (j < cp.n_cath) {
                const double ga = off ? 0.0 : scale * (gc[(size_t)m * cp.n_cath + j] - gdota);
                gN[(size_t)j * cp.n_points + m] = on[j] ? ga * W[j] : 0.0;
                S[j] += ga * a[j];
            }
    }
    __syncwarp();
    cluster_wait();
    double* first = cl.map_shared_rank(&part[0][0], 0);
#pragma unroll
    for (int j = 0; j < kMaxCath; ++j)
        if (j < cp.n_cath) {
            const double t = warp_sum(S[j]);
            if (threadIdx.x == 0) first[cl.block_rank() * kMaxCath + j] = t;
        }
    cl.sync();
    const int j = threadIdx.x;
    if (cl.block_rank() == 0 && j < cp.n_cath) {
        double t = 0.0;
        for (int b = 0; b < kCluster; ++b) t += part[b][j];
        const double nref = N[(size_t)j * cp.n_points + cp.ref];
        if (on[j]) gN[(size_t)j * cp.n_points + cp.ref] += -t / nref;
        gP[j] = cp.R[j] != 0.0 ? t / cp.R[j] * cp.dRdP[j] : 0.0;
    }
}

// dL/dcount[j][c] = dL/dN[j][patch(c)]
__global__ void scatter_kernel(const double* gN, const int32_t* patch, double* gcounts, int n_cells, int n_points)
{
    const int j = blockIdx.y;
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)n_cells; c += gridDim.x * blockDim.x) {
        const int m = patch[c];
        gcounts[(size_t)j * n_cells + c] = m >= 0 && m < n_points ? gN[(size_t)j * n_points + m] : 0.0;
    }
}

// grid of the kernels that run over every cell of every cathode
dim3 cell_grid(int n_cells, int n_cath)
{
    const int bx = (n_cells + 255) / 256;
    return dim3((unsigned)(bx < 1216 ? bx : 1216), (unsigned)n_cath);
}

sput_status adj_fail(sput_status s, const char* msg)
{
    sput::set_last_error(msg);
    return s;
}

sput_status comp_params(int n_cath, int n_cells, int n_points, int ref, const double* cal, const double* power,
                        CompParams& cp)
{
    if (n_cath < 1 || n_cath > kMaxCath) return adj_fail(SPUT_ERR_INVALID_ARG, "n_cathodes must be 1..16");
    if (n_cells < 1 || n_points < 1 || ref < 0 || ref >= n_points) return adj_fail(SPUT_ERR_INVALID_ARG, "bad sizes");
    if (!cal || !power) return adj_fail(SPUT_ERR_INVALID_ARG, "NULL calibration or power");
    std::memset(&cp, 0, sizeof cp);
    cp.n_cath = n_cath;
    cp.n_cells = n_cells;
    cp.n_points = n_points;
    cp.ref = ref;
    for (int j = 0; j < n_cath; ++j) {
        const double* q = cal + 6 * j;  // P_a, R_a, P_b, R_b, density, mass
        if (q[2] == q[0] || !(q[5] > 0.0)) return adj_fail(SPUT_ERR_INVALID_ARG, "bad calibration row");
        const double slope = (q[3] - q[1]) / (q[2] - q[0]);
        cp.R[j] = q[1] + slope * (power[j] - q[0]);
        cp.dRdP[j] = slope;
        cp.w[j] = q[4] / q[5];
    }
    return SPUT_OK;
}

}  // namespace

extern "C" {

sput_status sput_backward(const sput_scene* scene, const double* grad_counts, const double* score_tally,
                          double* grad_log_pressure, void* stream)
{
    sput::NvtxRange nvtx("sput_backward");
    if (!scene || !grad_counts || !score_tally || !grad_log_pressure) return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    sput_tally_layout L;
    sput_status st = sput_tally_layout_get(scene, &L);
    if (st != SPUT_OK) return st;
    const long long n_cells = (long long)L.nx * L.ny;
    lr_backward_kernel<<<L.n_instances * kCluster, kReduceThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        grad_counts, score_tally, grad_log_pressure, n_cells);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return adj_fail(SPUT_ERR_CUDA, cudaGetErrorString(e));
    return SPUT_OK;
}

}  // extern "C"

namespace {

sput_status emax_backward_launch(const sput_scene* scene, const double* grad_counts, const void* counts,
                                 const void* counts_cutoff, double* grad_ion_energy, double* grad_power,
                                 const VoltParams& vp, void* stream)
{
    sput_tally_layout L;
    sput_status st = sput_tally_layout_get(scene, &L);
    if (st != SPUT_OK) return st;
    if (grad_power && L.n_instances > kMaxCath)
        return adj_fail(SPUT_ERR_INVALID_ARG, "the voltage path supports at most 16 instances");
    const long long n_cells = (long long)L.nx * L.ny;
    const sput::DevInstance* inst = sput::scene_device_instances(scene);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (L.count_type == SPUT_COUNT_INT64)
        emax_backward_kernel<<<L.n_instances * kCluster, kReduceThreads, 0, s>>>(grad_counts, static_cast<const long long*>(counts),
                                                           static_cast<const long long*>(counts_cutoff), inst,
                                                           grad_ion_energy, n_cells, grad_power, vp);
    else
        emax_backward_kernel<<<L.n_instances * kCluster, kReduceThreads, 0, s>>>(grad_counts, static_cast<const int*>(counts),
                                                           static_cast<const int*>(counts_cutoff), inst,
                                                           grad_ion_energy, n_cells, grad_power, vp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return adj_fail(SPUT_ERR_CUDA, cudaGetErrorString(e));
    return SPUT_OK;
}

// slope dV/dP of each voltage line (P_a, V_a, P_b, V_b); E_i = e V, so dE_i/dP in eV/W
sput_status voltage_slopes(int n, const double* voltage, double* slope)
{
    if (n < 1 || !voltage) return adj_fail(SPUT_ERR_INVALID_ARG, "NULL voltage lines or no instance");
    for (int j = 0; j < n; ++j) {
        const double* q = voltage + 4 * j;
        if (!(q[2] != q[0]) || !std::isfinite(q[0]) || !std::isfinite(q[1]) || !std::isfinite(q[2]) ||
            !std::isfinite(q[3]))
            return adj_fail(SPUT_ERR_INVALID_ARG, "voltage line needs two finite points at distinct powers");
        slope[j] = (q[3] - q[1]) / (q[2] - q[0]);
    }
    return SPUT_OK;
}

}  // namespace

extern "C" {

sput_status sput_emax_backward(const sput_scene* scene, const double* grad_counts, const void* counts,
                               const void* counts_cutoff, double* grad_ion_energy, void* stream)
{
    sput::NvtxRange nvtx("sput_emax_backward");
    if (!scene || !grad_counts || !counts || !counts_cutoff || !grad_ion_energy)
        return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    VoltParams vp;
    std::memset(&vp, 0, sizeof vp);
    return emax_backward_launch(scene, grad_counts, counts, counts_cutoff, grad_ion_energy, nullptr, vp, stream);
}

sput_status sput_ion_energy(int n, const double* voltage, const double* power, double* ion_energy)
{
    if (!power || !ion_energy) return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    if (n > 4096) return adj_fail(SPUT_ERR_INVALID_ARG, "at most 4096 lines");
    for (int j = 0; j < n; ++j) {
        double slope;
        sput_status st = voltage_slopes(1, voltage + 4 * j, &slope);
        if (st != SPUT_OK) return st;
        if (!std::isfinite(power[j])) return adj_fail(SPUT_ERR_INVALID_ARG, "power must be finite");
        const double* q = voltage + 4 * j;
        ion_energy[j] = q[1] + slope * (power[j] - q[0]);  // singly charged ions: eV = e * volts
    }
    return n >= 1 ? SPUT_OK : adj_fail(SPUT_ERR_INVALID_ARG, "no voltage line");
}

sput_status sput_voltage_backward(const sput_scene* scene, const double* voltage, const double* grad_counts,
                                  const void* counts, const void* counts_cutoff, double* grad_ion_energy,
                                  double* grad_power, void* stream)
{
    sput::NvtxRange nvtx("sput_voltage_backward");
    if (!scene || !grad_counts || !counts || !counts_cutoff || !grad_ion_energy || !grad_power)
        return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    sput_tally_layout L;
    sput_status st = sput_tally_layout_get(scene, &L);
    if (st != SPUT_OK) return st;
    if (L.n_instances > kMaxCath) return adj_fail(SPUT_ERR_INVALID_ARG, "the voltage path supports at most 16 instances");
    VoltParams vp;
    std::memset(&vp, 0, sizeof vp);
    st = voltage_slopes(L.n_instances, voltage, vp.dEdP);
    if (st != SPUT_OK) return st;
    return emax_backward_launch(scene, grad_counts, counts, counts_cutoff, grad_ion_energy, grad_power, vp, stream);
}

sput_status sput_composition(int n_cathodes, int n_cells, int n_points, const int64_t* counts, const int32_t* patch_of_cell,
                             int ref_point, const double* calibration, const double* power, double* patch_counts,
                             double* composition, void* stream)
{
    CompParams cp;
    sput_status st = comp_params(n_cathodes, n_cells, n_points, ref_point, calibration, power, cp);
    if (st != SPUT_OK) return st;
    if (!counts || !patch_of_cell || !patch_counts || !composition) return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(patch_counts, 0, sizeof(double) * (size_t)n_cathodes * n_points, s);
    if (e != cudaSuccess) return adj_fail(SPUT_ERR_CUDA, cudaGetErrorString(e));
    patch_sum_kernel<<<cell_grid(n_cells, n_cathodes), 256, 0, s>>>(reinterpret_cast<const long long*>(counts),
                                                                   patch_of_cell, patch_counts, n_cells, n_points);
    composition_kernel<<<(n_points + 31) / 32, 32, 0, s>>>(patch_counts, composition, cp);
    e = cudaGetLastError();
    if (e != cudaSuccess) return adj_fail(SPUT_ERR_CUDA, cudaGetErrorString(e));
    return SPUT_OK;
}

sput_status sput_composition_backward(int n_cathodes, int n_cells, int n_points, const double* patch_counts,
                                      const int32_t* patch_of_cell, int ref_point, const double* calibration,
                                      const double* power, const double* grad_composition, double* grad_patch,
                                      double* grad_counts, double* grad_power, void* stream)
{
    sput::NvtxRange nvtx("sput_composition_backward");
    CompParams cp;
    sput_status st = comp_params(n_cathodes, n_cells, n_points, ref_point, calibration, power, cp);
    if (st != SPUT_OK) return st;
    if (!patch_counts || !patch_of_cell || !grad_composition || !grad_patch || !grad_counts || !grad_power)
        return adj_fail(SPUT_ERR_INVALID_ARG, "NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    composition_backward_kernel<<<kCluster, 32, 0, s>>>(patch_counts, grad_composition, grad_patch, grad_power, cp);
    scatter_kernel<<<cell_grid(n_cells, n_cathodes), 256, 0, s>>>(grad_patch, patch_of_cell, grad_counts, n_cells,
                                                                 n_points);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return adj_fail(SPUT_ERR_CUDA, cudaGetErrorString(e));
    return SPUT_OK;
}

}  // extern "C"
