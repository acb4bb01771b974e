// sput_transport.cu -- persistent Monte Carlo transport kernel for sm_103a.
//
// One thread carries one sputtered atom at a time; a warp refills its dead
// lanes from a warp-private pool of tickets that it takes in chunks from one
// global counter, so every lane runs exactly one free flight per loop
// iteration (Sec. "The SIMTRA model": launch, free flight, surface test,
// binary collision, repeated until the atom lands).  A run's last atoms, and
// small runs, go to drain_kernel, which carries one atom with several lanes.
// The geometry is staged in shared memory; the rate, cross-section and
// deflection tables and the cell masks are read through L1/L2.  The scattering
// angle comes from a bicubic table of ln tan(chi/2) built from the classical
// deflection integral, and from Gauss-Mehler quadrature in FP32 outside the
// table's range.  Counts are integer atomics (bit-exact, order independent);
// energy and score sums are FP64 atomics.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cstdint>
#include <map>
#include <mutex>
#include <utility>

#include "sput_internal.h"

namespace sput {

namespace {

constexpr unsigned kFull = 0xffffffffu;
// kernel instances: the exact transport, with the temperature score, or with the
// diffusion shortcut for thermalised atoms (the two options exclude each other)
enum { kModePlain = 0, kModeScoreT = 1, kModeWalk = 2 };

// ----------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of two 32x32
// multiplies with the published multipliers, keyed by the seed's key schedule
// (Weyl increments), which the host writes into the kernel parameters
// (set_philox_keys): each round's key is an operand from the parameter bank, not
// an addition.  Inlined: an out-of-line call made the caller save registers
// around it at 64 registers a thread.
__device__ __forceinline__ uint4 philox(const Params& P, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ P.rk0[r];
        c1 = lo1;
        c2 = hi0 ^ c3 ^ P.rk1[r];
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// RN in ]0,1]: ((x >> 8) + 1) 2^-24, exact in FP32
__device__ __forceinline__ float rn(uint32_t x) { return (float)((x >> 8) + 1u) * 5.9604644775390625e-8f; }

// ------------------------------------------------------------- checked build
// Built with SPUT_CHECKED, every table window, cell, primitive, instance,
// counter and record index is tested against its buffer before the access: an
// index outside sets kStatusBadIndex in the run's status word and the access
// is skipped (a read falls back to index 0, a write is dropped), so the run
// ends normally and the call reports SPUT_ERR_DEVICE_CHECK.  The regular build
// compiles every test to true.
__device__ __forceinline__ bool idx_ok(unsigned int* status, long long i, long long n)
{
#ifdef SPUT_CHECKED
    if (i >= 0 && i < n) return true;
    if (status) atomicOr(status, kStatusBadIndex);  // the probe kernel runs without a status word
    return false;
#else
    (void)status;
    (void)i;
    (void)n;
    return true;
#endif
}

// ------------------------------------------------------------- MUFU functions
// Approximate functions for arguments that are no denormals: the forms that flush them spare the
// scaling around the MUFU (a comparison and two or three instructions each, some 25 in a flight
// and its collision) and give the same result for all others.
__device__ __forceinline__ float fast_lg2(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_div(float a, float b)
{
    float y;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
__device__ __forceinline__ float fast_ln(float x) { return fast_lg2(x) * 0.69314718056f; }
__device__ __forceinline__ float fast_exp(float x) { return fast_ex2(x * 1.44269504089f); }

// ------------------------------------------------------------- tables
// Cell and position of a table coordinate x in [0, n], top = 2^23 + n - 1: i = min(floor(x), n - 1),
// t = x - i.  The sum with 2^23, rounded down, holds floor(x) in its mantissa; a conversion to
// integer and back would go through the XU pipe, at a quarter of the rate and five times the
// latency.
__device__ __forceinline__ void table_cell(float x, float top, int& i, float& t)
{
    const float r = fminf(__fadd_rd(x, 8388608.0f), top);
    i = __float_as_int(r) & 0x7fffff;
    t = x - (r - 8388608.0f);
}

__device__ __forceinline__ float cubic(const float4& c, float t) { return fmaf(t, fmaf(t, fmaf(t, c.w, c.z), c.y), c.x); }

struct TableView {
    const float4* bm;
    const float* xh;
    const float4* w;
    const float4* gm;  // Gauss-Mehler nodes: kGMHalf of the kGMNodes rule, then kGMHalfLo of the kGMNodesLo rule
    const DevPair* pairs;
    const DevGeom* geoms;
    int n_w;           // entries of w (bounds of the checked build)
    float bm_n, bm_top;  // pieces of bm, and 2^23 + pieces - 1
    float bm_lo, bm_inv_h;
    unsigned int* status;
};

__device__ __forceinline__ float bmax_eval(const TableView& T, float ln_eps)
{
    int i;
    float t;
    table_cell(fminf(fmaxf((ln_eps - T.bm_lo) * T.bm_inv_h, 0.0f), T.bm_n), T.bm_top, i, t);
    return cubic(__ldg(T.bm + i), t);
}

__device__ __forceinline__ float xh_eval(const TableView& T, float ln_eps)
{
    int i;
    float t;
    table_cell(fminf(fmaxf((ln_eps - T.bm_lo) * T.bm_inv_h, 0.0f), T.bm_n), T.bm_top, i, t);
    return fmaf(t, T.xh[i + 1] - T.xh[i], T.xh[i]);
}

// The rate tables' coordinate w = ln(1 + v/s), from the MUFU logarithm: its error
// (about 4e-7 absolute) moves K, A and B far less than their interpolation error.
__device__ __forceinline__ float w_of(const DevPair& pr, float v) { return fast_ln(1.0f + v * pr.inv_s); }

// K(v), A(v), B(v) and G(v) of a pair: cubic pieces in w = ln(1 + v/s).  K, A and B lie beside one
// another (three float4 per piece), so one cell lookup serves all three.  The tables are read
// through L1 from global memory (a few KB per pair, L1-resident), which keeps them out of
// shared memory so that four blocks fit on an SM.
enum { kTabK = 0, kTabA = 1, kTabB = 2 };

__device__ __forceinline__ void wtab_cell(const DevPair& pr, float v, int& i, float& t)
{
    table_cell(fminf(fmaxf(w_of(pr, v) * pr.w_inv_h, 0.0f), pr.w_n), pr.w_top, i, t);
}

__device__ __forceinline__ float wtab_at(const TableView& T, const DevPair& pr, int which, int i, float t)
{
    if (!idx_ok(T.status, (long long)pr.K_off + 3 * i + which, T.n_w)) return 0.0f;
    return cubic(__ldg(T.w + pr.K_off + 3 * i + which), t);
}

__device__ __forceinline__ float wtab_G(const TableView& T, const DevPair& pr, int i, float t)
{
    if (!idx_ok(T.status, (long long)pr.G_off + i, T.n_w)) return 0.0f;
    return cubic(__ldg(T.w + pr.G_off + i), t);
}

// sigma(g) g in A^2 km/s
// (kMoliere: known not to be hard spheres)
template <bool kMoliere>
__device__ __forceinline__ float h_of_g(const TableView& T, const DevPair& pr, float g, float g2)
{
    const float b = bmax_eval(T, fast_ln(pr.kappa * g2));
    return !kMoliere && pr.hard_sphere ? pr.sigma_scale * g : pr.sigma_scale * b * b * g;
}

// 1 - exp(-y) without cancellation for small y
__device__ __forceinline__ float one_minus_exp_neg(float y)
{
    if (y < 0.5f) {
        float s = 1.0f - y * (1.0f / 10.0f);
        s = 1.0f - y * (1.0f / 9.0f) * s;
        s = 1.0f - y * (1.0f / 8.0f) * s;
        s = 1.0f - y * (1.0f / 7.0f) * s;
        s = 1.0f - y * (1.0f / 6.0f) * s;
        s = 1.0f - y * (1.0f / 5.0f) * s;
        s = 1.0f - y * (1.0f / 4.0f) * s;
        s = 1.0f - y * (1.0f / 3.0f) * s;
        s = 1.0f - y * (1.0f / 2.0f) * s;
        return y * s;
    }
    return 1.0f - expf(-y);
}

// CM deflection for the Moliere potential in reduced units (eps, beta), in
// units of pi: apsis by Newton from the head-on lower bound max(beta, x_h),
// then the Gauss-Mehler sum chi / pi = (2 / N) sum_j D_j / (S_j (S_j + beta/x0))
// with N = kGMNodesLo below ln eps = kGMLoLnEps, else kGMNodes (2/N is a power
// of two, so the scaling is exact).  Roundings spelled out, as in the collision (sumsq_xyz).
__device__ float chi_over_pi_moliere(float eps, float ln_eps, float beta, float xh, const float4* gm)
{
    const float ie = 1.0f / eps;
    const float b2 = beta * beta;
    float x = fmaxf(beta, xh);
    // Terms of Phi with d_i = 1.2 and 6.0 are dropped, lane by lane, where their
    // share of the potential is below 1e-8: c_i d_i e^{-d_i x} < 1e-8 c_0 d_0 e^{-d_0 x}
    // for x > 23 (d = 1.2) and x > 4 (d = 6.0).  Both x-bounds hold from the start
    // of the apsis iteration onwards because x only grows from max(beta, x_h).
    const bool t1 = x < 23.0f, t2 = x < 4.0f;
    // loops are not unrolled: a compact kernel misses the instruction cache less
#pragma unroll 1
    for (int it = 0; it < kApsisIters; ++it) {
        float e0 = __fmul_rn(kMolC0, expf(-kMolD0 * x));
        float e1 = t1 ? kMolC1 * expf(-kMolD1 * x) : 0.0f;
        float e2 = t2 ? kMolC2 * expf(-kMolD2 * x) : 0.0f;
        float ph = __fadd_rn(__fadd_rn(e0, e1), e2);
        float dph = -fmaf(kMolD2, e2, fmaf(kMolD1, e1, __fmul_rn(kMolD0, e0)));
        float ix = __frcp_rn(x);
        float ix2 = ix * ix;
        float g = fmaf(-__fmul_rn(ph, ix), ie, fmaf(-b2, ix2, 1.0f));  // 1 - b2/x^2 - ph/(x eps)
        // 2 b2/x^3 - (dph x - ph)/(x^2 eps)
        float gp = fmaf(__fmul_rn(2.0f * b2, ix2), ix, -__fmul_rn(__fmul_rn(fmaf(dph, x, -ph), ix2), ie));
        x -= __fdividef(g, gp);
    }
    const float x0 = x;
    const float bt = beta / x0;
    const float iex = ie / x0;
    const bool u1 = x0 < 23.0f, u2 = x0 < 4.0f;
    const float p0 = kMolC0 * expf(-kMolD0 * x0) * iex;
    const float p1 = u1 ? kMolC1 * expf(-kMolD1 * x0) * iex : 0.0f;
    const float p2 = u2 ? kMolC2 * expf(-kMolD2 * x0) * iex : 0.0f;
    const float y0 = kMolD0 * x0, y1 = kMolD1 * x0, y2 = kMolD2 * x0;
    const bool lo = ln_eps < kGMLoLnEps;
    const float4* nodes = lo ? gm + kGMHalf : gm;
    const int nh = lo ? kGMHalfLo : kGMHalf;
    float s = 0.0f;
#pragma unroll 1
    for (int j = 0; j < nh; ++j) {
        const float4 nd = nodes[j];  // (u, 1/(1+u), u/(1-u^2), 1/u - 1)
        float D = p0 * fmaf(nd.z, one_minus_exp_neg(y0 * nd.w), nd.y);
        if (u1) D = fmaf(p1, fmaf(nd.z, one_minus_exp_neg(y1 * nd.w), nd.y), D);
        if (u2) D = fmaf(p2, fmaf(nd.z, one_minus_exp_neg(y2 * nd.w), nd.y), D);
        // S = sqrt(q), q = (beta/x0)^2 + D > 0; approximate reciprocal square root
        // and division (2 ulp) are well inside the quadrature error
        const float q = fmaf(bt, bt, D);
        const float S = __fmul_rn(q, rsqrtf(q));
        s += __fdividef(D, __fmul_rn(S, __fadd_rn(S, bt)));
    }
    return s * (lo ? 2.0f / (float)kGMNodesLo : 2.0f / (float)kGMNodes);
}

// Column and position of y = ln(b/b_max) <= 0 in the deflection table; false below it.
__device__ __forceinline__ bool chi_table_column(float y, int& j, float& ty)
{
    const bool coarse = y < kChiY1;
    const float fy = (y - (coarse ? kChiY0 : kChiY1)) * (coarse ? 1.0f / kChiHyC : 1.0f / kChiHyF);
    table_cell(fmaxf(fy, 0.0f), 8388608.0f + (float)((coarse ? kChiNyC : kChiNyF) - 1), j, ty);
    ty = fminf(ty, 1.0f);
    j += coarse ? 0 : kChiNyC;
    return y >= kChiY0;
}

// Deflection from the table: q = ln tan(chi/2) at x = ln eps in column j at ty, bicubic in the
// cell; false outside the table (then q is that of the nearest row: the caller integrates
// instead).  No branch, so that it overlaps with what the caller does beside it.
__device__ __forceinline__ bool chi_table_q(const float4* tab, unsigned int* status, float x, int j, float ty, float& q)
{
    const float fx = (x - kChiX0) * (1.0f / kChiHx);
    const bool in = fx >= 0.0f && fx < (float)kChiNx;
    int i;
    float tx;
    table_cell(fminf(fmaxf(fx, 0.0f), (float)kChiNx), 8388608.0f + (float)(kChiNx - 1), i, tx);
    const int cell = i * kChiNy + j;
    if (!idx_ok(status, cell, kChiCells)) return false;
    const float4* c = tab + 4 * cell;
    const float4 r0 = __ldg(c), r1 = __ldg(c + 1), r2 = __ldg(c + 2), r3 = __ldg(c + 3);
    const float c0 = cubic(r0, ty), c1 = cubic(r1, ty), c2 = cubic(r2, ty), c3 = cubic(r3, ty);
    q = fmaf(tx, fmaf(tx, fmaf(tx, c3, c2), c1), c0);
    return in;
}

// cos and sin of the deflection from q = ln tan(chi/2): with T = e^q,
// cos chi = (1 - T^2)/(1 + T^2), sin chi = 2T/(1 + T^2)
__device__ __forceinline__ void chi_cos_sin(float q, float& cc, float& sc)
{
    const float Tq = fast_exp(fminf(q, 40.0f));
    const float T2 = Tq * Tq;
    const float inv = fast_div(1.0f, 1.0f + T2);
    cc = (1.0f - T2) * inv;
    sc = 2.0f * Tq * inv;
}

// (sin 2 pi u, cos 2 pi u) for u in (0, 1] from the MUFU sine and cosine, whose
// absolute error bound (about 2^-21.4) holds on [-pi, pi]: 2 pi u = 2 pi (u - 1/2) + pi,
// and u - 1/2 is exact for u = m 2^-24
__device__ __forceinline__ void neg_sincos_2pi_fast(float u, float* ns, float* nc)
{
    __sincosf(6.283185307179586f * (u - 0.5f), ns, nc);
}
__device__ __forceinline__ void sincos_2pi_fast(float u, float* s, float* c)
{
    float ns, nc;
    neg_sincos_2pi_fast(u, &ns, &nc);
    *s = -ns;
    *c = -nc;
}

// -ln u for u in (0, 1] from the MUFU logarithm (absolute error about 2^-21.4 near 1,
// 3 ulp elsewhere), clamped at 0 where the approximation rounds above zero
__device__ __forceinline__ float neg_log_fast(float u) { return fmaxf(-fast_ln(u), 0.0f); }

// sqrt(x) for x >= 0 as x / sqrt(x) from the MUFU reciprocal square root (about 2 ulp); 0 at 0
__device__ __forceinline__ float sqrt_fast(float x) { return x > 0.0f ? x * fast_rsqrt(x) : 0.0f; }

// orthonormal pair perpendicular to unit n (Duff et al., JCGT 6(1), 2017)
__device__ __forceinline__ void onb(float nx, float ny, float nz, float3& b1, float3& b2)
{
    float sgn = copysignf(1.0f, nz);
    float a = fast_div(-1.0f, sgn + nz);
    float b = nx * ny * a;
    b1 = make_float3(1.0f + sgn * nx * nx * a, sgn * b, -sgn * nx);
    b2 = make_float3(b, sgn + ny * ny * a, -ny);
}

// Sums of products with their roundings spelled out.  An atom's collisions are computed in more
// than one kernel, and its path has to be the same in each of them: what is fused to an FMA is
// therefore not left to the compiler, which decides it by the surrounding code.
__device__ __forceinline__ float sumsq_xyz(float x, float y, float z)
{
    return fmaf(z, z, fmaf(y, y, __fmul_rn(x, x)));
}
__device__ __forceinline__ float sumsq_yxz(float x, float y, float z)
{
    return fmaf(z, z, fmaf(x, x, __fmul_rn(y, y)));
}
// a b + c d, the second product rounded first
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return fmaf(a, b, __fmul_rn(c, d)); }

// ------------------------------------------------------------- launch
struct Lane {
    float px, py, pz, dx, dy, dz, speed, score;
    float scoreT;  // d ln p(path)/dT (kernel instance with the temperature score only)
    bool diff;     // thermalised: random walk of the diffusion shortcut
    uint32_t pid, inst, k;  // k flights begun: k - 1 collisions while the k-th lasts
    // of the instance (load_conditions)
    float ng14;
    uint32_t strm;
    int geom, pair;  // geometry index (its record is read from TableView::geoms), gas pair
    int target;      // local index of the emitting target
};

// The instance's conditions that a flight needs, 16 bytes through L1.  The transport reads them
// anew for every flight instead of carrying them in registers from one to the next.
__device__ __forceinline__ void load_conditions(Lane& S, const Params& P)
{
    const uint4 c = __ldg(reinterpret_cast<const uint4*>(P.inst + S.inst));
    S.ng14 = __uint_as_float(c.x);
    S.strm = c.y;
    const int geom = (int)(c.z & 0xffffu), pair = (int)(c.z >> 16);
    S.geom = idx_ok(P.status, geom, P.n_geoms) ? geom : 0;
    S.pair = idx_ok(P.status, pair, P.n_pairs) ? pair : 0;
    S.target = (int)c.w;
}

__device__ __forceinline__ float racetrack_r(const DevCathode& C, const float4* rt_tab, int rt_n, int n_rt_all,
                                            unsigned int* status, float u)
{
    // inverse radial CDF: cubic pieces in sqrt(u) below the median, in
    // sqrt(1-u) above it (1 - u is exact for RN = m 2^-24)
    const bool upper = u > 0.5f;
    const float q = upper ? 1.0f - u : u;
    const float x = sqrtf(q) * ((float)rt_n * 1.41421356237309515f);
    const int i = min((int)x, rt_n - 1);
    const float t = x - (float)i;
    int k = C.rt_tab + (upper ? rt_n : 0) + i;
    if (!idx_ok(status, k, n_rt_all)) k = 0;
    const float4 c = rt_tab[k];
    return fminf(fmaxf(fmaf(t, fmaf(t, fmaf(t, c.w, c.z), c.y), c.x), 0.0f), C.rt_R);
}

__device__ float cosine_sum_mu(const DevCathode& C, float u)
{
    if (!C.cos_general) return sqrtf(u);
    // bisection on the polynomial CDF sum c_i mu^{i+1}/(i+1)
    const float tgt = u * C.coef_norm;
    float lo = 0.0f, hi = 1.0f;
    for (int it = 0; it < 26; ++it) {
        float m = 0.5f * (lo + hi);
        float F = C.coef[5] * (1.0f / 6.0f);
        F = fmaf(F, m, C.coef[4] * (1.0f / 5.0f));
        F = fmaf(F, m, C.coef[3] * (1.0f / 4.0f));
        F = fmaf(F, m, C.coef[2] * (1.0f / 3.0f));
        F = fmaf(F, m, C.coef[1] * (1.0f / 2.0f));
        F = fmaf(F, m, C.coef[0]);
        F *= m;
        if (F < tgt) lo = m;
        else hi = m;
    }
    return 0.5f * (lo + hi);
}

// Inverse CDF of a piecewise-uniform density over n cells: F[0..n] the
// cumulative weights (F[0] = 0, F[n] = 1), u in ]0,1].  Returns the first cell
// i with F[i+1] >= u (cells of zero weight are never returned) and the position
// t in ]0,1] of u inside it.
__device__ int table_pick(const float* F, int n, float u, float& t)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (F[mid + 1] >= u) hi = mid;
        else lo = mid + 1;
    }
    const float f0 = F[lo], d = F[lo + 1] - f0;
    t = d > 0.0f ? fminf(fmaxf((u - f0) / d, 0.0f), 1.0f) : 1.0f;
    return lo;
}

// Joint table draw (kept out of line: rare, and off the registers of the hot loop):
// mu from the marginal CDF F (u_mu), E from the conditional CDF of the drawn mu cell (u_E).
__device__ __noinline__ void table_launch(const float* F, int nmu, int nE, float dE, float u_mu, float u_E, float& mu,
                                          float& E)
{
    float tm, te;
    const int i = table_pick(F, nmu, u_mu, tm);
    const int k = table_pick(F + (nmu + 1) + i * (nE + 1), nE, u_E, te);
    mu = ((float)i + tm) / (float)nmu;
    E = ((float)k + te) * dE;
}

__device__ void launch_state(const Params& P, const float4* rt_tab, uint32_t inst, uint32_t pid, float& px,
                             float& py, float& pz, float& dx, float& dy, float& dz, float& E)
{
    const DevInstance& I = P.inst[inst];
    const DevCathode& C = P.cath[I.cathode];
    const uint4 w0 = philox(P, pid, I.stream, 0u, 0u);
    const uint4 w1 = philox(P, pid, I.stream, 0u, 1u);
    const float r = racetrack_r(C, rt_tab, P.rt_n, P.n_rt_all, P.status, rn(w0.x));
    float sa, ca;
    sincospif(2.0f * rn(w0.y), &sa, &ca);
    float mu;
    if (C.lt_off >= 0 &&
        idx_ok(P.status, (long long)C.lt_off + (C.lt_nmu + 1) + (long long)C.lt_nmu * (C.lt_nE + 1) - 1, P.n_lt_all)) {
        table_launch(P.lt_tab + C.lt_off, C.lt_nmu, C.lt_nE, C.lt_dE, rn(w0.w), rn(w0.z), mu, E);
    } else {
        // Thompson inverse CDF at u_E; E_max itself in a boundary run
        const float s = P.launch_at_cutoff ? I.thompson_q : sqrtf(rn(w0.z)) * I.thompson_q;
        E = I.U_s * s / (1.0f - s);
        mu = cosine_sum_mu(C, rn(w0.w));
    }
    float sp, cp;
    sincospif(2.0f * rn(w1.x), &sp, &cp);
    const float st = sqrtf((1.0f - mu) * (1.0f + mu));
    const float rc = r * ca, rs = r * sa, tc = st * cp, ts = st * sp;
    px = C.c[0] + rc * C.e1[0] + rs * C.e2[0];
    py = C.c[1] + rc * C.e1[1] + rs * C.e2[1];
    pz = C.c[2] + rc * C.e1[2] + rs * C.e2[2];
    dx = tc * C.e1[0] + ts * C.e2[0] + mu * C.n[0];
    dy = tc * C.e1[1] + ts * C.e2[1] + mu * C.n[1];
    dz = tc * C.e1[2] + ts * C.e2[2] + mu * C.n[2];
}

// ------------------------------------------------------------- geometry
// distance to the chamber walls from inside (0 behind a wall, infinite for a zero or NaN direction)
__device__ __forceinline__ float hit_box(const Params& P, float px, float py, float pz, float dx, float dy, float dz)
{
    // approximate quotients (2 ulp): a hit distance needs no correctly rounded division
    const float qx = fast_div((dx > 0.0f ? P.box_hi[0] : P.box_lo[0]) - px, dx);
    const float qy = fast_div((dy > 0.0f ? P.box_hi[1] : P.box_lo[1]) - py, dy);
    const float qz = fast_div((dz > 0.0f ? P.box_hi[2] : P.box_lo[2]) - pz, dz);
    const float tx = fabsf(dx) > 0.0f ? qx : CUDART_INF_F;
    const float ty = fabsf(dy) > 0.0f ? qy : CUDART_INF_F;
    const float tz = fabsf(dz) > 0.0f ? qz : CUDART_INF_F;
    return fmaxf(fminf(tx, fminf(ty, tz)), 0.0f);
}

// kBox: the primitive may be a chamber box
template <bool kBox>
__device__ __forceinline__ float hit_prim(const DevPrim& Q, const Params& P, float px, float py, float pz, float dx,
                                          float dy, float dz)
{
    float t = CUDART_INF_F;
    if (kBox && Q.kind == SPUT_PRIM_BOX) {
        t = hit_box(P, px, py, pz, dx, dy, dz);
    } else if (Q.kind == SPUT_PRIM_CYLINDER) {
        const float wx = px - Q.cx, wy = py - Q.cy, wz = pz - Q.cz;
        const float wa = wx * Q.ux + wy * Q.uy + wz * Q.uz;
        const float da = dx * Q.ux + dy * Q.uy + dz * Q.uz;
        const float wpx = wx - wa * Q.ux, wpy = wy - wa * Q.uy, wpz = wz - wa * Q.uz;
        const float dpx = dx - da * Q.ux, dpy = dy - da * Q.uy, dpz = dz - da * Q.uz;
        const float A = dpx * dpx + dpy * dpy + dpz * dpz;
        const float B = 2.0f * (wpx * dpx + wpy * dpy + wpz * dpz);
        const float Cc = wpx * wpx + wpy * wpy + wpz * wpz - Q.p0sq;
        const float disc = B * B - 4.0f * A * Cc;
        if (A > 0.0f && disc >= 0.0f) {
            const float sq = sqrtf(disc);
            const float q = -0.5f * (B + copysignf(sq, B));
            float r1 = fast_div(q, A), r2 = q != 0.0f ? fast_div(Cc, q) : r1;
            const float tlo = fminf(r1, r2), thi = fmaxf(r1, r2);
            if (tlo > 0.0f && fabsf(fmaf(tlo, da, wa)) <= Q.p1) t = tlo;
            else if (thi > 0.0f && fabsf(fmaf(thi, da, wa)) <= Q.p1) t = thi;
        }
    } else {
        const float den = dx * Q.nx + dy * Q.ny + dz * Q.nz;
        if (den != 0.0f) {
            const float num = (Q.cx - px) * Q.nx + (Q.cy - py) * Q.ny + (Q.cz - pz) * Q.nz;
            const float tt = fast_div(num, den);
            if (tt > 0.0f) {
                const float qx = fmaf(tt, dx, px) - Q.cx, qy = fmaf(tt, dy, py) - Q.cy, qz = fmaf(tt, dz, pz) - Q.cz;
                const float a1 = qx * Q.ux + qy * Q.uy + qz * Q.uz;
                const float a2 = qx * Q.vx + qy * Q.vy + qz * Q.vz;
                bool in;
                if (Q.kind == SPUT_PRIM_RECT) in = fabsf(a1) <= Q.p0 && fabsf(a2) <= Q.p1;
                else {
                    const float r2 = a1 * a1 + a2 * a2;
                    in = r2 >= Q.p0sq && r2 <= Q.p1 * Q.p1;
                }
                if (in) t = tt;
            }
        }
    }
    return t;
}

// ------------------------------------------------------------- particle start
// A prepared launch: position, direction and speed of particle (inst, pid).
struct Launch {
    float px, py, pz, dx, dy, dz, speed;
    uint32_t inst, pid;
};
constexpr int kLaunchWords = 9;  // 32-bit words of a Launch in a warp's shared-memory queue

__device__ Launch prepare_launch(const Params& P, uint32_t inst, uint32_t pid)
{
    if (!idx_ok(P.status, inst, P.n_inst)) inst = 0;
    const DevCathode& C = P.cath[P.inst[inst].cathode];
    Launch L;
    float E;
    launch_state(P, P.rt_tab, inst, pid, L.px, L.py, L.pz, L.dx, L.dy, L.dz, E);
    L.speed = C.v_per_sqrtE * sqrtf(E);
    L.inst = inst;
    L.pid = pid;
    return L;
}

// The lane takes up the prepared particle.
__device__ void start_from(Lane& S, const Params& P, const Launch& L)
{
    S.inst = L.inst;
    S.pid = L.pid;
    S.px = L.px;
    S.py = L.py;
    S.pz = L.pz;
    S.dx = L.dx;
    S.dy = L.dy;
    S.dz = L.dz;
    S.speed = L.speed;
    // failure-path test aid (SPUT_RUN_INJECT_NONFINITE): a non-finite state that the
    // flight step retires with the non-finite status bit
    if (P.inject_nonfinite && L.pid == 0u) S.speed = CUDART_NAN_F;
    S.k = 0u;
    S.score = 0.0f;
    S.scoreT = 0.0f;
    S.diff = false;
}

__device__ void start_particle(Lane& S, const Params& P, uint32_t inst, uint32_t pid)
{
    start_from(S, P, prepare_launch(P, inst, pid));
}

// ------------------------------------------------------------- one flight
enum { kStepNone = -1, kStepCollided = 0, kStepLanded = 1, kStepTimedOut = 2 };

struct StepOut {
    float t;        // landing: distance to the hit; otherwise the flight length
    int prim;       // landing: local primitive index
    int attempts;   // partner attempts of this collision
    int nonfinite;  // the state became NaN/Inf
    float Gv;       // d ln K / d ln s at the flight's speed (temperature score only)
};

// Inverse mean free path at the atom's speed (cell i, t of its pair's tables) and the flight
// length, nl = -ln u; Gv = d ln K / d ln s at its speed (temperature score only).
template <int kMode>
__device__ __forceinline__ void flight_length(const Lane& S, const Params& P, const TableView& T, const DevPair& pr,
                                              int i, float t, float nl, float& inv_lam, float& ell, float& Gv)
{
    // n_g <sigma g>/v (thermal) or n_g sigma(v) (gas at rest)
    const float Kv = wtab_at(T, pr, kTabK, i, t);
    inv_lam = P.gas_thermal ? S.ng14 * Kv / S.speed : S.ng14 * Kv;
    // diffusion shortcut: exponential steps of mean lambda_D, 1/lambda_D = n sigma_D
    if (kMode == kModeWalk && S.diff) inv_lam = S.ng14 * pr.sigma_D;
    ell = S.ng14 > 0.0f ? fast_div(nl, inv_lam) : CUDART_INF_F;
    if (kMode == kModeScoreT) Gv = wtab_G(T, pr, i, t);
}

// Terms of the path scores.  Pressure: a flight of length l that ends in a collision adds
// 1 - l/lambda, a landing takes t/lambda.  Temperature: the same times d ln(n_g K(v)/v)/dT =
// (-1 + G/2)/T (n_g = p/(k_B T), G = d ln K/d ln s), and per collision the partner density
// f_T(V) sigma(g) g / K(v): d ln/dT = (|V|^2/(2 s^2) - 3/2 - G/2)/T, here without its 1/T.
// Rounded as written wherever they are used.
__device__ __forceinline__ float score_gain(float ell, float inv_lam) { return fmaf(-ell, inv_lam, 1.0f); }
__device__ __forceinline__ float score_T_rate(const Params& P, float Gv) { return fmaf(0.5f, Gv, -1.0f) * P.inv_T; }
__device__ __forceinline__ float score_T_partner(const Params& P, float V2, float Gv)
{
    return fmaf(-0.5f, Gv, fmaf(0.5f * V2, P.inv_s2, -1.5f));
}

// Free flight k+1 of the atom in S: its Philox block w (word 0 the free path; words 1 and 2,
// the impact parameter and azimuth, are used by the collision; word 3 is unused), the
// inverse mean free path, the flight length and the envelope EA + EB rho of the partner rejection
// at its end (the speed does not change on the way).
template <int kMode>
__device__ void flight_begin(Lane& S, const Params& P, const TableView& T, const DevPair* pairs, StepOut& out,
                             uint4& w, float& inv_lam, float& ell, float& EA, float& EB)
{
    S.k += 1u;
    w = philox(P, S.pid, S.strm, S.k, 0u);
    const DevPair& pr = pairs[S.pair];
    int i;
    float t;
    wtab_cell(pr, S.speed, i, t);
    flight_length<kMode>(S, P, T, pr, i, t, neg_log_fast(rn(w.x)), inv_lam, ell, out.Gv);
    if (P.gas_thermal) {
        EA = wtab_at(T, pr, kTabA, i, t);
        EB = wtab_at(T, pr, kTabB, i, t);
    }
}

// The emitting target's local index on the first flight (it is skipped then: the atom
// leaves its plane), else -1.
__device__ __forceinline__ int excluded_prim(const Lane& S) { return S.k == 1u ? S.target : -1; }

// A warp's scratch in shared memory: the pairs of the surface test, and what the partner
// sampling hands to the lanes that try an atom's attempts.
constexpr int kAskers = 8;
union WarpScratch {
    uint2 list[32];
    struct {
        float4 v[kAskers];   // v, EA
        uint4 ids[kAskers];  // particle id, stream, flight, next attempt
        uint2 p[kAskers];    // EB, pair
    } ask;
};

// Nearest hit by a loop over the geometry's primitives, ties to the lowest index.  Every
// primitive whose bounding sphere lies within min(ell, best t) is tested (margin covers
// FP32 rounding): no hit beyond that can be the landing.
__device__ __forceinline__ void nearest_hit_loop(const Lane& S, const Params& P, const TableView& T,
                                                 const DevPrim* prims, float ell, float& tb, int& hb)
{
    const DevGeom G = T.geoms[S.geom];
    const int excl = excluded_prim(S);
    for (int li = 0; li < G.count; ++li) {
        if (li == excl) continue;
        if (!idx_ok(P.status, G.begin + li, P.n_prims)) break;
        const DevPrim& Q = prims[G.begin + li];
        if (Q.kind != SPUT_PRIM_BOX) {
            const float ex = Q.bx - S.px, ey = Q.by - S.py, ez = Q.bz - S.pz;
            const float reach = fminf(ell, tb) * 1.0001f + Q.br + 1e-3f;
            if (ex * ex + ey * ey + ez * ez > reach * reach) continue;
        }
        const float t = hit_prim<true>(Q, P, S.px, S.py, S.pz, S.dx, S.dy, S.dz);
        if (t < tb) {
            tb = t;
            hb = li;
        }
    }
}

// grid coordinate x's cell, the nearest one of n when x lies outside (0 for NaN)
__device__ __forceinline__ unsigned grid_clamp(float x, int n)
{
    return (unsigned)fminf(fmaxf(x, 0.0f), (float)(n - 1));
}

// Nearest hit of every active lane by the cell masks, the whole warp together.
//   * The chamber walls, if the geometry has them, are tested first, so the flight is a segment
//     of length L = min(ell, wall) inside the box.
//   * It is cut into pieces of at most 4 cell edges (most flights are one piece).  All of a
//     piece lies within R, half its length, of its centre: the mask of the centre's cell at
//     the smallest level r 2^k >= R holds every primitive it can reach (usually none: most
//     flights pass far from any surface).
//   * The (lane, primitive) pairs of all lanes are tested 32 at a time, one per lane,
//     whichever atom they belong to: a loop per lane would run as long as the busiest
//     lane's, and a loop over the geometry runs each test for the few lanes near it.
// A primitive outside the mask has no hit at t <= L, so the nearest hit and its tie-break
// (lowest index) are those of the loop above.  kWords: 32-bit words of a mask.
// The transport is bound by instruction issue, and the loop took 43 % (16 primitives, 0.5 Pa)
// to 67 % (64 primitives, 3 Pa) of the kernel: a warp ran 9.2 of 16 primitives' tests per
// step although 0.12 per atom cross the primitive at all.  Masks of the midpoint leave 8
// pairs per warp and step (0.5 Pa), so one round does.  Measured loop -> masks (GB300, before
// what followed): quaternary 4e7 atoms 67.2 -> 58.8 ms, 64 primitives at 3 Pa 1e6 atoms
// 118 -> 59 ms, with the diffusion shortcut 4e6 atoms 61.3 -> 24.7 ms.
template <int kWords>
__device__ __forceinline__ void nearest_hit_masks(bool active, const Lane& S, const Params& P, const TableView& T,
                                                  const DevPrim* prims, uint2* list, float ell, float& tb, int& hb)
{
    const int lane = threadIdx.x & 31;
    unsigned lo = 0u, hi = 0u;  // candidates 0..31 and 32..63
    int begin = 0;
    if (active) {
        const DevGeom G = T.geoms[S.geom];
        begin = G.begin;
        const int box = G.box();
        tb = hit_box(P, S.px, S.py, S.pz, S.dx, S.dy, S.dz);
        tb = box >= 0 ? tb : CUDART_INF_F;
        hb = tb < CUDART_INF_F ? box : -1;
        const float L = fminf(ell, tb);
        // 1 + floor(L / (4 h)) pieces (floor as in table_cell; at most kCellMaxPieces, also for NaN)
        float pieces = fminf(__fadd_rd(L * P.cell_inv_seg, 8388608.0f) - 8388607.0f, (float)kCellMaxPieces);
        const float R = 0.5f * fast_div(L, pieces);
        // the smallest level: max(0, ceil(log2(R / r))) from the exponent bits
        const int k = max(0, (int)((__float_as_uint(R * P.cell_inv_r) + 0x7fffffu) >> 23) - 127);
        // grid coordinates of the start; step of the centres
        const float sx = fmaf(S.px, P.cell_inv_h, P.cell_off[0]), sy = fmaf(S.py, P.cell_inv_h, P.cell_off[1]),
                    sz = fmaf(S.pz, P.cell_inv_h, P.cell_off[2]);
        const float Rh = R * P.cell_inv_h;
        for (float c = Rh; pieces > 0.0f; pieces -= 1.0f, c += 2.0f * Rh) {
            // floors of the coordinates; a negative one wraps to a large unsigned number
            unsigned ix = __float_as_uint(__fadd_rd(fmaf(c, S.dx, sx), 8388608.0f)) - 0x4b000000u;
            unsigned iy = __float_as_uint(__fadd_rd(fmaf(c, S.dy, sy), 8388608.0f)) - 0x4b000000u;
            unsigned iz = __float_as_uint(__fadd_rd(fmaf(c, S.dz, sz), 8388608.0f)) - 0x4b000000u;
            bool in = k < kCellLevels && ix < (unsigned)P.cell_n[0] && iy < (unsigned)P.cell_n[1] &&
                      iz < (unsigned)P.cell_n[2];
            if (!in) {
                // A centre outside the grid (without walls, or by rounding at one) takes the cell
                // nearest to it: the chamber is convex and what the flight may hit lies in it, so
                // that cell is no farther from any of it than the centre.
                ix = grid_clamp(fmaf(c, S.dx, sx), P.cell_n[0]);
                iy = grid_clamp(fmaf(c, S.dy, sy), P.cell_n[1]);
                iz = grid_clamp(fmaf(c, S.dz, sz), P.cell_n[2]);
                in = k < kCellLevels;
            }
            if (in) {
                const int cell = (int)((iz * P.cell_n[1] + iy) * P.cell_n[0] + ix);
                const uint32_t* m = P.cell_mask + G.cell_base;
                const int e = cell * kCellLevels + k;
                if (!idx_ok(P.status, G.cell_base + (P.cell_half ? (long long)e / 2 : (long long)kWords * e + kWords - 1),
                            P.n_cell_words)) {
                    // (the checked build reports it)
                } else if (kWords == 1) {
                    lo |= P.cell_half ? __ldg(reinterpret_cast<const unsigned short*>(m) + e) : __ldg(m + e);
                } else {
                    const uint2 m2 = __ldg(reinterpret_cast<const uint2*>(m) + e);
                    lo |= m2.x;
                    hi |= m2.y;
                }
            } else {
                // longer than kCellMaxPieces pieces: no walls stop it
                lo = G.count >= 32 ? ~0u : (1u << G.count) - 1u;
                if (kWords == 2) hi = G.count >= 64 ? ~0u : G.count > 32 ? (1u << (G.count - 32)) - 1u : 0u;
                if (box >= 0 && box < 32) lo &= ~(1u << box);
                if (kWords == 2 && box >= 32) hi &= ~(1u << (box - 32));
            }
        }
        const int excl = excluded_prim(S);
        if (excl >= 0 && excl < 32) lo &= ~(1u << excl);
        if (kWords == 2 && excl >= 32) hi &= ~(1u << (excl - 32));
    }
    const unsigned lt = (1u << lane) - 1u;
    for (;;) {
        // The lanes list their candidates, one each per turn, up to 32 pairs a round.  `turn` finds the
        // lane's place of a turn; the turns are gone through again to take the hits.
        const unsigned lo0 = lo, hi0 = hi;
        int total = 0;
        for (;;) {
            const bool any = (kWords == 2 ? lo | hi : lo) != 0u;
            const unsigned m = __ballot_sync(kFull, any);
            if (m == 0u || total == 32) break;
            const int at = total + __popc(m & lt);
            if (any && at < 32) {
                int li;
                if (kWords == 1 || lo) {
                    li = __ffs(lo) - 1;
                    lo &= lo - 1u;
                } else {
                    li = 31 + __ffs(hi);
                    hi &= hi - 1u;
                }
                list[at].x = (uint32_t)(begin + li) << 5 | (uint32_t)lane;
            }
            total = min(32, total + __popc(m));
        }
        if (total == 0) return;
        __syncwarp();
        const bool mine = lane < total;
        const uint32_t pr = mine ? list[lane].x : (uint32_t)lane;
        const int src = (int)(pr & 31u);
        const float px = __shfl_sync(kFull, S.px, src), py = __shfl_sync(kFull, S.py, src),
                    pz = __shfl_sync(kFull, S.pz, src);
        const float dx = __shfl_sync(kFull, S.dx, src), dy = __shfl_sync(kFull, S.dy, src),
                    dz = __shfl_sync(kFull, S.dz, src);
        if (mine)
            list[lane].y = __float_as_uint(idx_ok(P.status, pr >> 5, P.n_prims)
                                               ? hit_prim<false>(prims[pr >> 5], P, px, py, pz, dx, dy, dz)
                                               : CUDART_INF_F);
        __syncwarp();
        unsigned l0 = lo0, h0 = hi0;
        for (int t0 = 0; t0 < total;) {
            const bool any = (kWords == 2 ? l0 | h0 : l0) != 0u;
            const unsigned m = __ballot_sync(kFull, any);
            const int at = t0 + __popc(m & lt);
            if (any && at < 32) {
                const uint2 e = list[at];
                const float t = __uint_as_float(e.y);
                const int li = (int)(e.x >> 5) - begin;
                if (t < tb || (t == tb && li < hb)) {
                    tb = t;
                    hb = li;
                }
                if (kWords == 1 || l0) l0 &= l0 - 1u;
                else h0 &= h0 - 1u;
            }
            t0 += __popc(m);
        }
        __syncwarp();  // (what writes the scratch next does so after these reads)
        if (total < 32) return;
    }
}

// The flight's end.  Landing: S keeps the pre-flight position and out.t is the hit
// distance.  Otherwise the atom moves to the collision point.
template <int kMode>
__device__ int flight_end(Lane& S, const Params& P, StepOut& out, float inv_lam, float ell, float tb, int hb)
{
    constexpr bool kScoreT = kMode == kModeScoreT;
    out.nonfinite = 0;
    out.prim = -1;
    const float aT = kScoreT ? score_T_rate(P, out.Gv) : 0.0f;
    if (hb >= 0 && tb <= ell) {
        S.score = fmaf(-tb, inv_lam, S.score);
        if (kScoreT) S.scoreT = fmaf(-(aT * tb), inv_lam, S.scoreT);
        out.t = tb;
        out.prim = hb;
        return kStepLanded;
    }
    out.t = ell;
    S.px = fmaf(ell, S.dx, S.px);
    S.py = fmaf(ell, S.dy, S.py);
    S.pz = fmaf(ell, S.dz, S.pz);
    const float gain = score_gain(ell, inv_lam);
    S.score += gain;
    if (kScoreT) S.scoreT = fmaf(aT, gain, S.scoreT);
    if (!isfinite(S.px + S.py + S.pz + S.speed)) {
        out.nonfinite = 1;
        return kStepTimedOut;
    }
    if ((long long)S.k > P.max_collisions) return kStepTimedOut;
    return kStepCollided;
}

// position of the n-th (0-based) set bit of mask; mask has more than n set bits
__device__ __forceinline__ int nth_set_bit(unsigned mask, int n)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1)
        if (__popc(mask & ((1u << (pos + w)) - 1u)) <= n) pos += w;
    return pos;
}

// One attempt of the partner rejection below: the proposal's normals and their norms, and
// the uniform of its test.  Independent of the atom's velocity.
struct Attempt {
    float z1, z2, z3;
    float r3;     // |(z1, z2, z3)|: rho of the Maxwellian branch
    float rho_w;  // |(z1, z2, z3, z4)|: rho of the weighted branch
    float sc_w;   // scale of (z1, z2, z3) in the weighted branch
    float u;
};

__device__ __forceinline__ Attempt attempt_draw(const Params& P, uint32_t pid, uint32_t strm, uint32_t k, uint32_t a)
{
    const uint4 wn = philox(P, pid, strm, k, 1u + a);
    const float R0 = sqrt_fast(2.0f * neg_log_fast(rn(wn.x)));
    const float R1 = sqrt_fast(2.0f * neg_log_fast(rn(wn.z)));
    float s1, c1, s3, c3;
    sincos_2pi_fast(rn(wn.y), &s1, &c1);
    sincos_2pi_fast(rn(wn.w), &s3, &c3);
    Attempt d;
    d.z1 = R0 * c1;
    d.z2 = R0 * s1;
    d.z3 = R1 * c3;
    const float z4 = R1 * s3;
    // low bytes of words 0, 1, 2 as one more 24-bit uniform
    const uint32_t lowb = ((wn.x & 0xffu) << 24) | ((wn.y & 0xffu) << 16) | ((wn.z & 0xffu) << 8);
    d.u = rn(lowb);
    const float r32 = sumsq_xyz(d.z1, d.z2, d.z3);
    const float ir3 = r32 > 0.0f ? fast_rsqrt(r32) : 0.0f;
    d.r3 = r32 * ir3;
    d.rho_w = sqrt_fast(r32 + z4 * z4);
    d.sc_w = P.s_gas * (d.rho_w * ir3);
    return d;
}

// Whether the attempt takes the rho-weighted branch when the pair's envelope is EA + EB rho.
__device__ __forceinline__ bool attempt_weighted(const Attempt& d, float EA, float EB, float& ut, float& Bm)
{
    Bm = __fmul_rn(EB, (float)kEnvM);
    ut = __fmul_rn(d.u, __fadd_rn(EA, Bm));
    return ut <= Bm;
}

// The attempt's gas velocity in a branch.
__device__ __forceinline__ void attempt_velocity(const Params& P, const Attempt& d, bool weighted, float& cx, float& cy,
                                                 float& cz)
{
    const float sc = weighted ? d.sc_w : P.s_gas;
    cx = __fmul_rn(sc, d.z1);
    cy = __fmul_rn(sc, d.z2);
    cz = __fmul_rn(sc, d.z3);
}

// h(g) = sigma(g) g between the atom's velocity v and the gas velocity c
template <bool kMoliere>
__device__ __forceinline__ float attempt_h(const TableView& T, const DevPair& pr, float vx, float vy, float vz, float cx,
                                           float cy, float cz)
{
    const float g2 = sumsq_yxz(__fsub_rn(vx, cx), __fsub_rn(vy, cy), __fsub_rn(vz, cz));
    return h_of_g<kMoliere>(T, pr, sqrt_fast(g2), g2);
}

// Acceptance: the branch's own uniform, rescaled to (0, 1], times the envelope against h.
__device__ __forceinline__ bool attempt_accept(const Attempt& d, bool weighted, float ut, float Bm, float EA, float EB,
                                               float hg)
{
    const float env = fmaf(EB, weighted ? d.rho_w : d.r3, EA);
    return weighted ? ut * env <= Bm * hg : __fsub_rn(ut, Bm) * env <= EA * hg;
}

// Gas partners of every lane with `need`, drawn by the whole warp: the
// Maxwellian f(V) weighted by h(g) = sigma(g) g, by rejection from the
// proposal f(V) (EA + EB rho), rho = |V|/s, where EA + EB rho bounds h over the
// relative speeds a partner of speed rho s can give (the pair's envelope tables
// at the atom's speed).  The proposal is the Maxwellian with weight EA and, with
// weight EB E[rho], its rho-weighted form, whose speed follows the chi law with
// 4 degrees of freedom.  Attempt a of a particle uses its own Philox block 1 + a:
// the upper 24 bits of the four words give two Box-Muller pairs z1..z4, the low
// bytes of words 0-2 one more uniform u that selects the branch
// (u (EA + EB E[rho]) <= EB E[rho]: rho-weighted) and, rescaled within the
// branch, is the acceptance uniform.  Maxwellian branch: V = s (z1, z2, z3);
// rho-weighted branch: V = s |z| (z1, z2, z3)/|(z1, z2, z3)|.  The first
// accepted attempt is kept (attempt A-1 if none is).  While most lanes wait for a partner, each
// tries its own next attempt; then the pending particles' next attempts are spread over the
// warp (2^k consecutive attempts per particle), so the result is the sequential
// rejection loop's result while the lanes stay busy.  Must be called by all 32 lanes together.
__device__ void partner_sample_warp(bool need, const Params& P, const TableView& T, const DevPair* pairs,
                                    uint32_t pid, uint32_t strm, uint32_t k, int pair, float vx, float vy, float vz,
                                    float EA, float EB, WarpScratch* ws, float& Vx, float& Vy, float& Vz, int& attempts)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int A = P.max_attempts;
    unsigned pending = __ballot_sync(kFull, need);
    int next_a = 0;
    Vx = Vy = Vz = 0.0f;
    attempts = 0;
    while (pending) {
        // many lanes pending: each tries its next attempt itself; few: the whole warp tries theirs,
        // 2^shift consecutive attempts each
        const bool own = __popc(pending) > kAskers;
        const bool asks = (pending >> lane) & 1u;
        uint32_t o_pid = pid, o_strm = strm, o_k = k;
        int a = asks ? next_a : A, shift = 0, rank = 0;
        if (!own) {
            const int np = __popc(pending);
            shift = __clz(np - 1) - 27;  // 5 - ceil(log2 np)
            rank = __popc(pending & lt);
            if (asks) {
                ws->ask.v[rank] = make_float4(vx, vy, vz, EA);
                ws->ask.ids[rank] = make_uint4(pid, strm, k, (uint32_t)next_a);
                ws->ask.p[rank] = make_uint2(__float_as_uint(EB), (uint32_t)pair);
            }
            __syncwarp();
            const uint4 q = ws->ask.ids[lane >> shift];
            o_pid = q.x;
            o_strm = q.y;
            o_k = q.z;
            a = lane >> shift < np ? (int)q.w + (lane & ((1 << shift) - 1)) : A;
        }
        bool acc = false;
        float cx = 0.0f, cy = 0.0f, cz = 0.0f;
        if (a < A) {
            const Attempt d = attempt_draw(P, o_pid, o_strm, o_k, (uint32_t)a);
            float o_vx = vx, o_vy = vy, o_vz = vz, o_A = EA, o_B = EB;
            int op = pair;
            if (!own) {
                const float4 q = ws->ask.v[lane >> shift];
                const uint2 r = ws->ask.p[lane >> shift];
                o_vx = q.x;
                o_vy = q.y;
                o_vz = q.z;
                o_A = q.w;
                o_B = __uint_as_float(r.x);
                op = (int)r.y;
            }
            if (!idx_ok(T.status, op, P.n_pairs)) op = 0;
            float ut, Bm;
            const bool weighted = attempt_weighted(d, o_A, o_B, ut, Bm);
            attempt_velocity(P, d, weighted, cx, cy, cz);
            const float hg = attempt_h<false>(T, pairs[op], o_vx, o_vy, o_vz, cx, cy, cz);
            acc = attempt_accept(d, weighted, ut, Bm, o_A, o_B, hg) || a == A - 1;
        }
        const unsigned accm = __ballot_sync(kFull, acc);
        if (!own) __syncwarp();  // (a vote does not order memory: the scratch is written again after these reads)
        if (own) {
            if (acc) {
                Vx = cx;
                Vy = cy;
                Vz = cz;
                attempts = a + 1;
            }
            ++next_a;
            pending &= ~accm;
            continue;
        }
        int src = lane, first = 0;
        bool done = false;
        if (asks) {
            const int lanes = 1 << shift, at = rank << shift;
            const unsigned hit = accm & ((kFull >> (32 - lanes)) << at);
            if (hit) {
                src = __ffs(hit) - 1;
                first = src - at;
                done = true;
            } else {
                next_a += lanes;
            }
        }
        const float sx = __shfl_sync(kFull, cx, src);
        const float sy = __shfl_sync(kFull, cy, src);
        const float sz = __shfl_sync(kFull, cz, src);
        if (done) {
            Vx = sx;
            Vy = sy;
            Vz = sz;
            attempts = next_a + first + 1;
        }
        pending &= ~__ballot_sync(kFull, done);
    }
}

// The draws of a collision, from its flight's Philox block.
struct Impact {
    float ub;        // uniform of the impact parameter b = b_max sqrt(ub)
    int j;           // column of ln(ub)/2 in the deflection table and position in it; below the
    float ty;        // table 0 and -1
    float nsp, ncp;  // negated sine and cosine of the azimuth
};

__device__ __forceinline__ Impact impact_draw(const uint4& w)
{
    Impact I;
    I.ub = rn(w.y);
    if (!chi_table_column(0.5f * logf(I.ub), I.j, I.ty)) {
        I.j = 0;
        I.ty = -1.0f;
    }
    neg_sincos_2pi_fast(rn(w.z), &I.nsp, &I.ncp);
    return I;
}

// Cosine and sine of the CM deflection off the table: hard spheres, or the scattering integral.
__device__ __forceinline__ void deflect_off_table(const TableView& T, const DevPair& pr, float eps, float le, float ub,
                                                  float& cc, float& sc)
{
    if (pr.hard_sphere) {
        sincospif(acosf(sqrtf(ub)) * (2.0f / 3.14159265358979f), &sc, &cc);
    } else {
        const float beta = bmax_eval(T, le) * sqrtf(ub);
        sincospif(chi_over_pi_moliere(eps, le, beta, xh_eval(T, le), T.gm), &sc, &cc);
    }
}

// Binary collision in the CM frame: rotate g = v - V by (chi, psi), |g| kept; the atom's speed and
// direction (of velocity v) become those after it.  kUsual (the scene has a deflection table):
// straight-line code for what nearly every collision is, on the table, with a relative speed
// and a speed afterwards whose squares do not underflow; otherwise it returns false, with the
// result void, and the caller computes the collision without kUsual.
template <int kMode, bool kUsual>
__device__ __forceinline__ bool scatter(float& speed, float& dx, float& dy, float& dz, const Params& P,
                                        const TableView& T, const DevPair& pr, float vx, float vy, float vz, float Vx,
                                        float Vy, float Vz, const Impact& I)
{
    const float gx = __fsub_rn(vx, Vx), gy = __fsub_rn(vy, Vy), gz = __fsub_rn(vz, Vz);
    // (the temperature-score instance rounds this sum in the other order, as its results always were)
    const float g2 = kMode == kModeScoreT ? sumsq_yxz(gx, gy, gz) : sumsq_xyz(gx, gy, gz);
    const float ig = kUsual ? fast_rsqrt(g2) : rsqrtf(g2);
    const float g = g2 * ig;
    const float hx = gx * ig, hy = gy * ig, hz = gz * ig;
    const float eps = pr.kappa * g2;
    const float le = logf(eps);
    float sc, cc, q = 0.0f;
    bool on_table = false;
    if (kUsual || P.chi_tab) {
        on_table = chi_table_q(P.chi_tab, P.status, le, I.j, I.ty, q);
        chi_cos_sin(q, cc, sc);
    }
    if (!kUsual && g2 > 0.0f && !(on_table && I.ty >= 0.0f)) deflect_off_table(T, pr, eps, le, I.ub, cc, sc);
    const float sp = -I.nsp, cp = -I.ncp;
    float3 b1, b2;
    onb(hx, hy, hz, b1, b2);
    const float gpx = __fmul_rn(g, dot2(cc, hx, sc, dot2(sp, b2.x, cp, b1.x)));
    const float gpy = __fmul_rn(g, dot2(cc, hy, sc, dot2(sp, b2.y, cp, b1.y)));
    const float gpz = __fmul_rn(g, dot2(cc, hz, sc, dot2(sp, b2.z, cp, b1.z)));
    const float nvx = fmaf(pr.m2M, gpx, dot2(pr.m1M, vx, pr.m2M, Vx));
    const float nvy = fmaf(pr.m2M, gpy, dot2(pr.m1M, vy, pr.m2M, Vy));
    const float nvz = fmaf(pr.m2M, gpz, dot2(pr.m1M, vz, pr.m2M, Vz));
    if (kUsual) {
        const float sp2 = sumsq_yxz(nvx, nvy, nvz);
        const float is = fast_rsqrt(sp2);
        speed = sp2 * is;
        dx = nvx * is;
        dy = nvy * is;
        dz = nvz * is;
        // (2e-30: above the limit of the scaling below, however the sums round; the NaN of g2 = 0
        // fails it too)
        return on_table && I.ty >= 0.0f && sp2 > 2e-30f;
    }
    // an atom slowed to ~1e-15 km/s or below (gas at rest) would underflow the
    // squares: scale by the exact power of two 2^60 first
    const float up = sumsq_xyz(nvx, nvy, nvz) < 1e-30f ? 0x1p60f : 1.0f;
    const float ux = nvx * up, uy = nvy * up, uz = nvz * up;
    const float sp2 = sumsq_yxz(ux, uy, uz);
    const float is = rsqrtf(sp2);
    const float sn = sp2 * is;
    const bool moves = sp2 > 0.0f;
    if (g2 > 0.0f) {
        speed = !moves ? 0.0f : up == 1.0f ? sn : sn * 0x1p-60f;
        if (moves) {  // at rest: the direction is kept
            dx = ux * is;
            dy = uy * is;
            dz = uz * is;
        }
    }
    return true;
}

// Isotropic direction of the diffusion shortcut's walk from the flight block's words 1 and 2.
__device__ __forceinline__ void walk_direction(const uint4& w, float& dx, float& dy, float& dz)
{
    const float mu = 2.0f * rn(w.y) - 1.0f;
    const float st = sqrtf(fmaxf(0.0f, (1.0f - mu) * (1.0f + mu)));
    float sp, cp;
    sincospif(2.0f * rn(w.z), &sp, &cp);
    dx = st * cp;
    dy = st * sp;
    dz = mu;
}

// E (eV) of an atom of instance inst at this speed
__device__ __forceinline__ float energy_of(const Params& P, uint32_t inst, float speed)
{
    return P.cath[P.inst[inst].cathode].E_per_v2 * speed * speed;
}

// One flight of every active lane of the warp (flight, surface test, then for
// the lanes that collide: warp-wide partner sampling and the scattering).
// Must be called by all 32 lanes together; inactive lanes return kStepNone.
// kMasks: words of the surface test's cell masks (0: the counted loop); ws: the warp's scratch.
template <int kMode, int kMasks>
__device__ int flight_step_warp(bool active, Lane& S, const Params& P, const TableView& T, const DevPrim* prims,
                                const DevPair* pairs, WarpScratch* ws, StepOut& out)
{
    load_conditions(S, P);
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    int res = kStepNone;
    out.attempts = 0;
    constexpr bool kScoreT = kMode == kModeScoreT;
    if (kScoreT) out.Gv = 0.0f;
    float inv_lam = 0.0f, ell = 0.0f, EA = 0.0f, EB = 0.0f, tb = CUDART_INF_F;
    int hb = -1;
    if (active) flight_begin<kMode>(S, P, T, pairs, out, w, inv_lam, ell, EA, EB);
    if (kMasks) nearest_hit_masks<kMasks ? kMasks : 1>(active, S, P, T, prims, ws->list, ell, tb, hb);
    else if (active) nearest_hit_loop(S, P, T, prims, ell, tb, hb);
    if (active) res = flight_end<kMode>(S, P, out, inv_lam, ell, tb, hb);
    // a thermalised atom (diffusion shortcut) turns isotropically at the end of its step
    const bool walk = kMode == kModeWalk && res == kStepCollided && S.diff;
    const bool coll = res == kStepCollided && !walk;
    const DevPair pr = pairs[S.pair];
    const float vx = __fmul_rn(S.speed, S.dx), vy = __fmul_rn(S.speed, S.dy), vz = __fmul_rn(S.speed, S.dz);
    float Vx = 0.0f, Vy = 0.0f, Vz = 0.0f;
    if (P.gas_thermal) {
        partner_sample_warp(coll, P, T, pairs, S.pid, S.strm, S.k, S.pair, vx, vy, vz, EA, EB, ws, Vx,
                            Vy, Vz, out.attempts);
        if (kScoreT && coll)
            S.scoreT = fmaf(score_T_partner(P, sumsq_xyz(Vx, Vy, Vz), out.Gv), P.inv_T, S.scoreT);
    }
    if (coll) {
        const Impact I = impact_draw(w);
        float ns = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;
        bool usual = false;
        // (in a gas at rest atoms slow down below the table and most collisions would be computed
        // twice: 1e6 single-Ni atoms 3.08 ms without the first form, 3.33 with it)
        if (P.usual) usual = scatter<kMode, true>(ns, nx, ny, nz, P, T, pr, vx, vy, vz, Vx, Vy, Vz, I);
        if (usual) {
            S.speed = ns;
            S.dx = nx;
            S.dy = ny;
            S.dz = nz;
        } else {
            scatter<kMode, false>(S.speed, S.dx, S.dy, S.dz, P, T, pr, vx, vy, vz, Vx, Vy, Vz, I);
        }
        if (kMode == kModeWalk && energy_of(P, S.inst, S.speed) < P.E_switch) S.diff = true;
    } else if (walk) {
        walk_direction(w, S.dx, S.dy, S.dz);
    }
    return res;
}

// Adds the lanes' statistics to the run's; particles = landed + timed out, flights = landed +
// timed out + collisions.  Called by whole warps.
__device__ __forceinline__ void add_stats(const Params& P, uint32_t landed, uint32_t timed, unsigned long long coll,
                                          uint32_t att)
{
    unsigned long long v[kNumStats] = {landed + timed, landed, timed, landed + timed + coll, coll, att};
#pragma unroll
    for (int i = 0; i < kNumStats; ++i) {
        unsigned long long x = v[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(P.stats + i, x);
    }
}

// ------------------------------------------------------------- hand-over
// Atoms between two flights, in Params::pool, which holds what one run hands over.  Runs of a scene
// must not overlap; if they do all the same, each may clear the other's counters and find its
// atoms, or bytes of an earlier run, in the slots.  Results are then void, and the status word says
// so where it shows: an atom that finds no slot is dropped (to carry it on in its lane took 4x1e7
// quaternary atoms 48.0 instead of 45.8 ms, by spills), and what is read from a slot is used as an
// index only after a test (pool_holds).
__device__ __forceinline__ void pool_store(const Params& P, bool have, const Lane& S)
{
    const unsigned m = __ballot_sync(kFull, have);
    const int lane = threadIdx.x & 31;
    unsigned base = P.pool_slots;
    // (not added to once full: the count cannot wrap around)
    if (lane == 0 && m && *static_cast<volatile unsigned*>(P.pool_count) < P.pool_slots)
        base = atomicAdd(P.pool_count, (unsigned)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (!have) return;
    const unsigned i = base + __popc(m & ((1u << lane) - 1u));
    if (i >= P.pool_slots) {
        atomicOr(P.status, kStatusHandOver);
        return;
    }
    float4* q = P.pool + 4 * (size_t)i;
    q[0] = make_float4(S.px, S.py, S.pz, S.speed);
    q[1] = make_float4(S.dx, S.dy, S.dz, S.score);
    q[2] = make_float4(__uint_as_float(S.pid), __uint_as_float(S.inst), __uint_as_float(S.k),
                       __uint_as_float(S.diff ? 1u : 0u));
    q[3] = make_float4(S.scoreT, 0.0f, 0.0f, 0.0f);
}

// Whether a slot holds an atom of this run: its ticket, which the tallies and records are indexed by.
__device__ __forceinline__ bool pool_holds(const Params& P, uint32_t inst, uint32_t pid)
{
    if (inst < (uint32_t)P.n_inst && P.prefix[inst] + pid - P.ticket_begin < P.ticket_end - P.ticket_begin) return true;
    atomicOr(P.status, kStatusHandOver);
    return false;
}

// ------------------------------------------------------------- tallies
__device__ __forceinline__ void write_record(const Params& P, const Lane& S, int prim, int cell, float E, float cosang)
{
    const unsigned long long t = P.prefix[S.inst] + S.pid - P.ticket_begin;
    if (!idx_ok(P.status, (long long)t, (long long)(P.ticket_end - P.ticket_begin))) return;
    sput_record rec;
    rec.prim = prim;
    rec.cell = cell;
    rec.energy = E;
    rec.cos_angle = cosang;
    rec.n_collisions = S.k - 1u;
    rec.score = S.score;
    P.records[t] = rec;
}

// Landing of the atom in S (pre-flight position) on primitive hb at distance tb; s_cnt: the
// block's counters when they are privatised (P.smem_counters).
template <int kMode>
__device__ __forceinline__ void tally_landed(const Params& P, const Lane& S, const DevGeom* geoms, const DevPrim* prims,
                                             unsigned int* s_cnt, float tb, int hb)
{
    // every landing counts on its primitive; few (a tenth) reach the substrate
    if (!idx_ok(P.status, hb, P.max_prims)) {
        // dropped: the checked build reports it
    } else if (s_cnt) atomicAdd(&s_cnt[S.inst * (P.max_prims + 1) + hb], 1u);
    else if (P.prim_counts)
        atomicAdd(reinterpret_cast<unsigned long long*>(P.prim_counts) + (size_t)S.inst * P.max_prims + hb, 1ull);
    const DevGeom G = geoms[S.geom];
    const bool substrate = hb == G.substrate();
    if (!substrate && !P.records) return;
    const float E = energy_of(P, S.inst, S.speed);
    int cell = -1;
    float cosang = 0.0f;
    if (substrate) {
        const DevPrim& Q = prims[G.begin + hb];
        const float dn = S.dx * Q.nx + S.dy * Q.ny + S.dz * Q.nz;
        if (dn < 0.0f) {
            const float qx = fmaf(tb, S.dx, S.px) - Q.cx, qy = fmaf(tb, S.dy, S.py) - Q.cy,
                        qz = fmaf(tb, S.dz, S.pz) - Q.cz;
            const float a1 = qx * Q.ux + qy * Q.uy + qz * Q.uz;
            const float a2 = qx * Q.vx + qy * Q.vy + qz * Q.vz;
            const float fx = (a1 + P.half_u) * P.cells_per_mm_u;
            const float fy = (a2 + P.half_v) * P.cells_per_mm_v;
            if (fx >= 0.0f && fy >= 0.0f && fx <= (float)P.nx && fy <= (float)P.ny) {
                const int ix = min((int)fx, P.nx - 1), iy = min((int)fy, P.ny - 1);
                cell = iy * P.nx + ix;
            }
            cosang = -dn;
        }
    }
    const int ncell = P.nx * P.ny;
    if (cell >= 0 && idx_ok(P.status, (long long)S.inst * ncell + cell, (long long)P.n_inst * ncell)) {
        const size_t ci = (size_t)S.inst * ncell + cell;
        if (P.counts) {
            if (P.count64) atomicAdd(reinterpret_cast<unsigned long long*>(P.counts) + ci, 1ull);
            else atomicAdd(reinterpret_cast<unsigned int*>(P.counts) + ci, 1u);
        }
        if (P.energy) atomicAdd(P.energy + ci, (double)E);
        if (P.score) atomicAdd(P.score + ci, (double)S.score);
        if (kMode == kModeScoreT) atomicAdd(P.score_T + ci, (double)S.scoreT);
        if (P.hist_E) {
            int b = min(max((int)(E * P.ebin_per_eV), 0), P.n_ebins - 1);
            atomicAdd(reinterpret_cast<unsigned long long*>(P.hist_E) + (size_t)S.inst * P.n_ebins + b, 1ull);
        }
        if (P.hist_A) {
            const float th = acosf(fminf(cosang, 1.0f)) * (57.29577951308232f / 90.0f);
            int b = min(max((int)(th * (float)P.n_abins), 0), P.n_abins - 1);
            atomicAdd(reinterpret_cast<unsigned long long*>(P.hist_A) + (size_t)S.inst * P.n_abins + b, 1ull);
        }
    }
    if (P.records) write_record(P, S, hb, cell, E, cosang);
}

__device__ __forceinline__ void tally_timed_out(const Params& P, const Lane& S, unsigned int* s_cnt, int nonfinite)
{
    if (nonfinite) atomicOr(P.status, kStatusNonFinite);
    if (s_cnt) atomicAdd(&s_cnt[S.inst * (P.max_prims + 1) + P.max_prims], 1u);
    else if (P.timed_out) atomicAdd(reinterpret_cast<unsigned long long*>(P.timed_out) + S.inst, 1ull);
    if (P.records) write_record(P, S, -1, -1, energy_of(P, S.inst, S.speed), 0.0f);
}

// ------------------------------------------------------------- kernel
struct SmemLayout {
    size_t prims, geoms, pairs, prefix, gm, pool, queue, scratch, counters, total;
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

__host__ __device__ inline SmemLayout smem_layout(const Params& p)
{
    SmemLayout L;
    size_t o = 0;
    L.prims = o;
    o = align16(o + sizeof(DevPrim) * p.n_prims);
    L.geoms = o;
    o = align16(o + sizeof(DevGeom) * p.n_geoms);
    L.pairs = o;
    o = align16(o + sizeof(DevPair) * p.n_pairs);
    L.prefix = o;
    o = align16(o + sizeof(unsigned long long) * (p.n_inst + 1));
    L.gm = o;
    o = align16(o + sizeof(float4) * (kGMHalf + kGMHalfLo));
    L.pool = o;
    o = align16(o + sizeof(unsigned long long) * 4 * p.block_warps);
    L.queue = o;
    o = align16(o + sizeof(uint32_t) * kLaunchWords * 32 * p.block_warps);
    L.scratch = o;
    o = align16(o + sizeof(WarpScratch) * p.block_warps);
    L.counters = o;
    o = align16(o + (p.smem_counters ? sizeof(unsigned int) * (size_t)p.n_inst * (p.max_prims + 1) : 0));
    L.total = o;
    return L;
}

__device__ __forceinline__ void copy16(void* dst, const void* src, size_t bytes)
{
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    for (size_t i = threadIdx.x; i < bytes / 16; i += blockDim.x) d[i] = s[i];
    const unsigned char* sb = reinterpret_cast<const unsigned char*>(src);
    unsigned char* db = reinterpret_cast<unsigned char*>(dst);
    for (size_t i = (bytes / 16) * 16 + threadIdx.x; i < bytes; i += blockDim.x) db[i] = sb[i];
}

// Persistent warp pool.  Four blocks of 256 threads per SM (32 warps, 64 registers a
// thread): the issue-bound loop gains more from the extra warps than it loses to the
// few spills at 64 registers (five blocks at 48 registers: quaternary 48.7 against 46.8 ms); the
// lane state is kept small for it (the instance's conditions read at each flight, the ticket
// recomputed from (instance, id), the warp's ticket pool in shared memory).  Bound by
// instruction issue: 50 warp instructions per collision on the quaternary scene, issue slots
// 80 % busy.
template <int kMode, int kMasks>
__global__ void __launch_bounds__(256, 4) transport_kernel(const Params P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const SmemLayout L = smem_layout(P);
    DevPrim* s_prims = reinterpret_cast<DevPrim*>(smem + L.prims);
    DevGeom* s_geoms = reinterpret_cast<DevGeom*>(smem + L.geoms);
    DevPair* s_pairs = reinterpret_cast<DevPair*>(smem + L.pairs);
    unsigned long long* s_prefix = reinterpret_cast<unsigned long long*>(smem + L.prefix);
    float4* s_gm = reinterpret_cast<float4*>(smem + L.gm);
    unsigned long long* s_pool = reinterpret_cast<unsigned long long*>(smem + L.pool);
    uint32_t* s_queue = reinterpret_cast<uint32_t*>(smem + L.queue);
    unsigned int* s_cnt = P.smem_counters ? reinterpret_cast<unsigned int*>(smem + L.counters) : nullptr;

    copy16(s_prims, P.prims, sizeof(DevPrim) * P.n_prims);
    copy16(s_geoms, P.geoms, sizeof(DevGeom) * P.n_geoms);
    copy16(s_pairs, P.pairs, sizeof(DevPair) * P.n_pairs);
    copy16(s_prefix, P.prefix, sizeof(unsigned long long) * (P.n_inst + 1));
    if (threadIdx.x < kGMHalf) s_gm[threadIdx.x] = P.gm[threadIdx.x];
    else if (threadIdx.x < kGMHalf + kGMHalfLo) s_gm[threadIdx.x] = P.gm_lo[threadIdx.x - kGMHalf];
    const int n_cnt = P.smem_counters ? P.n_inst * (P.max_prims + 1) : 0;
    for (int i = threadIdx.x; i < n_cnt; i += blockDim.x) s_cnt[i] = 0u;
    __syncthreads();

    TableView T;
    T.bm = P.bm_tab;
    T.xh = P.xh_tab;  // (off the deflection table only: stays in global memory)
    T.w = P.w_tab;
    T.gm = s_gm;
    T.pairs = s_pairs;
    T.geoms = s_geoms;
    T.bm_n = P.bm_n;
    T.bm_top = 8388608.0f + (P.bm_n - 1.0f);
    T.n_w = P.n_w_all;
    T.bm_lo = P.bm_lo;
    T.bm_inv_h = P.bm_inv_h;
    T.status = P.status;

    const int lane = threadIdx.x & 31;
    const unsigned lane_lt = (1u << lane) - 1u;
    Lane S;
    S.px = S.py = S.pz = S.dx = S.dy = S.dz = S.speed = S.score = S.scoreT = 0.0f;
    S.pid = S.inst = S.k = 0u;
    S.geom = S.pair = 0;
    S.strm = 0u;
    S.target = -1;
    S.ng14 = 0.0f;
    bool alive = false;

    // per-lane statistics; particles = landed + timed out, flights = landed + timed out + collided
    uint32_t c_landed = 0, c_timed = 0, c_coll = 0, c_att = 0;
    // the warp's ticket pool [next, end) lives in shared memory (warp-uniform, read only
    // when the warp refills); the pool is exhausted once its end reaches ticket_end
    // and its queue of prepared launches: s_wpool[2] entries of kLaunchWords words
    unsigned long long* s_wpool = s_pool + 4 * (threadIdx.x >> 5);
    uint32_t* s_wqueue = s_queue + kLaunchWords * 32 * (threadIdx.x >> 5);
    WarpScratch* s_wscratch = reinterpret_cast<WarpScratch*>(smem + L.scratch) + (threadIdx.x >> 5);
    if (lane == 0) s_wpool[0] = s_wpool[1] = s_wpool[2] = 0ull;
    __syncwarp();

    for (;;) {
        // ---------------------------------------------------- refill (warp-uniform)
        // Dead lanes take prepared launches from the warp's queue at once.  When the
        // queue runs short, the whole warp prepares the next launches together, one
        // per lane, so the launch code runs with every lane busy instead of once for
        // a few dead lanes while the others wait.
        const unsigned need = __ballot_sync(kFull, !alive);
        if (need) {
            const unsigned n = __popc(need);
            const unsigned rank = __popc(need & lane_lt);
            unsigned qn = (unsigned)s_wpool[2];  // prepared launches in the queue (warp-uniform)
            if (qn < n) {
                // the whole warp prepares launches for up to 32 - qn new tickets, one per lane,
                // so that the launch code runs with every lane busy
                const unsigned want = 32u - qn;
                unsigned long long pool_next = s_wpool[0], pool_end = s_wpool[1];
                const bool exhausted = pool_end == P.ticket_end;
                const unsigned long long avail = pool_end - pool_next;
                unsigned long long t = ~0ull;
                if ((unsigned)lane < want && lane < avail) t = pool_next + lane;
                if (want > avail && !exhausted) {
                    const unsigned long long more = want - avail;
                    const unsigned long long grab = more > (unsigned long long)P.chunk ? more : (unsigned long long)P.chunk;
                    unsigned long long base = 0ull;
                    if (lane == 0) base = atomicAdd(P.ticket_counter, grab);
                    base = __shfl_sync(kFull, base, 0) + P.ticket_begin;
                    if ((unsigned)lane < want && lane >= avail && base + (lane - avail) < P.ticket_end)
                        t = base + (lane - avail);
                    const unsigned long long ne = base + grab < P.ticket_end ? base + grab : P.ticket_end;
                    const unsigned long long nn = base + more < ne ? base + more : ne;
                    pool_next = nn;
                    pool_end = ne;
                } else {
                    pool_next += (want < avail ? want : avail);
                }
                if (t != ~0ull) {
                    // ticket -> (instance, particle id) by binary search over the instance prefix
                    int lo = 0, hi = P.n_inst;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (s_prefix[mid] <= t) lo = mid;
                        else hi = mid;
                    }
                    const Launch Ln = prepare_launch(P, (uint32_t)lo, (uint32_t)(t - s_prefix[lo]));
                    uint32_t* e = s_wqueue + kLaunchWords * (qn + lane);
                    e[0] = __float_as_uint(Ln.px);
                    e[1] = __float_as_uint(Ln.py);
                    e[2] = __float_as_uint(Ln.pz);
                    e[3] = __float_as_uint(Ln.dx);
                    e[4] = __float_as_uint(Ln.dy);
                    e[5] = __float_as_uint(Ln.dz);
                    e[6] = __float_as_uint(Ln.speed);
                    e[7] = Ln.inst;
                    e[8] = Ln.pid;
                }
                qn += __popc(__ballot_sync(kFull, t != ~0ull));  // the lanes with tickets are a prefix
                __syncwarp();
                if (lane == 0) {
                    s_wpool[0] = pool_next;
                    s_wpool[1] = pool_end;
                }
            }
            // the dead lanes take launches from the top of the queue
            if (!alive && rank < qn) {
                const uint32_t* e = s_wqueue + kLaunchWords * (qn - 1u - rank);
                Launch Ln;
                Ln.px = __uint_as_float(e[0]);
                Ln.py = __uint_as_float(e[1]);
                Ln.pz = __uint_as_float(e[2]);
                Ln.dx = __uint_as_float(e[3]);
                Ln.dy = __uint_as_float(e[4]);
                Ln.dz = __uint_as_float(e[5]);
                Ln.speed = __uint_as_float(e[6]);
                Ln.inst = e[7];
                Ln.pid = e[8];
                start_from(S, P, Ln);
                alive = true;
            }
            __syncwarp();
            if (lane == 0) s_wpool[2] = qn - (n < qn ? n : qn);
            __syncwarp();
            // no tickets left and few atoms alive (or every atom, when the run is small):
            // hand them over to drain_kernel, which follows
            if (P.pool && (P.drain_live >= 32 || (qn < n && 32 - (int)(n - qn) <= P.drain_live))) {
                pool_store(P, alive, S);
                alive = false;
                if (qn >= n) continue;  // every lane got an atom: there may be more tickets
            }
        }
        if (!__any_sync(kFull, alive)) break;

        // ---------------------------------------------------- one flight (all lanes together)
        StepOut so;
        const int res = flight_step_warp<kMode, kMasks>(alive, S, P, T, s_prims, s_pairs, s_wscratch, so);
        c_att += so.attempts;
        if (res == kStepLanded) {
            tally_landed<kMode>(P, S, s_geoms, s_prims, s_cnt, so.t, so.prim);
            ++c_landed;
            c_coll += S.k - 1u;
            alive = false;
        } else if (res == kStepTimedOut) {
            tally_timed_out(P, S, s_cnt, so.nonfinite);
            ++c_timed;
            c_coll += S.k - 1u;
            alive = false;
        }
    }

    // ---------------------------------------------------- flush counters
    add_stats(P, c_landed, c_timed, c_coll, c_att);
    if (P.smem_counters) {
        __syncthreads();
        for (int i = threadIdx.x; i < n_cnt; i += blockDim.x) {
            const unsigned int c = s_cnt[i];
            if (!c) continue;
            const int inst = i / (P.max_prims + 1), li = i % (P.max_prims + 1);
            if (li < P.max_prims) {
                if (P.prim_counts)
                    atomicAdd(reinterpret_cast<unsigned long long*>(P.prim_counts) + (size_t)inst * P.max_prims + li,
                              (unsigned long long)c);
            } else if (P.timed_out) {
                atomicAdd(reinterpret_cast<unsigned long long*>(P.timed_out) + inst, (unsigned long long)c);
            }
        }
    }
}

// ------------------------------------------------------------- the last atoms
// Atoms handed over by transport_kernel: the whole of a small run, and the last ones of a large
// one.  Trajectories are long-tailed (0.5 Pa: median 12 collisions, longest of 1e5 atoms 734;
// 3 Pa: 270 and 9652 of 1e6), so a run's end, or all of a small one, lasts as long as the
// longest trajectory takes, one dependent step after the other: 3.3 us per step in a sparse warp
// of transport_kernel.  Here G = 8, 16 or 32 lanes carry one atom, G flights at a time, so that
// what does not depend on the trajectory is done in parallel and little is left on the chain:
//   1. the lanes draw the batch's random numbers (flight l and its first four partner
//      attempts in lane l) into shared memory;
//   2. the collisions, one after the other.  The gas is homogeneous, so velocities follow from
//      the collisions alone: where the atom is does not enter.  Eight lanes compute the
//      collision with each of four attempts in either branch of its proposal while the envelope
//      is looked up and tested, and the accepted lane's velocity is taken (0.1 % of the
//      collisions need more attempts); lane f keeps the velocity before flight f;
//   3. lane f works out flight f: the free path, the position (a running sum over the
//      flights), the surface test.  The first flight that lands ends the atom; the
//      collisions drawn beyond it are dropped.
// A warp starts with as many lanes per atom as the pool's size allows, and once the pool is
// empty the lanes of finished atoms join the others'.  Every number is computed as in the
// single-lane step, so the results are bit-identical.
// Bound by the latency of the chain, 1200 cycles (0.6 us) per step, a third of it waiting for the
// deflection table in L1 or L2.  Measured on a GB300 without and with the drain when it came:
// single Ni 3e3 atoms 1.8 -> 0.53 ms (now 0.35), 1e5 2.4 -> 1.26 ms (0.91), quaternary 4e5
// 3.0 -> 1.8 ms (1.3), 64 primitives at 3 Pa 1e6 atoms 59 -> 47 ms (38).  Which atoms of a run
// come here: hand_over in sput_api.cpp.
constexpr int kDrawn = 4;
constexpr int kMinGroupLog2 = 3;

struct DrainWarp {                // by the flight's lane
    float4 z[32][kDrawn];         // z1, z2, z3, u of an attempt
    float4 rho[32][kDrawn];       // r3, rho_w, sc_w
    Impact hit[32];               // the collision after the flight
    float4 walk[32];              // direction after the flight (diffusion shortcut)
    uint2 list[32];               // of nearest_hit_masks
};

struct DrainLayout {
    size_t prims, geoms, pairs, gm, warps, total;
};

__host__ __device__ inline DrainLayout drain_layout(const Params& p)
{
    DrainLayout L;
    size_t o = 0;
    L.warps = o;
    o = align16(o + sizeof(DrainWarp) * (kDrainThreads / 32));
    L.prims = o;
    o = align16(o + sizeof(DevPrim) * p.n_prims);
    L.geoms = o;
    o = align16(o + sizeof(DevGeom) * p.n_geoms);
    L.pairs = o;
    o = align16(o + sizeof(DevPair) * p.n_pairs);
    L.gm = o;
    o = align16(o + sizeof(float4) * (kGMHalf + kGMHalfLo));
    L.total = o;
    return L;
}

// The batch's collisions, one after the other (2. above): S goes through them; F, in lane f of the
// group, keeps the velocity before flight f, and att and V2 its partner's attempts and |V|^2.
// kFast: thermal gas and a deflection table, so that a step is one run of straight-line code in
// which the loads and the MUFU overlap.
template <int kMode, bool kFast>
__device__ __forceinline__ void drain_collisions(Lane& S, Lane& F, const Params& P, const TableView& T,
                                                 const DrainWarp& W, const DevPair& pr, bool have, int head, int l,
                                                 int G, uint32_t& att, float& V2)
{
    constexpr bool kScoreT = kMode == kModeScoreT;
    const bool thermal = kFast || P.gas_thermal;
    const int A = P.max_attempts;
    const int my_a = l & (kDrawn - 1);
    const bool my_branch = (l & kDrawn) != 0;
#pragma unroll 1
    for (int f = 0; f < G; ++f) {
        if (l == f) {
            F.speed = S.speed;
            F.dx = S.dx;
            F.dy = S.dy;
            F.dz = S.dz;
            F.diff = S.diff;
        }
        const bool walk = kMode == kModeWalk && S.diff;
        bool pend = have && !walk;
        if (kMode == kModeWalk && walk) {
            const float4 d = W.walk[head + f];
            S.dx = d.x;
            S.dy = d.y;
            S.dz = d.z;
        }
        if (kMode == kModeWalk && !__any_sync(kFull, pend)) continue;
        const float vx = __fmul_rn(S.speed, S.dx), vy = __fmul_rn(S.speed, S.dy), vz = __fmul_rn(S.speed, S.dz);
        float EA = 0.0f, EB = 0.0f;
        if (thermal) {
            int i;
            float t;
            wtab_cell(pr, S.speed, i, t);
            EA = wtab_at(T, pr, kTabA, i, t);
            EB = wtab_at(T, pr, kTabB, i, t);
        }
        const Impact h = W.hit[head + f];
        const float4 z = W.z[head + f][my_a], r = W.rho[head + f][my_a];
        Attempt d;
        d.z1 = z.x;
        d.z2 = z.y;
        d.z3 = z.z;
        d.u = z.w;
        d.r3 = r.x;
        d.rho_w = r.y;
        d.sc_w = r.z;
        for (int a = my_a;;) {
            // the collision with this lane's attempt in its branch, and whether it is the one
            float cx = 0.0f, cy = 0.0f, cz = 0.0f;
            bool acc = true;
            if (thermal) attempt_velocity(P, d, my_branch, cx, cy, cz);
            float ns = S.speed, nx = S.dx, ny = S.dy, nz = S.dz;
            const bool usual = scatter<kMode, kFast>(ns, nx, ny, nz, P, T, pr, vx, vy, vz, cx, cy, cz, h);
            if (thermal) {
                float ut, Bm;
                const bool weighted = attempt_weighted(d, EA, EB, ut, Bm);
                const float hg = attempt_h<kFast>(T, pr, vx, vy, vz, cx, cy, cz);
                const bool ok = attempt_accept(d, my_branch, ut, Bm, EA, EB, hg);
                acc = (a < A) & (weighted == my_branch) & (ok | (a == A - 1));
            }
            // the first accepted attempt, in either branch
            const unsigned m = __ballot_sync(kFull, acc) >> head;
            const unsigned first = (m | m >> kDrawn) & ((1u << kDrawn) - 1u);
            int src = first ? __ffs(first) - 1 : 0;
            const uint32_t n_att = (uint32_t)(a - my_a + src) + 1u;
            if (!((m >> src) & 1u)) src += kDrawn;
            if (kFast && !usual) {  // rare
                ns = S.speed;
                nx = S.dx;
                ny = S.dy;
                nz = S.dz;
                scatter<kMode, false>(ns, nx, ny, nz, P, T, pr, vx, vy, vz, cx, cy, cz, h);
            }
            ns = __shfl_sync(kFull, ns, head + src);
            nx = __shfl_sync(kFull, nx, head + src);
            ny = __shfl_sync(kFull, ny, head + src);
            nz = __shfl_sync(kFull, nz, head + src);
            const float c2 = kScoreT ? __shfl_sync(kFull, sumsq_xyz(cx, cy, cz), head + src) : 0.0f;
            if (pend && first) {
                S.speed = ns;
                S.dx = nx;
                S.dy = ny;
                S.dz = nz;
                if (l == f) {
                    att = thermal ? n_att : 0u;
                    V2 = c2;
                }
                if (kMode == kModeWalk && energy_of(P, S.inst, S.speed) < P.E_switch) S.diff = true;
                pend = false;
            }
            if (!__any_sync(kFull, pend)) break;
            // rare: none of the drawn attempts; the group draws four more
            a += kDrawn;
            d = attempt_draw(P, S.pid, S.strm, S.k + 1u + f, (uint32_t)a);
        }
    }
}

template <int kMode, int kMasks>
__global__ void __launch_bounds__(kDrainThreads, 2) drain_kernel(const Params P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool kScoreT = kMode == kModeScoreT;
    // (one lane's reading, so that a warp agrees on it whatever becomes of the counter)
    const unsigned n_pool = min(__shfl_sync(kFull, *P.pool_count, 0), P.pool_slots);
    const unsigned n_warps = gridDim.x * (kDrainThreads / 32);
    const unsigned per_warp = (n_pool + n_warps - 1u) / n_warps;
    int lg = per_warp <= 1u ? 5 : per_warp <= 2u ? 4 : kMinGroupLog2;  // log2 of the lanes per atom
    if ((unsigned long long)blockIdx.x * (kDrainThreads / 32) * (32u >> lg) >= n_pool) return;

    const DrainLayout L = drain_layout(P);
    DevPrim* s_prims = reinterpret_cast<DevPrim*>(smem + L.prims);
    DevGeom* s_geoms = reinterpret_cast<DevGeom*>(smem + L.geoms);
    DevPair* s_pairs = reinterpret_cast<DevPair*>(smem + L.pairs);
    float4* s_gm = reinterpret_cast<float4*>(smem + L.gm);
    DrainWarp& W = reinterpret_cast<DrainWarp*>(smem + L.warps)[threadIdx.x >> 5];
    // the lanes of a group without an atom go through the collisions with the others: what they read
    // has to be a table column from the start (shared memory begins with anything)
    W.hit[threadIdx.x & 31] = Impact{1.0f, 0, 0.0f, 0.0f, 0.0f};
    copy16(s_prims, P.prims, sizeof(DevPrim) * P.n_prims);
    copy16(s_geoms, P.geoms, sizeof(DevGeom) * P.n_geoms);
    copy16(s_pairs, P.pairs, sizeof(DevPair) * P.n_pairs);
    if (threadIdx.x < kGMHalf) s_gm[threadIdx.x] = P.gm[threadIdx.x];
    else if (threadIdx.x < kGMHalf + kGMHalfLo) s_gm[threadIdx.x] = P.gm_lo[threadIdx.x - kGMHalf];
    __syncthreads();

    TableView T;
    T.bm = P.bm_tab;
    T.xh = P.xh_tab;  // (off the deflection table only: stays in global memory)
    T.w = P.w_tab;
    T.gm = s_gm;
    T.pairs = s_pairs;
    T.geoms = s_geoms;
    T.bm_n = P.bm_n;
    T.bm_top = 8388608.0f + (P.bm_n - 1.0f);
    T.n_w = P.n_w_all;
    T.bm_lo = P.bm_lo;
    T.bm_inv_h = P.bm_inv_h;
    T.status = P.status;

    const int lane = threadIdx.x & 31;
    Lane S;  // the group's atom, the same in its lanes
    S.px = S.py = S.pz = S.dx = S.dy = S.dz = S.speed = S.score = S.scoreT = 0.0f;
    S.pid = S.inst = S.k = 0u;
    S.geom = S.pair = 0;
    S.strm = 0u;
    S.target = -1;
    S.ng14 = 0.0f;
    S.diff = false;
    bool have = false, more = true;  // more: the pool may hold further atoms (warp-uniform)
    uint32_t c_landed = 0, c_timed = 0, c_coll = 0, c_att = 0;

    for (;;) {
        int head = lane >> lg << lg, l = lane - head;  // the group's first lane, lane in the group
        // ---------------------------------------------------- next atoms
        while (more && __any_sync(kFull, !have)) {
            unsigned i = 0u;
            if (!have && l == 0) i = atomicAdd(P.pool_next, 1u);
            i = __shfl_sync(kFull, i, head);
            more = !__any_sync(kFull, !have && i >= n_pool);
            const float4* q = P.pool + 4 * (size_t)i;
            float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (!have && i < n_pool) c = q[2];
            if (!have && i < n_pool && pool_holds(P, __float_as_uint(c.y), __float_as_uint(c.x))) {
                const float4 a = q[0], b = q[1];
                S.px = a.x;
                S.py = a.y;
                S.pz = a.z;
                S.speed = a.w;
                S.dx = b.x;
                S.dy = b.y;
                S.dz = b.z;
                S.score = b.w;
                S.pid = __float_as_uint(c.x);
                S.inst = __float_as_uint(c.y);
                S.k = __float_as_uint(c.z);
                S.diff = __float_as_uint(c.w) != 0u;
                if (kScoreT) S.scoreT = q[3].x;
                load_conditions(S, P);
                have = true;
            }
        }
        if (!more) {
            // half as many atoms as groups or fewer: twice as many lanes each
            const unsigned heads = __ballot_sync(kFull, have && l == 0);
            const int live = __popc(heads);
            if (live == 0) break;
            if (lg < 5 && 2 * live <= 32 >> lg) {
                do ++lg;
                while (lg < 5 && 2 * live <= 32 >> lg);
                const int to = lane >> lg;
                have = to < live;
                const int src = nth_set_bit(heads, have ? to : 0);
                S.px = __shfl_sync(kFull, S.px, src);
                S.py = __shfl_sync(kFull, S.py, src);
                S.pz = __shfl_sync(kFull, S.pz, src);
                S.dx = __shfl_sync(kFull, S.dx, src);
                S.dy = __shfl_sync(kFull, S.dy, src);
                S.dz = __shfl_sync(kFull, S.dz, src);
                S.speed = __shfl_sync(kFull, S.speed, src);
                S.score = __shfl_sync(kFull, S.score, src);
                if (kScoreT) S.scoreT = __shfl_sync(kFull, S.scoreT, src);
                if (kMode == kModeWalk) S.diff = __shfl_sync(kFull, (int)S.diff, src) != 0;
                S.pid = __shfl_sync(kFull, S.pid, src);
                S.inst = __shfl_sync(kFull, S.inst, src);
                S.k = __shfl_sync(kFull, S.k, src);
                S.geom = __shfl_sync(kFull, S.geom, src);
                S.target = __shfl_sync(kFull, S.target, src);
                S.pair = __shfl_sync(kFull, S.pair, src);
                S.ng14 = __shfl_sync(kFull, S.ng14, src);
                S.strm = __shfl_sync(kFull, S.strm, src);
                head = lane >> lg << lg;
                l = lane - head;
            }
        }
        const int G = 1 << lg;

        // ---------------------------------------------------- 1. random numbers
        float nl = 0.0f;  // -ln u of the free path of flight l
        if (have) {
            const uint32_t k = S.k + 1u + l;
            const uint4 w = philox(P, S.pid, S.strm, k, 0u);
            nl = neg_log_fast(rn(w.x));
            W.hit[lane] = impact_draw(w);
            if (kMode == kModeWalk) {
                float4 d = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                walk_direction(w, d.x, d.y, d.z);
                W.walk[lane] = d;
            }
            if (P.gas_thermal) {
#pragma unroll 2
                for (int a = 0; a < kDrawn; ++a) {
                    const Attempt d = attempt_draw(P, S.pid, S.strm, k, (uint32_t)a);
                    W.z[lane][a] = make_float4(d.z1, d.z2, d.z3, d.u);
                    W.rho[lane][a] = make_float4(d.r3, d.rho_w, d.sc_w, 0.0f);
                }
            }
        }
        __syncwarp();

        // ---------------------------------------------------- 2. collisions
        Lane F;  // flight l: the velocity before it, later its position and scores
        F.pid = S.pid;
        F.inst = S.inst;
        F.geom = S.geom;
        F.target = S.target;
        F.pair = S.pair;
        F.ng14 = S.ng14;
        F.k = S.k + 1u + l;
        F.speed = F.dx = F.dy = F.dz = 0.0f;
        F.diff = false;
        uint32_t att = 0u;
        float V2 = 0.0f;
        const DevPair& pr = s_pairs[S.pair];
        if (P.usual) drain_collisions<kMode, true>(S, F, P, T, W, pr, have, head, l, G, att, V2);
        else drain_collisions<kMode, false>(S, F, P, T, W, pr, have, head, l, G, att, V2);

        // ---------------------------------------------------- 3. flights
        float inv_lam = 0.0f, ell = 0.0f, Gv = 0.0f;
        if (have) {
            int i;
            float t;
            wtab_cell(pr, F.speed, i, t);
            flight_length<kMode>(F, P, T, pr, i, t, nl, inv_lam, ell, Gv);
        }
        // positions and scores before each flight: running sums over the batch, in order
        const float gain = score_gain(ell, inv_lam);
        const float aT = kScoreT ? score_T_rate(P, Gv) : 0.0f;
        const float cT = kScoreT ? score_T_partner(P, V2, Gv) : 0.0f;
        F.px = S.px;
        F.py = S.py;
        F.pz = S.pz;
        F.score = S.score;
        F.scoreT = S.scoreT;
#pragma unroll 8
        for (int f = 0; f < G; ++f) {
            const int src = head + f;
            const float e = __shfl_sync(kFull, ell, src);
            S.px = fmaf(e, __shfl_sync(kFull, F.dx, src), S.px);
            S.py = fmaf(e, __shfl_sync(kFull, F.dy, src), S.py);
            S.pz = fmaf(e, __shfl_sync(kFull, F.dz, src), S.pz);
            const float gn = __shfl_sync(kFull, gain, src);
            S.score += gn;
            if (kScoreT) {
                S.scoreT = fmaf(__shfl_sync(kFull, aT, src), gn, S.scoreT);
                if (P.gas_thermal) S.scoreT = fmaf(__shfl_sync(kFull, cT, src), P.inv_T, S.scoreT);
            }
            if (l > f) {
                F.px = S.px;
                F.py = S.py;
                F.pz = S.pz;
                F.score = S.score;
                F.scoreT = S.scoreT;
            }
        }
        float tb = CUDART_INF_F;
        int hb = -1;
        if (kMasks) nearest_hit_masks<kMasks ? kMasks : 1>(have, F, P, T, s_prims, W.list, ell, tb, hb);
        else if (have) nearest_hit_loop(F, P, T, s_prims, ell, tb, hb);
        StepOut out;
        out.Gv = Gv;
        int res = kStepNone;
        if (have) res = flight_end<kMode>(F, P, out, inv_lam, ell, tb, hb);
        const unsigned ends = (__ballot_sync(kFull, res == kStepLanded || res == kStepTimedOut) >> head) &
                              (0xffffffffu >> (32 - G));
        const int last = ends ? __ffs(ends) - 1 : G;
        if (have && l < last) c_att += att;
        if (have && l == last) {
            if (res == kStepLanded) {
                tally_landed<kMode>(P, F, s_geoms, s_prims, nullptr, out.t, out.prim);
                ++c_landed;
            } else {
                tally_timed_out(P, F, nullptr, out.nonfinite);
                ++c_timed;
            }
            c_coll += F.k - 1u;
        }
        S.k += G;
        if (ends) have = false;
        __syncwarp();
    }
    add_stats(P, c_landed, c_timed, c_coll, c_att);
}

// ------------------------------------------------------------- probes
template <int kMode>
__device__ int trace_step(int words, bool active, Lane& S, const Params& P, const TableView& T, WarpScratch* ws, StepOut& out)
{
    return words == 0   ? flight_step_warp<kMode, 0>(active, S, P, T, P.prims, P.pairs, ws, out)
           : words == 1 ? flight_step_warp<kMode, 1>(active, S, P, T, P.prims, P.pairs, ws, out)
                        : flight_step_warp<kMode, 2>(active, S, P, T, P.prims, P.pairs, ws, out);
}

__global__ void probe_kernel(const Params P, int what, int idx, int n, const double* x, double* y)
{
    __shared__ float4 s_gm[kGMHalf + kGMHalfLo];
    __shared__ WarpScratch s_ws[4];  // (launched with 128 threads)
    if (threadIdx.x < kGMHalf) s_gm[threadIdx.x] = P.gm[threadIdx.x];
    else if (threadIdx.x < kGMHalf + kGMHalfLo) s_gm[threadIdx.x] = P.gm_lo[threadIdx.x - kGMHalf];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    TableView T;
    T.bm = P.bm_tab;
    T.xh = P.xh_tab;
    T.w = P.w_tab;
    T.gm = s_gm;
    T.pairs = P.pairs;
    T.geoms = P.geoms;
    T.bm_n = P.bm_n;
    T.bm_top = 8388608.0f + (P.bm_n - 1.0f);
    T.n_w = P.n_w_all;
    T.bm_lo = P.bm_lo;
    T.bm_inv_h = P.bm_inv_h;
    T.status = P.status;
    if (what == SPUT_PROBE_TRACE) {
        // state after each flight of particle x[i] of instance idx, kTraceRows rows of 10;
        // the flight step is warp-collective, so lanes past n take part without a particle
        const bool valid = i < n;
        Lane S;
        S.px = S.py = S.pz = S.dx = S.dy = S.dz = S.speed = S.score = S.scoreT = 0.0f;
        S.pid = S.inst = S.k = 0u;
        S.geom = S.pair = 0;
        S.strm = 0u;
        S.target = -1;
        S.ng14 = 0.0f;
        double* o = valid ? y + (size_t)i * kTraceRows * 10 : nullptr;
        if (valid) {
            start_particle(S, P, (uint32_t)idx, (uint32_t)x[i]);
            for (int r = 0; r < kTraceRows * 10; ++r) o[r] = 0.0;
            for (int r = 1; r < kTraceRows; ++r) o[r * 10 + 7] = -2.0;
            o[0] = S.px; o[1] = S.py; o[2] = S.pz; o[3] = S.dx; o[4] = S.dy; o[5] = S.dz; o[6] = S.speed;
            o[7] = -1.0;
        }
        bool running = valid;
        for (int r = 1; r < kTraceRows; ++r) {
            if (!__any_sync(kFull, running)) break;
            StepOut so;
            // (the surface test of the scene's masks where it has them, whatever a run would choose)
            WarpScratch* ws = &s_ws[threadIdx.x >> 5];
            const int words = P.cell_mask ? P.cell_words : 0;
            const int status = P.E_switch > 0.0f ? trace_step<kModeWalk>(words, running, S, P, T, ws, so)
                                                 : trace_step<kModePlain>(words, running, S, P, T, ws, so);
            if (running) {
                double* q = o + (size_t)r * 10;
                float px = S.px, py = S.py, pz = S.pz;
                if (status == kStepLanded) {
                    px = fmaf(so.t, S.dx, S.px);
                    py = fmaf(so.t, S.dy, S.py);
                    pz = fmaf(so.t, S.dz, S.pz);
                }
                q[0] = px; q[1] = py; q[2] = pz; q[3] = S.dx; q[4] = S.dy; q[5] = S.dz; q[6] = S.speed;
                q[7] = status; q[8] = status == kStepLanded ? so.prim : so.attempts; q[9] = so.t;
                if (status != kStepCollided) running = false;
            }
        }
        return;
    }
    if (i >= n) return;
    if (what == SPUT_PROBE_CHI) {
        const float eps = (float)x[2 * i], beta = (float)x[2 * i + 1];
        const float le = logf(eps);
        y[i] = 3.141592653589793 * (double)chi_over_pi_moliere(eps, le, beta, xh_eval(T, le), T.gm);
    } else if (what == SPUT_PROBE_CHI_U) {
        // the collision's path: table inside its range, direct integration outside
        const float eps = (float)x[2 * i], ub = (float)x[2 * i + 1];
        const float le = logf(eps);
        float q, ty;
        int j;
        const bool column = chi_table_column(0.5f * logf(ub), j, ty);
        if (chi_table_q(P.chi_tab, P.status, le, j, ty, q) && column) {
            y[i] = 2.0 * atan(exp((double)q));
        } else {
            const float beta = bmax_eval(T, le) * sqrtf(ub);
            y[i] = 3.141592653589793 * (double)chi_over_pi_moliere(eps, le, beta, xh_eval(T, le), T.gm);
        }
    } else if (what == SPUT_PROBE_BMAX) {
        y[i] = bmax_eval(T, logf((float)x[i]));
    } else if (what == SPUT_PROBE_K) {
        const DevPair pr = P.pairs[idx];
        const float v = (float)x[i];
        int c;
        float t;
        wtab_cell(pr, v, c, t);
        float val = wtab_at(T, pr, kTabK, c, t);
        if (!P.gas_thermal) val *= v;  // the table holds sigma(v) = K/v
        y[i] = val;
    } else if (what == SPUT_PROBE_M) {
        // rejection envelope (A, B) of the pair at speed v
        const DevPair pr = P.pairs[idx];
        int c;
        float t;
        wtab_cell(pr, (float)x[i], c, t);
        y[2 * i] = wtab_at(T, pr, kTabA, c, t);
        y[2 * i + 1] = wtab_at(T, pr, kTabB, c, t);
    } else if (what == SPUT_PROBE_LAUNCH) {
        float px, py, pz, dx, dy, dz, E;
        launch_state(P, P.rt_tab, (uint32_t)idx, (uint32_t)x[i], px, py, pz, dx, dy, dz, E);
        double* o = y + 7 * (size_t)i;
        o[0] = px;
        o[1] = py;
        o[2] = pz;
        o[3] = dx;
        o[4] = dy;
        o[5] = dz;
        o[6] = E;
    }
}

}  // namespace

size_t transport_smem_bytes(const Params& p) { return smem_layout(p).total; }

// What counts towards the largest scene: a block's tables, pools and launch queues at eight warps,
// and the cross-section table, the apsis table and the stream words as if they were staged
// too (the limit dates from when they were, and scenes are accepted by it still).
size_t transport_scene_bytes(const Params& p)
{
    Params q = p;
    q.block_warps = 8;
    q.smem_counters = 0;
    return smem_layout(q).total - align16(sizeof(WarpScratch) * 8) + sizeof(float4) * p.n_bm +
           align16(sizeof(float) * (p.n_bm + 1)) + align16(sizeof(uint32_t) * p.n_inst);
}

namespace {

using KernelFn = void (*)(const Params);

// the instances [mode][words of the cell masks, 0 = the counted loop]
#define SPUT_KERNELS(k, mode) {k<mode, 0>, k<mode, 1>, k<mode, 2>}
#define SPUT_KERNEL_TABLE(k) {SPUT_KERNELS(k, kModePlain), SPUT_KERNELS(k, kModeScoreT), SPUT_KERNELS(k, kModeWalk)}
const KernelFn kTransport[3][3] = SPUT_KERNEL_TABLE(transport_kernel);
const KernelFn kDrain[3][3] = SPUT_KERNEL_TABLE(drain_kernel);
#undef SPUT_KERNEL_TABLE
#undef SPUT_KERNELS

// the smallest occupancy of a kernel's instances
int min_blocks_per_sm(const KernelFn (&k)[3][3], int threads, size_t smem)
{
    int m = 1 << 30;
    for (int mode = 0; mode < 3; ++mode)
        for (int words = 0; words < 3; ++words) {
            int nb = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k[mode][words], threads, smem) != cudaSuccess)
                return 0;
            m = nb < m ? nb : m;
        }
    return m;
}

int instance_mode(const Params& p) { return p.score_T ? kModeScoreT : (p.E_switch > 0.0f ? kModeWalk : kModePlain); }

}  // namespace

#ifdef SPUT_CHECKED
// For the tests of the checked library: which surface test the last run enqueued by this thread
// took (words of its cell masks, 0: the counted loop), and which atoms it handed to the drain
// (Params::drain_live, 0: none).
thread_local int t_mask_words = -1, t_drain_live = -1;
extern "C" int sput_checked_mask_words() { return t_mask_words; }
extern "C" int sput_checked_drain_live() { return t_drain_live; }
// and how the next run enqueued by this thread finds the hand-over pool, as one overlapped by another
// run of its scene would: `room` slots left, behind `taken` (at most 255) whose bytes are all `byte`
thread_local unsigned t_pool_taken = 0, t_pool_room = 0;
thread_local int t_pool_byte = 0;
extern "C" void sput_checked_overlap(unsigned taken, unsigned room, int byte)
{
    t_pool_taken = taken;
    t_pool_room = room;
    t_pool_byte = byte;
}
// and how many words of its cell masks the runs of this thread may read (-1: all)
thread_local long long t_mask_limit = -1;
extern "C" void sput_checked_mask_limit(long long words) { t_mask_limit = words; }
static Params for_test(Params p)
{
    if (t_mask_limit >= 0 && t_mask_limit < p.n_cell_words) p.n_cell_words = t_mask_limit;
    if (t_pool_room && p.pool && t_pool_taken + t_pool_room <= p.pool_slots) p.pool_slots = t_pool_taken + t_pool_room;
    return p;
}
#endif

size_t drain_smem_bytes(const Params& p) { return drain_layout(p).total; }

int transport_max_blocks_per_sm(int threads, size_t smem) { return min_blocks_per_sm(kTransport, threads, smem); }

int transport_blocks_per_sm(const Params& p, int threads, size_t smem)
{
    int nb = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &nb, kTransport[instance_mode(p)][p.cell_mask ? p.cell_words : 0], threads, smem);
    return e == cudaSuccess ? nb : 0;
}

int drain_max_blocks_per_sm(size_t smem) { return min_blocks_per_sm(kDrain, kDrainThreads, smem); }

int transport_configure(int max_dynamic_smem)
{
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    for (int mode = 0; mode < 3; ++mode)
        for (int words = 0; words < 3; ++words) {
            cudaError_t e = cudaFuncSetAttribute(kTransport[mode][words], a, max_dynamic_smem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kDrain[mode][words], a, max_dynamic_smem);
            if (e != cudaSuccess) return (int)e;
        }
    return 0;
}

int transport_launch(const Params& run, int blocks, int threads, size_t smem, void* stream)
{
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
#ifdef SPUT_CHECKED
    const Params p = for_test(run);
    t_mask_words = p.cell_mask ? p.cell_words : 0;
    t_drain_live = p.pool ? p.drain_live : 0;
    if (p.pool && p.pool_slots != run.pool_slots) {
        cudaMemsetAsync(p.pool, t_pool_byte, 4 * sizeof(float4) * t_pool_taken, st);
        cudaMemsetAsync(p.pool_count, (int)(t_pool_taken & 0xffu), 1, st);
    }
#else
    const Params& p = run;
#endif
    kTransport[instance_mode(p)][p.cell_mask ? p.cell_words : 0]<<<blocks, threads, smem, st>>>(p);
    return (int)cudaGetLastError();
}

int drain_launch(const Params& run, int blocks, size_t smem, void* stream)
{
#ifdef SPUT_CHECKED
    const Params p = for_test(run);
    t_pool_room = 0;
#else
    const Params& p = run;
#endif
    kDrain[instance_mode(p)][p.cell_mask ? p.cell_words : 0]<<<blocks, kDrainThreads, smem,
                                                               reinterpret_cast<cudaStream_t>(stream)>>>(p);
    return (int)cudaGetLastError();
}

int probe_launch(const Params& p, int what, int idx, int n, const double* x_dev, double* y_dev, void* stream)
{
    if (n <= 0) return 0;
    probe_kernel<<<(n + 127) / 128, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(p, what, idx, n, x_dev, y_dev);
    return (int)cudaGetLastError();
}

// ------------------------------------------------------- static run scratch
// Run scratch for sput_run_noalloc: ticket counter, statistics and status word
// in module memory, so that a run needs no device allocation at all.  Every
// device that loads the library holds these kStaticScratchBytes until the
// process exits.  In host code the name below is only a stand-in for the
// device symbol; its device address is looked up with the device current.
static __device__ __align__(256) unsigned long long g_static_run_scratch[kStaticScratchBytes / 8];

namespace {
// The address is cached per CUDA context, identified by the driver's context
// id: a context torn down and created again (cudaDeviceReset) gets a new id,
// so a stale address is never reused.  The two driver entry points are taken
// through the runtime, which needs no link against the driver library.
typedef CUresult (*PfnCtxGetCurrent)(CUcontext*);
typedef CUresult (*PfnCtxGetId)(CUcontext, unsigned long long*);

int current_context_id(unsigned long long* id)
{
    static PfnCtxGetCurrent get_current = nullptr;
    static PfnCtxGetId get_id = nullptr;
    if (!get_current || !get_id) {
        void* f0 = nullptr;
        void* f1 = nullptr;
        cudaDriverEntryPointQueryResult q0, q1;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f0, 12000, cudaEnableDefault, &q0);
        if (e == cudaSuccess)
            e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f1, 12000, cudaEnableDefault, &q1);
        if (e != cudaSuccess) return (int)e;
        if (q0 != cudaDriverEntryPointSuccess || q1 != cudaDriverEntryPointSuccess || !f0 || !f1)
            return (int)cudaErrorNotSupported;
        get_current = reinterpret_cast<PfnCtxGetCurrent>(f0);
        get_id = reinterpret_cast<PfnCtxGetId>(f1);
    }
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return (int)cudaErrorDeviceUninitialized;
    if (get_id(ctx, id) != CUDA_SUCCESS) return (int)cudaErrorDeviceUninitialized;
    return 0;
}
}  // namespace

int static_scratch_address(int device, unsigned long long** out)
{
    static std::mutex mu;
    static std::map<std::pair<int, unsigned long long>, unsigned long long*> cache;
    std::lock_guard<std::mutex> lock(mu);
    unsigned long long ctx_id = 0;
    int e0 = current_context_id(&ctx_id);
    if (e0 != 0) return e0;
    const auto key = std::make_pair(device, ctx_id);
    auto it = cache.find(key);
    if (it != cache.end()) {
        *out = it->second;
        return 0;
    }
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_run_scratch);
    if (e != cudaSuccess) return (int)e;
    cache[key] = reinterpret_cast<unsigned long long*>(ptr);
    *out = cache[key];
    return 0;
}

}  // namespace sput
