"""Composition map, its backward pass and the likelihood-ratio contraction at the sizes where their
grids and clusters can go wrong (one point, the edges of a warp and of a cluster's threads, one and
sixteen cathodes, an empty reference point, a rate of zero), against plain FP64 numpy.
Tolerance: sums of at most 4e4 products, rounded in another order, are within 4e4 x 1.1e-16 of
their absolute sum."""

import ctypes as C

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _p(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("n_cath,n_points,n_cells", [(1, 1, 1), (2, 31, 333), (3, 33, 1000), (4, 256, 40001),
                                                     (4, 257, 65536), (16, 342, 5001), (5, 1500, 20000)])
@pytest.mark.parametrize("special", ["plain", "empty_reference", "zero_rate"])
def test_composition_and_backward(n_cath, n_points, n_cells, special):
    import torch

    from paper_2411_14413_gb300 import _native as N

    rng = np.random.default_rng(n_cath * 1000 + n_points)
    patch = rng.integers(-1, n_points, n_cells).astype(np.int32)
    patch[: min(n_points, n_cells)] = np.arange(min(n_points, n_cells))
    counts = rng.integers(1, 500, (n_cath, n_cells))
    ref = n_points // 2
    if n_cells < n_points:
        ref = 0
    cal = np.stack([[5.0, 0.01 + 0.01 * j, 35.0, 0.05 + 0.02 * j, 8.0 + j, 58.0 + 10 * j] for j in range(n_cath)])
    power = 10.0 + rng.random(n_cath) * 20.0
    if special == "empty_reference":
        counts[n_cath - 1, patch == ref] = 0
    if special == "zero_rate":
        # dyadic, so that the rate is 0 exactly however the host fuses the line's evaluation
        cal[0, :4], power[0] = (12.0, -0.25, 28.0, 0.25), 20.0
    g = rng.standard_normal((n_points, n_cath))
    dev = {k: torch.as_tensor(v, device="cuda") for k, v in (("c", counts), ("p", patch), ("g", g))}
    out = {k: torch.full(s, 7.0, dtype=torch.float64, device="cuda") for k, s in
           (("N", (n_cath, n_points)), ("comp", (n_points, n_cath)), ("gN", (n_cath, n_points)),
            ("gc", (n_cath, n_cells)), ("gP", (n_cath,)))}
    lib, st = N.load(), C.c_void_p(torch.cuda.current_stream().cuda_stream)
    hp = [x.ctypes.data_as(C.c_void_p) for x in (cal, power)]
    N.check(lib.sput_composition(n_cath, n_cells, n_points, _p(dev["c"]), _p(dev["p"]), ref, *hp, _p(out["N"]),
                                 _p(out["comp"]), st), "composition")
    N.check(lib.sput_composition_backward(n_cath, n_cells, n_points, _p(out["N"]), _p(dev["p"]), ref, *hp, _p(dev["g"]),
                                          _p(out["gN"]), _p(out["gc"]), _p(out["gP"]), st), "backward")
    got = {k: v.cpu().numpy() for k, v in out.items()}

    inside = patch >= 0
    Nj = np.stack([np.bincount(patch[inside], weights=c[inside], minlength=n_points) for c in counts])
    slope = (cal[:, 3] - cal[:, 1]) / (cal[:, 2] - cal[:, 0])
    R = cal[:, 1] + slope * (power - cal[:, 0])
    w = cal[:, 4] / cal[:, 5]
    nref = Nj[:, ref]
    on = nref > 0
    W = np.where(on, R * w / np.where(on, nref, 1.0), 0.0)
    a = W[:, None] * Nj
    A = a.sum(axis=0)
    ok = A > 0
    As = np.where(ok, A, 1.0)
    comp = np.where(ok, 100.0 * a / As, 0.0)
    ga = np.where(ok, 100.0 / As * (g.T - (g.T * comp).sum(axis=0) / 100.0), 0.0)
    gN = np.where(on[:, None], ga * W[:, None], 0.0)
    S = (ga * a).sum(axis=1)
    gN[:, ref] += np.where(on, -S / np.where(on, nref, 1.0), 0.0)
    gP = np.where(R != 0, S / np.where(R != 0, R, 1.0), 0.0) * slope
    gc = np.where(inside, gN[:, np.where(inside, patch, 0)], 0.0)
    assert np.array_equal(got["N"], Nj)
    scale = n_points * 1e-15
    for k, want in (("comp", comp.T), ("gN", gN), ("gc", gc), ("gP", gP)):
        tol = scale * (1.0 + np.abs(want).max() + (np.abs(ga * a).sum() if k != "comp" else 0.0) /
                       max(1e-300, np.abs(R[R != 0]).min(initial=np.inf) if k == "gP" else 1.0))
        assert np.abs(got[k] - want).max() <= tol, (k, np.abs(got[k] - want).max(), tol)


@pytest.mark.parametrize("nx,ny", [(1, 1), (7, 73), (64, 64), (4097, 1), (200, 201)])
def test_contractions(nx, ny):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N

    sc = workloads.scene_quaternary(n_per_cathode=10, nx=nx, ny=ny)
    tr = pkg.Transport(sc)
    n = nx * ny
    rng = np.random.default_rng(n)
    g, score = rng.standard_normal((4, n)), rng.standard_normal((4, n))
    c0, c1 = rng.integers(0, 1000, (4, n)), rng.integers(0, 1000, (4, n))
    d = [torch.as_tensor(x, device="cuda") for x in (g, score, c0, c1)]
    out = torch.full((4,), 7.0, dtype=torch.float64, device="cuda")
    lib, st = N.load(), C.c_void_p(torch.cuda.current_stream().cuda_stream)
    N.check(lib.sput_backward(tr.h, _p(d[0]), _p(d[1]), _p(out), st), "backward")
    tol = n * 1.2e-16 * (np.abs(g * score).sum(axis=1) + 1e-300)
    assert np.all(np.abs(out.cpu().numpy() - (g * score).sum(axis=1)) <= tol)
    first = out.clone()
    N.check(lib.sput_backward(tr.h, _p(d[0]), _p(d[1]), _p(out), st), "backward")
    assert torch.equal(first, out)  # the order of the sum does not depend on timing
    N.check(lib.sput_emax_backward(tr.h, _p(d[0]), _p(d[2]), _p(d[3]), _p(out), st), "emax")
    el = [c["element"] for c in sc.cathodes]
    Mg = sc.gas.mass
    want, tol = np.empty(4), np.empty(4)
    for j, e in enumerate(el):
        kL = 0.4 * 4 * Mg * e.mass / (Mg + e.mass) ** 2
        Em = kL * 400.0 - e.U_s
        f = kL * 2 * e.U_s / (Em * (Em + e.U_s))
        want[j] = f * (g[j] * (c1[j] - c0[j])).sum()
        # (the cut-off is rebuilt from FP32 scene values)
        tol[j] = 1e-5 * abs(want[j]) + n * 1.2e-16 * f * np.abs(g[j] * (c1[j] - c0[j])).sum()
    assert np.all(np.abs(out.cpu().numpy() - want) <= tol)
    tr.close()
