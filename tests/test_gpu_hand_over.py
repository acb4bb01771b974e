"""Which atoms of a run go to the drain: none where trajectories are short, all of a small run where they
are long, a warp's last ones in between and of large runs.  The choice changes no result: across
its lines integer tallies, statistics and records equal those of a run without the drain."""

import ctypes as C

import pytest

import workloads

pytestmark = pytest.mark.gpu

NONE, LAST, ALL = 0, 12, 32


def _choice(sc, **opts):
    """Params::drain_live of a run, from the bounds-checked library, and its status word."""
    import torch

    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    lib = N.load(path=N.CHECKED_LIB_PATH)
    d, keep = api.scene_desc(sc)
    h = C.c_void_p()
    assert lib.sput_scene_create(C.byref(d), 0, C.byref(h)) == 0
    timed_out = torch.zeros((len(sc.instances),), dtype=torch.int64, device="cuda")
    tal, st = N.sput_tallies(), N.sput_run_stats()
    tal.timed_out = timed_out.data_ptr()
    rc = lib.sput_run(h, C.byref(api.run_opts(seed=5, **opts)), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                      C.byref(tal), C.byref(st))
    live = lib.sput_checked_drain_live()
    lib.sput_scene_destroy(h)
    assert rc == 0 and st.device_status == 0
    return live


@pytest.mark.parametrize("pressure,n,physics,want", [
    (0.0, 1, {}, NONE), (0.0, 100_000, {}, NONE), (0.0, 1_000_000, {}, NONE), (0.05, 100_000, {}, NONE),
    (0.05, 3_000, {}, ALL), (0.2, 20_000, {}, ALL), (0.2, 100_000, {}, LAST), (0.5, 3_000, {}, ALL),
    (0.5, 100_000, {}, ALL), (0.5, 1_000_000, {}, LAST), (1.0, 100_000, {"gas_motion": "stationary"}, NONE),
    (0.5, 100_000, {"interaction": "hard_sphere", "gas_motion": "stationary"}, LAST),
    (0.1, 100_000, {"thermal_switch_eV": 0.1}, NONE), (0.5, 100_000, {"thermal_switch_eV": 0.1}, LAST)])
def test_choice(pressure, n, physics, want):
    assert _choice(workloads.scene_single_ni(n=n, pressure=pressure, physics=dict(physics, max_collisions=50))) == want


def test_one_instance_with_long_trajectories():
    """One dense instance among empty chambers keeps the hand-over of the last atoms."""
    sc = workloads.scene_quaternary(n_per_cathode=50_000, pressure=0.0)
    assert _choice(sc) == NONE
    sc.instances[0]["pressure"] = 1.0
    assert _choice(sc) == LAST


@pytest.mark.parametrize("pressure", [0.0, 0.02, 0.1, 0.3])
@pytest.mark.parametrize("n", [1, 300, 30_000, 160_000])
def test_same_results(pressure, n):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import api

    tr = pkg.Transport(workloads.scene_single_ni(n=n, pressure=pressure), records=True)
    stream = torch.cuda.current_stream().cuda_stream
    st_a = api.sput_run_noalloc(tr.h, api.run_opts(seed=3), stream, tr._tal)
    want = {k: v.clone() for k, v in tr.t.items()}
    st_b = api.sput_run(tr.h, api.run_opts(seed=3), stream, tr._tal)
    for k, v in tr.t.items():
        if v.dtype == torch.float64:
            assert torch.allclose(want[k], v, rtol=1e-12, atol=1e-12), k
        else:
            assert torch.equal(want[k], v), k
    for f in ("particles", "landed", "timed_out", "flights", "collisions", "attempts"):
        assert getattr(st_a, f) == getattr(st_b, f), f
    tr.close()


@pytest.mark.parametrize("mode", ["plain", "score_T", "walk"])
@pytest.mark.parametrize("name", ["single_ni", "quaternary", "large"])
def test_atoms_on_their_way(name, mode):
    """More atoms than the pool holds: what a warp hands over has flights, scores and, with the
    diffusion shortcut, the walk behind it.  Seven primitives (the loop), 16 and 64 (masks of one and
    two words)."""
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import api

    n = torch.cuda.get_device_properties(0).multi_processor_count * 1024 + 1
    kw = {"n_per_cathode": n // 4 + 1} if name == "quaternary" else {"n": n}
    kw["physics"] = {"thermal_switch_eV": 0.1} if mode == "walk" else {}
    sc = workloads.scene_by_name(name, pressure=0.6, **kw)
    assert _choice(sc) == LAST
    tr = pkg.Transport(sc, records=True, energy=True, score=True, score_T=mode == "score_T")
    stream = torch.cuda.current_stream().cuda_stream
    st_a = api.sput_run_noalloc(tr.h, api.run_opts(seed=29), stream, tr._tal)
    want = {k: v.clone() for k, v in tr.t.items()}
    tr.t["records"].fill_(7)
    st_b = api.sput_run(tr.h, api.run_opts(seed=29), stream, tr._tal)
    for k, v in tr.t.items():
        if v.dtype == torch.float64:
            assert torch.allclose(want[k], v, rtol=1e-12, atol=1e-12 * float(want[k].abs().max() + 1e-300)), k
        else:
            assert torch.equal(want[k], v), k
    for f in ("particles", "landed", "timed_out", "flights", "collisions", "attempts"):
        assert getattr(st_a, f) == getattr(st_b, f), f
    tr.close()
