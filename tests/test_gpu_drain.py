"""The drain of a run's last atoms (several lanes per atom, a batch of flights at a time) against
the step of one atom per lane.  sput_run_noalloc transports without the drain and serves as the
reference; both follow each atom through the same numbers, so integer tallies, statistics and
per-particle records agree bit for bit.  Sizes: one atom, the edges of the lanes per atom and of
the pool; options: every kernel instance, few collisions (ends inside the first batch, at its
edges, just beyond), few partner attempts (below, at and above the four that are drawn ahead),
boundary launches, non-finite starts, a ticket range."""

import copy

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _both(sc, score_T=False, **opts):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    tr = pkg.Transport(sc, records=True, energy=True, score=True, score_T=score_T)
    stream = torch.cuda.current_stream().cuda_stream
    out = []
    for run in (api.sput_run_noalloc, api.sput_run):
        tr.t["records"].fill_(7)
        st = run(tr.h, api.run_opts(seed=23, **opts), stream, tr._tal, False) if opts.get("flags") else \
            run(tr.h, api.run_opts(seed=23, **opts), stream, tr._tal)
        torch.cuda.synchronize()
        out.append(({k: v.clone() for k, v in tr.t.items()}, st))
    tr.close()
    (a, sa), (b, sb) = out
    for k in a:
        if a[k].dtype == torch.float64:
            assert torch.allclose(a[k], b[k], rtol=1e-12, atol=1e-12 * float(a[k].abs().max() + 1e-300)), k
        else:
            assert torch.equal(a[k], b[k]), k
    if sa is not None:
        for f in ("particles", "landed", "timed_out", "flights", "collisions", "attempts"):
            assert getattr(sa, f) == getattr(sb, f), f
    return b, sb


@pytest.mark.parametrize("n", [1, 2, 7, 33, 1000, 20_000])
def test_small_runs(n):
    got, st = _both(workloads.scene_single_ni(n=n, pressure=0.7))
    assert st.particles == n


@pytest.mark.parametrize("off", [0, 1])
def test_pool_edge(off):
    import torch

    n = torch.cuda.get_device_properties(0).multi_processor_count * 1024 + off
    got, st = _both(workloads.scene_single_ni(n=n, pressure=0.5))
    assert st.particles == n


@pytest.mark.parametrize("mode", ["plain", "score_T", "walk"])
@pytest.mark.parametrize("name", ["single_ni", "quaternary", "large"])
def test_instances(name, mode):
    kw = {"n_per_cathode": 1500} if name == "quaternary" else {"n": 3000}
    if mode == "walk":
        kw["physics"] = {"thermal_switch_eV": 0.1}
    _both(workloads.scene_by_name(name, pressure=2.0, **kw), score_T=mode == "score_T")


@pytest.mark.parametrize("max_collisions", [0, 1, 7, 8, 9, 31, 32, 33])
def test_few_collisions(max_collisions):
    for n in (50, 20_000):
        got, st = _both(workloads.scene_single_ni(n=n, pressure=2.0, physics={"max_collisions": max_collisions}))
        assert st.timed_out > 0


@pytest.mark.parametrize("max_attempts", [1, 3, 4, 5, 9, 64])
def test_few_attempts(max_attempts):
    _both(workloads.scene_quaternary(n_per_cathode=4000, pressure=1.0, physics={"max_attempts": max_attempts}))


@pytest.mark.parametrize("physics", [{"interaction": "hard_sphere"}, {"gas_motion": "stationary"},
                                     {"interaction": "hard_sphere", "gas_motion": "stationary"}])
def test_other_physics(physics):
    _both(workloads.scene_single_ni(n=5000, physics=dict(physics, max_collisions=150)))


def test_flags_and_range():
    from paper_2411_14413_gb300 import _native as N

    sc = workloads.scene_quaternary(n_per_cathode=3000)
    _both(sc, flags=N.SPUT_RUN_LAUNCH_AT_CUTOFF)
    _both(sc, flags=N.SPUT_RUN_INJECT_NONFINITE)
    _both(sc, flags=N.SPUT_RUN_NO_CELL_MASKS)
    _both(sc, ticket_begin=2900, ticket_end=6100)
    table = copy.deepcopy(workloads.scene_single_ni_table(n=3000, pressure=1.0))
    got, _ = _both(table)
    assert int(np.asarray(got["timed_out"].sum().cpu())) == 0


@pytest.mark.parametrize("n", [1, 5, 33, 5491])
@pytest.mark.parametrize("physics", [{}, {"gas_motion": "stationary", "max_collisions": 100}])
def test_idle_groups_stay_in_bounds(n, physics):
    """Groups without an atom go through a warp's collisions too.  The bounds-checked library must
    report no index outside its table for them, whatever the shared memory held before: here what
    a transport with large tables left in it."""
    import ctypes as C

    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    lib = N.load(path=N.CHECKED_LIB_PATH)
    dirty = pkg.Transport(workloads.scene_tilt_pressure_sweep(n_range=(300, 1000)))
    sc = workloads.scene_large_shielded(n=n, pressure=0.8, nx=31, ny=17, physics=physics)
    d, keep = api.scene_desc(sc)
    h = C.c_void_p()
    assert lib.sput_scene_create(C.byref(d), 0, C.byref(h)) == 0
    counts = torch.zeros((1, 17, 31), dtype=torch.int64, device="cuda")
    tal = N.sput_tallies()
    tal.counts = counts.data_ptr()
    for seed in range(3):
        dirty.run(seed=seed, want_stats=False, flags=N.SPUT_RUN_SMEM_COUNTERS)
        st = N.sput_run_stats()
        rc = lib.sput_run(h, C.byref(api.run_opts(seed=seed)), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                          C.byref(tal), C.byref(st))
        assert rc == 0 and st.device_status == 0 and st.particles == n
    lib.sput_scene_destroy(h)
    dirty.close()
