"""The pool through which the transport hands atoms to the drain, when it is not as one run alone leaves
it (overlapping runs of a scene, which are not allowed, clear each other's counters).  The
bounds-checked library prepares it: some slots taken and filled with bytes that make no atom of
the run, then so many left.  Slots that hold none of the run's atoms are left out and reported,
so every tally equals that of the run by itself; once the pool is full, the atoms that find no slot are
left out and reported, and every other one is tallied once."""

import ctypes as C

import pytest

import workloads

pytestmark = pytest.mark.gpu


def _run(sc, overlap=None, **opts):
    import torch

    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    lib = N.load(path=N.CHECKED_LIB_PATH)
    d, keep = api.scene_desc(sc)
    h = C.c_void_p()
    assert lib.sput_scene_create(C.byref(d), 0, C.byref(h)) == 0
    lay = N.sput_tally_layout()
    assert lib.sput_tally_layout_get(h, C.byref(lay)) == 0
    t = {"counts": torch.zeros((lay.n_instances, lay.ny, lay.nx), dtype=torch.int64 if lay.count_type else torch.int32,
                               device="cuda"),
         "prim_counts": torch.zeros((lay.n_instances, lay.max_prims), dtype=torch.int64, device="cuda"),
         "timed_out": torch.zeros((lay.n_instances,), dtype=torch.int64, device="cuda"),
         "records": torch.zeros((lay.n_tickets, 6), dtype=torch.int32, device="cuda")}
    tal, st = N.sput_tallies(), N.sput_run_stats()
    for k, v in t.items():
        setattr(tal, k, v.data_ptr())
    if overlap:
        lib.sput_checked_overlap(*overlap)
    lib.sput_run(h, C.byref(api.run_opts(seed=8, **opts)), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                 C.byref(tal), C.byref(st))
    live = lib.sput_checked_drain_live()
    lib.sput_scene_destroy(h)
    return t, st, live


SCENES = {"all": lambda: workloads.scene_single_ni(n=3000, pressure=0.5),
          "last": lambda: workloads.scene_single_ni(n=100_000, pressure=0.2),
          "masks": lambda: workloads.scene_quaternary(n_per_cathode=1500, pressure=1.0),
          "walk": lambda: workloads.scene_large_shielded(n=3000, pressure=1.0, nx=31, ny=17,
                                                         physics={"thermal_switch_eV": 0.1})}


@pytest.mark.parametrize("taken,byte", [(1, 255), (200, 127), (255, 1)])
@pytest.mark.parametrize("scene", SCENES)
def test_foreign_slots(scene, taken, byte):
    import torch

    sc = SCENES[scene]()
    want, st_a, live = _run(sc)
    assert st_a.device_status == 0 and live == (12 if scene == "last" else 32)
    got, st_b, _ = _run(sc, (taken, 100_000, byte))
    assert st_b.device_status == 4
    for k in want:
        assert torch.equal(want[k], got[k]), k
    for f in ("particles", "landed", "timed_out", "flights", "collisions", "attempts"):
        assert getattr(st_a, f) == getattr(st_b, f), f


@pytest.mark.parametrize("taken,room", [(0, 1), (0, 31), (0, 33), (255, 100)])
@pytest.mark.parametrize("scene", SCENES)
def test_full_pool(scene, taken, room):
    sc = SCENES[scene]()
    got, st, live = _run(sc, (taken, room, 255))
    assert st.device_status == 4
    n = sum(i["n"] for i in sc.instances)
    assert room <= st.particles < n and (scene == "last" or st.particles == room)
    assert int(got["prim_counts"].sum() + got["timed_out"].sum()) == st.particles
    # (a landed or timed-out atom leaves its energy in the record)
    assert int((got["records"][:, 2] != 0).sum()) == st.particles


def test_ticket_outside_the_range():
    """Slots of zeros: instance 0, particle 0, which another range of tickets does not hold."""
    import torch

    sc = SCENES["all"]()
    want, st_a, _ = _run(sc, ticket_begin=1000, ticket_end=2500)
    got, st_b, _ = _run(sc, (100, 10_000, 0), ticket_begin=1000, ticket_end=2500)
    assert (st_a.device_status, st_b.device_status) == (0, 4)
    for k in want:
        assert torch.equal(want[k], got[k]), k
