"""The surface test by cell masks for geometries without chamber walls, whose atoms leave the grid and
may come back: the same flights as the loop over every primitive, bit for bit, and no index
outside its table (bounds-checked library).  Sizes: one and two mask words and their edges;
vacuum (no end to a flight), a few flights per chamber, a fraction of a cell per flight.  A
primitive that sticks out of the chamber box leaves the loop in place."""

import copy
import ctypes as C

import pytest

import workloads

pytestmark = pytest.mark.gpu


def _scene(n_prims, pressure, n=20_000):
    sc = copy.deepcopy(workloads.scene_large_shielded(n=n, pressure=pressure, nx=31, ny=17,
                                                      physics={"max_collisions": 300}))
    sc.prims = sc.prims[1:n_prims + 1]
    sc.geometries[0]["substrate"] -= 1
    sc.cathodes[0]["target"] -= 1
    sc.geometries[0]["prim_count"] = len(sc.prims)
    assert sc.geometries[0]["prim_count"] == n_prims
    return sc


def _checked_run(sc, flags=0):
    """Status word of a run through the bounds-checked library, and its words per cell mask."""
    import torch

    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    lib = N.load(path=N.CHECKED_LIB_PATH)
    d, keep = api.scene_desc(sc)
    h = C.c_void_p()
    assert lib.sput_scene_create(C.byref(d), 0, C.byref(h)) == 0
    counts = torch.zeros((1, 17, 31), dtype=torch.int64, device="cuda")
    tal, st = N.sput_tallies(), N.sput_run_stats()
    tal.counts = counts.data_ptr()
    lib.sput_run(h, C.byref(api.run_opts(seed=5, flags=flags)), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                 C.byref(tal), C.byref(st))
    words = lib.sput_checked_mask_words()
    lib.sput_scene_destroy(h)
    return st.device_status, words


@pytest.mark.parametrize("pressure", [0.0, 0.3, 3.0])
@pytest.mark.parametrize("n_prims", [9, 16, 17, 32, 33, 63])
def test_masks_match_loop(n_prims, pressure):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N

    sc = _scene(n_prims, pressure)
    tr = pkg.Transport(sc, records=True)
    tr.run(seed=5, flags=N.SPUT_RUN_NO_CELL_MASKS, want_stats=False)
    want = {k: v.clone() for k, v in tr.t.items()}
    tr.run(seed=5, flags=N.SPUT_RUN_CELL_MASKS, want_stats=False)
    for k, v in tr.t.items():
        if v.dtype == torch.float64:
            assert torch.allclose(want[k], v, rtol=1e-12, atol=0), k
        else:
            assert torch.equal(want[k], v), k
    tr.close()
    # in vacuum the atoms that hit nothing end as non-finite (bit 0); no index is out of range (bit 1)
    status, words = _checked_run(sc, N.SPUT_RUN_CELL_MASKS)
    assert status & 2 == 0 and (pressure == 0.0 or status == 0)
    assert words == (1 if n_prims <= 32 else 2)


def test_default():
    """Many primitives and short flights take the masks by default, with or without walls."""
    assert _checked_run(_scene(63, 0.5)) == (0, 2)
    out = _scene(63, 0.5)
    last = out.prims[-1]
    out.box_hi = tuple(float(x) for x in out.box_hi[:2]) + (float(last["center"][2]),)
    assert _checked_run(out) == (0, 0)


@pytest.mark.parametrize("n_prims", [16, 32, 63])
def test_mask_reads_are_checked(n_prims):
    """The bounds-checked library reports a mask index behind the masks' end."""
    from paper_2411_14413_gb300 import _native as N

    lib = N.load(path=N.CHECKED_LIB_PATH)
    lib.sput_checked_mask_limit.argtypes = [C.c_longlong]
    sc = _scene(n_prims, 0.3, n=2000)
    try:
        lib.sput_checked_mask_limit(1000)
        assert _checked_run(sc, N.SPUT_RUN_CELL_MASKS)[0] == 2
    finally:
        lib.sput_checked_mask_limit(-1)
    assert _checked_run(sc, N.SPUT_RUN_CELL_MASKS)[0] == 0
