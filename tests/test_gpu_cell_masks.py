"""The surface test by cell masks against the loop over every primitive, where the masks can go
wrong: geometries at the edges of the mask words (9, 32, 33, 63, 64 primitives), chamber walls
that are not the first primitive, flights across the whole chamber (vacuum) and of a fraction of
a cell (3 Pa), a chamber whose sides are no multiple of the cells'.  Both tests find the nearest
hit of the same flights, so integer tallies and per-particle records agree bit for bit."""

import copy

import pytest

import workloads

pytestmark = pytest.mark.gpu


def _scene(n_prims, pressure, box_last, chamber):
    n = {0.0: 60_000, 0.3: 60_000, 3.0: 4_000}[pressure]
    sc = copy.deepcopy(workloads.scene_large_shielded(n=n, pressure=pressure))
    sc.prims = sc.prims[:n_prims]
    if box_last:
        sc.prims = sc.prims[1:] + sc.prims[:1]
        sc.geometries[0]["substrate"] -= 1
        sc.cathodes[0]["target"] -= 1
    sc.geometries[0]["prim_count"] = n_prims
    if chamber is not None:
        sc.box_lo, sc.box_hi = chamber
    return sc


@pytest.mark.parametrize("box_last", [False, True])
@pytest.mark.parametrize("pressure", [0.0, 0.3, 3.0])
@pytest.mark.parametrize("n_prims,chamber", [(7, None), (9, None), (16, None), (17, None), (32, ((-211.0, -187.5, -100.0), (203.0, 199.0, 171.3))),
                                             (33, None), (63, ((-300.0, -150.0, -95.0), (155.0, 160.0, 640.0))),
                                             (64, None)])
def test_masks_match_loop(n_prims, chamber, pressure, box_last):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N

    tr = pkg.Transport(_scene(n_prims, pressure, box_last, chamber), records=True)
    st_a = tr.run(seed=5, flags=N.SPUT_RUN_NO_CELL_MASKS)
    want = {k: v.clone() for k, v in tr.t.items()}
    st_b = tr.run(seed=5, flags=N.SPUT_RUN_CELL_MASKS)
    for k, v in tr.t.items():
        if v.dtype == torch.float64:
            assert torch.allclose(want[k], v, rtol=1e-12, atol=0), k
        else:
            assert torch.equal(want[k], v), k
    assert (st_a.flights, st_a.collisions, st_a.attempts) == (st_b.flights, st_b.collisions, st_b.attempts)
    tr.close()
