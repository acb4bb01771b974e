"""A scene with more geometries than an index of 16 bits holds is refused like any other whose tables do
not fit a block's shared memory: its indices must not be used in packed form before that.  (Used
so, geometry 66000 of one gas pair reads the host's pair table behind its end.)"""

import copy

import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_refused():
    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N

    sc = copy.deepcopy(workloads.scene_large_shielded(n=100, pressure=0.5, nx=8, ny=8))
    sc.prims = sc.prims + sc.prims[-2:]  # 66 primitives: no cell masks to build
    sc.geometries = [dict(sc.geometries[0], prim_count=len(sc.prims)) for _ in range(70_000)]
    sc.instances[0]["geometry"] = 66_000
    with pytest.raises(N.SputError) as e:
        pkg.Transport(sc)
    assert N.STATUS_NAMES[e.value.status] == "SPUT_ERR_UNSUPPORTED"
