"""The largest scenes that a block's shared memory takes, where the room for the warps' queues runs
out: accepted at the limit, refused one primitive beyond it, and the run with as many warps as
fit gives the tallies of one with a single warp per block."""

import importlib.util
import os

import pytest

import workloads

pytestmark = pytest.mark.gpu


def _scene(n_prims, physics):
    here = os.path.dirname(os.path.abspath(__file__))
    spec = importlib.util.spec_from_file_location("limits", os.path.join(here, "test_gpu_limits.py"))
    limits = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(limits)
    return limits._with_wall_tiles(workloads.scene_large_shielded(n=2000, pressure=0.5, physics=physics), n_prims - 64,
                                   seed=3)


@pytest.mark.parametrize("n_prims,physics", [(2540, None), (2780, {"interaction": "hard_sphere"})])
def test_largest_scene(n_prims, physics):
    import torch

    import paper_2411_14413_gb300 as pkg
    from paper_2411_14413_gb300 import _native as N

    tr = pkg.Transport(_scene(n_prims, physics), energy=False)
    st = tr.run(seed=4, block_threads=256)
    want = {k: v.clone() for k, v in tr.t.items()}
    assert st.particles == 2000 and st.device_status == 0
    tr.run(seed=4, block_threads=32)
    for k, v in tr.t.items():
        assert torch.equal(want[k], v), k
    tr.close()
    with pytest.raises(N.SputError) as e:
        pkg.Transport(_scene(n_prims + 1, physics), energy=False)
    assert N.STATUS_NAMES[e.value.status] == "SPUT_ERR_UNSUPPORTED"


@pytest.mark.parametrize("flags", [1, 2])
def test_counters_of_many_instances(flags):
    """Counters in shared memory (2), in global memory (1), and where the default puts them."""
    import torch

    import paper_2411_14413_gb300 as pkg

    tr = pkg.Transport(workloads.scene_tilt_pressure_sweep(n_range=(300, 2000)))
    tr.run(seed=6)
    want = {k: v.clone() for k, v in tr.t.items()}
    tr.run(seed=6, flags=flags)
    for k, v in tr.t.items():
        assert torch.equal(want[k], v), k
    tr.close()
