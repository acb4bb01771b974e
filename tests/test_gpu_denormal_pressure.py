"""Pressures so low that the inverse mean free path is a denormal number: every atom flies as in vacuum,
also the few (one in 2^24) whose free path is drawn as zero times that."""

import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pressure", [1e-36, 1e-37, 1e-39, 1e-42])
def test_as_in_vacuum(pressure):
    import torch

    import paper_2411_14413_gb300 as pkg

    n = 200_000_000  # 12 such draws expected
    out = []
    for p in (0.0, pressure):
        tr = pkg.Transport(workloads.scene_single_ni(n=n, pressure=p))
        st = tr.run(seed=1)
        assert st.device_status == 0 and st.landed == n and st.collisions == 0
        out.append({k: v.clone() for k, v in tr.t.items()})
        tr.close()
    for k in ("counts", "prim_counts", "timed_out"):
        assert torch.equal(out[0][k], out[1][k]), k
