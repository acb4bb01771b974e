"""The autotuner times the transport kernel, whose launch shape it chooses, on samples of any size:
also on those that an ordinary run would hand to the drain at once."""

import ctypes as C

import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sample", [(1_000_000, 8_000), (1_000_000, 200_000), (3_000, 100_000)])
def test_small_samples_time_the_transport(n, sample):
    import torch

    from paper_2411_14413_gb300 import _native as N
    from paper_2411_14413_gb300 import api

    lib = N.load(path=N.CHECKED_LIB_PATH)
    d, keep = api.scene_desc(workloads.scene_single_ni(n=n, pressure=0.5))
    h = C.c_void_p()
    assert lib.sput_scene_create(C.byref(d), 0, C.byref(h)) == 0
    timed_out = torch.zeros((1,), dtype=torch.int64, device="cuda")
    tal, out = N.sput_tallies(), N.sput_tune_result()
    tal.timed_out = timed_out.data_ptr()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    o = api.run_opts(seed=1)
    assert lib.sput_autotune(h, C.byref(o), stream, C.byref(tal), sample, C.byref(out)) == 0
    assert lib.sput_checked_drain_live() == 12
    assert out.n_candidates > 1 and out.best_rate == max(out.cand_rate[:out.n_candidates]) > 0
    # an ordinary run of so many atoms goes to the drain at once, before and after tuning
    o.ticket_end = min(n, 3_000)
    assert lib.sput_run(h, C.byref(o), stream, C.byref(tal), None) == 0
    assert lib.sput_checked_drain_live() == 32
    torch.cuda.synchronize()
    lib.sput_scene_destroy(h)
