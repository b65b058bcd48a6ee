"""Batches that do not fit one wave: events with very different segment spacing,
whose track constants must never meet another event's segments, searched wave
by wave while the autotuner runs and afterwards."""
import numpy as np
import pytest
import torch

import paper_2507_07816_gb300 as tcw
import tcw_synth as syn
from test_gpu_batched import check_against_oracle, make_batch, run_batched

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_det,dtype", [(1, np.float32), (2, np.float16)])
def test_autotuned_in_several_waves(n_det, dtype):
    events, bank = make_batch(81 + n_det, n_det, dtype, False, [40, 300, 9, 520])
    for i, e in enumerate(events):
        # segments 4 s, 20 s, 60 s and 7 s apart, T0 a little into the data
        step = (4.0, 20.0, 60.0, 7.0)[i]
        e.t_mid = e.t_mid[0] + step * np.arange(len(e.t_mid))
        e.T0 = float(e.t_mid[0] + 5.5 * step)
    k = 6
    s, val, idx = run_batched(events, bank, k)
    assert s.batch_info()["waves"] == 1
    s.close()
    s, val2, idx2 = run_batched(events, bank, k, options=[(tcw.OPT_BATCH_MEMORY, 1 << 20)])
    info = s.batch_info()
    assert info["waves"] >= 2 and info["autotuned"] == 1
    check_against_oracle(events, bank, val2, idx2, k)
    np.testing.assert_allclose(val2, val, rtol=0, atol=1e-4)
    s.close()


def long_events(seed, sizes, n_seg):
    events, bank = make_batch(seed, 1, np.float16, False, sizes, n_tmpl=60, n_bin=400)
    r = np.random.default_rng(seed)
    for e in events:
        d = syn.random_detectors(r, 1)[0]
        e.t_mid = e.t_mid[0] + 4.0 * np.arange(n_seg)
        e.velocity = d.velocity(e.t_mid)[None]
        e.rho = r.standard_exponential((1, n_seg, 400), dtype=np.float32).astype(np.float16)
        e.T0 = float(e.t_mid[0] - 2.0)
    return events, bank


def loaded(events, bank, options=()):
    s = tcw.Search(0)
    s.set_option(tcw.OPT_AUTOTUNE, 0)
    for o, v in options:
        s.set_option(o, v)
    s.define_bank(bank.f0, bank.tau, bank.n, 0.0)
    s.load_events(events, events[0].f_min, events[0].df)
    return s


def test_rows_count_towards_the_wave_budget():
    """Events of 112 MB of Doppler rows each and little else, 260 MB per wave."""
    events, bank = long_events(91, [1000] * 6, 4000)
    s = loaded(events, bank)
    val, idx = s.search_batched(4)
    assert s.batch_info()["waves"] == 1
    s.close()
    s = loaded(events, bank, [(tcw.OPT_BATCH_MEMORY, 260_000_000)])
    free = torch.cuda.mem_get_info()[0]
    val2, idx2 = s.search_batched(4)
    used = free - torch.cuda.mem_get_info()[0]
    assert s.batch_info()["waves"] == 3
    s.close()
    np.testing.assert_array_equal(val, val2)
    np.testing.assert_array_equal(idx, idx2)
    assert used < 260e6 + 300e6   # and the scratch of one context


def test_rows_that_do_not_fit_leave_the_group_kernel():
    """Device memory for the group kernel's buffers but not for 1.8 GB of rows."""
    events, bank = long_events(92, [2000] * 4, 8000)
    s = loaded(events, bank)
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 900_000_000, dtype=torch.uint8, device="cuda:0")
    try:
        val, idx = s.search_batched(4)
    finally:
        del hog
        torch.cuda.empty_cache()
    s.close()
    s = loaded(events, bank)
    val2, idx2 = s.search_batched(4)
    s.close()
    np.testing.assert_allclose(val, val2, rtol=0, atol=1e-3)
