"""Batches that do not fit one wave: events with very different segment spacing,
whose track constants must never meet another event's segments, searched wave
by wave while the autotuner runs and afterwards."""
import numpy as np
import pytest

import paper_2507_07816_gb300 as tcw
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
