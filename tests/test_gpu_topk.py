"""Selection of the k best templates (tcw_topk.cu) around its 2048 sorted
candidates: rows that fit, rows narrowed by Psi, and rows whose k-th value is
shared by thousands of templates, which only the caller index tells apart."""
import numpy as np
import pytest

import paper_2507_07816_gb300 as tcw
import tcw_synth as syn
from _parity import assert_topk_consistent

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tmpl,in_band,k", [(1, 1, 1), (31, 31, 31), (2048, 2048, 1024), (2049, 2049, 1),
                                              (7000, 7000, 1024), (7000, 20, 50), (7000, 3000, 1024),
                                              (70000, 30, 1000)])
def test_k_best_in_order(n_tmpl, in_band, k):
    r = syn.rng(1000 + n_tmpl + in_band)
    t = syn.segment_times(12, 4.0)
    dets = syn.random_detectors(r, 1)
    vel = np.stack([d.velocity(t) for d in dets])
    bank = syn.random_bank(r, n_tmpl, f0_range=(520.0, 1100.0), tau_range=(3500, 35000))
    bank.f0[r.permutation(n_tmpl)[in_band:]] = 5000.0   # never in the band: Psi is -inf
    p = syn.Problem(syn.exponential_noise(r, (1, 12, 2600)), t, None, vel, 500.0, 0.25, float(t[0] - 2.0),
                    syn.random_sky(r, 3), bank, [], dets, name="topk")
    s = tcw.Search(0)
    s.set_option(tcw.OPT_KEEP_STATS, 1)
    s.load_problem(p)
    val, idx = s.search(k)
    psi = s.statistics()["psi"]
    s.close()
    assert np.isfinite(psi).sum() == 3 * in_band
    assert_topk_consistent(psi, idx, val, k)
