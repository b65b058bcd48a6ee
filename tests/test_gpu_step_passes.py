"""The step-function search over observations that take several passes, whose sums
move from one sky order to the next in the difference cells of a template block:
every kind of value, blocks of 32 templates (up to 512 skies), of 16 (more) and of
4, against the FP64 oracle.  TCW_OPT_BANK_CHUNK = 4096 makes the bank one work
item, for which step_block keeps the largest block; with chunks of one block a
small bank takes blocks of 4."""
import numpy as np
import pytest

import oracle
import paper_2507_07816_gb300 as tcw
import tcw_synth as syn
from _parity import assert_topk_consistent
from test_gpu_step_limits import run, stepped

pytestmark = pytest.mark.gpu
TH = 1.6


def long_problem(seed, n_det, n_sky, n_tmpl, dtype, n_seg=840, t_step=60.0, n_bin=1000, bank=None):
    """14 h, T0 inside the data, templates past both band edges, weights 0.06-1.5."""
    r = syn.rng(seed)
    t = syn.segment_times(n_seg, t_step)
    dets = syn.random_detectors(r, n_det)
    vel = np.stack([d.velocity(t) for d in dets])
    rho = syn.exponential_noise(r, (n_det, n_seg, n_bin)).astype(dtype)
    w = syn.uniform_weights(r, n_det, n_seg)
    w[:, n_seg // 3] = 0.06
    if bank is None:
        bank = syn.random_bank(r, n_tmpl, f0_range=(495.0, 500.0 + 0.25 * n_bin + 5), tau_range=(3500, 35000))
    return syn.Problem(rho, t, w, vel, 500.0, 0.25, float(t[0] + 0.05 * n_seg * t_step), syn.random_sky(r, n_sky), bank,
                       [], dets, name="passes")


KINDS = {"f32": (np.float32, 0, 1, None), "f16": (np.float16, 0, 1, None), "f32 amp": (np.float32, 4, 1, None),
         "f16 amp": (np.float16, 4, 1, None), "two bins": (np.float32, 0, 2, None), "two bins f16 amp": (np.float16, 3, 2, None),
         "count": (np.float32, 0, 1, TH), "count two bins amp": (np.float16, 2, 2, TH)}


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("n_sky,n_det,chunk", [(300, 1, 4096), (512, 2, 4096), (513, 2, 4096), (900, 1, 4096),
                                               (1100, 2, 4096), (700, 2, 1)])
def test_passes(kind, n_sky, n_det, chunk):
    dtype, amp, bins, th = KINDS[kind]
    p = long_problem(3000 + n_sky, n_det, n_sky, 70, dtype)
    val, idx, st, info = run(p, options=[(tcw.OPT_BANK_CHUNK, chunk), (tcw.OPT_AMPLITUDE_POWER, amp),
                                         (tcw.OPT_TRACK_BINS, bins)],
                             statistic=None if th is None else (tcw.STAT_NUMBER_COUNT, th))
    S, W1, W2, psi = oracle.search_stats(np.asarray(p.rho, np.float64), p.f_min, p.df, p.t_mid, p.weights, p.velocity,
                                         p.nhat, p.bank.f0, p.bank.tau, p.bank.n, p.T0, amp_power=amp, track_bins=bins,
                                         rho_th=th)
    assert info.kernel == tcw.KERNEL_GROUP
    # templates of a few lookups keep the grid's rounding beside their small sums
    many = W1 > 0.05 * W1.max()
    assert stepped({"S": st["S"][many]}, [S[many]])
    for k, ref in (("S", S), ("W1", W1), ("W2", W2)):
        assert np.all(np.abs(st[k] - ref) <= 1e-5 * ref + 1e-6), k
    fin = np.isfinite(psi)
    assert np.array_equal(fin, np.isfinite(st["psi"]))
    assert np.all(np.abs(st["psi"][many] - psi[many]) <= 2.0 ** -23 * np.abs(psi[many]) + 2.0 ** -21)
    assert np.all(np.abs(st["psi"][fin] - psi[fin]) <= 1e-5 * (np.abs(psi) + np.sqrt(W1) + 1)[fin])
    assert_topk_consistent(st["psi"], idx, val, 3)


@pytest.mark.parametrize("n_det,dtype,th", [(1, np.float16, None), (2, np.float32, None), (2, np.float32, TH)])
def test_batched_events_of_several_passes(n_det, dtype, th):
    """Events with blocks of 32 and of 16 templates, of several passes and of one."""
    first = long_problem(3100 + n_det, n_det, 400, 60, dtype)
    events = [first] + [long_problem(3110 + n_det + i, n_det, n_sky, 0, dtype, n_seg=n_seg, bank=first.bank)
                        for i, (n_sky, n_seg) in enumerate([(900, 700), (1030, 400), (40, 60)])]
    s = tcw.Search(0)
    s.set_option(tcw.OPT_AUTOTUNE, 0)
    if th is not None:
        s.set_statistic(tcw.STAT_NUMBER_COUNT, th)
    b = first.bank
    s.define_bank(b.f0, b.tau, b.n, 0.0)
    s.load_events(events, first.f_min, first.df)
    val, idx = s.search_batched(5)
    s.close()
    row = 0
    for e in events:
        psi = oracle.search_stats(np.asarray(e.rho, np.float64), e.f_min, e.df, e.t_mid, e.weights, e.velocity, e.nhat,
                                  b.f0, b.tau, b.n, e.T0, rho_th=th)[3]
        n = len(e.nhat)
        v, i = val[row:row + n], idx[row:row + n]
        ref = np.take_along_axis(psi, i, 1)
        fin = np.isfinite(ref)
        assert np.array_equal(fin, np.isfinite(v))
        assert np.all(np.abs(v[fin] - ref[fin]) <= 2.0 ** -23 * np.abs(ref[fin]) + 2.0 ** -20)
        best = -np.sort(-psi, 1)[:, :5]
        assert np.all(np.abs(best[fin] - ref[fin]) <= 2.0 ** -22 * np.abs(best[fin]) + 2.0 ** -19)
        row += n


@pytest.mark.parametrize("n_det", [1, 2])
def test_thresholds_among_the_skies(n_det):
    """Velocities of one direction and skies nearly across it, so that their shifts span a
    few 1e-6 bins, and tracks of constant frequency at the bins' edges: nearly every
    lookup is within the fp32 thresholds' error, and the exact ones decide it."""
    r = syn.rng(3200 + n_det)
    n_seg, n_sky, n_tmpl = 70, 60, 64
    p = long_problem(3210, n_det, n_sky, n_tmpl, np.float32, n_seg=n_seg, t_step=4.0, n_bin=3000)
    p.velocity[:] = np.array([29000.0, 0.0, 0.0])
    a = r.uniform(-2e-5, 2e-5, n_sky)
    ph = r.uniform(0, 2 * np.pi, n_sky)
    q = np.sqrt(1 - a * a)
    p.nhat = np.ascontiguousarray(np.stack([a, q * np.cos(ph), q * np.sin(ph)], -1))
    p.bank.tau[:] = 1e18   # no drift over the segments
    p.bank.n[:] = 3.0
    edge = p.f_min + (np.arange(n_tmpl) * 40 + 100.5) * p.df
    p.bank.f0[:] = edge * (1 + 2e-9 * r.uniform(-1, 1, n_tmpl))
    p.T0 = float(p.t_mid[0] - 2.0)
    val, idx, st, info = run(p)
    S, W1, W2, psi = oracle.search_stats(p.rho, p.f_min, p.df, p.t_mid, p.weights, p.velocity, p.nhat, p.bank.f0,
                                         p.bank.tau, p.bank.n, p.T0)
    assert info.kernel == tcw.KERNEL_GROUP
    # skies on both sides of the edges
    assert (np.abs(S - S[:1]).max(0) > 1).mean() > 0.5
    # a track within 2^-30 bins of an edge may go either way
    D = p.nhat @ p.velocity[0, 0] / 299792458.0
    x = (p.bank.f0[None] * (1 + D[:, None]) - p.f_min) / p.df
    clear = np.abs(x - np.floor(x) - 0.5) > 2.0 ** -29
    assert clear.mean() > 0.9 and (np.abs(x - np.floor(x) - 0.5) < 5e-6).mean() > 0.5
    assert stepped({"S": st["S"][clear]}, [S[clear]])
