"""The step-function search (tcw_step.cu) against the FP64 oracle where its
geometry can go wrong: sky lists around a block of 8, around the 511 / 512
skies where a block of templates shrinks from 32 to 16, and around the
1024-sky chunk; single and ragged segment counts; an observation long enough
for several passes with their own sky order; more segments than one carry of
the low words; maps whose powers are too large for fixed-point sums; and maps
with infinities, whose search must equal the kernel that sums in fp32."""
import numpy as np
import pytest

import oracle
import paper_2507_07816_gb300 as tcw
import tcw_synth as syn
from _parity import assert_stats_close, assert_topk_consistent, oracle_stats

pytestmark = pytest.mark.gpu


def problem(seed, n_det, n_seg, n_sky, n_tmpl, t_step=4.0, n_bin=3000, dtype=np.float32, weights=True, t0=0.0):
    """Random bank over the whole band and past both edges; segments t_step apart."""
    r = syn.rng(seed)
    df, f_min = 0.25, 500.0
    t = syn.segment_times(n_seg, t_step)
    T0 = float(t[0] - 2.0 + t0 * n_seg * t_step)
    dets = syn.random_detectors(r, n_det)
    vel = np.stack([d.velocity(t) for d in dets])
    rho = syn.exponential_noise(r, (n_det, n_seg, n_bin)).astype(dtype)
    w = syn.uniform_weights(r, n_det, n_seg) if weights else None
    f_max = f_min + n_bin * df
    bank = syn.random_bank(r, n_tmpl, f0_range=(f_min - 5, f_max + 5), tau_range=(3500, 35000))
    return syn.Problem(rho, t, w, vel, f_min, df, T0, syn.random_sky(r, n_sky), bank, [], dets, name="step")


def search(p, k=3, options=()):
    s = tcw.Search(0)
    s.set_option(tcw.OPT_KEEP_STATS, 1)
    for o, v in options:
        s.set_option(o, v)
    s.load_problem(p)
    val, idx = s.search(k)
    st = s.statistics()
    info = s.info()
    s.close()
    return val, idx, st, info


def check(p, k=3, options=(), amp_power=0):
    val, idx, st, info = search(p, k, options)
    assert info.kernel == tcw.KERNEL_GROUP
    rho = np.asarray(p.rho, np.float64) if p.rho.dtype == np.float16 else None
    assert_stats_close((st["S"], st["W1"], st["W2"], st["psi"]), oracle_stats(p, rho=rho, amp_power=amp_power), p.name)
    assert_topk_consistent(st["psi"], idx, val, k)
    return st


@pytest.mark.parametrize("n_sky", [1, 7, 8, 9, 504, 505, 511, 513, 1024, 1025])
def test_sky_counts(n_sky):
    check(problem(200 + n_sky, 2, 70, n_sky, 70))


@pytest.mark.parametrize("n_seg,n_det", [(1, 1), (5, 2), (8, 1), (33, 2), (129, 1), (2100, 2)])
def test_segment_counts(n_seg, n_det):
    check(problem(300 + n_seg, n_det, n_seg, 20, 33, n_bin=1500))


@pytest.mark.parametrize("n_det,dtype,amp", [(1, np.float32, 0), (2, np.float32, 0), (2, np.float16, 4)])
def test_long_observations_take_several_passes(n_det, dtype, amp):
    # 14 h: the sky order changes along the way; T0 inside the data
    p = problem(400 + n_det, n_det, 840, 900, 40, t_step=60.0, n_bin=1000, dtype=dtype, t0=0.1)
    check(p, options=[(tcw.OPT_AMPLITUDE_POWER, amp)], amp_power=amp)


def test_tile_lengths_agree():
    p = problem(500, 2, 300, 600, 50)
    a = check(p)
    for tile in (8, 128):
        b = check(p, options=[(tcw.OPT_TILE_SEGMENTS, tile)])
        np.testing.assert_allclose(b["psi"], a["psi"], rtol=0, atol=1e-5)


@pytest.mark.parametrize("scale", [1e-12, 1e9])
def test_powers_of_any_scale(scale):
    """Weights and powers far from 1: the fixed-point unit follows them, or the
    search sums in fp32."""
    p = problem(600, 1, 100, 30, 40)
    p.rho = (p.rho * np.float32(scale)).astype(np.float32) if scale > 1 else p.rho
    if scale < 1:
        p.weights = (p.weights * np.float32(scale)).astype(np.float32)
    val, idx, st, info = search(p)
    oS, oW1, oW2, oP = oracle_stats(p)
    ok = oW2 > 0
    assert np.all(np.abs(st["S"] - oS) <= 1e-5 * oS)
    assert np.all(np.abs(st["W1"] - oW1) <= 1e-5 * oW1) and np.all(np.abs(st["W2"] - oW2) <= 1e-5 * oW2)
    assert np.all(np.abs(st["psi"][ok] - oP[ok]) <= 1e-5 * (oS[ok] / np.sqrt(oW2[ok])) + 1e-5)


def test_infinite_powers_stay_with_their_lookups():
    p = problem(700, 1, 60, 40, 60)
    p.rho[0, 20, ::97] = np.inf
    val, idx, st, info = search(p)
    S = oracle_stats(p)[0]
    fin = np.isfinite(S)
    assert 0 < fin.sum() < S.size
    # lookups that never touch an infinite bin are finite and right
    sel = fin & np.isfinite(st["S"])
    assert sel.sum() > 0.9 * fin.sum()
    assert np.all(np.abs(st["S"][sel] - S[sel]) <= 1e-5 * S[sel] + 1e-6)
    assert not np.isfinite(st["S"][~fin]).any()


def test_skies_at_a_bin_boundary_take_the_exact_thresholds():
    """Detectors at rest and a bank of constant frequencies on bin edges and a few
    ulp around them: every lookup lies within the error of the fp32 thresholds."""
    p = problem(800, 2, 70, 20, 64, weights=True)
    p.velocity[:] = 0.0
    p.bank.tau[:] = 1e12
    p.bank.n[:] = 3.0
    e = p.f_min + (np.arange(64) * 11 + 40.5) * p.df
    p.bank.f0[:] = e * (1.0 + (np.arange(64) % 9 - 4) * 1e-8)
    check(p)


def test_long_sfts_take_short_tiles():
    # 32 s segments at 500-1250 Hz: up to 2.4 bins of Doppler shift, five boundaries per lookup
    r = syn.rng(900)
    t = syn.segment_times(90, 32.0)
    dets = syn.random_detectors(r, 2)
    vel = np.stack([d.velocity(t) for d in dets])
    bank = syn.random_bank(r, 60, f0_range=(505.0, 745.0), tau_range=(3500, 35000))
    p = syn.Problem(syn.exponential_noise(r, (2, 90, 8000)), t, syn.uniform_weights(r, 2, 90), vel, 500.0, 1 / 32.0,
                    float(t[0] - 16.0), syn.random_sky(r, 300), bank, [], dets, name="32 s")
    check(p)


@pytest.mark.parametrize("cluster,width", [(3, 1e-12), (4, 1e-12), (5, 1e-7), (40, 1e-4)])
def test_crowded_skies(cluster, width):
    """Skies in clusters narrower than a bucket of thresholds (below and above the 3
    skies of a fast window), at distances from below to far above the thresholds'
    error."""
    p = problem(1100 + cluster, 2, 40, 120, 50)
    r = syn.rng(1200 + cluster)
    n = np.repeat(p.nhat[::cluster], cluster, axis=0)[:120] + width * r.normal(size=(120, 3))
    p.nhat = np.ascontiguousarray(n / np.linalg.norm(n, axis=1, keepdims=True))
    check(p)


@pytest.mark.parametrize("n_tmpl,n_seg,n_sky,n_det", [(300, 700, 12, 2), (300, 700, 1024, 1), (9000, 64, 20, 2),
                                                      (9000, 64, 600, 2)])
def test_block_sizes(n_tmpl, n_seg, n_sky, n_det):
    """Blocks of 4 templates for few templates over long data, of 32 and 16 for many."""
    check(problem(1300 + n_sky + n_tmpl, n_det, n_seg, n_sky, n_tmpl, n_bin=2000))
