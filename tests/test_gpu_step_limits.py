"""Where the step-function search (tcw_step.cu) ends: inputs at its limits, and
beyond them the kernels that it hands over to."""
import numpy as np
import pytest
import torch

import oracle
import paper_2507_07816_gb300 as tcw
import tcw_synth as syn
from _parity import assert_stats_close, assert_topk_consistent, oracle_stats

pytestmark = pytest.mark.gpu


def run(p, k=3, options=(), statistic=None):
    """Search of p: values, indices, statistics, info."""
    s = tcw.Search(0)
    s.set_option(tcw.OPT_KEEP_STATS, 1)
    for o, v in options:
        s.set_option(o, v)
    if statistic:
        s.set_statistic(*statistic)
    s.load_problem(p)
    val, idx = s.search(k)
    st, info = s.statistics(), s.info()
    s.close()
    return val, idx, st, info


def stepped(st, ora):
    """Whether the step-function search ran: its S are exact sums rounded once (0.5
    ulp, and 0.02 for the fixed-point grid), those of the group kernel sums in fp32."""
    ulp = np.spacing(np.abs(ora[0]).astype(np.float32)).astype(np.float64)
    return bool(np.all(np.abs(st["S"].astype(np.float64) - ora[0]) <= 0.52 * ulp))


def check(p, k=3, options=(), amp_power=0):
    val, idx, st, info = run(p, k, options)
    rho = np.asarray(p.rho, np.float64) if p.rho.dtype == np.float16 else None
    ora = oracle_stats(p, rho=rho, amp_power=amp_power)
    assert info.kernel == tcw.KERNEL_GROUP
    assert_stats_close((st["S"], st["W1"], st["W2"], st["psi"]), ora, p.name)
    assert_topk_consistent(st["psi"], idx, val, k)
    return stepped(st, ora)


@pytest.mark.parametrize("n_bin,step", [(2 ** 23 - 1100, True), (2 ** 23 + 64, False)])
def test_wide_bands(n_bin, step):
    """Detectors nearly at rest over bands of 2^23 bins.  Up to there bins are placed
    in fp32; the templates are at the top of the band.  Beyond, another kernel runs
    (its bins are fp32 estimates too: templates at the band's bottom)."""
    r = syn.rng(2000)
    n_seg, df = 12, 0.25
    t = syn.segment_times(n_seg, 4.0)
    v = r.normal(size=(2, n_seg, 3))
    v *= 46.0 / np.linalg.norm(v, axis=-1, keepdims=True)
    f_min, f_max = 1000 * df, (1000 + n_bin) * df
    lo, hi = (0.97 * f_max, f_max + 5) if step else (f_min + 1e3, f_min + 2e4)
    bank = syn.random_bank(r, 60, f0_range=(lo, hi), tau_range=(3500, 35000))
    rho = np.tile(syn.exponential_noise(r, (1, 1, n_bin)), (2, n_seg, 1))
    p = syn.Problem(rho, t, syn.uniform_weights(r, 2, n_seg), v, f_min, df, float(t[0] - 2.0), syn.random_sky(r, 12),
                    bank, [], [], name="wide")
    assert check(p) == step


@pytest.mark.parametrize("statistic,bins,amp", [("power", 1, 0), ("power", 2, 0), ("power", 1, 4), ("power", 1, 7),
                                                ("count", 1, 0)])
def test_psi_is_rounded_once(statistic, bins, amp):
    """A few skies far apart (too wide a group for the group kernel): Psi is Eq. 4 of
    exact sums, rounded once to fp32 (2^-24 relative, 2^-25 for its pieces), as from
    sums in FP64.  The sums' grid is 2^-25 or finer here, 0.3 of it per value: 6 sigma
    of that are 2^-23 of sigma = sqrt(W2) when the weights' rms is at least 0.25.
    Amplitude weights are rounded twice to fp32 per lookup, independently: below 2^-24
    of a sum of 50 of them and of its squares' at 6 sigma, beside the sums' own 2^-24."""
    r = syn.rng(2100)
    n_seg = 1500
    t = syn.segment_times(n_seg, 4.0)
    dets = syn.random_detectors(r, 2)
    vel = np.stack([d.velocity(t) for d in dets])
    bank = syn.random_bank(r, 300, f0_range=(495.0, 1255.0), tau_range=(3500, 35000))
    rho = 2 * syn.exponential_noise(r, (2, n_seg, 3000))    # off the noise's mean: Psi up to 50
    p = syn.Problem(rho, t, syn.uniform_weights(r, 2, n_seg), vel, 500.0, 0.25, float(t[0] - 2.0),
                    syn.random_sky(r, 12), bank, [], dets, name="far apart")
    val, idx, st, info = run(p, options=[(tcw.OPT_TRACK_BINS, bins), (tcw.OPT_AMPLITUDE_POWER, amp)],
                             statistic=(tcw.STAT_NUMBER_COUNT, 1.6) if statistic == "count" else None)
    assert info.kernel == tcw.KERNEL_GROUP
    S, W1, W2, psi = oracle.search_stats(p.rho, p.f_min, p.df, p.t_mid, p.weights, p.velocity, p.nhat, bank.f0, bank.tau,
                                         bank.n, p.T0, amp_power=amp, track_bins=bins,
                                         rho_th=1.6 if statistic == "count" else None)
    assert_topk_consistent(st["psi"], idx, val, 3)
    ok = W2 >= 0.0625 * W1.max() / 16
    assert ok.mean() > 0.5 and np.abs(psi[ok]).max() > 20
    assert np.all(np.abs(st["W1"] - W1)[ok] <= 2.0 ** -23 * W1[ok])
    assert np.all(np.abs(st["W2"] - W2)[ok] <= 2.0 ** -23 * W2[ok])
    assert np.all(np.abs(st["psi"][ok] - psi[ok]) <= (2.0 ** -24 + 2.0 ** -25) * np.abs(psi[ok]) + 2.0 ** -23)


def test_two_bin_sums_are_not_rounded():
    """Bins of 1 + 2^-23 and 1 - 2^-24 in turn: every pair sums to 2 + 2^-24, which fp32
    rounds to 2.  Psi is n 2^-24 / sqrt(2 n), 2e-6 here, and 0 from rounded sums."""
    r = syn.rng(2200)
    n_seg = 1500
    t = syn.segment_times(n_seg, 4.0)
    dets = syn.random_detectors(r, 2)
    vel = np.stack([d.velocity(t) for d in dets])
    bank = syn.random_bank(r, 60, f0_range=(800.0, 1200.0), tau_range=(3500, 35000))
    row = np.where(np.arange(3000) % 2 == 0, 1 + 2.0 ** -23, 1 - 2.0 ** -24).astype(np.float32)
    p = syn.Problem(np.broadcast_to(row, (2, n_seg, 3000)).copy(), t, None, vel, 500.0, 0.25, float(t[0] - 2.0),
                    syn.random_sky(r, 12), bank, [], dets, name="pairs")
    for amp in (0, 2):
        _, _, st, info = run(p, options=[(tcw.OPT_TRACK_BINS, 2), (tcw.OPT_AMPLITUDE_POWER, amp)])
        assert info.kernel == tcw.KERNEL_GROUP
        psi = oracle.search_stats(p.rho, p.f_min, p.df, p.t_mid, p.weights, p.velocity, p.nhat, bank.f0, bank.tau, bank.n,
                                  p.T0, track_bins=2, amp_power=amp)[3]
        assert np.abs(psi).max() > 1.5e-6
        assert np.all(np.abs(st["psi"] - psi) <= 2.0 ** -23)


def small(seed, n_det=1, n_seg=300, n_sky=40, n_tmpl=60, n_bin=3000, weights=True):
    r = syn.rng(seed)
    t = syn.segment_times(n_seg, 4.0)
    dets = syn.random_detectors(r, n_det)
    vel = np.stack([d.velocity(t) for d in dets])
    f_max = 500.0 + n_bin * 0.25
    bank = syn.random_bank(r, n_tmpl, f0_range=(495.0, f_max + 5), tau_range=(3500, 35000))
    w = syn.uniform_weights(r, n_det, n_seg) if weights else None
    return syn.Problem(syn.exponential_noise(r, (n_det, n_seg, n_bin)), t, w, vel, 500.0, 0.25, float(t[0] - 2.0),
                       syn.random_sky(r, n_sky), bank, [], dets, name="small")


@pytest.mark.parametrize("scale", [1e-3, 1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("part", ["all", "band", "odd bins"])
def test_quiet_maps(scale, part):
    """Powers far below 1, everywhere, in the lower half of the band, or in all bins of a
    map whose rows begin with a bin of 1: S is as close as fp32 sums have it."""
    p = small(2300)
    if part == "all":
        p.rho *= np.float32(scale)
    elif part == "band":
        p.rho[:, :, :1500] *= np.float32(scale)
    else:
        p.rho *= np.float32(scale)
        p.rho[:, :, 0] = 1.0
    val, idx, st, info = run(p)
    S, W1, W2, psi = oracle_stats(p)
    assert info.kernel == tcw.KERNEL_GROUP
    assert np.all(np.abs(st["S"] - S) <= 1e-5 * S)
    fin = np.isfinite(psi)
    assert np.array_equal(fin, np.isfinite(st["psi"]))
    assert np.all(np.abs(st["psi"][fin] - psi[fin]) <= 1e-5 * (np.sqrt(W1) + 1)[fin])


@pytest.mark.parametrize("n_bin", [3000, 3001, 31])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
def test_lines_and_gaps_keep_the_fast_search(n_bin, dtype):
    """A loud line in one bin of every row, and rows and stretches of zeros: powers that
    the fixed-point grid spans."""
    p = small(2400 + n_bin, n_det=2, n_bin=n_bin)
    p.rho[:, 10:20] = 0.0
    p.rho[:, :, n_bin // 3:n_bin // 2] = 0.0
    p.rho[:, :, n_bin // 2 + 3] = 2000.0
    p.rho = p.rho.astype(dtype)
    if n_bin == 31:
        p.bank.f0[:] = 500 + 7 * np.linspace(0.5, 1.1, len(p.bank.f0))
    assert check(p)


@pytest.mark.parametrize("w_low", [1.3 * 2.0 ** -3, 1.3 * 2.0 ** -9, 1.3 * 2.0 ** -13, 1.3 * 2.0 ** -18])
@pytest.mark.parametrize("statistic", ["power", "count"])
def test_templates_of_small_weights(statistic, w_low):
    """Weights 1 in the first half and w_low in the second, the only one where the
    templates are in the band: W1, W2 and Psi from the small weights alone."""
    p = small(2500, n_det=2, n_seg=64, n_sky=20, n_tmpl=50, n_bin=1500)
    p.t_mid = p.t_mid[0] + 60.0 * np.arange(64)
    p.weights = np.ones((2, 64), np.float32)
    p.weights[:, 30:] = w_low
    f_top = p.f_min + 1500 * p.df
    # above the band's top, Doppler shifts included, at segment 30
    drop = (60.0 * 30 / p.bank.tau + 1) ** (1 / (1 - p.bank.n))
    p.bank.f0[:] = f_top / drop * np.linspace(1.0005, 1.004, 50)
    stat = (tcw.STAT_NUMBER_COUNT, 1.0) if statistic == "count" else None
    val, idx, st, info = run(p, statistic=stat)
    S, W1, W2, psi = oracle.search_stats(p.rho, p.f_min, p.df, p.t_mid, p.weights, p.velocity, p.nhat, p.bank.f0,
                                         p.bank.tau, p.bank.n, p.T0, rho_th=1.0 if stat else None)
    low = (W1 > 0) & (W1 < 68 * w_low * 1.001)
    assert info.kernel == tcw.KERNEL_GROUP and low.sum() > 100 and (W2[low] > 0).all()
    assert np.all(np.abs(st["W1"] - W1)[low] <= 1e-6 * W1[low])
    assert np.all(np.abs(st["W2"] - W2)[low] <= 1e-6 * W2[low])
    assert np.all(np.abs(st["S"] - S)[low] <= 1e-5 * S[low])
    assert np.all(np.abs(st["psi"] - psi)[low] <= 1e-5 * (S / np.sqrt(np.maximum(W2, 1e-30)))[low] + 1e-5)


@pytest.mark.parametrize("gated", ["weights", "gap"])
@pytest.mark.parametrize("n_det", [1, 2])
def test_amplitude_weights_after_a_gap(gated, n_det):
    """Tracks whose first lookups come late, when (f/f0)^8 is down to 1e-6: the segments
    before have weight 0, or are missing while the track comes into the band."""
    r = syn.rng(2600 + n_det)
    t = 1.4e9 + 10.0 * np.arange(1200)
    if gated == "gap":
        t[4:] += 9000.0   # between two tiles
    dets = syn.random_detectors(r, n_det)
    vel = np.stack([d.velocity(t) for d in dets])
    w = syn.uniform_weights(r, n_det, 1200)
    if gated == "weights":
        w[:, :1100] = 0.0
    f0 = {"weights": (600.0, 1090.0), "gap": (1150.0, 1800.0)}[gated]
    bank = syn.random_bank(r, 50, f0_range=f0, tau_range=(500.0, 520.0), n_range=(3.0, 3.1))
    p = syn.Problem(syn.exponential_noise(r, (n_det, 1200, 4000)), t, w, vel, 100.0, 0.25, float(t[0] - 5.0),
                    syn.random_sky(r, 20), bank, [], dets, name="late")
    val, idx, st, info = run(p, options=[(tcw.OPT_AMPLITUDE_POWER, 8)])
    S, W1, W2, psi = oracle_stats(p, amp_power=8)
    on = W1 > 0
    assert info.kernel == tcw.KERNEL_GROUP and on.sum() > 500 and W1[on].max() < 1.0
    for k, ref in (("S", S), ("W1", W1), ("W2", W2)):
        assert np.all(np.abs(st[k] - ref) <= 1e-5 * ref), k
    assert np.all(np.abs(st["psi"] - psi)[on] <= 1e-5 * (S / np.sqrt(np.where(on, W2, 1)))[on] + 1e-5)


def long_list(seed, n_sky, n_seg=8000, n_bin=1500):
    """Thousands of skies over 8 h of one detector, few templates."""
    r = syn.rng(seed)
    t = syn.segment_times(n_seg, 4.0)
    dets = syn.random_detectors(r, 1)
    vel = np.stack([d.velocity(t) for d in dets])
    f_max = 500.0 + n_bin * 0.25
    bank = syn.random_bank(r, 64, f0_range=(600.0, f_max + 5), tau_range=(10000, 35000))
    rho = syn.exponential_noise(r, (1, n_seg, n_bin)).astype(np.float16)
    return syn.Problem(rho, t, syn.uniform_weights(r, 1, n_seg), vel, 500.0, 0.25, float(t[0] - 2.0),
                       syn.random_sky(r, n_sky), bank, [], dets, name="long list")


def test_rows_of_long_sky_lists_are_held_in_parts():
    """40000 skies x 8000 segments: 9 GB of Doppler rows, held 4 GiB at a time.  The
    sums are exact, so any sky's results are those of a short list."""
    p = long_list(2700, 40000)
    s = tcw.Search(0)
    s.set_option(tcw.OPT_KEEP_STATS, 1)
    s.load_problem(p)
    free = torch.cuda.mem_get_info()[0]
    val, idx = s.search(3)
    used = free - torch.cuda.mem_get_info()[0]
    st = s.statistics()
    some = np.argsort(p.nhat @ p.velocity[0, 4000])[::997]   # over all the parts
    p.nhat = np.ascontiguousarray(p.nhat[some])
    s.load_problem(p)
    val1, idx1 = s.search(3)
    st1 = s.statistics()
    s.close()
    assert used < (4 << 30) + 600e6
    for k in st:
        np.testing.assert_array_equal(st[k][some], st1[k])
    np.testing.assert_array_equal(val[some], val1)
    np.testing.assert_array_equal(idx[some], idx1)


def test_tables_that_do_not_fit_leave_the_group_kernel():
    """Device memory left for the group kernel's tables (0.4 GB) but not for the step
    kernel's rows (2 GB): the search runs as with memory to spare."""
    p = long_list(2800, 9000)
    s = tcw.Search(0)
    s.set_option(tcw.OPT_KEEP_STATS, 1)
    s.load_problem(p)
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 1_200_000_000, dtype=torch.uint8, device="cuda:0")
    try:
        val, idx = s.search(3)
        st = s.statistics()
    finally:
        del hog
        torch.cuda.empty_cache()
    val1, idx1 = s.search(3)
    st1 = s.statistics()
    s.close()
    np.testing.assert_allclose(st["S"], st1["S"], rtol=1e-5)
    np.testing.assert_allclose(st["W1"], st1["W1"], rtol=1e-5)
    np.testing.assert_allclose(st["psi"], st1["psi"], rtol=0, atol=1e-3)
    assert_topk_consistent(st["psi"], idx, val, 3)


@pytest.mark.parametrize("scale", [1e-9, 1e-6, 1e-3, 1e3, 1e9])
@pytest.mark.parametrize("amp", [0, 4])
def test_weights_of_any_scale_keep_the_fast_search(scale, amp):
    """The grids follow the weights' scale, on which Psi does not depend."""
    p = small(2900, n_det=2)
    p.weights = (p.weights * np.float32(scale)).astype(np.float32)
    val, idx, st, info = run(p, options=[(tcw.OPT_AMPLITUDE_POWER, amp)])
    S, W1, W2, psi = oracle_stats(p, amp_power=amp)
    assert info.kernel == tcw.KERNEL_GROUP
    many = W1 > 0.1 * W1.max()
    assert stepped({"S": st["S"][many]}, [S[many]])
    assert np.all(np.abs(st["W2"] - W2)[many] <= 2.0 ** -23 * W2[many])
    assert np.all(np.abs(st["psi"][many] - psi[many]) <= 2.0 ** -23 * np.abs(psi[many]) + 2.0 ** -22)
    assert_topk_consistent(st["psi"], idx, val, 3)


@pytest.mark.parametrize("delay,power", [(2000.0, 4), (6000.0, 4), (20000.0, 3), (20000.0, 4)])
def test_amplitude_weights_long_after_the_start(delay, power):
    """Data that begin well after T0, when (f/f0)^p is down to 0.02: their grids resolve it."""
    p = small(2950 + power, n_det=2, n_tmpl=200)
    p.T0 = float(p.t_mid[0] - delay)
    p.bank.f0[:] = 500.0 + np.linspace(30, 745, 200)
    p.bank.f0[:] *= (delay / p.bank.tau + 1) ** (1 / (p.bank.n - 1))
    val, idx, st, info = run(p, options=[(tcw.OPT_AMPLITUDE_POWER, power)])
    S, W1, W2, psi = oracle_stats(p, amp_power=power)
    assert info.kernel == tcw.KERNEL_GROUP
    many = W1 > 0.02 * W1.max()
    assert many.mean() > 0.5 and stepped({"S": st["S"][many]}, [S[many]])
    assert np.all(np.abs(st["W1"] - W1)[many] <= 2.0 ** -23 * W1[many])
    assert np.all(np.abs(st["W2"] - W2)[many] <= 2.0 ** -23 * W2[many])
    assert np.all(np.abs(st["psi"][many] - psi[many]) <= 2.0 ** -23 * np.abs(psi[many]) + 2.0 ** -20)
    assert_topk_consistent(st["psi"], idx, val, 3)
