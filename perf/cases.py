"""Performance cases of the track-statistic search: what a user has it do.

Each case is one call (or one training pass) through the public entry points
of ``paper_2507_07816_gb300`` on synthetic data: whitened noise (Exp(1) power)
with a few injected tracks, circular-orbit detectors with their own rotation,
random or lattice template banks over the parameter ranges of the search, and
Fibonacci, random or clustered sky lists.  Sizes are those of the repository's
configurations, its benchmark and its density study, and the odd ones between
them.  Over many skies the loudest template of each direction is kept (a map of
the sky's maxima, as the noise threshold of a search takes it); a directed
search keeps its ten best.

``exact`` evaluates Eq. 1, Eq. 2, the nearest bin and Eq. 4 in plain FP64
torch.
"""
import math
import os

import numpy as np
import torch

import paper_2507_07816_gb300 as tcw

DEV = "cuda:0"
C_LIGHT = 299792458.0
ORBIT_V = 29784.7          # m/s
ORBIT_RATE = 2.0 * math.pi / (365.25 * 86400.0)
SIDEREAL = 7.2921159e-5
OBLIQUITY = math.radians(23.4393)
RHO_TH = 1.6               # number-count threshold
WEIGHTS_FILE = os.path.join(os.path.dirname(os.path.abspath(tcw.__file__)), "triage_weights.npz")
EXACT_LOOKUPS = 6.0e10     # exact() evaluates searches up to this many lookups


def _search(name, **kw):
    c = {"name": name, "kind": "search", "n_det": 2, "n_seg": 10000, "n_bin": 10000, "t_sft": 4.0, "f_min": 500.0,
         "dtype": "f32", "bank": "random", "n_tmpl": 20000, "sky": "fibonacci", "n_sky": 1024, "k": 1,
         "weights": False, "amp": 0, "statistic": "power", "bins": 1, "stats": False, "t0": 0.0}
    c.update(kw)
    return c


def listed():
    return [
        # one source of known position over a small 2.3 h map, every statistic kept: the smallest call
        _search("directed-small", n_det=1, n_seg=256, n_bin=4096, t_sft=32.0, bank="lattice", n_tmpl=5120, n_sky=1,
                sky="random", k=10, weights=True, stats=True),
        # the same directed search with the full bank and 11 h of data, one direction
        _search("directed-long", n_det=1, n_tmpl=200000, n_sky=1, sky="random", k=10, weights=True),
        # a dozen known targets spread over the sky, full statistics for the follow-up
        _search("targets", n_seg=2001, n_bin=8000, n_tmpl=301, n_sky=12, sky="random", k=3, stats=True,
                weights=True),
        # a region of the sky with ragged sizes everywhere and data that start before the source
        _search("region-ragged", n_seg=9973, n_bin=10007, n_tmpl=9001, n_sky=301, sky="region", k=1, weights=True,
                t0=0.03),
        # the all-sky search of two detectors over the full bank: the largest call
        _search("allsky", n_tmpl=200000, k=1),
        # Eq. 3's amplitude weighting over a triage-sized sky list
        _search("amplitude", n_tmpl=20011, n_sky=128, k=1, weights=True, amp=4),
        # the number-count statistic over the whole sky
        _search("count", n_tmpl=40000, k=1, statistic="count", weights=True),
        # fast tracks: two bins per lookup, one detector, an FP16 map, a random sky list
        _search("two-bin-f16", n_det=1, n_tmpl=30011, n_sky=777, sky="random", k=1, bins=2, dtype="f16"),
        # many events of uneven length in one call (FP16 maps, one detector, own sky lists)
        {"name": "batched", "kind": "batched", "n_events": 8, "n_det": 1, "seg_lo": 2000, "seg_hi": 9000,
         "n_bin": 10000, "t_sft": 4.0, "f_min": 500.0, "dtype": "f16", "n_tmpl": 12000, "sky_lo": 100, "sky_hi": 800,
         "k": 1, "triaged": False},
        # the learned triage of one event at its shipped operating point
        {"name": "triaged", "kind": "triaged", "n_det": 2, "n_seg": 10000, "n_bin": 10000, "t_sft": 4.0,
         "f_min": 500.0, "dtype": "f32", "n_tmpl": 200000, "n_sky": 1024, "k": 1},
        # the density study's search: 24 h of 8 s segments, a bank generated on the device
        {"name": "generated", "kind": "generated", "n_seg": 10800, "n_bin": 5280, "t_sft": 8.0, "f_min": 550.0,
         "bank": "random", "n_tmpl": 400000, "n_sky": 64, "k": 2},
        # one training pass of the triage network (forward, loss, backward)
        {"name": "train", "kind": "train", "batch": 4096},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["search", "batched", "triaged", "generated", "train"], [10, 2, 1, 1, 1])[0]
    if kind == "train":
        return {"kind": "train", "batch": _logint(rng, 32, 16384)}
    if kind == "batched":
        return {"kind": "batched", "n_events": rng.randint(2, 12), "n_det": rng.choice([1, 2]), "seg_lo": 1500,
                "seg_hi": _logint(rng, 3000, 9000), "n_bin": rng.randint(6000, 10000), "t_sft": 4.0, "f_min": 500.0,
                "dtype": rng.choice(["f16", "f32"]), "n_tmpl": _logint(rng, 2000, 12000), "sky_lo": 100,
                "sky_hi": _logint(rng, 120, 1300), "k": 1, "triaged": rng.random() < 0.3}
    if kind == "triaged":
        return {"kind": "triaged", "n_det": rng.choice([1, 2]), "n_seg": _logint(rng, 3000, 10000),
                "n_bin": rng.randint(8000, 10000), "t_sft": 4.0, "f_min": 500.0, "dtype": rng.choice(["f32", "f16"]),
                "n_tmpl": _logint(rng, 20000, 200000), "n_sky": rng.randint(256, 1024), "k": 1}
    if kind == "generated":
        return {"kind": "generated", "n_seg": rng.randint(3000, 10800), "n_bin": 5280, "t_sft": 8.0, "f_min": 550.0,
                "bank": rng.choice(["random", "lattice"]), "n_tmpl": _logint(rng, 30000, 400000),
                "n_sky": rng.randint(64, 256), "k": 1}
    for _ in range(1000):
        long_sft = rng.random() < 0.1
        count = rng.random() < 0.2
        n_sky = _logint(rng, 1, 1500)
        k = max(1, min(10, int(math.sqrt(100.0 / n_sky))))
        c = _search("", n_det=rng.choice([1, 2]), n_seg=256 if long_sft else _logint(rng, 500, 12000),
                    n_bin=4096 if long_sft else rng.randint(5000, 10000), t_sft=32.0 if long_sft else 4.0,
                    dtype=rng.choice(["f32", "f32", "f16"]), bank="lattice" if long_sft else "random",
                    n_tmpl=_logint(rng, 300, 200000), sky=rng.choice(["fibonacci", "random", "region"]), n_sky=n_sky,
                    k=k, weights=count or rng.random() < 0.5, amp=0 if count else rng.choice([0, 0, 0, 4]),
                    statistic="count" if count else "power", bins=rng.choice([1, 1, 1, 2]),
                    stats=n_sky <= 16 and rng.random() < 0.3, t0=rng.choice([0.0, 0.0, 0.05]))
        del c["name"]
        lookups = c["n_sky"] * c["n_tmpl"] * c["n_det"] * c["n_seg"]
        # a pass costs no more than the largest listed one; short lists of targets spread
        # over the sky are followed up with small banks
        if lookups > 3.5e12 or (1 < c["n_sky"] < 100 and c["sky"] != "region" and lookups > 6e6 * c["n_sky"]):
            continue
        if c["n_det"] * c["n_seg"] * c["n_bin"] > 2.1e8:
            continue
        return c
    raise RuntimeError("no case drawn")


# ------------------------------------------------------------------ inputs
def _velocities(r, n_det, t):
    """Detector velocities [n_det][n_seg][3]: a common orbit, each detector's own rotation."""
    orb = r.uniform(0.0, 2.0 * math.pi)
    out = np.empty((n_det, len(t), 3))
    ce, se = math.cos(OBLIQUITY), math.sin(OBLIQUITY)
    for d in range(n_det):
        a = ORBIT_RATE * t + orb
        b = SIDEREAL * t + r.uniform(0.0, 2.0 * math.pi)
        rot = 465.0 * math.cos(r.uniform(-1.0, 1.0))
        vx, vy = -ORBIT_V * np.sin(a), ORBIT_V * np.cos(a)
        out[d] = np.stack([vx - rot * np.sin(b), ce * vy + rot * np.cos(b), se * vy], -1)
    return out


def _sky(r, kind, n):
    if kind == "fibonacci":
        i = np.arange(n) + 0.5
        z, phi = 1.0 - 2.0 * i / n, i * math.pi * (3.0 - math.sqrt(5.0)) + r.uniform(0.0, 2.0 * math.pi)
        q = np.sqrt(1.0 - z * z)
        v = np.stack([q * np.cos(phi), q * np.sin(phi), z], -1)
    elif kind == "region":      # a patch a few degrees wide around one direction
        c = r.normal(size=3)
        v = c / np.linalg.norm(c) + 0.04 * r.normal(size=(n, 3))
    else:
        v = r.normal(size=(n, 3))
    return np.ascontiguousarray(v / np.linalg.norm(v, axis=1, keepdims=True))


def _bank(r, kind, n, f_lo, f_hi):
    if kind == "lattice":       # 5 braking indices, 16 spin-down times, f0 evenly spaced
        m = max(1, n // 80)
        nn, tt, ff = np.meshgrid(np.arange(3.0, 8.0), np.geomspace(3500.0, 35000.0, 16),
                                 np.linspace(f_lo + 60.0, f_hi - 4.0, m) + r.uniform(-0.01, 0.01, m), indexing="ij")
        return ff.ravel(), tt.ravel(), nn.ravel()
    return r.uniform(f_lo, f_hi, n), r.uniform(3500.0, 35000.0, n), r.uniform(3.0, 7.0, n)


def _event(c, seed, n_seg, n_sky, sky, t0_frac, weights, n_inj=3, snr=(8.0, 16.0)):
    """One event: (rho on the GPU, t_mid, weights, velocity, T0, nhat) with injected tracks."""
    r = np.random.default_rng([seed, 11])
    t = 1.4e9 + r.uniform(0.0, 3.0e7) + (np.arange(n_seg) + 0.5) * c["t_sft"]
    T0 = float(t[0] - 0.5 * c["t_sft"] + t0_frac * n_seg * c["t_sft"])
    D, n_bin, df = c.get("n_det", 1), c["n_bin"], 1.0 / c["t_sft"]
    vel = _velocities(r, D, t)
    nhat = _sky(r, sky, n_sky)
    w = r.uniform(0.5, 1.5, (D, n_seg)).astype(np.float32) if weights else None
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    rho = torch.empty((D, n_seg, n_bin), dtype=torch.float32, device=DEV).exponential_(generator=g)
    f_hi = c["f_min"] + n_bin * df
    on = t >= T0
    for _ in range(n_inj):
        f0, tau, n = r.uniform(0.5 * (c["f_min"] + f_hi), f_hi), r.uniform(7000.0, 35000.0), r.uniform(3.0, 7.0)
        s = nhat[int(r.integers(0, n_sky))]
        f = f0 * (np.where(on, t - T0, 0.0) / tau + 1.0) ** (1.0 / (1.0 - n))
        k = np.floor((f[None] * (1.0 + vel @ s / C_LIGHT) - c["f_min"]) / df + 0.5).astype(np.int64)
        dd, jj = np.nonzero((k >= 0) & (k < n_bin) & on[None])
        if not len(dd):
            continue
        lam = ((f / f0) ** 4)[jj]
        mu = np.sqrt(2.0 * r.uniform(*snr) * lam * math.sqrt(len(dd)) / lam.sum())
        p = ((r.normal(size=len(dd)) + mu) ** 2 + r.normal(size=len(dd)) ** 2) / 2.0
        ix = tuple(torch.as_tensor(a, device=DEV) for a in (dd, jj, k[dd, jj]))
        rho[ix] = torch.as_tensor(p, dtype=torch.float32, device=DEV)
    if c.get("dtype") == "f16":
        rho = rho.half()
    return rho, t, w, vel, T0, nhat


class _Event:
    def __init__(self, parts):
        self.rho, self.t_mid, self.weights, self.velocity, self.T0, self.nhat = parts


def _case_event(c, seed):
    r = np.random.default_rng([seed, 5])
    kind = c["kind"]
    f_hi = c["f_min"] + c["n_bin"] / c["t_sft"]
    if kind == "search":
        ev = _event(c, seed, c["n_seg"], c["n_sky"], c["sky"], c["t0"], c["weights"])
        return ev, _bank(r, c["bank"], c["n_tmpl"], c["f_min"], f_hi)
    if kind == "generated":
        return _event(c, seed, c["n_seg"], c["n_sky"], "random", 0.0, False), None
    return (_event(c, seed, c["n_seg"], c["n_sky"], "fibonacci", 0.0, False, n_inj=1),
            _bank(r, "random", c["n_tmpl"], c["f_min"], f_hi))


def _batch_events(c, seed):
    r = np.random.default_rng([seed, 3])
    sizes = np.random.default_rng([c["n_events"], c["seg_hi"], c["sky_hi"]])     # the case's, not the seed's
    evs = []
    for i in range(c["n_events"]):
        n_seg = int(sizes.integers(c["seg_lo"], c["seg_hi"] + 1))
        n_sky = int(sizes.integers(c["sky_lo"], c["sky_hi"] + 1))
        evs.append(_event(c, seed * 101 + i, n_seg, n_sky, "random", float(r.uniform(0.0, 0.1)), False, n_inj=1))
    return evs, _bank(r, "random", c["n_tmpl"], c["f_min"], c["f_min"] + c["n_bin"] / c["t_sft"])


def _gen_spec(c, seed):
    lo, hi = (1000.0, 3500.0, 3.0), (1200.0, 35000.0, 7.0)
    if c["bank"] == "lattice":
        m = max(1, c["n_tmpl"] // 200)
        return tcw.bank_spec(tcw.BANK_LATTICE, (lo[0] + (seed % 997) * 1e-3,) + lo[1:], hi, n_f0=m, n_tau=20, n_n=10)
    return tcw.bank_spec(tcw.BANK_RANDOM, lo, hi, n_tmpl=c["n_tmpl"], seed=seed)


def _train_inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    n = c["batch"]
    # log(1 + count) histograms: a bell over the bins, a few counts in the tail of positives
    x = torch.linspace(-4.0, 12.0, 128, device=DEV)
    counts = torch.poisson(2.0e4 * torch.exp(-0.5 * x * x).expand(n, 128).contiguous(), generator=g)
    y = (torch.rand(n, device=DEV, generator=g) < 0.1).float()
    counts[:, 80:] += y[:, None] * (torch.rand((n, 48), device=DEV, generator=g) < 0.05)
    theta = tcw.Mlp.initial(seed % 65536)
    return torch.log1p(counts).contiguous(), y, theta


# ------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        x, y, theta = _train_inputs(c, seed)
        return {"case": c, "mlp": tcw.Mlp(theta, device=DEV), "x": x, "y": y}
    s = tcw.Search(0)
    st = {"case": c, "search": s}
    if kind in ("triaged", "batched"):
        st["mlp"] = tcw.Mlp.load(WEIGHTS_FILE, device=DEV)
        s.set_option(tcw.OPT_TRIAGE_TEMPLATES, 12)
    if kind == "batched":
        evs, bank = _batch_events(c, seed)
        torch.cuda.synchronize()
        s.define_bank(*bank, 0.0)
        s.load_events([_Event(e) for e in evs], c["f_min"], 1.0 / c["t_sft"])
        return st
    (rho, t, w, vel, T0, nhat), bank = _case_event(c, seed)
    torch.cuda.synchronize()
    if kind == "search":
        s.set_option(tcw.OPT_AMPLITUDE_POWER, c["amp"])
        s.set_option(tcw.OPT_TRACK_BINS, c["bins"])
        s.set_option(tcw.OPT_KEEP_STATS, 1 if c["stats"] else 0)
        if c["statistic"] == "count":
            s.set_statistic(tcw.STAT_NUMBER_COUNT, RHO_TH)
    s.load_spectrogram(rho, c["f_min"], 1.0 / c["t_sft"], t, w)
    s.load_velocity(vel)
    if bank is not None:
        s.define_bank(*bank, T0)
    else:
        st["spec"], st["T0"] = _gen_spec(c, seed), T0
    s.define_sky(nhat)
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "train":
        m, x = state["mlp"], state["x"]
        h1, h2, y = m.forward(x)
        loss, dy = m.bce(y, state["y"], 9.0)
        return {"y": y, "loss": loss, "grad": m.backward(x, h1, h2, dy)}
    s = state["search"]
    if kind == "batched":
        if c["triaged"]:
            psi, idx, searched = s.search_batched_triaged(state["mlp"], 0, -4.0, 12.0, 0.35, c["k"])
            return {"psi": psi, "idx": idx, "searched": searched}
        psi, idx = s.search_batched(c["k"])
        return {"psi": psi, "idx": idx}
    if kind == "triaged":
        psi, idx, searched = s.search_triaged(state["mlp"], 32, -4.0, 12.0, 0.35, c["k"])
        return {"psi": psi, "idx": idx, "searched": searched}
    if kind == "generated":
        psi, idx = s.search_generated(state["spec"], state["T0"], c["k"])
        return {"psi": psi, "idx": idx}
    psi, idx = s.search(c["k"])
    out = {"psi": psi, "idx": idx}
    if c["stats"]:
        out["stats"] = s.statistics()
    return out


# ------------------------------------------------------------------ work
def _search_work(c, n_seg, n_sky, n_tmpl, out_cols):
    """The map is read once and the entries kept are written; every template's track is
    evaluated once per segment (Eq. 1, about 20 operations), every detector adds at least
    one weighted power per (template, segment), and every (sky, template) is finished once."""
    D = c.get("n_det", 1)
    esz = 2 if c.get("dtype") == "f16" else 4
    nbytes = D * n_seg * c["n_bin"] * esz + 24.0 * n_tmpl + 24.0 * n_sky + 24.0 * D * n_seg + 12.0 * n_sky * out_cols
    return nbytes, n_tmpl * n_seg * (20.0 + 4.0 * D) + 4.0 * n_sky * n_tmpl


def work(case):
    c, kind = case, case["kind"]
    if kind == "train":
        n = c["batch"]
        return {"bytes": 4.0 * n * (128 + 2) + 8.0 * 99073, "flops": 6.0 * n * (128 * 256 + 256 * 256 + 256)}
    if kind == "batched":
        seg, sky = (c["seg_lo"] + c["seg_hi"]) / 2, (c["sky_lo"] + c["sky_hi"]) / 2
        b, f = _search_work(c, seg, sky, c["n_tmpl"], c["k"])
        return {"bytes": b * c["n_events"], "flops": f * c["n_events"]}
    b, f = _search_work(c, c["n_seg"], c["n_sky"], c["n_tmpl"], c["k"])
    if c.get("stats"):
        b += 16.0 * c["n_sky"] * c["n_tmpl"]
    if kind == "triaged":       # a coarse Psi at every 32nd sky, then the chosen skies' templates
        f = c["n_tmpl"] * c["n_seg"] * (20.0 + 4.0 * c["n_det"]) + 4.0 * c["n_tmpl"] * (c["n_sky"] / 32)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact
def _exact_psi(c, ev, bank):
    """S, W1, W2, Psi [n_sky][n_tmpl] of Eq. 4 in FP64."""
    rho, t, w, vel, T0, nhat = ev
    f8 = dict(dtype=torch.float64, device=DEV)
    f0, tau, n = (torch.as_tensor(np.ascontiguousarray(a), **f8) for a in bank)
    ex = 1.0 / (1.0 - n)
    S, B = nhat.shape[0], f0.shape[0]
    D, n_seg, n_bin = rho.shape
    df, two = 1.0 / c["t_sft"], c.get("bins", 1) == 2
    count = c.get("statistic") == "count"
    dop = torch.as_tensor(np.einsum("djk,sk->djs", vel, nhat) / C_LIGHT, **f8)
    out = [torch.zeros((S, B), **f8) for _ in range(3)]
    step = max(1, int(4e7 // S))
    for b0 in range(0, B, step):
        sl = slice(b0, min(B, b0 + step))
        acc = [torch.zeros((S, f0[sl].shape[0]), **f8) for _ in range(3)]
        for j in range(n_seg):
            if t[j] < T0:
                continue
            u = ((t[j] - T0) / tau[sl] + 1.0) ** ex[sl]
            f, amp = f0[sl] * u, u ** c.get("amp", 0)
            for d in range(D):
                x = (f[None, :] * (1.0 + dop[d, j][:, None]) - c["f_min"]) / df
                k = torch.floor(x + (0.0 if two else 0.5))
                ok = (k >= 0) & (k + (1 if two else 0) < n_bin)
                k = torch.where(ok, k, torch.zeros_like(k)).long()
                row = rho[d, j].double()
                if count:
                    row = (row > RHO_TH).double()
                v = row[k]
                if two:
                    v = v + row[torch.clamp(k + 1, max=n_bin - 1)]
                wt = (1.0 if w is None else float(w[d, j])) * amp[None, :] * ok
                acc[0] += wt * v
                acc[1] += wt
                acc[2] += wt * wt
        for o, a in zip(out, acc):
            o[:, sl] = a
    q = math.exp(-RHO_TH) if count else 1.0
    nb = 2.0 if two else 1.0
    var = nb * (q * (1.0 - q) if count else 1.0) * out[2]
    psi = torch.where(var > 0, (out[0] - nb * q * out[1]) / torch.sqrt(torch.clamp(var, min=1e-300)),
                      torch.full_like(var, -math.inf))
    return out + [psi]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        x, lab, theta = _train_inputs(c, seed)
        th = torch.as_tensor(theta, device=DEV)
        sizes = [(128, 256), (256,), (256, 256), (256,), (256, 1), (1,)]
        p, o = [], 0
        for s in sizes:
            m = int(np.prod(s))
            v = th[o:o + m].reshape(s)
            # the forward and backward passes read bfloat16 weights
            p.append((v.bfloat16() if len(s) == 2 else v).double().requires_grad_())
            o += m
        h = torch.relu(x.double() @ p[0] + p[1])
        h = torch.relu(h @ p[2] + p[3])
        y = (h @ p[4] + p[5])[:, 0]
        loss = torch.nn.functional.binary_cross_entropy_with_logits(
            y, lab.double(), pos_weight=torch.tensor(9.0, dtype=torch.float64, device=DEV))
        loss.backward()
        return {"y": y.detach(), "loss": loss.detach().reshape(1), "grad": torch.cat([v.grad.reshape(-1) for v in p])}
    if kind != "search" or c["n_sky"] * c["n_tmpl"] * c["n_det"] * c["n_seg"] > EXACT_LOOKUPS:
        return None
    # about 12 small kernels per (detector, segment) of every block of templates
    if c["n_seg"] * c["n_det"] * max(1.0, c["n_sky"] * c["n_tmpl"] / 4e7) > 24000:
        return None
    ev, bank = _case_event(c, seed)
    S, W1, W2, psi = _exact_psi(c, ev, bank)
    out = {"psi": torch.topk(psi, c["k"], dim=1).values, "idx": None}
    if c["stats"]:
        out["stats"] = {"S": S, "W1": W1, "W2": W2, "psi": psi}
    return out
