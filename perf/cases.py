"""Timed cases of the F-map: what a program does with this library, through its
public entry points, from one 200 x 200 map to 1024 templates over a
2000 x 2000 grid.

A case is a dict of plain numbers.  ``kind`` is ``"map"`` (one plan: atoms on
the device in, map and summaries out), ``"batch"`` (many uneven instances in
one captured graph) or ``"serve"`` (a burst of requests from host memory).

Inputs follow the data model of ``synth`` (Gaussian noise atoms of one or two
detectors with the sidereal antenna pattern and missing SFTs, some templates
with an injected transient), drawn on the GPU from the seed alone, at GPS
timestamps.
"""

import math

import numpy as np
import torch

import paper_1805_05652_gb300 as fm
from paper_1805_05652_gb300 import binding as fb

T_SFT = 1800
GPS0 = 1126051217              # first SFT's start
OMEGA = 2.0 * math.pi / 86164.0
RECT, EXP, TABLE = fb.FMAP_RECT, fb.FMAP_EXP, fb.FMAP_TABLE
WINDOWS = {"rect": RECT, "exp": EXP, "table": TABLE}
# form of a plan: window, precision, plan flags
FORMS = {"rect": ("rect", "fp64", 0),
         "rec": ("exp", "fp64", fb.FMAP_PLAN_EXP_RECURRENCE),
         "bf16x3": ("exp", "bf16x3", 0),
         "tf32": ("exp", "tf32", 0),
         "table": ("table", "bf16x3", 0)}
TABLE_POINTS = 257
CHUNK_BYTES = 1 << 30          # working arrays of exact()


def _map(name, form, T, n, n_t0, n_tau, dt0=T_SFT, dtau=T_SFT, det=1, presence=1.0, sky=False):
    c = dict(kind="map", form=form, T=T, n=n, n_t0=n_t0, n_tau=n_tau, dt0=dt0, dtau=dtau, det=det,
             presence=presence, sky=sky)
    return dict(c, name=name) if name else c


def listed():
    return [
        # One candidate, one detector with 10 % gaps: the call of an
        # interactive follow-up, where latency and launches count.
        _map("rect_small", "rect", 1, 200, 200, 200, presence=0.9),
        # The same for an exponential transient, ragged sizes.
        _map("exp_small", "rec", 1, 331, 150, 177, presence=0.9),
        # A narrow frequency band of a post-glitch search, two detectors
        # merged, rectangular windows at steps of a few SFTs' length.
        _map("rect_band", "rect", 16, 2000, 1000, 1000, 2700, 2700, det=2, presence=0.9),
        # The same band with exponential windows by the decayed recurrence
        # (the library's FP64-class form)
        _map("exp_band", "rec", 16, 2000, 1000, 1000, det=2, presence=0.9),
        # and by the tensor-core contraction.
        _map("exp_band_bf16x3", "bf16x3", 16, 2000, 1000, 1000, det=2, presence=0.9),
        # A year of SFTs, a few templates: longer than the recurrence takes.
        _map("exp_year_tf32", "tf32", 5, 17520, 411, 389, 18 * T_SFT, 12 * T_SFT, det=2,
             presence=0.8),
        # Candidates at different sky positions: antenna rows of their own.
        _map("exp_sky", "rec", 24, 977, 403, 389, sky=True, det=2, presence=0.9),
        # A window function of the user's own, sampled.
        _map("table_band", "table", 8, 1000, 301, 500, det=2, presence=0.9),
        # Many templates of one sky position, the throughput calls.
        _map("rect_templates", "rect", 1024, 5000, 2000, 2000),
        _map("exp_templates", "rec", 1024, 5000, 2000, 2000),
        # Uneven instances (both windows) in one graph-captured batch.
        dict(name="uneven_batch", kind="batch", items=48, layout=7, n_lo=100, n_hi=8000, g_lo=50,
             g_hi=2000),
        # A burst of follow-up requests to the server, from host memory.
        dict(name="serve_burst", kind="serve", items=12, layout=11, n_lo=100, n_hi=8000, g_lo=50,
             g_hi=2000, t_hi=64),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    k = rng.random()
    if k < 0.1:
        g_hi = rng.randint(300, 2000)
        return dict(kind="batch", items=rng.randint(8, 64), layout=rng.randint(0, 1 << 20),
                    n_lo=100, n_hi=_log_int(rng, 800, 8000), g_lo=50, g_hi=g_hi)
    if k < 0.2:
        return dict(kind="serve", items=rng.randint(3, 16), layout=rng.randint(0, 1 << 20),
                    n_lo=100, n_hi=_log_int(rng, 800, 8000), g_lo=50, g_hi=rng.randint(300, 2000),
                    t_hi=rng.randint(1, 64))
    form = rng.choice(["rect", "rect", "rec", "rec", "rec", "bf16x3", "tf32", "table"])
    n = _log_int(rng, 100, 9000 if form in ("rect", "rec") else
                 17520 if form != "table" else 2000)
    n_t0, n_tau = _log_int(rng, 50, 2000), _log_int(rng, 50, 2000)
    if form == "table":
        n_t0, n_tau = min(n_t0, 500), min(n_tau, 500)
    det = rng.randint(1, 2)
    presence = rng.choice([1.0, 0.9, 0.8])
    sky = rng.random() < 0.15
    # templates: log-uniform within a bound on the map and, for the
    # contractions, on the window terms
    cells = n_t0 * n_tau
    t_hi = min(1024, 4_000_000_000 // cells)
    if form in ("bf16x3", "tf32", "table"):
        t_hi = min(t_hi, int(2e11 / (cells * min(n, 3 * n_tau))))
    if sky:
        t_hi = min(t_hi, 32, 60_000_000 // cells)
    T = _log_int(rng, 1, max(1, t_hi))
    # grid steps: one SFT, or spanning the data in integer seconds
    span = int(n / max(0.1, presence)) * T_SFT
    if rng.random() < 0.5:
        dt0 = dtau = T_SFT
    else:
        dt0 = max(1, span // n_t0)
        dtau = max(1, span // (n_tau if form == "rect" else 3 * n_tau))
    return _map(None, form, T, n, n_t0, n_tau, dt0, dtau, det, presence, sky)


# ---------------------------------------------------------------- inputs ----

def _times(gen, n, det, presence):
    """Slots that hold an SFT of at least one detector (int64 [n], on a T_SFT
    lattice) and which detectors are there ([det][n])."""
    dev = gen.device
    if presence >= 1.0:
        return torch.arange(n, device=dev) * T_SFT, torch.ones((det, n), dtype=torch.bool,
                                                               device=dev)
    n_slots = int(1.3 * n / (1.0 - (1.0 - presence) ** det)) + 64
    pres = torch.rand((det, n_slots), generator=gen, device=dev) < presence
    slots = torch.nonzero(pres.any(0)).flatten()[:n]
    return slots * T_SFT, pres[:, slots]


def _window_weight(kind, x):
    """Amplitude at x = (t - t0) / tau >= 0 of an injected transient."""
    if kind == RECT:
        return (x < 1.0).to(x.dtype)
    return torch.where(x < 3.0, torch.exp(-x), torch.zeros_like(x))


def _atoms(gen, n, T, det, presence, window, sky=False, first=GPS0):
    """Atoms of T templates: timestamps [n] int64, antenna rows [3][n] (or
    [T][3][n]) and data rows [T][4][n] float32."""
    dev = gen.device
    t, pres = _times(gen, n, det, presence)
    n_sky = T if sky else 1
    ph = torch.rand((n_sky, det, 2, 1), generator=gen, device=dev, dtype=torch.float64) * 2 * math.pi
    ts = (t + (first - GPS0)).to(torch.float64)
    m = pres.to(torch.float64)
    a = (0.4 + 0.3 * torch.cos(OMEGA * ts + ph[:, :, 0])) * m       # [n_sky][det][n]
    b = (0.2 + 0.3 * torch.sin(OMEGA * ts + ph[:, :, 1])) * m
    antenna = torch.stack([(a * a).sum(1), (b * b).sum(1), (a * b).sum(1)], 1).to(torch.float32)
    fafb = torch.empty((T, 4, n), dtype=torch.float32, device=dev)
    every = max(1, T // 8)                                          # injected templates
    span = float(t[-1] + T_SFT)
    inj = torch.rand((T, 3), generator=gen, device=dev, dtype=torch.float64).cpu().tolist()
    amp = torch.randn((T, 4), generator=gen, device=dev, dtype=torch.float64)
    step = max(1, (1 << 24) // (det * n))
    for lo in range(0, T, step):
        hi = min(T, lo + step)
        z = torch.randn((2, hi - lo, det, n), generator=gen, device=dev) * math.sqrt(0.5)
        aa, bb = (a[lo:hi], b[lo:hi]) if sky else (a, b)
        for j in range(lo, hi):
            if j % every:
                continue
            t0, tau = inj[j][0] * 0.5 * span, (0.02 + 0.2 * inj[j][1]) * span
            x = (t.to(torch.float64) - t0) / tau
            w = torch.where(x >= 0, _window_weight(window, x.clamp(min=0)), torch.zeros_like(x))
            ja, jb = (a[j], b[j]) if sky else (a[0], b[0])
            h = torch.stack([ja * amp[j, 0] + jb * amp[j, 2], ja * amp[j, 1] + jb * amp[j, 3]]) * w
            s = torch.sqrt((100.0 + 160.0 * inj[j][2]) / (2.0 * (h * h).sum() + 1e-12))
            z[:, j - lo] += (h * s).to(torch.float32)
        fafb[lo:hi, 0] = (aa * z[0]).sum(1).to(torch.float32)
        fafb[lo:hi, 1] = (aa * z[1]).sum(1).to(torch.float32)
        fafb[lo:hi, 2] = (bb * z[0]).sum(1).to(torch.float32)
        fafb[lo:hi, 3] = (bb * z[1]).sum(1).to(torch.float32)
    return t + first, antenna.contiguous() if sky else antenna[0].contiguous(), fafb


def _window_table():
    """A Gaussian-shaped rise and fall, sampled on [0, 3] (units of tau)."""
    x = np.linspace(0.0, 3.0, TABLE_POINTS)
    return np.exp(-0.5 * ((x - 1.2) / 0.6) ** 2).astype(np.float32)


def _grid(window, n_t0, n_tau, dt0, dtau):
    """(t0_min, dt0, n_t0, tau_min, dtau, n_tau, T_sft, window)"""
    return (GPS0, dt0, n_t0, T_SFT if window == EXP else 2 * T_SFT, dtau, n_tau, T_SFT, window)


def _items(case):
    """Sizes of a batch's instances or a burst's requests."""
    rng = np.random.default_rng(case["layout"])
    out = []
    for _ in range(case["items"]):
        n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        n_t0, n_tau = (int(rng.integers(case["g_lo"], case["g_hi"] + 1)) for _ in range(2))
        window = int(rng.integers(0, 2))
        T = int(rng.integers(1, case["t_hi"] + 1)) if "t_hi" in case else 1
        if case["kind"] == "batch":   # whole SFTs
            dt0, dtau = (T_SFT * max(1, round(n / k)) for k in (n_t0, n_tau))
        else:                         # integer seconds over the data's span
            dt0, dtau = (max(1, int(n / 0.9) * T_SFT // k) for k in (n_t0, n_tau))
        out.append((n, T, _grid(window, n_t0, n_tau, dt0, dtau)))
    return out


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _inputs(case, seed):
    """The atoms of every problem of a case: a list of (grid, t, antenna, fafb)."""
    gen = _generator(seed)
    if case["kind"] == "map":
        window = WINDOWS[FORMS[case["form"]][0]]
        grid = _grid(window, case["n_t0"], case["n_tau"], case["dt0"], case["dtau"])
        return [(grid, *_atoms(gen, case["n"], case["T"], case["det"], case["presence"], window,
                               case["sky"]))]
    # (batches: gap-free data of one detector; requests: 10 % gaps)
    presence = 1.0 if case["kind"] == "batch" else 0.9
    return [(g, *_atoms(gen, n, T, 1, presence, g[7])) for n, T, g in _items(case)]


# --------------------------------------------------------------- the calls --

def _columns(summary):
    """The summaries' fields (max 2F, log Bayes factor, cell (m, n), valid
    cells) of a uint8 [T][32] buffer.  The candidates' ranking statistics are
    both kept in single precision (logB is stated to 1e-4)."""
    return {"max2F": summary.view(torch.float32)[:, 0],
            "logB": summary.view(torch.float64)[:, 2].to(torch.float32),
            "cell": summary.view(torch.int32)[:, 1:3],
            "n_valid": summary.view(torch.int64)[:, 3]}


def prepare(case, seed):
    problems = _inputs(case, seed)
    if case["kind"] == "map":
        grid, t, antenna, fafb = problems[0]
        _, precision, flags = FORMS[case["form"]]
        if case["sky"]:
            flags |= fb.FMAP_PLAN_PER_TEMPLATE_ANTENNA
        plan = fm.Plan(grid, case["n"], case["T"], precision, flags)
        if grid[7] == TABLE:
            fb.fmap_plan_window_table(plan.handle, _window_table())
        m = torch.empty((case["T"], case["n_t0"], case["n_tau"]), dtype=torch.float32,
                        device="cuda")
        s = torch.empty((case["T"], 32), dtype=torch.uint8, device="cuda")
        return dict(kind="map", plan=plan, atoms=(t, antenna, fafb), map=m, summary=s)
    if case["kind"] == "batch":
        # the instances' maps and summaries in one buffer each
        sizes = [g[2] * g[5] * x.shape[0] for g, _, _, x in problems]
        at = np.concatenate([[0], np.cumsum([(s + 63) // 64 * 64 for s in sizes])])
        row = np.concatenate([[0], np.cumsum([x.shape[0] for _, _, _, x in problems])])
        m = torch.zeros(int(at[-1]), dtype=torch.float32, device="cuda")
        s = torch.zeros((int(row[-1]), 32), dtype=torch.uint8, device="cuda")
        items = [fb.fmap_batch_item(fb.make_grid(g),
                                    fb.make_atoms(t.shape[0], x.shape[0], True, t, a, x),
                                    m.data_ptr() + 4 * int(at[i]), s.data_ptr() + 32 * int(row[i]))
                 for i, (g, t, a, x) in enumerate(problems)]
        torch.cuda.synchronize()
        return dict(kind="batch", batch=_Batch(items), keep=problems, map=m, summary=s)
    host = [(g, t.cpu().numpy(), a.cpu().numpy(), x.cpu().numpy()) for g, t, a, x in problems]
    server = fm.Server(device_mem_budget=12 << 30, pinned_bytes=256 << 20, max_inflight=8,
                       exp_mode="auto")
    return dict(kind="serve", server=server, requests=host)


class _Batch:
    """Owns a batch handle."""

    handle = None

    def __init__(self, items):
        self.handle = fb.fmap_batch_plan(items, 0, fb.FMAP_BATCH_AUTOTUNE)

    def __del__(self):
        fb.fmap_batch_destroy(self.handle)


def run(state):
    if state["kind"] == "map":
        m, s = state["plan"].compute(*state["atoms"], out_map=state["map"],
                                     out_summary=state["summary"])
        return {"map": m, **_columns(s)}
    if state["kind"] == "batch":
        fb.fmap_batch_run(state["batch"].handle)
        return {"map": state["map"], **_columns(state["summary"])}
    server = state["server"]
    tickets = [server.submit(*r) for r in state["requests"]]
    s = np.concatenate([server.poll(k)[1] for k in tickets])
    return {"max2F": s["max2F"], "logB": s["logB"].astype(np.float32),
            "cell": np.stack([s["m"], s["n"]], 1), "n_valid": s["n_valid"]}


# ------------------------------------------------- what a pass has to do ----

def _terms(n, grid, presence):
    """Atoms summed over all windows of one template (App. A's N_sums)."""
    _, dt0, n_t0, tau_min, dtau, n_tau, t_sft, window = grid
    span = n / presence * t_sft
    left = np.maximum(0.0, span - dt0 * np.arange(n_t0, dtype=np.float64))
    length = (tau_min + dtau * np.arange(n_tau, dtype=np.float64)) * (1.0 if window == RECT else 3.0)
    return float(np.minimum(left[:, None], length[None, :]).sum()) / t_sft * presence


def work(case):
    """Bytes: every atom read once, every map cell and summary written once.
    Flops per template: rectangular windows, prefix sums (4 N) and 4
    differences and 17 for 2F per cell; exponential ones, the decayed
    recurrence (2 x 4 N per tau) and 12 for the sums and 17 for 2F per cell;
    sampled windows have no recurrence: 2 x 4 per atom of each window."""
    if case["kind"] == "map":
        window = WINDOWS[FORMS[case["form"]][0]]
        probs = [(case["n"], case["T"], _grid(window, case["n_t0"], case["n_tau"], case["dt0"],
                                              case["dtau"]))]
        presence = 1.0 - (1.0 - case["presence"]) ** case["det"]
        n_ant, maps = case["T"] if case["sky"] else 1, True
    else:
        probs, n_ant = _items(case), 1
        presence, maps = 1.0 if case["kind"] == "batch" else 0.9, case["kind"] == "batch"
    by = fl = 0.0
    for n, T, g in probs:
        cells = g[2] * g[5]
        by += 8 * n + 12 * n * n_ant + 16 * n * T + 32 * T + (4 * cells * T if maps else 0)
        if g[7] == RECT:
            fl += T * (4 * n + 21 * cells)
        elif g[7] == EXP:
            fl += T * (8 * n * g[5] + 29 * cells)
        else:
            fl += T * (8 * _terms(n, g, presence) + 17 * cells)
    return {"bytes": by, "flops": fl}


# --------------------------------------------- the same results in 64 bits --

def _rect_sums(x, i0, j):
    """Window sums [..., n_t0, n_tau] of rows x [..., n]: exact fixed-point
    prefix sums (2^-42 units), differenced."""
    p = torch.zeros((*x.shape[:-1], x.shape[-1] + 1), dtype=torch.int64, device=x.device)
    torch.cumsum(torch.round(x.to(torch.float64) * 2.0 ** 42).to(torch.int64), -1, out=p[..., 1:])
    return (p[..., j] - p[..., i0].unsqueeze(-1)).to(torch.float64) * 2.0 ** -42


def _exp_sums(x, t, i0, j, t0, tau, power):
    """Window sums [..., n_t0, k] with w^power, w = e^{-(t - t0)/tau}, for k
    values of tau: suffix sums by doubling, in 64 bits."""
    n = x.shape[-1]
    r = power / tau.to(torch.float64)                                # [k]
    e = x.to(torch.float64).unsqueeze(-2).expand(*x.shape[:-1], tau.shape[0], n).clone()
    s = 1
    while s < n:
        d = torch.exp(-(t[s:] - t[:-s]).to(torch.float64) * r[:, None])
        e = torch.cat([e[..., :-s] + d * e[..., s:], e[..., -s:]], -1)
        s *= 2
    e = torch.cat([e, torch.zeros((*e.shape[:-1], 1), dtype=e.dtype, device=e.device)], -1)
    e = e.transpose(-1, -2)                                          # [..., n + 1, k]
    tp = torch.cat([t, t[-1:]])                                      # (e[n] = 0: any time does)
    k = torch.arange(tau.shape[0], device=x.device)
    ti = tp[i0][:, None]
    pre = torch.exp(-(ti - t0[:, None]).clamp(min=0).to(torch.float64) * r)   # [n_t0][k]
    tail = torch.exp(-(tp[j] - ti).clamp(min=0).to(torch.float64) * r)
    out = pre * (e[..., i0, :] - tail * e[..., j, k])
    return torch.where(j > i0[:, None], out, torch.zeros_like(out))


def _table_sums(x, t, i0, j, t0, tau, power):
    """The same with the sampled window, summed directly per tau."""
    w = torch.from_numpy(_window_table()).to(x.device).to(torch.float64)
    a = torch.arange(t.shape[0], device=x.device)
    cols = []
    for k in range(tau.shape[0]):
        u = (t[None, :] - t0[:, None]).to(torch.float64) * ((TABLE_POINTS - 1) / (3.0 * float(tau[k])))
        f = u.clamp(0, TABLE_POINTS - 1).floor().clamp(max=TABLE_POINTS - 2).to(torch.int64)
        v = w[f] + (u - f) * (w[f + 1] - w[f])
        inside = (a[None, :] >= i0[:, None]) & (a[None, :] < j[:, k, None]) & (u <= TABLE_POINTS - 1)
        v = torch.where(inside, v, torch.zeros_like(v)) ** power
        cols.append((x.to(torch.float64).reshape(-1, x.shape[-1]) @ v.T).reshape(*x.shape[:-1], -1))
    return torch.stack(cols, -1)


def _exact_map(grid, t, antenna, fafb, want_map):
    """The map [T][n_t0][n_tau] (None unless wanted) and per template max 2F
    and logB, in 64 bits."""
    t0_min, dt0, n_t0, tau_min, dtau, n_tau, t_sft, window = grid
    dev, T, n = t.device, fafb.shape[0], t.shape[0]
    t0 = t0_min + dt0 * torch.arange(n_t0, device=dev)
    tau = tau_min + dtau * torch.arange(n_tau, device=dev)
    length = tau if window == RECT else 3 * tau
    i0 = torch.searchsorted(t, t0)
    j = torch.searchsorted(t, t0[:, None] + length[None, :] - t_sft, right=True)
    j = torch.maximum(j, i0[:, None])
    per_tau = 8 * 4 * 4 * max(n, n_t0)
    k_step = n_tau if window == RECT else max(1, min(n_tau, CHUNK_BYTES // per_tau))

    def sums(x, lo, hi, power):
        if window == RECT:
            return _rect_sums(x, i0, j[:, lo:hi])
        f = _exp_sums if window == EXP else _table_sums
        return f(x, t, i0, j[:, lo:hi], t0, tau[lo:hi], power)

    out = torch.zeros((T, n_t0, n_tau), dtype=torch.float64, device=dev) if want_map else None
    top, bayes = [], []
    shared = antenna.dim() == 2
    kept = {}
    for q in range(T):
        row = out[q] if want_map else torch.zeros((n_t0, n_tau), dtype=torch.float64, device=dev)
        ok = torch.empty((n_t0, n_tau), dtype=torch.bool, device=dev)
        for lo in range(0, n_tau, k_step):
            hi = min(n_tau, lo + k_step)
            if not shared or lo not in kept:
                A, B, C = sums(antenna if shared else antenna[q], lo, hi, 2)
                D = A * B - C * C
                good = (j[:, lo:hi] - i0[:, None] >= 2) & (D > 0)
                kept[lo] = (A, B, C, torch.where(good, D, torch.ones_like(D)), good)
            A, B, C, D, good = kept[lo]
            ar, ai, br, bi = sums(fafb[q], lo, hi, 1)
            f = 2.0 * (B * (ar * ar + ai * ai) + A * (br * br + bi * bi)
                       - 2.0 * C * (ar * br + ai * bi)) / D
            row[:, lo:hi] = torch.where(good, f, torch.zeros_like(f))
            ok[:, lo:hi] = good
        v = row[ok]
        top.append(v.max())
        bayes.append(torch.logsumexp(0.5 * v, 0) - math.log(v.numel()))
    return out, torch.stack(top), torch.stack(bayes)


def exact(case, seed):
    if case["kind"] == "map" and case["form"] == "table" and case["n_tau"] * case["n_t0"] > 300_000:
        return None
    problems = _inputs(case, seed)
    maps, top, bayes = [], [], []
    for p in problems:
        m, a, b = _exact_map(*p, want_map=case["kind"] != "serve")
        maps.append(m)
        top.append(a)
        bayes.append(b)
    out = {"max2F": torch.cat(top), "logB": torch.cat(bayes), "cell": None, "n_valid": None}
    if case["kind"] == "serve":
        return {k: None if v is None else v.cpu().numpy() for k, v in out.items()}
    if case["kind"] == "map":
        return {"map": maps[0], **out}
    flat = torch.cat([torch.nn.functional.pad(m.reshape(-1), (0, -m.numel() % 64)) for m in maps])
    return {"map": flat, **out}
