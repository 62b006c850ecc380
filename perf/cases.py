"""Performance cases of the OPMM library, through its Python entry points.

Each case is one call (or one burst of calls) that a program built on this
library makes, at sizes of the benchmark's workloads and around them:

  fit       search of a batch of recorded saccades: a one-shot opmm_fit_batch,
            or the execution of a plan kept for batches of one shape
  seeded    surrogate-seeded search with the plain search as fallback
  serve     a burst of single saccades through the request loop
  train     training steps of the surrogate network (forward and backward)
  predict   the network's OPC estimate of a batch
  simulate  trajectories of many OPC vectors
  score     objective of many OPC vectors against one recording
  refine    Levenberg-Marquardt refinement of given OPC vectors
  detect    I-VT saccade detection on a raw position stream

The recordings are synthetic: a hidden OPC vector within 20% of the nominal
one, its trajectory from the FP64 plant below (plain torch, none of the
library's code) and 0.05 deg of Gaussian noise, at the rates, windows and
amplitudes of the workloads package.
"""
import math

import numpy as np
import torch

import paper_2007_09884_gb300 as G

NP = 18
SE_AG, SE_ANT, LT_AG, LT_ANT, NC_AG, NC_ANT, BP, B_AG, B_ANT, J = range(10)
TAC_AG, TAC_ANT, TDE_AG, TDE_ANT, NC_FIX, H_AG, H_ANT, PW = range(10, 18)
TABLE1 = [2.5, 2.5, 1.2, 1.2, 0.8, 0.5, 0.06, 0.046, 0.022, 0.000043, 11.7, 2.4, 2.0, 1.9, 14.0, 55.0, 0.5, 0.0]
NOISE_DEG = 0.05
ONSET_MS, TAIL_MS = 10.0, 20.0
HIDDEN, LAYERS = 512, 4
N_WEIGHTS = LAYERS * (HIDDEN * HIDDEN + HIDDEN) + NP * HIDDEN + NP
# searches of the benchmark: seeded search in a 5% box, plain search for its misses
SEEDED = dict(candidates=1024, iterations=20, box_lo=0.95, box_hi=1.05, init_step=0.025)
FALLBACK = dict(candidates=4096, iterations=30)
DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one freshly recorded 10 deg saccade, 1 kHz, Table 1's own pulse height: the smallest search
        dict(name="fit_single", kind="fit", n=1, candidates=4096, iterations=20, hz=1000, lmin=150, lmax=150, amp=10.0,
             model=18, plan=False, device=False, table1=True),
        # the plain batched search, the largest call: one laboratory's saccades per execution of a kept plan
        dict(name="fit_batch", kind="fit", n=1024, candidates=65536, iterations=30, hz=1000, lmin=60, lmax=200, amp=0.0,
             model=18, plan=True, device=False, table1=False),
        # recordings of mixed rates, directions and lengths from several trackers, traces already on the device
        dict(name="fit_uneven", kind="fit", n=2500, candidates=16384, iterations=30, hz=0, lmin=40, lmax=400, amp=0.0,
             model=18, plan=True, device=True, table1=False),
        # the 9-parameter model on a session's saccades, one-shot
        dict(name="fit_model9", kind="fit", n=201, candidates=16384, iterations=30, hz=1000, lmin=60, lmax=200, amp=0.0,
             model=9, plan=False, device=False, table1=False),
        # high-throughput fitting: network estimate, narrow search, plain search where that misses 0.1 deg
        dict(name="fit_seeded", kind="seeded", n=2000),
        # real-time use: a burst of single saccades arrives at the request loop, every result is collected
        dict(name="serve_burst", kind="serve", n=384, seeded=True, round_iters=5),
        # training the surrogate on saccades generated on the device
        dict(name="train", kind="train", steps=96, batch=4096),
        # the network alone over a held-out set
        dict(name="predict", kind="predict", n=10000),
        # trajectories of candidate vectors for inspection: 64 vectors of each of 1,021 saccades
        dict(name="simulate", kind="simulate", n=1021, per=64),
        # a caller's own search step: one generation of candidates against one recording
        dict(name="score", kind="score", m=32768, samples=150, hz=1000),
        # gradient refinement of a batch after its search
        dict(name="refine", kind="refine", n=1024, iterations=10, model=18),
        # 16.7 hours of raw 1 kHz positions, already on the device
        dict(name="detect", kind="detect", samples=60000011, hz=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "seeded", "serve", "train", "predict", "simulate", "score", "refine",
                       "detect"])
    if kind == "fit":
        model = 9 if rng.random() < 0.25 else 18
        hz = rng.choice([0, 250, 500, 1000])
        top = max(work(c)["flops"] for c in listed())
        while True:
            c = dict(kind=kind, n=_log(rng, 1, 3000), candidates=_log(rng, 22, 65536), iterations=rng.randint(3, 40), hz=hz,
                     lmin=60 if hz == 1000 else 40, lmax=rng.randint(120, 400), amp=0.0, model=model,
                     plan=rng.random() < 0.5, device=rng.random() < 0.5, table1=False)
            if work(c)["flops"] <= top:
                return c
    if kind == "seeded":
        return dict(kind=kind, n=_log(rng, 1, 4000))
    if kind == "serve":
        seeded = rng.random() < 0.7
        return dict(kind=kind, n=_log(rng, 1, 800 if seeded else 200), seeded=seeded, round_iters=rng.randint(3, 10))
    if kind == "train":
        return dict(kind=kind, steps=rng.randint(1, 120), batch=128 * rng.randint(1, 40))
    if kind == "predict":
        return dict(kind=kind, n=_log(rng, 1, 20000))
    if kind == "simulate":
        return dict(kind=kind, n=_log(rng, 1, 2000), per=_log(rng, 1, 100))
    if kind == "score":
        return dict(kind=kind, m=_log(rng, 100, 300000), samples=rng.randint(60, 400), hz=rng.choice([250, 500, 1000]))
    if kind == "refine":
        return dict(kind=kind, n=_log(rng, 1, 2000), iterations=rng.randint(3, 12), model=9 if rng.random() < 0.25 else 18)
    return dict(kind=kind, samples=_log(rng, 5000, 60000000), hz=rng.choice([250, 500, 1000]))


# ------------------------------------------------------------------ FP64 plant
def _plant(p, fs, nsub):
    """Single-substep RK4 matrices (I + Q) of the pulse and the step phase, their plant matrices, the substep."""
    n = p.shape[0]
    h = 1.0 / (fs * nsub)

    def matrix(tau_a, tau_n):
        A = torch.zeros(n, 6, 6, dtype=F64, device=DEV)
        kp = p[:, NC_AG] + p[:, NC_ANT]
        A[:, 0, 1] = 1.0
        A[:, 1, 0] = -(p[:, SE_AG] + p[:, SE_ANT] + kp) / p[:, J]
        A[:, 1, 1] = -p[:, BP] / p[:, J]
        A[:, 1, 2] = p[:, SE_AG] / p[:, J]
        A[:, 1, 3] = -p[:, SE_ANT] / p[:, J]
        A[:, 2, 0] = p[:, SE_AG] / p[:, B_AG]
        A[:, 2, 2] = -(p[:, SE_AG] + p[:, LT_AG]) / p[:, B_AG]
        A[:, 2, 4] = 1.0 / p[:, B_AG]
        A[:, 3, 0] = -p[:, SE_ANT] / p[:, B_ANT]
        A[:, 3, 3] = -(p[:, SE_ANT] + p[:, LT_ANT]) / p[:, B_ANT]
        A[:, 3, 5] = 1.0 / p[:, B_ANT]
        A[:, 4, 4] = -1000.0 / tau_a
        A[:, 5, 5] = -1000.0 / tau_n
        return A

    return matrix(p[:, TAC_AG], p[:, TDE_ANT]), matrix(p[:, TDE_AG], p[:, TAC_ANT]), h


def _mm(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _mv(a, v):
    return (a * v[:, None, :]).sum(2)


def _rk4(A, h):
    """One RK4 step of e' = A e as a matrix, the step length per row."""
    eye = torch.eye(6, dtype=F64, device=DEV)
    Z = A * h[:, None, None]
    W = eye + Z / 4
    W = eye + _mm(Z, W) / 3
    W = eye + _mm(Z, W) / 2
    return eye + _mm(Z, W)


def _power(M, k):
    """M^k, the exponent per row."""
    out = torch.eye(6, dtype=F64, device=DEV).expand_as(M).clone()
    k = k.clone()
    while bool((k > 0).any()):
        out = torch.where((k & 1).bool()[:, None, None], _mm(out, M), out)
        k = k >> 1
        M = _mm(M, M)
    return out


def _levels(p, th):
    ta, tn = p[:, NC_FIX] + p[:, NC_AG] * th, p[:, NC_FIX] - p[:, NC_ANT] * th
    return (ta * (1 + p[:, LT_AG] / p[:, SE_AG]) + p[:, LT_AG] * th,
            tn * (1 + p[:, LT_ANT] / p[:, SE_ANT]) - p[:, LT_ANT] * th)


def _rest(p, fa, fn):
    ag, an = p[:, SE_AG] / (p[:, SE_AG] + p[:, LT_AG]), p[:, SE_ANT] / (p[:, SE_ANT] + p[:, LT_ANT])
    th = (ag * fa - an * fn) / (p[:, NC_AG] + p[:, NC_ANT] + ag * p[:, LT_AG] + an * p[:, LT_ANT])
    ta, tn = ag * (fa - p[:, LT_AG] * th), an * (fn + p[:, LT_ANT] * th)
    return torch.stack([th, torch.zeros_like(th), th + ta / p[:, SE_AG], tn / p[:, SE_ANT] - th, fa, fn], 1)


def _trajectories(p, L, onset, fs, th0, thf):
    """theta [n][max L] in FP64 of OPC vectors p [n][18] on their saccades (RK4 at about 0.1 ms, the substep that
    holds the pulse end split there).  The plant is linear within a phase, so one sample is one 6 x 6 map."""
    n = p.shape[0]
    sign = torch.where(thf < th0, -1.0, 1.0).to(F64)
    a, b = sign * th0, sign * thf
    nsub = torch.floor(1.0e4 / fs + 0.5).clamp(min=1)
    A1, A2, h = _plant(p, fs, nsub)
    Q1, Q2 = _rk4(A1, h), _rk4(A2, h)
    k = nsub.long()
    P1, P2 = _power(Q1, k), _power(Q2, k)
    s0, s2 = _rest(p, *_levels(p, a)), _rest(p, *_levels(p, b))
    s1 = _rest(p, p[:, H_AG], p[:, H_ANT])
    tau = (p[:, PW] * fs * nsub / 1000.0).clamp(0.0, 1.0e9)
    whole = torch.floor(tau)
    frac = tau - whole
    n1 = torch.div(whole.long(), k, rounding_mode="floor")
    sub = whole.long() - n1 * k
    before = _mm(_rk4(A1, frac * h), _power(Q1, sub))
    after = _mm(_power(Q2, (k - 1 - sub).clamp(min=0)), _rk4(A2, h - frac * h))
    Ms, bs = _mm(after, before), _mv(after, s1 - s2)
    lmax = int(L.max())
    out = a[:, None].expand(n, lmax).clone()
    e = s0 - s1
    for j in range(1, lmax):
        i = j - onset - 1                      # index of the sample interval that ends at sample j
        pulse, switch = i < n1, i == n1
        nxt = torch.where(pulse[:, None], _mv(P1, e), _mv(P2, e))
        nxt = torch.where(switch[:, None], _mv(Ms, e) + bs, nxt)
        moving = i >= 0
        e = torch.where(moving[:, None], nxt, e)
        th = torch.where(pulse, s1[:, 0], s2[:, 0]) + e[:, 0]
        out[:, j] = torch.where(moving, th, out[:, j])
    return sign[:, None] * out


_PULSE = {}


def _pulse(A):
    """Agonist pulse whose default saccade 0 -> A (1 kHz, 250 ms) peaks at A, interpolated in a table over A; the
    step level where that already reaches A.  theta is linear in the pulse height, so two trajectories per table
    entry give the peak at any height."""
    if not _PULSE:
        grid = torch.linspace(0.5, 45.0, 512, dtype=F64, device=DEV)
        n = grid.numel()
        p = torch.tensor(TABLE1, dtype=F64, device=DEV).expand(n, NP).clone()
        p[:, PW] = 2.2 * grid + 21.0 - 6.0
        one = torch.ones(n, dtype=F64, device=DEV)
        fixed = ((251 * one).long(), (0 * one).long(), 1000 * one, 0 * one, grid)
        p[:, H_AG] = 0.0
        base = _trajectories(p, *fixed)
        p[:, H_AG] = 1.0
        slope = _trajectories(p, *fixed) - base
        lo = _levels(p, grid)[0]
        a, b = lo.clone(), lo * 1024
        for _ in range(60):
            mid = 0.5 * (a + b)
            hit = (base[:, 1:] + mid[:, None] * slope[:, 1:]).amax(1) >= grid
            a, b = torch.where(hit, a, mid), torch.where(hit, mid, b)
        _PULSE["grid"], _PULSE["h"] = grid, torch.where((base + lo[:, None] * slope)[:, 1:].amax(1) >= grid, lo, 0.5 * (a + b))
    g, h = _PULSE["grid"], _PULSE["h"]
    x = ((A - g[0]) / (g[-1] - g[0]) * (g.numel() - 1)).clamp(0, g.numel() - 1)
    j = x.floor().long().clamp(max=g.numel() - 2)
    f = x - j
    return (1 - f) * h[j] + f * h[j + 1]


def _nominal(A, table1=False):
    p = torch.tensor(TABLE1, dtype=F64, device=DEV).expand(A.numel(), NP).clone()
    p[:, PW] = 2.2 * A + 21.0 - 6.0
    if not table1:
        p[:, H_AG] = _pulse(A)
    return p


# ------------------------------------------------------------------ recordings
class Recordings:
    """n synthetic saccades: descriptors (numpy), the nominal and the hidden OPC vectors, noisy traces [n][max L]
    (float32, on the device)."""

    def __init__(self, n, seed, hz=0, lmin=40, lmax=400, amp=0.0, table1=False):
        # rates and window lengths belong to the case, the recordings to the seed
        g = np.random.default_rng([0x09884, n, hz, lmin, lmax])
        fs = np.full(n, float(hz)) if hz else g.choice([250.0, 500.0, 1000.0], n)
        # a window holds onset, a saccade of at least 1 deg and the tail
        room = ONSET_MS + TAIL_MS + 21.0 + 2.2 * 1.05
        low = np.maximum(lmin, np.ceil(room * fs / 1000.0).astype(np.int64) + 1)
        L = low + np.floor(g.random(n) * (np.maximum(lmax, low) - low + 1)).astype(np.int64)
        g = np.random.default_rng([0x09884, seed])
        onset = np.ceil(ONSET_MS * 1e-3 * fs - 1e-9).astype(np.int64)
        top = np.minimum(40.0, (1000.0 * (L - onset) / fs - TAIL_MS - 21.0) / 2.2)
        A = np.float32(np.exp(g.random(n) * np.log(np.maximum(top, 1.0)))).astype(np.float64)
        if amp:
            A = np.full(n, float(amp))
        side = np.where(g.random(n) < 0.5, -1.0, 1.0) if not amp else np.ones(n)
        mult = g.uniform(0.8, 1.2, (n, NP))
        self.n, self.fs, self.L, self.onset = n, fs, L, onset
        self.th0, self.thf, self.A = np.zeros(n), side * A, A
        self.dur = np.float32(2.2 * A + 21.0)
        self.args = tuple(torch.as_tensor(v, device=DEV) for v in (L, onset, fs, self.th0, self.thf))
        self.nominal = _nominal(torch.as_tensor(A, device=DEV), table1)
        self.hidden = (self.nominal * torch.as_tensor(mult, device=DEV)).float()
        self.clean = _trajectories(self.hidden.to(F64), *self.args)
        gen = torch.Generator(device=DEV).manual_seed(seed)
        noise = torch.randn(self.clean.shape, generator=gen, device=DEV, dtype=F64)
        self.y = (self.clean + NOISE_DEG * noise).float()

    def batch(self, device=False):
        """As a program holds them: one array per saccade in host memory, or one packed device tensor."""
        if device:
            keep = torch.arange(self.y.shape[1], device=DEV)[None, :] < self.args[0][:, None]
            traces, offsets = self.y[keep], np.concatenate([[0], np.cumsum(self.L)[:-1]])
        else:
            y = self.y.cpu().numpy()
            traces, offsets = [np.ascontiguousarray(y[i, :self.L[i]]) for i in range(self.n)], None
        return G.make_batch(traces, self.fs, self.onset, self.th0, self.thf, self.dur, n_samples=self.L, offsets=offsets)

    def singles(self):
        y = self.y.cpu().numpy()
        return [G.make_batch([np.ascontiguousarray(y[i, :self.L[i]])], [self.fs[i]], [self.onset[i]], [self.th0[i]],
                             [self.thf[i]], [self.dur[i]]) for i in range(self.n)]


# ------------------------------------------------------------------ the surrogate's weights
def _features(rec):
    """Features [n][512] in FP64: 256 points 1 ms apart from onset, linear interpolation held at the window's end,
    in the positive frame over the amplitude; 10 x the per-ms differences."""
    L, onset, fs, th0, thf = rec.args
    sign = torch.where(thf < th0, -1.0, 1.0).to(F64)
    i = torch.arange(257, device=DEV, dtype=F64)
    s = torch.minimum(onset[:, None] + i[None, :] * fs[:, None] / 1000.0, (L - 1)[:, None].to(F64))
    k0 = s.floor().long()
    k1 = torch.minimum(k0 + 1, (L - 1)[:, None])
    w = s - k0
    y = rec.y.to(F64)
    pos = (sign[:, None] * ((1 - w) * y.gather(1, k0) + w * y.gather(1, k1)) - (sign * th0)[:, None])
    pos = pos / (sign * (thf - th0)).clamp(min=0.5)[:, None]
    vel = 10.0 * (pos[:, 1:] - pos[:, :-1])
    vel[:, 255] = 0.0
    return torch.cat([pos[:, :256], vel], 1)


def _unflatten(w):
    out, o = [], 0
    for rows in [HIDDEN] * LAYERS + [NP]:
        out.append((w[o:o + rows * HIDDEN].view(rows, HIDDEN), w[o + rows * HIDDEN:o + rows * HIDDEN + rows]))
        o += rows * HIDDEN + rows
    return out


def _network(w, x):
    layers = _unflatten(w)
    for W, b in layers[:-1]:
        x = torch.nn.functional.gelu(x @ W.t() + b)
    return x @ layers[-1][0].t() + layers[-1][1]


_WEIGHTS = []


def _weights():
    """The weights that a program loads: trained once per process, in plain torch, on 49,152 recordings; the target
    is ln(multiplier) / 0.2."""
    if not _WEIGHTS:
        rec = Recordings(49152, 4242)
        x = _features(rec).float()
        t = ((rec.hidden.to(F64) / rec.nominal).log() / 0.2).float()
        gen = torch.Generator(device=DEV).manual_seed(1)
        w = ((2 * torch.rand(N_WEIGHTS, generator=gen, device=DEV) - 1) / math.sqrt(HIDDEN)).requires_grad_()
        opt = torch.optim.Adam([w], lr=1e-3)
        for step in range(360):
            rows = torch.randint(0, x.shape[0], (2048,), generator=gen, device=DEV)
            loss = (_network(w, x[rows]) - t[rows]).square().mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
        _WEIGHTS.append(w.detach().cpu().numpy())
    return _WEIGHTS[0]


# ------------------------------------------------------------------ contexts
class Context:
    """A library context, destroyed with its last holder."""

    def __init__(self, weights=False, init_seed=None):
        self.h = G.opmm_create(0)
        if weights or init_seed is not None:
            G.opmm_surrogate_init(self.h, init_seed or 0)
        if weights:
            G.opmm_surrogate_set_params(self.h, _weights())

    def __del__(self):
        if getattr(self, "h", None):
            G.opmm_destroy(self.h)


_SHARED = {}


def _shared(weights=False):
    """The context that a program opens once."""
    if weights not in _SHARED:
        _SHARED[weights] = Context(weights)
    return _SHARED[weights]


# ------------------------------------------------------------------ raw streams
def _stream(n, hz, seed):
    """Raw positions: fixations of 150-1200 ms within 40 deg with 0.005 deg of noise, raised-cosine saccades of 1-30 deg
    and main-sequence duration between them, blinks (NaN): some inside a fixation, some over a whole saccade.  Where the
    eye goes belongs to the case, the noise to the seed; no saccade is as near to the 4 deg that a kept one needs, nor
    to a blink or the end, that the noise would decide whether it is kept, so every seed has the same events."""
    g = np.random.default_rng([0x1F7, n, hz])
    m = int(n / (0.67 * hz)) + 8
    step = g.uniform(1.0, 30.0, m)
    step = np.where((step > 3.4) & (step < 4.6), step + 1.2, step)
    pos = np.zeros(m + 1)
    side = g.random(m)
    for i in range(m):                          # toward the side with room, else to either
        right = pos[i] + step[i] <= 20.0 and (side[i] < 0.5 or pos[i] - step[i] < -20.0)
        pos[i + 1] = pos[i] + step[i] if right or pos[i] - step[i] < -20.0 else pos[i] - step[i]
    fix = np.floor(g.uniform(0.15, 1.2, m) * hz).astype(np.int64)
    dur = np.maximum(2, np.rint((2.2 * step + 21.0) * hz / 1000.0)).astype(np.int64)
    start = np.concatenate([[0], np.cumsum(fix + dur)])
    still = n - 2 * hz                          # the eye rests for the last two seconds
    inside = (fix >= 0.6 * hz) & (g.random(m) < 0.2)
    over = ~inside & (g.random(m) < 0.05)
    length = np.floor(g.uniform(0.08, 0.2, m) * hz).astype(np.int64)
    b0 = np.where(inside, start[:-1] + int(0.2 * hz), start[:-1] + fix - 20)[inside | over]
    b1 = b0 + np.where(inside, length, dur + 40)[inside | over]
    dev = lambda v: torch.as_tensor(v, device=DEV)  # noqa: E731
    edge = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    edge.index_add_(0, dev(b0.clip(0, max(0, still - hz))), torch.ones(b0.size, dtype=torch.int32, device=DEV))
    edge.index_add_(0, dev(b1.clip(0, max(0, still - hz))), -torch.ones(b1.size, dtype=torch.int32, device=DEV))
    start, fix, dur, pos = dev(start), dev(fix), dev(dur), dev(pos)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    out = torch.empty(n, dtype=torch.float32, device=DEV)
    for k0 in range(0, n, 1 << 23):
        k = torch.arange(k0, min(n, k0 + (1 << 23)), device=DEV)
        at = k.clamp(max=max(0, still))
        seg = torch.searchsorted(start, at, right=True) - 1
        t = (at - start[seg] - fix[seg] + 1).clamp(min=0).to(F64) / dur[seg]
        x = pos[seg] + (pos[seg + 1] - pos[seg]) * 0.5 * (1 - torch.cos(math.pi * t))
        out[k0:k0 + k.numel()] = x.float() + 0.005 * torch.randn(k.numel(), generator=gen, device=DEV)
    out[torch.cumsum(edge, 0)[:n] > 0] = float("nan")
    return out


# ------------------------------------------------------------------ prepare / run
def _fit_options(case):
    return dict(candidates=case["candidates"], iterations=case["iterations"], seed=0, model=case["model"],
                pulse_init=G.OPMM_PULSE_TABLE1 if case["table1"] else G.OPMM_PULSE_CALIBRATED)


def _fit_recordings(case, seed):
    return Recordings(case["n"], seed, case["hz"], case["lmin"], case["lmax"], case["amp"], case["table1"])


def _candidates(rec, per, seed):
    """`per` OPC vectors for each saccade, log-uniform in the search's default box [0.5, 2] around the nominal."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    u = math.log(2.0) * (2 * torch.rand(rec.n, per, NP, generator=gen, device=DEV, dtype=F64) - 1)
    return (rec.nominal[:, None, :] * u.exp()).reshape(-1, NP).float().contiguous()


def _simulate_recordings(case, seed):
    return Recordings(case["n"], seed)


def _score_recordings(case, seed):
    return Recordings(1, seed, case["hz"], case["samples"], case["samples"])


def prepare(case, seed):
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind == "fit":
        s["ctx"] = _shared()
        batch = _fit_recordings(case, seed).batch(case["device"])
        if case["plan"]:
            s["plan"] = G.opmm_plan_create(s["ctx"].h, batch, **_fit_options(case))
        s["batch"], s["options"] = batch, _fit_options(case)
    elif kind == "seeded":
        s["ctx"], s["batch"] = _shared(True), Recordings(case["n"], seed).batch()
    elif kind == "serve":
        s["ctx"] = Context(weights=case["seeded"])
        fit = dict(SEEDED, use_surrogate=True) if case["seeded"] else dict(candidates=16384, iterations=30)
        G.opmm_serve_start(s["ctx"].h, G.serve_opts(max_slots=1024, max_samples=400, round_iters=case["round_iters"]), **fit)
        s["requests"] = Recordings(case["n"], seed).singles()
    elif kind == "train":
        s["ctx"] = Context(init_seed=seed)
        s["steps"], s["size"], s["seed"] = case["steps"], case["batch"], seed
    elif kind == "predict":
        s["ctx"], s["batch"] = _shared(True), Recordings(case["n"], seed).batch()
    elif kind == "simulate":
        rec = _simulate_recordings(case, seed)
        s["ctx"], s["batch"] = _shared(), rec.batch()
        s["opc"] = _candidates(rec, case["per"], seed)
        s["index"] = np.repeat(np.arange(rec.n, dtype=np.int32), case["per"])
        s["out"] = torch.empty(int(rec.L.sum()) * case["per"], dtype=torch.float32, device=DEV)
    elif kind == "score":
        rec = _score_recordings(case, seed)
        s["ctx"], s["batch"] = _shared(), rec.batch(True)
        s["opc"] = _candidates(rec, case["m"], seed)
        s["out"] = torch.empty(case["m"], dtype=torch.float32, device=DEV)
    elif kind == "refine":
        rec = Recordings(case["n"], seed)
        g = np.random.default_rng([0x5EF, seed])
        # starts as near as a search leaves them; the 9-parameter model scales the nominal drive and shared pairs
        m = g.uniform(0.9, 1.1, (rec.n, NP))
        start = rec.hidden.cpu().numpy() * m
        if case["model"] == 9:
            start = rec.nominal.cpu().numpy() * m
            start[:, SE_ANT], start[:, LT_ANT] = start[:, SE_AG], start[:, LT_AG]
        s["ctx"], s["batch"], s["start"] = _shared(), rec.batch(), start.astype(np.float32)
        s["options"] = dict(iterations=case["iterations"], model=case["model"])
    else:
        s["ctx"], s["stream"], s["hz"] = _shared(), _stream(case["samples"], case["hz"], seed), float(case["hz"])
    torch.cuda.synchronize()
    return s


def run(s):
    kind, ctx = s["kind"], s["ctx"].h
    if kind == "fit":
        return G.opmm_plan_execute(s["plan"]) if "plan" in s else G.opmm_fit_batch(ctx, s["batch"], **s["options"])
    if kind == "seeded":
        return G.opmm_fit_batch_seeded(ctx, s["batch"], SEEDED, FALLBACK, 0.1)
    if kind == "serve":
        tickets = [G.opmm_serve_submit(ctx, b) for b in s["requests"]]
        got = [G.opmm_serve_poll(ctx, t)[0] for t in tickets]
        return {k: np.stack([r[k] for r in got]) for k in got[0]}
    if kind == "train":
        losses = G.opmm_surrogate_train(ctx, s["steps"], batch=s["size"], lr=1e-3, weight_decay=1e-4, data_seed=s["seed"])
        return losses, G.opmm_surrogate_get_params(ctx)
    if kind == "predict":
        return G.opmm_surrogate_predict(ctx, s["batch"])
    if kind == "simulate":
        return G.opmm_simulate(ctx, s["opc"], s["batch"], s["index"], s["out"])
    if kind == "score":
        return G.opmm_score(ctx, s["opc"], s["batch"], 0, s["out"])
    if kind == "refine":
        return G.opmm_refine_batch(ctx, s["batch"], s["start"], **s["options"])
    events = G.opmm_detect_saccades(ctx, s["stream"], s["hz"])
    return {k: events[k] for k in events.dtype.names}


# ------------------------------------------------------------------ work
def _sim_flops(samples, nsub):
    """FP32 operations of one candidate: parameters and step matrices 700, powering to one sample 332 a product, 55 a
    sample after onset, the sample that holds the pulse end."""
    products = 0 if nsub <= 1 else nsub.bit_length() - 1 + bin(nsub).count("1") - 1
    return 700 + 332 * products + 55 * samples + 52 * nsub + 158


def _mean_sim_flops(hz, lmin, lmax):
    rates = [hz] if hz else [250, 500, 1000]
    total = 0.0
    for f in rates:
        low = max(lmin, math.ceil(53.31 * f / 1000.0) + 1)
        total += _sim_flops(0.5 * (low + max(lmax, low)) - 1 - math.ceil(0.01 * f), round(1.0e4 / f))
    return total / len(rates)


def _search(n, candidates, iterations, dim, per_sim):
    simplices = candidates // (dim + 4)
    return n * simplices * (dim + 1 + (dim + 4) * iterations) * per_sim


def work(case):
    """Traces and OPC vectors read once, results written once; the candidates that the search is asked to simulate."""
    kind = case["kind"]
    row = 120.0                                  # one fit result
    uneven = 4.0 * 230                           # one trace of 40-400 samples
    net = 2.0 * (LAYERS * HIDDEN * HIDDEN + NP * HIDDEN)
    if kind == "fit":
        trace = 2.0 * (case["lmin"] + case["lmax"])
        return {"bytes": case["n"] * (trace + row),
                "flops": _search(case["n"], case["candidates"], case["iterations"], case["model"],
                                 _mean_sim_flops(case["hz"], case["lmin"], case["lmax"]))}
    per_sim = _mean_sim_flops(0, 40, 400)
    if kind == "seeded":
        n = case["n"]
        return {"bytes": n * (uneven + row) + 4.0 * N_WEIGHTS, "flops": n * net + _search(n, 1024, 20, NP, per_sim)}
    if kind == "serve":
        n = case["n"]
        fit = (1024, 20) if case["seeded"] else (16384, 30)
        return {"bytes": n * (uneven + row), "flops": _search(n, *fit, NP, per_sim) + (n * net if case["seeded"] else 0.0)}
    if kind == "train":
        m = case["steps"] * case["batch"]
        # forward, output-layer gradients, four weight gradients, three error products; weights and moments per step
        flop = net + 4.0 * NP * HIDDEN + 2.0 * 7 * HIDDEN * HIDDEN
        return {"bytes": case["steps"] * 24.0 * N_WEIGHTS, "flops": m * flop}
    if kind == "predict":
        return {"bytes": case["n"] * (uneven + 4.0 * NP) + 2.0 * N_WEIGHTS, "flops": case["n"] * net}
    if kind == "simulate":
        m = case["n"] * case["per"]
        return {"bytes": m * (4.0 * NP + uneven), "flops": m * per_sim}
    if kind == "score":
        return {"bytes": case["m"] * 4.0 * (NP + 1),
                "flops": case["m"] * _mean_sim_flops(case["hz"], case["samples"], case["samples"])}
    if kind == "refine":
        sims = 2 * case["model"] + 1
        normal = (case["model"] * (case["model"] + 1) / 2 + case["model"]) * 2.0 * 230
        return {"bytes": case["n"] * (uneven + row + 4.0 * NP),
                "flops": case["n"] * case["iterations"] * (sims * per_sim + normal)}
    return {"bytes": 4.0 * case["samples"] + 64.0 * case["samples"] / (0.74 * case["hz"]), "flops": 6.0 * case["samples"]}


# ------------------------------------------------------------------ exact
def _detected(x, hz):
    """The I-VT definition: decisions in FP32 on FP32 samples (as it is stated), the reported numbers in 64 bits."""
    n = x.numel()
    valid = (x >= -90.0) & (x <= 90.0)
    step = (x[1:] - x[:-1]).abs()
    fast = valid[1:] & valid[:-1] & (step * np.float32(hz) > 30.0)       # fast[k - 1]: step k
    zero = torch.zeros(1, dtype=torch.bool, device=DEV)
    a = (fast & ~torch.cat([zero, fast[:-1]])).nonzero()[:, 0] + 1       # first fast step of each run
    b = (fast & ~torch.cat([fast[1:], zero])).nonzero()[:, 0] + 2        # first slow step after it
    s, e = a - 1, b - 1
    run_of = torch.cumsum((fast & ~torch.cat([zero, fast[:-1]])).int(), 0).long() - 1
    speed = (x[1:].to(F64) - x[:-1].to(F64)).abs() * hz
    peak = torch.zeros(a.numel(), dtype=F64, device=DEV).scatter_reduce_(0, run_of[fast], speed[fast], "amax")
    amp = (x[e].to(F64) - x[s].to(F64)).abs()
    dur = (e - s).to(F64) * 1000.0 / hz
    ws, we = s - 10, e + 40
    bad = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum((~valid).long(), 0)])
    ok = (dur.float() >= 6.0) & ((x[e] - x[s]).abs() >= 4.0) & (ws >= 0) & (we <= n - 1)
    ok &= bad[(we + 1).clamp(0, n)] == bad[ws.clamp(0, n)]
    cols = dict(onset=s, end=e, window_start=ws, n_samples=we - ws + 1, onset_index=s - ws, theta_start_deg=x[s].to(F64),
                theta_end_deg=x[e].to(F64), amplitude_deg=amp, duration_ms=dur, peak_velocity_dps=peak, reserved=0 * s)
    return {k: v[ok].cpu().numpy() for k, v in cols.items()}


def exact(case, seed):
    """None for the searches, the refinement and the training: the path they take depends on the rounding of every
    step before, so 64 bits give another path and not another rounding of this one."""
    kind = case["kind"]
    if kind == "simulate":
        rec = _simulate_recordings(case, seed)
        opc = _candidates(rec, case["per"], seed)
        args = tuple(v.repeat_interleave(case["per"], 0) for v in rec.args)
        out = _trajectories(opc.to(F64), *args)
        return out[torch.arange(out.shape[1], device=DEV)[None, :] < args[0][:, None]], None
    if kind == "score":
        rec = _score_recordings(case, seed)
        opc = _candidates(rec, case["m"], seed)
        out = _trajectories(opc.to(F64), *(v.expand(opc.shape[0]) for v in rec.args))
        return (out - rec.y.to(F64)).square().mean(1)
    if kind == "predict":
        rec = Recordings(case["n"], seed)
        y = _network(torch.as_tensor(_weights(), device=DEV).to(F64), _features(rec))
        return rec.nominal * (0.2 * y).exp()
    if kind == "detect":
        return _detected(_stream(case["samples"], case["hz"], seed), float(case["hz"]))
    return None
