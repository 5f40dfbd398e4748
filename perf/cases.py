"""What this library's users have it do, as cases that can be timed and checked.

A case names one use of a public entry point of ``paper_1811_09711_gb300.vamp``
and the sizes and options of the problem it is used on:

* ``run``     a whole adaptation run: the grid file of an unadapted problem is
              loaded, then every iteration samples, rebins and updates the
              channel weights;
* ``step``    one adaptation iteration on adapted grids, the state coming from
              and going back to pinned host buffers (what a driver program does
              that keeps the grids, or one that exchanges them between ranks);
* ``events``  unweighted events from adapted grids, into device memory;
* ``batch``   one iteration of many uneven problems in one launch, and their
              grids for the grid files;
* ``serve``   a burst of integrate-then-generate requests through the server;
* ``static``  one pass of the entry point that allocates nothing.

Problems are drawn as in ``problems.py`` (Breit-Wigner and power-law channels,
Dirichlet peak weights, Gaussian factors of width 0.2); their grids are adapted
here, in 64 bits by plain torch (:class:`_Method`), which also says what every
output is (:func:`exact`).  FP64 contexts hand on their results as they are;
FP32-eval contexts compute weights in single precision, so what they sum up to
is handed on in single precision.
"""
import math

import numpy as np
import torch

from paper_1811_09711_gb300 import problems as P
from paper_1811_09711_gb300 import vamp as V

GAUSS_SIGMA, GAUSS_CENTRE = 0.2, 0.5
GEN_BATCH = 1 << 20      # calls per generation batch (the library's default)
STEP_ITERATION = 3       # an iteration that does not enter the combination yet
LOOKUPS_EXACT = 2.5e10   # grid lookups that exact() does in a few seconds


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(kind, prec, d, k, n, calls, maps="bw", name=None, **kw):
    c = {"kind": kind, "prec": prec, "d": d, "k": k, "n": n, "calls": calls, "maps": maps, "iterations": 1,
         "same_peaks": True, "signed": False, "equiv": False, "smooth": False, "second_moment": False,
         "stratified": False, "events": 0, "problems": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the single-channel VEGAS problem, 5 x 1e4 calls from uniform grids: the smallest run there is
        _case("run", "fp64", 4, 1, 20, 10_000, "id", "run_gauss_d4_k1_fp64", iterations=5),
        # a few symmetric channels with equivalences and smoothed bin weights, 3e4 calls: a small call with options
        _case("step", "fp32", 6, 3, 20, 30_000, "ring", "step_ring_d6_k3_fp32", equiv=True, smooth=True),
        # Breit-Wigner x Gauss, six resonances, 1e6 calls: the ordinary iteration
        _case("step", "fp32", 8, 6, 50, 1_000_000, "bw", "step_bw_d8_k6_fp32"),
        # the same problem in FP64, three iterations enqueued without a host wait
        _case("run", "fp64", 8, 6, 50, 1_000_000, "bw", "run_bw_d8_k6_fp64", iterations=3),
        # the collider-like problem, 64 channels, 1e7 calls: the headline workload, in both precisions
        _case("step", "fp32", 14, 64, 100, 10_000_000, "mixed", "step_collider_d14_k64_fp32"),
        _case("step", "fp64", 14, 64, 100, 10_000_000, "mixed", "step_collider_d14_k64_fp64"),
        # pseudo-stratified VEGAS in few dimensions
        _case("step", "fp32", 4, 1, 20, 1_000_000, "id", "step_stratified_d4_fp32", stratified=True),
        # unweighted events from the adapted collider (FP32-eval) and from the resonances (FP64)
        _case("events", "fp32", 14, 64, 100, 1_000_000, "mixed", "events_collider_fp32", events=50_000),
        _case("events", "fp64", 8, 6, 50, 200_000, "bw", "events_bw_fp64", events=200_000),
        # 32 uneven problems advanced together (d 2..16, 1..64 channels, 1e4..1e7 calls: a parameter scan)
        _case("batch", "fp32", 0, 0, 0, 10_000_000, "bw", "batch_32_fp32", problems=32),
        # a burst of requests: adapt, then unweighted events, FP64
        _case("serve", "fp64", 0, 0, 0, 300_000, "bw", "serve_8_fp64", problems=8, iterations=3, events=5_000),
        # a pass for a caller that owns all device memory
        _case("static", "fp32", 8, 6, 50, 200_000, "bw", "static_bw_d8_k6_fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step", "run", "events", "batch", "serve", "static"], [10, 3, 4, 2, 1, 1])[0]
    prec = "fp64" if kind in ("run", "serve") else rng.choice(["fp32", "fp32", "fp64"])
    if kind in ("batch", "serve"):
        return _case(kind, prec, 0, 0, 0, _log_int(rng, 100_000, 3_000_000 if kind == "batch" else 300_000), "bw",
                     problems=rng.randint(3, 24 if kind == "batch" else 10), iterations=3 if kind == "serve" else 1,
                     events=_log_int(rng, 1_000, 10_000) if kind == "serve" else 0)
    d, n = rng.randint(2, 16), rng.randint(10, 120)
    k = _log_int(rng, 1, 64)
    maps = rng.choice(["bw", "bw", "mixed"]) if d >= 4 else "bw"
    c = _case(kind, prec, d, k, n, 0, maps)
    if kind in ("step", "run") and rng.random() < 0.15:
        c["maps"], c["k"], c["equiv"] = "ring", rng.randint(2, min(d, 8)), True
    elif rng.random() < 0.1:
        c["maps"], c["k"] = "id", 1
    if kind != "events":
        c["same_peaks"] = rng.random() < 0.85 or c["maps"] == "id"
        c["signed"] = c["k"] > 1 and not c["equiv"] and rng.random() < 0.15
    if kind in ("step", "run"):
        c["smooth"] = rng.random() < 0.2
        c["second_moment"] = rng.random() < 0.2
        c["stratified"] = d <= 8 and rng.random() < 0.2
        c["iterations"] = rng.randint(2, 5) if kind == "run" else 1
    if kind == "events":
        c["calls"] = 200_000 if c["k"] * c["d"] < 200 else 1_000_000
        c["events"] = _log_int(rng, 1_000, 50_000 if prec == "fp32" else 200_000)
        return c
    # at most the work of the largest listed case, and of its calls in single precision
    most = 1e7 * _call_ops(14, 64, 3) / (_call_ops(c["d"], c["k"], 3) * c["iterations"])
    c["calls"] = _log_int(rng, 10_000, max(20_000, min(1e7, 0.8 * most)))
    if kind == "static":
        c["calls"] = min(c["calls"], 1_000_000)
    return c


def _call_ops(d, k, mapped):
    """Operations of one call: lookups of every channel, inverse maps, channel terms, forward map, random words."""
    return 8 * k * d + 15 * mapped * k + 7 * k + 8 * d + 60 * -(-d // 4) + 10


def _sub_cases(case):
    """The problems of a batch or of a burst of requests, drawn as uneven instances (their sizes from the case alone)."""
    rng = np.random.default_rng(5000 + case["problems"])
    out = []
    for _ in range(case["problems"]):
        d = int(rng.integers(2, 17))
        k = max(1, int(round(math.exp(rng.uniform(0.0, math.log(64.0))))))
        calls = int(round(math.exp(rng.uniform(math.log(1e4), math.log(case["calls"])))))
        events = int(round(math.exp(rng.uniform(math.log(1e3), math.log(max(1e3, case["events"]))))))
        out.append(_case("step", case["prec"], d, k, int(rng.choice([20, 50, 100])), calls, "bw",
                         events=events if case["events"] else 0, iterations=case["iterations"]))
    return out


def work(case):
    subs = _sub_cases(case) if case["problems"] > 1 else [case]
    byt = flops = 0.0
    for c in subs:
        d, k, n = c["d"], c["k"], c["n"]
        ops = _call_ops(d, k, {"id": 0, "bw": 1, "ring": 1, "mixed": 3}[c["maps"]])
        state = 8 * (k * d * (n + 1) + 2 * k)
        rec = 8 * ((4 * d + 7) // 8) + 8
        if case["kind"] == "events":
            calls = c["events"]  # every call an event at best
        else:
            calls = c["calls"] * c["iterations"]
        flops += calls * ops
        byt += 2 * state + c["events"] * rec + 64 * c["iterations"]
        if case["kind"] == "static":
            byt += 8 * k * d * n - state
    return {"bytes": byt, "flops": flops}


# ---------------------------------------------------------------------------
# problems, drawn from the seed
# ---------------------------------------------------------------------------
def _problem(case, seed):
    rng = np.random.default_rng(seed)
    d, k = case["d"], case["k"]
    ms = P.MapSet.identity(k)
    if case["maps"] == "ring":
        ms.n_mapped[:] = 1
        ms.coord[:, 0] = np.arange(k)
        ms.kind[:, 0] = P.MAP_BW
        ms.a[:, 0] = 0.5
        ms.b[:, 0] = math.exp(rng.uniform(math.log(1e-3), math.log(1e-2)))
    elif case["maps"] == "bw":
        ms.n_mapped[:] = 1
        ms.coord[:, 0] = rng.integers(0, d, size=k) if k > d else rng.choice(d, size=k, replace=False)
        ms.kind[:, 0] = P.MAP_BW
        ms.a[:, 0] = rng.uniform(0.2, 0.8, size=k)
        ms.b[:, 0] = np.exp(rng.uniform(math.log(1e-3), math.log(1e-2), size=k))
    elif case["maps"] == "mixed":
        for c in range(k):
            nm = 2 + c % 3
            ms.n_mapped[c] = nm
            ms.coord[c, :nm] = rng.choice(d, size=nm, replace=False)
            for s in range(nm):
                bw = rng.uniform() < 0.5
                ms.kind[c, s] = P.MAP_BW if bw else P.MAP_POW
                ms.a[c, s] = rng.uniform(0.2, 0.8) if bw else 0.0
                ms.b[c, s] = math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))
    peaks = ms.copy()
    if not case["same_peaks"]:  # resonances a little beside and wider than the channels'
        bw = peaks.kind == P.MAP_BW
        peaks.a[bw] += 0.5 * peaks.b[bw]
        peaks.b[bw] *= 1.5
    w = rng.exponential(1.0, size=k)
    w = w / w.sum()
    if case["maps"] == "ring":
        w[:] = 1.0 / k
    if case["signed"]:
        w[-1] *= -0.3
    sigma, norm = (0.1, P.GAUSS_NORM_REAL_LINE) if case["maps"] == "id" else (GAUSS_SIGMA, P.GAUSS_NORM_UNIT)
    return P.Problem(
        name="drawn", d=d, n_bins=case["n"], channels=ms, peak_weight=w, peaks=peaks, gauss_sigma=sigma,
        gauss_centre=GAUSS_CENTRE, gauss_norm=norm, seed=int(rng.integers(0, 2**63)),
        request_id=int(rng.integers(0, 2**31)), smooth=int(case["smooth"]), omega_mode=int(case["second_moment"]),
        gen_batch=GEN_BATCH, iterations=case["iterations"], calls=case["calls"],
        combine_from=1 if case["kind"] == "run" else STEP_ITERATION + 1, n_events=case["events"],
        stratified=int(case["stratified"]), equivalences=P.rotation_equivalences(k, d) if case["equiv"] else None)


# ---------------------------------------------------------------------------
# the method in 64 bits, in plain torch: adapts the grids that cases start
# from, and says what their outputs are
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _mul32(a, x):
    """High and low 32 bits of a 32-bit constant times 32-bit words held in int64."""
    hi = (a * (x >> 16) + ((a * (x & 0xFFFF)) >> 16)) >> 16
    return hi & _M32, (a * x) & _M32


def _philox(call, block, field, request, key):
    x, y = call & _M32, torch.full_like(call, block)
    z, w = torch.full_like(call, field), torch.full_like(call, request)
    k0, k1 = key & _M32, (key >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        h0, l0 = _mul32(0xD2511F53, x)
        h1, l1 = _mul32(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
    return x, y, z, w


class _Method:
    """One problem's adaptation state and steps (§3 of the paper), FP64 on the GPU."""

    CHUNK = 1 << 18  # calls evaluated together

    def __init__(self, pr):
        self.pr, self.dev = pr, "cuda"
        self.d, self.K, self.n = pr.d, pr.n_channels, pr.n_bins
        t = {"dtype": torch.float64, "device": self.dev}
        uniform = torch.tensor([j / self.n for j in range(self.n + 1)], **t)
        self.edges = uniform.repeat(self.K, self.d, 1).contiguous()
        self.alpha = torch.full((self.K,), 1.0 / self.K, **t)
        self.shift = torch.zeros(self.K, **t)
        self.w_max, self.history = 0.0, []
        s, c = pr.gauss_sigma, pr.gauss_centre
        if pr.gauss_norm == P.GAUSS_NORM_REAL_LINE:
            self.z = s * math.sqrt(2 * math.pi)
        else:
            self.z = s * math.sqrt(math.pi / 2) * (math.erf((1 - c) / (s * math.sqrt(2)))
                                                   + math.erf(c / (s * math.sqrt(2))))

    # -- one call ---------------------------------------------------------
    @staticmethod
    def _bw(m, g):
        t0 = math.atan(m / g)
        return t0, math.atan((1 - m) / g) + t0

    def _words(self, call, field, nw):
        out = []
        for b in range(-(-nw // 4)):
            out += _philox(call, b, field, self.pr.request_id, self.pr.seed)
        return out[:nw]

    def _evaluate(self, ch, groups, words, digits=None, nr=None):
        """p, f, g and forward bins of the calls with channels ch; groups: (channel, where its calls are)."""
        d, K, n, pr = self.d, self.K, self.n, self.pr
        flat, N = self.edges.view(-1), ch.shape[0]
        x, jf = [], []
        own = torch.ones(N, dtype=torch.float64, device=self.dev)
        for k in range(d):
            if digits is None:
                t = (2 * words[k] + 1) * n
                j, fr = t >> 33, (t & ((1 << 33) - 1)).double() * 2.0**-33
            else:
                den = nr << 33
                t = ((digits[k] << 33) + 2 * words[k] + 1) * n
                j = torch.div(t, den, rounding_mode="floor")
                fr = (t - j * den).double() / den.double()
            at = (ch * d + k) * (n + 1) + j
            e0, e1 = flat[at], flat[at + 1]
            x.append(e0 + fr * (e1 - e0))
            jf.append(j)
            own /= n * (e1 - e0)
        p = [v.clone() for v in x]
        ms = pr.channels
        for c, sel in groups:
            for s in range(int(ms.n_mapped[c])):
                k, m, g = int(ms.coord[c, s]), float(ms.a[c, s]), float(ms.b[c, s])
                v = x[k][sel]
                if ms.kind[c, s] == P.MAP_BW:
                    t0, A = self._bw(m, g)
                    v = m + g * torch.tan(A * v - t0)
                    jac = (g / A) / ((v - m) ** 2 + g * g)
                else:
                    jac = 1.0 / (5.0 * v**4)
                    v = (v**5).clamp_min(np.finfo(np.float64).tiny)
                p[k][sel] = v
                own[sel] *= jac
        # densities of every channel at its own coordinates (Eq. 30)
        g_c = torch.ones(K, N, dtype=torch.float64, device=self.dev)
        for k in range(d):
            xs = p[k].repeat(K, 1)
            for c in range(K):
                for s in range(int(ms.n_mapped[c])):
                    if int(ms.coord[c, s]) == k:
                        m, g = float(ms.a[c, s]), float(ms.b[c, s])
                        if ms.kind[c, s] == P.MAP_BW:
                            t0, A = self._bw(m, g)
                            xs[c] = (torch.atan((p[k] - m) / g) + t0) / A
                            g_c[c] *= (g / A) / ((p[k] - m) ** 2 + g * g)
                        else:
                            xs[c] = p[k] ** 0.2
                            g_c[c] *= 0.2 * p[k] ** -0.8
            e = self.edges[:, k, :].contiguous()
            dens = 1.0 / (n * (e[:, 1:] - e[:, :-1]))
            j = (torch.searchsorted(e, xs, right=True) - 1).clamp_(0, n - 1)
            g_c *= torch.gather(dens, 1, j)
        g_c.scatter_(0, ch[None, :], own[None, :])
        gsum = (self.alpha[:, None] * g_c).sum(0)
        # the integrand's peaks
        f = torch.zeros(N, dtype=torch.float64, device=self.dev)
        gauss = [torch.exp(-((v - pr.gauss_centre) ** 2) / (2 * pr.gauss_sigma**2)) / self.z for v in p]
        pk = pr.peaks
        for q in range(pr.n_peaks):
            t = torch.full((N,), float(pr.peak_weight[q]), dtype=torch.float64, device=self.dev)
            mapped = {int(pk.coord[q, s]): s for s in range(int(pk.n_mapped[q]))}
            for k in range(d):
                if k not in mapped:
                    t *= gauss[k]
                    continue
                m, g = float(pk.a[q, mapped[k]]), float(pk.b[q, mapped[k]])
                if pk.kind[q, mapped[k]] == P.MAP_BW:
                    t *= (g / self._bw(m, g)[1]) / ((p[k] - m) ** 2 + g * g)
                else:
                    t *= (p[k] + g) ** -0.8 / (5.0 * ((1 + g) ** 0.2 - g**0.2))
            f += t
        return p, f, gsum, jf

    # -- one pass ------------------------------------------------------------
    def _allocate(self, calls):
        """Calls, cells per axis, calls per cell of every channel."""
        out = []
        for a in self.alpha.tolist():
            nc = max(self.pr.n_min, math.floor(a * calls)) if a > 0 else 0
            m, s = 1, nc
            if self.pr.stratified and nc >= 2:
                m = max(1, int((nc / 2) ** (1.0 / self.d)) - 1)
                while 2 * (m + 1) ** self.d <= nc:
                    m += 1
                s = nc // m**self.d
                nc = s * m**self.d
            out.append((nc, m, s))
        return out

    def sample(self, calls, iteration):
        d, K, n, pr, strat = self.d, self.K, self.n, self.pr, bool(self.pr.stratified)
        self.Nc = self._allocate(calls)
        nc, axis, per_cell = torch.tensor(self.Nc, device=self.dev).T
        ends = np.cumsum([v[0] for v in self.Nc])
        first, total = nc.cumsum(0) - nc, int(ends[-1])
        cell0 = (axis**d).cumsum(0) - axis**d
        cells = torch.zeros(int(cell0[-1] + axis[-1] ** d) if strat else 0, dtype=torch.float64, device=self.dev)
        D = torch.zeros(K * d * n, dtype=torch.float64, device=self.dev)
        s1, s2 = torch.zeros(2, K, dtype=torch.float64, device=self.dev)
        wm = 0.0
        for a in range(0, total, self.CHUNK):
            call = torch.arange(a, min(total, a + self.CHUNK), device=self.dev)
            ch = torch.searchsorted(nc.cumsum(0), call, right=True)
            lo, hi = np.searchsorted(ends, [a, a + call.shape[0] - 1], side="right")
            groups = [(c, slice(max(0, int(ends[c] - self.Nc[c][0]) - a), int(ends[c]) - a))
                      for c in range(lo, hi + 1) if self.Nc[c][0]]
            digits = None
            if strat:
                m = axis[ch]
                cell = torch.div(call - first[ch], per_cell[ch], rounding_mode="floor")
                digits = [torch.div(cell, m**k, rounding_mode="floor") % m for k in range(d)]
            p, f, g, jf = self._evaluate(ch, groups, self._words(call, iteration, d), digits, axis[ch])
            w = f / g
            dv = w - self.shift[ch]
            s1 += torch.bincount(ch, weights=dv, minlength=K)
            s2 += torch.bincount(ch, weights=dv * dv, minlength=K)
            wm = max(wm, float(w.abs().max()))
            for k in range(d):
                D += torch.bincount((ch * d + k) * n + jf[k], weights=w * w, minlength=K * d * n)
            if strat:
                cells += torch.bincount(cell0[ch] + cell, weights=dv, minlength=cells.shape[0])
        self.D = D.view(K, d, n)
        self.Ic, self.Vc, self.Wc = [0.0] * K, [0.0] * K, [0.0] * K
        shifts, s1, s2 = self.shift.tolist(), s1.tolist(), s2.tolist()
        for c, (nc, m, s) in enumerate(self.Nc):
            if nc == 0:
                shifts[c] = 0.0
                continue
            m1, m2 = s1[c] / nc, s2[c] / nc
            self.Ic[c] = shifts[c] + m1
            if strat:
                q = cells[int(cell0[c]):int(cell0[c]) + m**d]
                self.Vc[c] = max(0.0, (s2[c] - float((q * q).sum()) / s) / (m**d * (s - 1.0))) if s >= 2 else 0.0
            elif nc > 1:
                self.Vc[c] = max(0.0, (m2 - m1 * m1) * nc / (nc - 1.0))
            self.Wc[c] = (m2 - m1 * m1) + self.Ic[c] ** 2
            shifts[c] = self.Ic[c]
        self.shift = torch.tensor(shifts, dtype=torch.float64, device=self.dev)
        al, live = self.alpha.tolist(), [c for c in range(K) if self.Nc[c][0]]
        I = sum(al[c] * self.Ic[c] for c in live)
        var = sum(al[c] ** 2 * self.Vc[c] / self.Nc[c][0] for c in live)
        self.w_max = wm
        if iteration >= pr.combine_from:
            self.history.append((I, var))
        comb, sig, chi = self._combine()
        return {"integral": I, "variance": var, "w_max": wm, "efficiency": I / wm if wm else 0.0, "n_calls": total,
                "combined": comb, "combined_sigma": sig, "chi2_dof": chi}

    def _combine(self):
        h = self.history
        if not h:
            return 0.0, 0.0, 0.0
        if any(v <= 0 for _, v in h):
            z = [i for i, v in h if v <= 0]
            return sum(z) / len(z), 0.0, 0.0
        sw = sum(1 / v for _, v in h)
        c = sum(i / v for i, v in h) / sw
        chi = sum((i - c) ** 2 / v for i, v in h) / (len(h) - 1) if len(h) > 1 else 0.0
        return c, math.sqrt(1 / sw), chi

    # -- adaptation -------------------------------------------------------------
    def refine(self):
        d, K, n, pr = self.d, self.K, self.n, self.pr
        D = self.D.clone()
        for r in (pr.equivalences if pr.equivalences is not None else []):
            for k in range(d):
                D[r[0], k] += self.D[r[1], r[2 + k]]  # identity kind
        if pr.smooth and n >= 2:
            S = D.clone()
            S[..., 1:-1] = (D[..., :-2] + D[..., 1:-1] + D[..., 2:]) / 3.0
            S[..., 0], S[..., -1] = (D[..., 0] + D[..., 1]) / 2.0, (D[..., -2] + D[..., -1]) / 2.0
            D = S
        om = D.sqrt().view(K * d, n)
        tot = om.sum(1, keepdim=True)
        r = om / tot.clamp_min(1e-300)
        safe = r.clamp(1e-300, 1 - 1e-13)
        m = ((safe - 1) / torch.log(safe)) ** pr.grid_alpha
        m = torch.where(r == 0, torch.zeros_like(m), torch.where((r - 1).abs() < 1e-12, torch.ones_like(m), m))
        C = torch.zeros(K * d, n + 1, dtype=torch.float64, device=self.dev)
        C[:, 1:] = m.cumsum(1)
        M = C[:, -1:]
        t = torch.arange(1, n, device=self.dev).double()[None, :] * M / n
        j = torch.searchsorted(C[:, 1:].contiguous(), t.contiguous()).clamp_(0, n - 1)
        e = self.edges.view(K * d, n + 1)
        lo, hi = torch.gather(e, 1, j), torch.gather(e, 1, j + 1)
        new = e.clone()
        new[:, 1:-1] = lo + (t - torch.gather(C, 1, j)) / torch.gather(m, 1, j) * (hi - lo)
        keep = (tot > 0) & (M > 0)
        self.edges = torch.where(keep, new, e).view(K, d, n + 1).contiguous()

    def update_alpha(self):
        al, om = self.alpha.tolist(), self.Wc if self.pr.omega_mode else self.Vc
        live = [al[c] > 0 and self.Nc[c][0] > 0 and om[c] > 0 for c in range(self.K)]
        u = [al[c] * om[c] ** self.pr.beta if live[c] else 0.0 for c in range(self.K)]
        su, mu = math.fsum(u), math.fsum(a for a, l in zip(al, live) if l)
        new = []
        for c in range(self.K):
            a = al[c]
            if a > 0 and self.Nc[c][0] > 0:
                a = u[c] / su * mu if live[c] else (0.0 if self.Ic[c] == 0.0 else a)
            new.append(a)
        tot = math.fsum(new)
        self.alpha = torch.tensor([a / tot for a in new] if tot > 0 else al, dtype=torch.float64, device=self.dev)

    def iterate(self, calls, iteration):
        r = self.sample(calls, iteration)
        self.refine()
        self.update_alpha()
        return r

    # -- unweighted events ----------------------------------------------------------
    def generate(self, n_events):
        pr, d = self.pr, self.d
        A = torch.cumsum(self.alpha, 0)
        ps, ws, n, used, over, batch = [], [], 0, 0, 0, 0
        while n < n_events:
            bmax, field = 0.0, 0x80000000 | batch
            for a in range(0, pr.gen_batch, self.CHUNK):
                call = torch.arange(a, min(pr.gen_batch, a + self.CHUNK), device=self.dev)
                words = self._words(call, field, d + 2)
                u = [(w.double() + 0.5) * 2.0**-32 for w in words[d:]]
                ch = torch.searchsorted(A, u[0] * A[-1], right=True).clamp_max(self.K - 1)
                p, f, g, _ = self._evaluate(ch, [(c, (ch == c).nonzero()[:, 0]) for c in range(self.K)], words[:d])
                w = f / g
                bmax = max(bmax, float(w.abs().max()))
                at = (u[1] * self.w_max < w.abs()).nonzero()[:, 0][: n_events - n]
                ps.append(torch.stack([v[at] for v in p], 1))
                ws.append(w[at])
                over += int((ws[-1].abs() > self.w_max).sum())
                n += int(at.shape[0])
                if n >= n_events:
                    used += a + int(at[-1]) + 1
                    break
            else:
                used += pr.gen_batch
            self.w_max, batch = max(self.w_max, bmax), batch + 1
        return torch.cat(ps), torch.cat(ws), {"n_written": n, "n_calls_used": used, "n_overweight": over}

    def state(self):
        return {"edges": self.edges.cpu().numpy(), "alpha": self.alpha.cpu().numpy(),
                "shift": self.shift.cpu().numpy(), "w_max": self.w_max}


def _adapted(pr, calls, iterations=3):
    """The problem's grids, weights and shifts after some iterations, on streams that no case samples from."""
    m = _Method(pr)
    for it in range(iterations):
        m.iterate(calls, 1000 + it)
    m.history.clear()
    return m


def _started(pr, case):
    """The grids a case starts from; events want them well adapted (a poor unweighting efficiency is no use to anyone)."""
    if case["kind"] == "events":
        return _adapted(pr, case["calls"], 6)
    return _adapted(pr, min(case["calls"], 100_000))


# ---------------------------------------------------------------------------
# what a program has in hand, and the pass
# ---------------------------------------------------------------------------
RESULT = ("integral", "variance", "w_max", "efficiency", "combined", "combined_sigma", "chi2_dof")
#: the order in which an asynchronous pass writes them
ROW = ("integral", "variance", "w_max", "efficiency", "n_calls", "combined", "combined_sigma", "chi2_dof")


def _prec(case):
    return V.PREC_FP64 if case["prec"] == "fp64" else V.PREC_FP32_EVAL


def _np_type(case):
    return np.float64 if case["prec"] == "fp64" else np.float32


def _results(rs, case):
    """Pass results (objects or dicts), one array per quantity."""
    get = (lambda r, k: r[k]) if isinstance(rs[0], dict) else getattr
    out = {k: np.array([get(r, k) for r in rs], _np_type(case)) for k in RESULT}
    out["n_calls"] = np.array([get(r, "n_calls") for r in rs], np.int64)
    return out


def _rows(out):
    """The quantities of asynchronous passes, as views of what they wrote."""
    return {k: out[:, i] for i, k in enumerate(ROW)}


def _state(st, case):
    t = _np_type(case)
    return {"edges": np.array(st["edges"], t), "alpha": np.array(st["alpha"], t), "shift": np.array(st["shift"], t),
            "w_max": np.array(st["w_max"], t)}


def _joined(states, case):
    """The states of many problems, end to end (the grid files of an iteration)."""
    return {k: np.concatenate([np.ravel(s[k]) for s in states]).astype(_np_type(case)) for k in states[0]}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        prs = [_problem(c, seed * 64 + i) for i, c in enumerate(_sub_cases(case))]
        b = V.Batch(prs, precision=_prec(case))
        calls = [p.calls for p in prs]
        b.iterate(calls, 0)  # the first iteration: it also picks the launch shape
        return {"case": case, "batch": b, "calls": calls, "it": 0}
    if kind == "serve":
        prs = [_problem(c, seed * 64 + i) for i, c in enumerate(_sub_cases(case))]
        srv = V.Server(max_slots=16, mem_budget_bytes=8 << 30, precision=_prec(case))
        recs = [torch.zeros(p.n_events, V.record_bytes(p.d), dtype=torch.uint8, device="cuda") for p in prs]
        states = [torch.zeros(p.n_channels * p.d * (p.n_bins + 1) + 2 * p.n_channels, dtype=torch.float64,
                              device="cuda") for p in prs]
        return {"case": case, "server": srv, "problems": prs, "records": recs, "states": states}
    pr = _problem(case, seed)
    if kind == "run":
        g = V.Vamp(pr, precision=_prec(case), stream=torch.cuda.current_stream())
        out = torch.zeros(case["iterations"], 9, dtype=torch.float64, device="cuda")
        return {"case": case, "vamp": g, "blob": g.checkpoint(), "out": out}
    m = _started(pr, case)
    if kind == "static":
        return {"case": case, "problem": pr, "edges": m.edges, "alpha": m.alpha, "shift": m.shift,
                "D": torch.zeros(pr.n_channels, pr.d, pr.n_bins, dtype=torch.float64, device="cuda")}
    g = V.Vamp(pr, precision=_prec(case), stream=torch.cuda.current_stream())
    st = m.state()
    if kind == "events":
        g.set_state(st["edges"], st["alpha"], st["shift"], st["w_max"])
        g.sample_pass(case["calls"], 2000)  # the last integration pass: it sets w_max
        rec = torch.zeros(case["events"], V.record_bytes(pr.d), dtype=torch.uint8, device="cuda")
        return {"case": case, "vamp": g, "records": rec}

    def pinned(a):
        t = torch.empty(a.shape, dtype=torch.float64, pin_memory=True)
        t.numpy()[...] = a
        return t.numpy()

    start = {k: pinned(st[k]) for k in ("edges", "alpha", "shift")}
    end = {k: pinned(st[k]) for k in start}
    return {"case": case, "vamp": g, "start": start, "end": end, "w_max": st["w_max"]}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        s["it"] = s["it"] % 3 + 1  # iterations 1, 2, 3 and again: none enters the combination yet
        rs = s["batch"].iterate(s["calls"], s["it"])
        return {"result": _results(rs, case), "state": _joined([s["batch"].get_state(i) for i in range(len(rs))], case)}
    if kind == "serve":
        return _run_serve(s)
    if kind == "static":
        pr = s["problem"]
        r = V.sample_pass_static(pr, _prec(case), s["edges"].data_ptr(), s["alpha"].data_ptr(), s["shift"].data_ptr(),
                                 case["calls"], STEP_ITERATION, stream=torch.cuda.current_stream().cuda_stream,
                                 D_out_ptr=s["D"].data_ptr())
        return {"result": _results([r], case), "D": s["D"] if case["prec"] == "fp64" else s["D"].float()}
    g = s["vamp"]
    if kind == "events":
        st = g.generate(case["events"], s["records"].data_ptr())
        return {"stats": st, **_events(s["records"], g.d, case)}
    if kind == "run":
        g.restore(s["blob"])
        if case["calls"] <= 100_000:  # small passes: the program looks at every result
            rs = []
            for it in range(case["iterations"]):
                rs.append(g.sample_pass(case["calls"], it))
                g.refine_grids()
                g.update_alpha()
            return {"result": _results(rs, case), "state": _state(g.get_state(), case)}
        for it in range(case["iterations"]):
            g.sample_pass_async(case["calls"], it, s["out"][it].data_ptr())
            g.refine_grids()
            g.update_alpha()
        return {"result": _rows(s["out"]), "state": _state(g.get_state(), case)}
    g.set_state(s["start"]["edges"], s["start"]["alpha"], s["start"]["shift"], s["w_max"])
    r = g.sample_pass(case["calls"], STEP_ITERATION)
    g.refine_grids()
    g.update_alpha()
    return {"result": _results([r], case), "state": _state(g.get_state(out=s["end"]), case)}


def _events(rec, d, case):
    w = rec[:, -8:].view(torch.float64)[:, 0]
    return {"p": rec[:, : 4 * d].view(torch.float32), "w": w if case["prec"] == "fp64" else w.float()}


def _run_serve(s):
    case, srv = s["case"], s["server"]
    ids = [srv.submit(p, p.iterations, p.calls, p.n_events, rec.data_ptr(), state_ptr=st.data_ptr())
           for p, rec, st in zip(s["problems"], s["records"], s["states"])]
    srv.wait_idle()
    got = {r.id: r for r in srv.poll()}
    rs = [got[i] for i in ids]
    return {"result": _results([r.result for r in rs], case), "state": s["states"],
            "used": np.array([r.events_calls_used for r in rs], np.int64),
            "over": np.array([r.events_overweight for r in rs], np.int64),
            "events": [_events(rec, p.d, case) for rec, p in zip(s["records"], s["problems"])]}


# ---------------------------------------------------------------------------
# the outputs in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind, wide = case["kind"], dict(case, prec="fp64")
    subs = _sub_cases(case) if case["problems"] > 1 else [case]
    passes = {"batch": 2, "run": case["iterations"], "serve": case["iterations"]}.get(kind, 1)
    if sum(c["calls"] * c["k"] * c["d"] * passes for c in subs) > LOOKUPS_EXACT:
        return None
    if kind == "batch":
        rs, states = [], []
        for i, c in enumerate(subs):
            m = _Method(_problem(c, seed * 64 + i))
            m.iterate(c["calls"], 0)
            rs.append(m.iterate(c["calls"], 1))
            states.append(m.state())
        return {"result": _results(rs, wide), "state": _joined(states, wide)}
    if kind == "serve":
        rs, states, used, over, evs = [], [], [], [], []
        for i, c in enumerate(subs):
            m = _Method(_problem(c, seed * 64 + i))
            for it in range(c["iterations"]):
                r = m.iterate(c["calls"], it)
            rs.append(r)
            states.append(torch.cat([m.edges.reshape(-1), m.alpha, m.shift]))
            p, w, st = m.generate(c["events"])
            used.append(st["n_calls_used"])
            over.append(st["n_overweight"])
            evs.append({"p": p.float(), "w": w})
        return {"result": _results(rs, wide), "state": states, "used": np.array(used, np.int64),
                "over": np.array(over, np.int64), "events": evs}
    pr = _problem(case, seed)
    if kind == "run":
        m = _Method(pr)
        rs = [m.iterate(case["calls"], it) for it in range(case["iterations"])]
        if case["calls"] <= 100_000:
            return {"result": _results(rs, wide), "state": _state(m.state(), wide)}
        rows = torch.tensor([[float(r[k]) for k in ROW] for r in rs], dtype=torch.float64)
        return {"result": _rows(rows), "state": _state(m.state(), wide)}
    m = _started(pr, case)
    if kind == "static":
        return {"result": {k: (np.zeros(1) if k in RESULT[4:] else v) for k, v in
                           _results([m.sample(case["calls"], STEP_ITERATION)], wide).items()}, "D": m.D}
    if kind == "events":
        if case["prec"] != "fp64":
            return None  # which calls are accepted is a decision of the single-precision weights
        m.sample(case["calls"], 2000)
        p, w, st = m.generate(case["events"])
        return {"stats": st, "p": p.float(), "w": w}
    r = m.iterate(case["calls"], STEP_ITERATION)
    return {"result": _results([r], wide), "state": _state(m.state(), wide)}
