"""What the library's speed is judged by: calls that its users make, over the sizes they make them at.

listed() gives the cases, draw(rng) further ones of the same ranges, prepare(case, seed) what a program holds
before the call (a context, inputs on the device or on the host), run(state) one pass through the public entry
points, work(case) the bytes and operations that such a pass cannot do without, exact(case, seed) the same
outputs in 64 bits by plain torch.

Kinds of pass:
  job       nodes, all frequency solves, window spectra and samples of one obstacle (one whole simulation)
  batch     the same for several star obstacles solved together in one context
  serve     two admitted batches in turn on one serving context: solve, first query, queries on resident fields
  query     one query at a few times on resident target fields, host buffers
  times     many times on resident target fields, device buffers
  sample    a new signal and new targets on resident densities (spectra, target fields, synthesis)
  static    the synthesis without allocation
  split     the synthesis with the low-frequency split
  conv      the scaled convolution for equispaced times
"""
import json
import math
import os

import numpy as np
import torch

from paper_1807_02718_gb300 import fh

PREC = {"fp64": fh.FH_FP64, "fp32": fh.FH_MIXED_FP32, "tf32": fh.FH_MIXED_TF32, "bf16": fh.FH_MIXED_BF16}
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
T0, H, SHIFT = -10.0, 10.0, 9.0


def listed():
    return [
        # the plain method's first configuration: a circle with a closed-form solution, 16 receivers
        dict(name="circle64_fp64", kind="job", curve="circle", prec="fp64", io="host", J=64, W=16.0, N=256,
             n_x=16, n_T=200, t_far=20.0, pulses=1, span=0.0, dt=0.01),
        # one long-signal simulation of the kite in plain FP64, the accuracy reference of every user
        dict(name="kite256_fp64", kind="job", curve="kite", prec="fp64", io="dev", J=256, W=40.0, N=0,
             n_x=1024, n_T=4096, t_far=1e4, pulses=40, span=400.0, dt=0.01),
        # the same simulation in the default mixed precision
        dict(name="kite256_bf16", kind="job", curve="kite", prec="bf16", io="dev", J=256, W=40.0, N=0,
             n_x=1024, n_T=4096, t_far=1e4, pulses=40, span=400.0, dt=0.01),
        # the wide-band simulation (the benchmark's default workload): N up to 1920
        dict(name="kite512_wide_bf16", kind="job", curve="kite", prec="bf16", io="dev", J=512, W=160.0, N=0,
             n_x=1024, n_T=4096, t_far=1e4, pulses=40, span=400.0, dt=0.005),
        # a design sweep: many star obstacles solved as one batch, TF32 factorisations
        dict(name="stars16_tf32", kind="batch", prec="tf32", P=16, J=128, W_lo=20.0, W_hi=100.0, n_x=256, n_T=512,
             t_far=1e4, pulses=5, span=60.0, dt=0.01),
        # a serving slot: uneven requests admitted in twos, every one a new obstacle
        dict(name="serve_bf16", kind="serve", prec="bf16", P=2, J=128, W_lo=10.0, W_hi=120.0, n_x=800, n_T=16,
             queries=4, t_far=1e4, pulses=5, span=60.0, dt=0.01),
        # a later query of a served request: the smallest call, latency only
        dict(name="query16_bf16", kind="query", curve="star", prec="bf16", J=128, W=60.0, n_x=777, n_T=16,
             t_far=1e4, pulses=5, span=60.0, dt=0.01),
        # a time series at all receivers on resident fields
        dict(name="times4096_bf16", kind="times", curve="kite", prec="bf16", J=256, W=40.0, n_x=1024, n_T=4096,
             t_far=1e4, pulses=40, span=400.0, dt=0.01),
        # another signal and receiver set for a solved obstacle, plain FP64, ragged sizes
        dict(name="sample_fp64", kind="sample", curve="kite", prec="fp64", J=201, W=30.0, n_x=333, n_T=1001,
             t_far=2e3, pulses=12, span=120.0, dt=0.01),
        # the split synthesis of the 256-frequency kite, the option for late-time accuracy in 2D
        dict(name="split256", kind="split", J=256, W=40.0, j_c=5, n_x=1024, n_T=4096, t_far=1e4, pulses=40,
             span=400.0, dt=0.01),
        # time traces on an equispaced grid for a set of receivers and windows
        dict(name="conv_64x16384", kind="conv", M=1000, L=16384, batch=64, dt=0.2),
        # one very long trace, not a power of two
        dict(name="conv_1x1e6", kind="conv", M=5000, L=1000000, batch=1, dt=0.2),
    ]


def _logi(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["job", "job", "job", "batch", "serve", "query", "times", "sample", "static", "split", "conv"])
    sig = dict(pulses=rng.randint(1, 40), span=round(rng.uniform(0.0, 400.0)) * 1.0, dt=0.01)
    if kind == "conv":
        M = 2 * _logi(rng, 5, 2500)
        batch = _logi(rng, 1, 128)
        L = 2 * _logi(rng, max(M, 64) // 2, max(M, min(500000, 600000 // batch)))
        return dict(kind=kind, M=M, L=max(L, M), batch=batch, dt=rng.choice([0.05, 0.2, 0.5]))
    if kind == "split":
        j_c = rng.randint(3, 8)
        n = 2 * _logi(rng, 10, 125) + 1
        return dict(kind=kind, J=n + j_c, W=round(rng.uniform(5, 40), 2), j_c=j_c, n_x=_logi(rng, 4, 1024),
                    n_T=_logi(rng, 16, 4096), t_far=float(_logi(rng, 50, 10000)), **sig)
    if kind == "static":
        J = _logi(rng, 24, 512)
        return dict(kind=kind, J=J, W=round(rng.uniform(5, 40), 2), n_x=_logi(rng, 2, 1024),
                    n_T=_logi(rng, 8, min(2048, 524288 // J)), t_far=float(_logi(rng, 50, 10000)), **sig)
    if kind in ("batch", "serve"):
        W = rng.uniform(10, 60)
        serve = kind == "serve"
        return dict(kind=kind, prec=rng.choice(["bf16", "bf16", "tf32"]), P=rng.randint(1, 4) if serve else rng.randint(2, 16),
                    J=_logi(rng, 32, 128), W_lo=round(W, 2), W_hi=round(W * rng.uniform(1, 2), 2),
                    n_x=_logi(rng, 16, 2048) if serve else _logi(rng, 16, 512), n_T=16 if serve else _logi(rng, 16, 1024),
                    t_far=1e4, pulses=rng.randint(2, 8), span=60.0, dt=0.01, **(dict(queries=rng.randint(1, 8)) if serve else {}))
    prec = rng.choice(["bf16", "bf16", "tf32", "fp32", "fp64"])
    slow = prec in ("fp64", "fp32")
    J = _logi(rng, 16, 256 if slow else 512)
    W = (J - 1) * rng.uniform(0.1, 0.5)     # frequency steps that resolve windows of width 2H = 20
    c = dict(kind=kind, curve=rng.choice(["kite", "star", "circle"]), prec=prec, J=J,
             W=round(min(W, 25.0 if slow else 100.0), 2),
             n_x=_logi(rng, 3, 1024), n_T=_logi(rng, 5, 4096), t_far=float(_logi(rng, 50, 10000)), **sig)
    if kind == "job":
        c.update(io=rng.choice(["host", "dev"]), N=0)
        if c["io"] == "host":
            c.update(n_x=_logi(rng, 3, 100), n_T=_logi(rng, 5, 500))
    elif kind == "query":
        c.update(n_T=_logi(rng, 1, 64))
    return c


# ------------------------------------------------------------------ inputs

class Curve:
    """Obstacle in the form the binding takes: circle, kite or star with harmonics (amp, phase)."""

    def __init__(self, kind, rng):
        self.kind = {"circle": fh.FH_CURVE_CIRCLE, "kite": fh.FH_CURVE_KITE, "star": fh.FH_CURVE_STAR}[kind]
        self.r0, self.center, self.amp, self.phase = 1.0, (0.0, 0.0), [], []
        if kind == "star":
            self.amp, self.phase = rng.uniform(0.0, 0.1, 5).tolist(), rng.uniform(0.0, 2 * math.pi, 5).tolist()

    def at(self, t):
        """z, z', z'' (complex) at parameters t (numpy)."""
        if self.kind == fh.FH_CURVE_KITE:
            return (np.cos(t) + 0.65 * np.cos(2 * t) - 0.65 + 1.5j * np.sin(t),
                    -np.sin(t) - 1.3 * np.sin(2 * t) + 1.5j * np.cos(t),
                    -np.cos(t) - 2.6 * np.cos(2 * t) - 1.5j * np.sin(t))
        r, dr, ddr = np.full_like(t, self.r0), np.zeros_like(t), np.zeros_like(t)
        for k, (a, p) in enumerate(zip(self.amp, self.phase), start=1):
            r, dr, ddr = r + a * np.cos(k * t + p), dr - k * a * np.sin(k * t + p), ddr - k * k * a * np.cos(k * t + p)
        e = np.exp(1j * t)
        return r * e, (dr + 1j * r) * e, (ddr + 2j * dr - r) * e


def _sizes(curve, omega, N):
    """Boundary sizes: N points, or (N = 0) 8 per wavelength rounded up to 32, at least 64."""
    if N:
        return np.full(omega.size, N, dtype=np.int32)
    z = curve.at(np.linspace(0.0, 2 * math.pi, 8193))[0]
    n = np.maximum(64, np.ceil(8.0 * omega * np.abs(np.diff(z)).sum() / (2 * math.pi)))
    return (np.ceil(n / 32) * 32).astype(np.int32)


def _signal(c, W, rng):
    """Sum of Gaussian pulses with centre frequencies well inside the band, samples on t0 + q dt."""
    n = int(math.ceil((SHIFT + c["span"] + 9.0 - T0) / c["dt"])) + 1
    t = T0 + c["dt"] * np.arange(n)
    a = np.zeros(n)
    hi = min(30.0, 0.75 * W)
    for d, f in zip(rng.uniform(0.0, c["span"], c["pulses"]) if c["span"] else np.zeros(c["pulses"]),
                    rng.uniform(hi / 6, hi, c["pulses"])):
        s = t - SHIFT - d
        q = slice(*np.searchsorted(s, [-12.0, 12.0]))
        a[q] += np.sin(f * s[q]) * np.exp(-0.5 * s[q] ** 2)
    return a


def _targets(n, rng):
    th = 2 * math.pi * (np.arange(n) + rng.uniform()) / n
    return np.stack([3.0 * np.cos(th), 3.0 * np.sin(th)], axis=1).ravel() + np.tile(rng.uniform(-0.1, 0.1, 2), n)


def _times(n, c, rng):
    """Three quarters over the signal's passage, the rest out to t_far."""
    near = min(c["span"] + 80.0, c["t_far"])
    m = n - n // 4
    return np.sort(np.concatenate([near * (np.arange(m) + rng.uniform()) / m, rng.uniform(0.0, c["t_far"], n - m)]))


def _problem(c, W, kind, rng):
    cur = Curve(kind, rng)
    om = np.linspace(0.0, W, c["J"])
    ang = rng.uniform(0, 2 * math.pi)
    return dict(curve=cur, omega=om, N=_sizes(cur, om, c.get("N", 0)), p=(math.cos(ang), math.sin(ang)),
                a=_signal(c, W, rng), x=_targets(c["n_x"], rng), T=_times(c["n_T"], c, rng))


def _problems(c, seed):
    """The problems of a case: one, or the batches of `batch` and `serve` (lists)."""
    rng = np.random.default_rng([seed, 11])
    if c["kind"] not in ("batch", "serve"):
        return [_problem(c, c["W"], c["curve"], rng)]
    # the band limits are spread evenly, so that cases of another seed cost the same
    Ws = np.linspace(c["W_lo"], c["W_hi"], c["P"] + 2)[1:-1]
    out = [_problem(c, float(W), "star", rng) for W in Ws]
    if c["kind"] == "serve":
        for q, pb in enumerate(out):
            pb["queries"] = [np.sort(rng.uniform(0.0, c["t_far"] * (0.02 if i % 2 else 1.0), c["n_T"])) for i in range(c["queries"])]
        other = [_problem(c, float(W) * 0.93, "star", rng) for W in Ws[::-1]]
        for pb in other:
            pb["queries"] = [np.sort(rng.uniform(0.0, c["t_far"] * (0.02 if i % 2 else 1.0), c["n_T"])) for i in range(c["queries"])]
        return [out, other]
    return out


def _dev(a):
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.float64).ravel() if np.iscomplexobj(a) else a.ravel()).cuda()


def _windows(t_last):
    K = 0
    while 1.5 * H * K - H < t_last:
        K += 1
    return 1.5 * H * np.arange(max(K, 1))


def _cutoff(u):
    v = torch.where((u > 0) & (u < 1), u, 0.5)
    return torch.where(u <= 0, 1.0, torch.where(u >= 1, 0.0, torch.exp(2.0 * torch.exp(-1.0 / v) / (v - 1.0))))


def _spectra(a, dt, omega):
    """Window centres and B[k, j] = int w(tau) a(s_k + tau) e^{i omega_j tau} dtau, trapezoidal, 64 bits."""
    s = _windows(T0 + (a.size - 1) * dt)
    Q = int(round(2 * H / dt))
    tau = -H + dt * torch.arange(Q + 1, dtype=torch.float64, device="cuda")
    w = torch.where(tau <= -H / 2, 1 - _cutoff((tau + H) / (H / 2)), torch.where(tau >= H / 2, _cutoff((tau - H / 2) / (H / 2)), 1.0))
    start = np.round((s - H - T0) / dt).astype(np.int64)
    pad = int(max(0, -start.min()))
    ext = np.concatenate([np.zeros(pad), a, np.zeros(max(0, int(start.max()) + Q + 1 - a.size))])
    ext = torch.from_numpy(ext).cuda()
    rows = torch.stack([ext[int(v) + pad:int(v) + pad + Q + 1] for v in start]) * w
    ph = torch.outer(tau, torch.as_tensor(omega, dtype=torch.float64, device="cuda"))
    return s, dt * torch.complex(rows @ torch.cos(ph), rows @ torch.sin(ph))


def _sing_points(wc):
    mu = wc * (np.arange(1, 5) / 4.0) ** 9.1
    x = np.cos(math.pi * np.arange(8) / 7)
    return np.concatenate([0.5 * (a + b) + 0.5 * (b - a) * x for a, b in zip(mu[:-1], mu[1:])])


def _hankel(x, order1=True):
    """H0 and H1 of the first kind at x >= 0, 64 bits: the ascending series below 5, the trapezoidal rule for the
    integral of e^{-v^2} (1 + i v^2 / 2x)^{-+1/2} up to 30, Hankel's expansion above."""
    h0 = torch.empty(x.shape, dtype=torch.complex128, device="cuda")
    h1 = torch.empty_like(h0) if order1 else None
    small, large = x < 5.0, x >= 30.0
    if bool(small.any()):
        v = x[small]
        q, lg = v * v / 4, torch.log(v / 2)
        j0, y0, j1, y1 = (torch.zeros_like(v) for _ in range(4))
        t0, t1, hk = torch.ones_like(v), torch.ones_like(v), 0.0
        for k in range(36):
            j0, y0 = j0 + t0, y0 - hk * t0
            j1, y1 = j1 + t1, y1 - (2 * hk + 1.0 / (k + 1) - 2 * np.euler_gamma) * t1 / 2
            hk += 1.0 / (k + 1)
            t0, t1 = -t0 * q / (k + 1) ** 2, -t1 * q / ((k + 1) * (k + 2))
        h0[small] = torch.complex(j0, (2 / math.pi) * ((lg + np.euler_gamma) * j0 + y0))
        if order1:
            h1[small] = torch.complex(j1 * v / 2, -2 / (math.pi * v) + (v / math.pi) * (lg * j1 + y1))
    for m, quad in ((~small & ~large, True), (large, False)):
        if not bool(m.any()):
            continue
        v = x[m]
        f0, f1 = (torch.zeros(v.shape, dtype=torch.complex128, device="cuda") for _ in range(2))
        if quad:
            h = 0.375
            for k in range(18):
                u = h * h * k * k
                w = math.exp(-u) * h * (1.0 if k else 0.5) * 2 / math.sqrt(math.pi)
                r = torch.sqrt(torch.complex(torch.ones_like(v), u / (2 * v)))
                f0 += w / r
                f1 += 2 * u * w * r
        else:
            i8 = 1.0 / (8 * v)
            t0, t1 = torch.ones_like(v), torch.ones_like(v)
            for k in range(22):
                for f, t in ((f0, t0), (f1, t1)):
                    (f.imag if k % 2 else f.real).add_(t if k % 4 < 2 else -t)
                t0, t1 = t0 * i8 * (-(2 * k + 1) ** 2 / (k + 1.0)), t1 * i8 * ((4 - (2 * k + 1) ** 2) / (k + 1.0))
        c, s = torch.cos(v), torch.sin(v)
        e = torch.complex(c + s, s - c) / torch.sqrt(math.pi * v)       # sqrt(2/(pi x)) e^{i (x - pi/4)}
        h0[m] = e * f0
        if order1:
            h1[m] = -1j * e * f1
    return h0, h1


def _synthesis_inputs(c, seed):
    """Signal spectra and the fields of three line sources inside the obstacle, from their closed form."""
    rng = np.random.default_rng([seed, 12])
    om = np.linspace(0.0, c["W"], c["J"])
    a, x, T = _signal(c, c["W"], rng), _targets(c["n_x"], rng), _times(c["n_T"], c, rng)
    src, amp = rng.uniform(-0.5, 0.5, (3, 2)), rng.uniform(0.3, 1.0, 3)
    xt = torch.from_numpy(x.reshape(-1, 2)).cuda()

    def fields(freqs):
        w = torch.as_tensor(freqs, dtype=torch.float64, device="cuda")
        v = 0
        for y, g in zip(src, amp):
            z = torch.outer(w, torch.linalg.norm(xt - torch.from_numpy(y).cuda(), dim=1))
            v = v + float(g) * _hankel(z, False)[0]
        return v
    V = torch.cat([torch.ones(1, c["n_x"], dtype=torch.complex128, device="cuda"), fields(om[1:])])
    s, B = _spectra(a, c["dt"], om)
    d = dict(om=om, s=s, B=B, V=V, T=T)
    if c["kind"] == "split":
        ws = _sing_points(float(om[c["j_c"]]))
        d.update(Bs=_spectra(a, c["dt"], ws)[1], Vs=fields(ws))
    return d


def _flat(z):
    return torch.view_as_real(z.contiguous()).reshape(-1)


def _coefficients(c, seed):
    """Fourier coefficients of pulses' spectra on a band (the paper's example), one row per trace."""
    rng = np.random.default_rng([seed, 13])
    A, delta, M = 3.5, 11.5, c["M"]
    P = 1.3 * 2 * A
    w = torch.from_numpy(delta + 2 * A * (np.arange(M) - M // 2) / M).cuda()
    w0, w1 = (torch.from_numpy(rng.uniform(lo, hi, (c["batch"], 1))).cuda() for lo, hi in ((9.5, 12.5), (4.0, 10.0)))
    F = torch.polar(torch.exp(-(w - w0) ** 2 / 4.0), -w1 * w)
    m = torch.arange(M, dtype=torch.float64, device="cuda") - M // 2
    ph = (-2 * math.pi / P) * torch.outer(w - delta, m)
    return F @ torch.polar(torch.ones_like(ph), ph) / M, A, P, P / (2 * math.pi) * c["dt"]


# ------------------------------------------------------------------ passes

def _context(c):
    pr = fh.Problem(torch.cuda.current_device(), PREC[c["prec"]])
    st = torch.cuda.Stream()
    fh.fh_set_stream(pr.ctx, st.cuda_stream)
    return pr, st


def prepare(case, seed):
    c = dict(case)
    s = dict(case=c)
    kind = c["kind"]
    if kind in ("job", "batch", "serve", "query", "times", "sample"):
        pbs = _problems(c, seed)
        s["pr"], s["stream"] = _context(c)
        s["problems"] = pbs
    if kind == "job" and c["io"] == "dev" or kind in ("times", "sample"):
        pb = pbs[0]
        s.update(a=_dev(pb["a"]), x=_dev(pb["x"]), T=_dev(pb["T"]), u=torch.empty(c["n_x"] * c["n_T"], dtype=torch.float64, device="cuda"))
    if kind == "batch":
        for pb in pbs:
            pb.update(d_a=_dev(pb["a"]), d_x=_dev(pb["x"]), d_T=_dev(pb["T"]), u=torch.empty(c["n_x"] * c["n_T"], dtype=torch.float64, device="cuda"))
    if kind in ("query", "times", "sample"):   # a solved obstacle whose densities (and fields) stay on the device
        pr, pb = s["pr"], pbs[0]
        pr.discretize(pb["curve"], pb["omega"], pb["N"], 1.0, pb["p"])
        pr.solve()
        if kind != "sample":
            pr.window_spectra(pb["a"], T0, c["dt"], H)
            pr.sample(pb["x"], pb["T"][:2])
    if kind in ("split", "static"):
        d = _synthesis_inputs(c, seed)
        s.update({k: _flat(d[k]) for k in ("B", "V", "Bs", "Vs") if k in d}, s=_dev(d["s"]), T=_dev(d["T"]),
                 u=torch.empty(c["n_x"] * c["n_T"], dtype=torch.float64, device="cuda"))
    if kind == "conv":
        cf, A, P, beta = _coefficients(c, seed)
        s.update(c=_flat(cf), A=A, P=P, beta=beta, d=torch.empty(2 * c["batch"] * c["L"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "conv":
        fh.fh_scaled_convolution(s["c"], c["M"], s["beta"], 1.0, c["L"] // 2, c["L"], s["A"], s["P"], s["d"],
                                 torch.cuda.current_stream().cuda_stream)
        return s["d"]
    if kind == "split":
        fh.fh_synthesize_sing(c["J"], c["W"], c["j_c"], s["s"], s["B"], s["Bs"], s["V"], s["Vs"], s["T"], s["u"],
                              torch.cuda.current_stream().cuda_stream)
        return s["u"]
    if kind == "static":
        fh.fh_synthesize_static(c["J"], c["W"], s["s"], s["B"], s["V"], s["T"], s["u"], torch.cuda.current_stream().cuda_stream)
        return s["u"]
    pr = s["pr"]
    if kind == "batch":
        pbs = s["problems"]
        fh.fh_discretize_batch(pr.ctx, [b["curve"] for b in pbs], [b["omega"] for b in pbs], [b["N"] for b in pbs], ps=[b["p"] for b in pbs])
        fh.fh_solve_frequencies(pr.ctx)
        for q, b in enumerate(pbs):
            fh.fh_window_spectra_p_dev(pr.ctx, q, b["d_a"], T0, c["dt"], H)
            fh.fh_sample_p_dev(pr.ctx, q, b["d_x"], b["d_T"], b["u"])
        return [b["u"] for b in pbs]
    if kind == "serve":
        out = []
        for pbs in s["problems"]:
            fh.fh_discretize_batch(pr.ctx, [b["curve"] for b in pbs], [b["omega"] for b in pbs], [b["N"] for b in pbs], ps=[b["p"] for b in pbs])
            fh.fh_solve_frequencies(pr.ctx)
            for q, b in enumerate(pbs):
                fh.fh_window_spectra_p(pr.ctx, q, b["a"], T0, c["dt"], H)
                first = fh.fh_sample_p(pr.ctx, q, b["x"], b["queries"][0])
                out.append([first] + [fh.fh_resample_p(pr.ctx, q, T, c["n_x"]) for T in b["queries"][1:]])
        return [np.concatenate(v, axis=1) for v in out]
    b = s["problems"][0]
    if kind == "job":
        pr.discretize(b["curve"], b["omega"], b["N"], 1.0, b["p"])
        pr.solve()
        if c["io"] == "host":
            pr.window_spectra(b["a"], T0, c["dt"], H)
            return pr.sample(b["x"], b["T"])
    if kind in ("job", "sample"):
        fh.fh_window_spectra_dev(pr.ctx, s["a"], T0, c["dt"], H)
        fh.fh_sample_dev(pr.ctx, s["x"], s["T"], s["u"])
        return s["u"]
    if kind == "times":
        fh.fh_resample_p_dev(pr.ctx, 0, s["T"], s["u"])
        return s["u"]
    return fh.fh_resample_p(pr.ctx, 0, b["T"], c["n_x"])


# ------------------------------------------------------------------ work

def work(case):
    """Inputs read once and outputs written once; matrix entries count as one complex number of the LU's type
    written and read, LU as 8/3 N^3, special functions as 30 operations, synthesis as its direct products."""
    c = dict(case)
    if c["kind"] == "conv":
        n = 2 ** math.ceil(math.log2(2 * c["L"]))
        return dict(bytes=16.0 * c["batch"] * (c["M"] + c["L"]), flops=5.0 * n * math.log2(n) * (4 * c["batch"] + 5))
    K = len(_windows(SHIFT + c["span"] + 9.0))
    io = 8.0 * c["n_x"] * c["n_T"] + 8.0 * (2 * c["n_x"] + c["n_T"]) + 16.0 * K * c["J"]
    syn = 4.0 * c["J"] * c["n_x"] * c["n_T"] + 8.0 * K * c["n_T"] * c["J"]
    if c["kind"] in ("split", "static", "times", "query"):
        return dict(bytes=io + 16.0 * c["J"] * c["n_x"], flops=syn)
    n_sig = (SHIFT + c["span"] + 9.0 - T0) / c["dt"]
    spec = 4.0 * K * (2 * H / c["dt"]) * c["J"]

    def one(W, solve, queries=1):
        L = {"kite": 9.53}.get(c.get("curve", "star"), 6.4)
        om = np.linspace(0.0, W, c["J"])[1:]
        N = np.full(om.size, float(c["N"])) if c.get("N") else np.ceil(np.maximum(64.0, 8 * om * L / (2 * math.pi)) / 32) * 32
        el = 16.0 if c["prec"] == "fp64" else 8.0
        b, f = queries * io + 8.0 * n_sig + 16.0 * N.sum(), queries * syn + spec + 38.0 * c["n_x"] * N.sum()
        if solve:
            b, f = b + 2 * el * (N ** 2).sum(), f + (8 / 3 * N ** 3).sum() + 60.0 * (N ** 2).sum()
        return np.array([b, f])
    if c["kind"] in ("batch", "serve"):
        Ws = np.linspace(c["W_lo"], c["W_hi"], c["P"] + 2)[1:-1]
        v = sum(one(float(W) * r, True, c.get("queries", 1)) for W in Ws for r in ((1.0, 0.93) if c["kind"] == "serve" else (1.0,)))
    else:
        v = one(c["W"], c["kind"] == "job")
    return dict(bytes=float(v[0]), flops=float(v[1]))


# ------------------------------------------------------------------ 64-bit values

def _kress(N):
    n = N // 2
    d = torch.arange(N, dtype=torch.int64, device="cuda")
    m = torch.arange(1, n, dtype=torch.int64, device="cuda")
    R = -(2 * math.pi / n) * (torch.cos((d[:, None] * m % N).double() * (math.pi / n)) / m).sum(1) - (math.pi / n ** 2) * (1.0 - 2.0 * (d % 2).double())
    ls = torch.log(4 * torch.sin(d.double() * (math.pi / N)) ** 2)
    ls[0] = 0.0
    idx = (d[:, None] - d[None, :]) % N
    return R[idx], ls[idx]


def _fields(pb):
    """Target fields V[j, x] of the combined-field densities, Nystrom method with Kress's weights."""
    xt = torch.from_numpy(pb["x"].reshape(-1, 2)).cuda()
    xt = torch.complex(xt[:, 0], xt[:, 1])
    V = torch.ones(pb["omega"].size, xt.numel(), dtype=torch.complex128, device="cuda")
    px, py = pb["p"]
    last = None
    for j in range(1, pb["omega"].size):
        N, k = int(pb["N"][j]), float(pb["omega"][j])
        if N != last:
            last, n = N, N // 2
            z, dz, ddz = (torch.from_numpy(v).cuda() for v in pb["curve"].at(math.pi * np.arange(N) / n))
            sp = dz.abs()
            R, ls = _kress(N)
            df = z[None, :] - z[:, None]
            r = df.abs().fill_diagonal_(1.0)
            Nil = dz.imag[:, None] * df.real - dz.real[:, None] * df.imag
            g = Nil * sp[None, :] / (sp[:, None] * r)
            rx = (xt[:, None] - z[None, :]).abs()
        x = k * r
        H0, H1 = _hankel(x)
        M = 0.25j * H0 * sp
        M1 = -H0.real * sp / (4 * math.pi)
        Lk = 0.25j * k * H1 * g
        L1 = -k / (4 * math.pi) * H1.real * g
        M2, L2 = M - M1 * ls, Lk - L1 * ls
        M1.diagonal().copy_(-sp / (4 * math.pi))
        M2.diagonal().copy_(torch.complex((-np.euler_gamma - torch.log(k * sp / 2)) / (2 * math.pi), torch.full_like(sp, 0.25)) * sp)
        L1.diagonal().zero_()
        L2.diagonal().copy_(((ddz.real * dz.imag - ddz.imag * dz.real) / (4 * math.pi * sp ** 2)).to(L2.dtype))
        A = R * (L1 - 1j * k * M1) + (math.pi / n) * (L2 - 1j * k * M2)
        A.diagonal().add_(0.5)
        pz = px * z.real + py * z.imag
        rhs = 1j * k * ((px * dz.imag - py * dz.real) / sp - 1.0) * torch.polar(torch.ones_like(pz), k * pz)
        q = torch.linalg.solve(A, rhs) * sp * (math.pi / n)
        V[j] = 0.25j * _hankel(k * rx, False)[0] @ q
    return V


def _sinc(v):
    """sin(pi v)/(pi v), the argument reduced before the product with pi."""
    r = torch.round(v)
    s = torch.sin(math.pi * (v - r)) * (1.0 - 2.0 * torch.remainder(r, 2.0))
    return torch.where(v == 0, 1.0, s / (math.pi * torch.where(v == 0, 1.0, v)))


def _synthesis(J, W, s, B, V, T):
    """u[x, t] = Re sum_p V[p, x] (mu_p / 2 pi) sum_k B[k, p] D_p(t - s_k), the band-limited transform."""
    h = J - 1
    M = 2 * h
    m = torch.arange(-h, h, device="cuda")
    ph = -2 * math.pi / M * (torch.outer(m, torch.arange(J, device="cuda")) % M).double()
    E = (2 * W / M) * torch.cat([torch.cos(ph), torch.sin(ph)], dim=1)
    mu = torch.full((J,), 2.0, dtype=torch.float64, device="cuda")
    mu[0] = mu[-1] = 1.0
    st, Tt = torch.from_numpy(s).cuda(), torch.from_numpy(T).cuda()
    G = []
    for t in Tt.split(32):
        y = W * (t[:, None] - st) * (1.0 / math.pi)
        D = _sinc(y[:, :, None] - m) @ E
        G.append((B * torch.complex(D[..., :J], D[..., J:])).sum(1))
    G = torch.cat(G) * mu / (2 * math.pi)
    return V.real.T @ G.real.T - V.imag.T @ G.imag.T


def _job_u(pb, dt, T, V=None):
    V = _fields(pb) if V is None else V
    s, B = _spectra(pb["a"], dt, pb["omega"])
    return _synthesis(pb["omega"].size, float(pb["omega"][-1]), s, B, V, T)


def _split_u(c, d):
    """FC(Gram) continuation and term-wise integrals on [w_c, W], Filon-Clenshaw-Curtis on (0, w_c]."""
    with open(os.path.join(ROOT, "oracle", "fc_gram_d6_c31.json")) as f:
        tab = json.load(f)
    At, Qt = (torch.tensor(tab[k], dtype=torch.float64, device="cuda") for k in ("A", "Q"))
    j_c, om, st, T = c["j_c"], d["om"], torch.from_numpy(d["s"]).cuda(), torch.from_numpy(d["T"]).cuda()
    n, wc, W = c["J"] - c["j_c"], float(om[c["j_c"]]), float(om[-1])
    E = At @ Qt.T                                       # 31 x 6: continuation of the right end's values
    X = torch.zeros(n + 31, n, dtype=torch.float64, device="cuda")
    X[:n] = torch.eye(n, dtype=torch.float64, device="cuda")
    X[n:, n - 6:] += E
    X[n:, :6] += E.flip(0).flip(1)
    L = n + 31
    m = torch.arange(-(L // 2), L // 2, device="cuda")
    l = torch.arange(L, device="cuda")
    ang = lambda num, den: torch.polar(torch.ones(num.shape, dtype=torch.float64, device="cuda"), (num % (2 * den)).double() * (math.pi / den))  # noqa: E731
    C = (ang(-2 * m[:, None] * l, L) @ X.to(torch.complex128)) * ang(m * (n - 1), L)[:, None] / L
    A, P, delta = 0.5 * (W - wc), L * (W / (c["J"] - 1)), 0.5 * (wc + W)
    mu = wc * (np.arange(1, 5) / 4.0) ** 9.1
    xg, wg = (torch.from_numpy(v).cuda() for v in np.polynomial.legendre.leggauss(24))
    k8 = np.arange(8)
    w8 = np.where((k8 == 0) | (k8 == 7), 0.5, 1.0)
    ch = torch.from_numpy((2.0 / 7) * np.cos(math.pi * np.outer(k8, k8) / 7) * w8[None, :] * w8[:, None]).cuda()  # [order, point]
    B = torch.cat([d["B"][:, j_c:], d["Bs"]], dim=1)
    V = torch.cat([d["V"][j_c:], d["Vs"]])
    G = []
    for t in T.split(16):
        tp = t[:, None] - st
        b = 2 * A * _sinc((2 * A / P) * (P / (2 * math.pi) * tp[:, :, None] - m))
        ph = -delta * tp
        D = [torch.complex(b @ C.real, b @ C.imag) * torch.polar(torch.ones_like(ph), ph)[:, :, None]]
        for a, e in zip(mu[:-1], mu[1:]):
            hh, dl = 0.5 * (e - a), 0.5 * (a + e)
            np_ = int(float(hh * tp.abs().max()) / 6.0) + 1
            ed = torch.linspace(-1.0, 1.0, np_ + 1, dtype=torch.float64, device="cuda")
            x = (0.5 * (ed[1:] - ed[:-1])[:, None] * xg + 0.5 * (ed[1:] + ed[:-1])[:, None]).reshape(-1)
            wt = (0.5 * (ed[1:] - ed[:-1])[:, None] * wg).reshape(-1)
            basis = (torch.cos(torch.arange(8, device="cuda")[:, None] * torch.arccos(x)) * wt).T @ ch      # node x point
            pe = -tp[:, :, None] * (dl + hh * x)
            D.append(hh * torch.complex(torch.cos(pe) @ basis, torch.sin(pe) @ basis))
        G.append((B * torch.cat(D, dim=2)).sum(1))
    G = torch.cat(G) / math.pi
    return V.real.T @ G.real.T - V.imag.T @ G.imag.T


def _turns(alpha, k, L):
    """e^{i pi alpha k^2 / L}, the phase reduced in extended precision."""
    v = np.asarray(k, dtype=np.longdouble)
    r = np.fmod(np.longdouble(alpha) * v * v / np.longdouble(L), np.longdouble(2))
    r = torch.from_numpy(r.astype(np.float64)).cuda() * math.pi
    return torch.polar(torch.ones_like(r), r)


def _frft(x, alpha):
    """sum_m x_m e^{-2 pi i alpha m p / L} for m, p = -L/2 .. L/2 - 1 (chirp factorisation)."""
    L = x.shape[-1]
    n = 2 ** math.ceil(math.log2(2 * L))
    ch = _turns(-alpha, np.arange(L) - L // 2, L)
    f = torch.zeros(n, dtype=torch.complex128, device="cuda")
    kern = _turns(alpha, np.arange(L), L)
    f[:L] = kern
    f[n - L + 1:] = kern[1:].flip(0)
    y = torch.fft.ifft(torch.fft.fft(x * ch, n=n) * torch.fft.fft(f))[..., :L]
    return y * ch


def _conv(c, seed):
    cf, A, P, beta = _coefficients(c, seed)
    L, M = c["L"], c["M"]
    x = torch.zeros(c["batch"], L, dtype=torch.complex128, device="cuda")
    x[:, L // 2 - M // 2:L // 2 + M // 2] = cf
    q = torch.arange(L, dtype=torch.float64, device="cuda") - L // 2
    Bp = _frft(2 * A * _sinc((2 * A / P) * q).to(torch.complex128), 1.0)
    v = np.fmod(2 * np.longdouble(beta) * (L // 2) * (np.arange(L) - L // 2).astype(np.longdouble) / L, np.longdouble(2))
    v = torch.from_numpy(v.astype(np.float64)).cuda() * math.pi
    return _flat(_frft(_frft(x, 1.0) * Bp * torch.polar(torch.ones_like(v), v), -beta) / L)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "conv":
        return _conv(c, seed)
    if kind == "split":
        return _split_u(c, _synthesis_inputs(c, seed)).reshape(-1)
    if kind == "static":
        d = _synthesis_inputs(c, seed)
        return _synthesis(c["J"], c["W"], d["s"], d["B"], d["V"], d["T"]).reshape(-1)
    pbs = _problems(c, seed)
    if kind == "batch":      # the first and the last obstacle
        return [_job_u(pb, c["dt"], pb["T"]).reshape(-1) if q in (0, len(pbs) - 1) else None for q, pb in enumerate(pbs)]
    if kind == "serve":
        flat = [pb for b in pbs for pb in b]
        return [_job_u(pb, c["dt"], np.concatenate(pb["queries"])) if q in (0, len(flat) - 1) else None for q, pb in enumerate(flat)]
    u = _job_u(pbs[0], c["dt"], pbs[0]["T"])
    return u.reshape(-1) if kind in ("times", "sample") or c.get("io") == "dev" else u
