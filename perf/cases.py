"""The work that a user of the library has it do, as measurable cases.

Each case is one call through the Python binding: a single-point evaluation
inside a fit, a spectrum at a point, batched scans in the fold's precisions, a
grouped launch over uneven detector configurations, the rank-8 evaluator with
its gradient, the profiled evaluation, and the learned surrogate's scan and
training.  Sizes are those of the 7Be-line, solar-set and uneven-configuration
workloads, with odd and ragged ones among them.  Inputs (sources, response,
backgrounds, pseudo-data, parameter points) are made from the seed; `exact`
evaluates the same quantities in 64 bits with torch alone.
"""

import math
import random

import numpy as np
import torch

import paper_2607_00488_gb300 as srw

M_E = 0.51099895
SIN2W, F_TAU, T_MIN = 0.23121, 0.5, 1e-3
# pi alpha^2 / m_e^2 over 2 G_F^2 m_e / pi for a moment of 1e-11 Bohr magnetons, MeV
KAPPA = (math.pi / (137.035999084 * M_E)) ** 2 / (2.0 * 1.1663787e-11**2 * M_E) * 1e-22
PRECISION = {"fp32": srw.SRW_FP32, "bf16": srw.SRW_BF16, "bf16x3": srw.SRW_BF16X3, "fp16x3": srw.SRW_FP16X3}
BOX_CENTRE, BOX_HALF = (0.0, 0.0, 0.0, 0.0, 1.5), (0.3, 0.3, 0.3, 0.3, 1.5)
HIDDEN = 256
_STREAM = []


# ------------------------------------------------------------------ the cases
def listed():
    line = {"sources": "line", "n_t": 256, "n_rec": 128, "exposure": 1e5, "res": 0.05, "mask": False}
    solar = {"sources": "solar", "n_t": 4096, "n_rec": 2048, "exposure": 1e5, "res": 0.05, "mask": False}
    odd = {"sources": "solar", "n_t": 3001, "n_rec": 1111, "exposure": 3e5, "res": 0.06, "mask": True}
    wide = {"sources": "solar", "n_t": 7001, "n_rec": 3333, "exposure": 1e6, "res": 0.08, "mask": False}
    return [
        # a minimiser on the 7Be line: one point per call from host memory, the smallest call there is
        {"name": "call_line_host", "kind": "call", "where": "host", **line},
        # a fit on the full solar set: one point per call, device memory
        {"name": "call_solar", "kind": "call", "where": "device", **solar},
        # the expected counts at one point (a plot, Asimov data): direct cross-section integrals, then the fold
        {"name": "spectrum_solar", "kind": "spectrum", "stage": 3, **solar},
        # an ensemble sampler's step: a few hundred walkers on an odd binning with dead bins
        {"name": "walkers_fp16x3", "kind": "scan", "precision": "fp16x3", "points": 300, **odd},
        # the dense scan of the parameter box on the solar set
        {"name": "scan_fp16x3", "kind": "scan", "precision": "fp16x3", "points": 65536, **solar},
        # a ragged scan of a large, poorly resolved configuration
        {"name": "scan_bf16x3", "kind": "scan", "precision": "bf16x3", "points": 5001, **wide},
        # the same scan where FP32 products are asked for
        {"name": "scan_fp32", "kind": "scan", "precision": "fp32", "points": 4096, **solar},
        # uneven detector configurations evaluated together
        {"name": "group_fp16x3", "kind": "group", "precision": "fp16x3", "n": 12, "sizes": 4, "scale": 1.0},
        # gradients for a sampler or a fit with many starting points
        {"name": "rank8_gradient", "kind": "rank8", "grad": True, "points": 65536, **solar},
        # the signal rate as a constrained nuisance, on a grid around the best fit (host arrays)
        {"name": "profiled", "kind": "profiled", "sigma": 0.05, "points": 8191, **solar},
        # the surrogate's values for a chunk of a dense scan
        {"name": "surrogate_scan", "kind": "surrogate", "points": 1 << 20, **solar},
        # training the surrogate: exact spectra, standardization, three epochs of Adam
        {"name": "surrogate_fit", "kind": "fit", "points": 65536, "batch": 4096, "epochs": 3, **solar},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "spectrum", "scan", "scan", "scan", "group", "rank8", "profiled", "surrogate", "fit"])
    if kind == "group":
        return {"kind": kind, "precision": rng.choice(["bf16x3", "fp16x3"]), "n": rng.randint(2, 12),
                "sizes": rng.randint(5, 10**6), "scale": round(math.exp(rng.uniform(math.log(0.1), 0.0)), 4)}
    c = {"kind": kind, "sources": "solar", "n_t": _log_int(rng, 257, 8192), "n_rec": _log_int(rng, 100, 4096),
         "exposure": round(10.0 ** rng.uniform(4, 6.5)), "res": round(rng.uniform(0.03, 0.08), 4),
         "mask": rng.random() < 0.4}
    if kind in ("call", "spectrum") and rng.random() < 0.3:
        c.update(sources="line", n_t=rng.randint(100, 600), n_rec=rng.randint(50, 300))
    size = c["n_t"] * c["n_rec"]
    if kind == "call":
        c["where"] = rng.choice(["host", "device"])
    elif kind == "spectrum":
        c["stage"] = rng.randint(0, 3)
    elif kind == "scan":
        c["precision"] = rng.choice(["fp32", "bf16", "bf16x3", "bf16x3", "fp16x3", "fp16x3"])
        most = (4096 if c["precision"] == "fp32" else 65536) * 4096 * 2048 // size
        c["points"] = _log_int(rng, 2, max(2, min(65536, most)))
    elif kind == "rank8":
        c.update(grad=rng.random() < 0.5, points=_log_int(rng, 10, 65536 if c["n_rec"] <= 2048 else 32768))
    elif kind == "profiled":
        c.update(sigma=rng.choice([0.0, 0.05]), points=_log_int(rng, 10, 8192 if c["n_rec"] <= 2048 else 4096))
    elif kind == "surrogate":
        c["points"] = _log_int(rng, 1000, (1 << 20) if c["n_rec"] <= 2048 else (1 << 19))
    elif kind == "fit":
        c.update(n_rec=min(c["n_rec"], 2048), n_t=min(c["n_t"], 4096), points=_log_int(rng, 3000, 65536),
                 batch=128 * rng.randint(4, 32), epochs=rng.randint(1, 3))
    return c


# ------------------------------------------------------------------ inputs from the seed
def _sources(kind):
    """(energies, weights, survival probabilities) per source."""
    if kind == "line":
        return [(np.array([0.862]), np.array([1.0]), np.array([0.55]))]

    def pee(e):
        return 0.55 - 0.25 * np.log(np.clip(e, 1.0, 5.0)) / math.log(5.0)

    out = []
    for q, rate in ((0.420, 6e10), (1.20, 3e8), (1.73, 2e8), (16.0, 5e6)):  # pp, 13N, 15O, 8B
        e = (np.arange(2000) + 0.5) * (q / 2000)
        w = e * e * (q - e) ** 2
        out.append((e, w / w.sum() * rate, pee(e)))
    for q, rate in ((0.862, 4.5e9), (0.384, 5e8), (1.44, 1.4e8)):  # the 7Be lines, pep
        out.append((np.array([q]), np.array([rate]), pee(np.array([q]))))
    return out


def _response(t_edges, rec_edges, res, tail, noise, gen):
    """Conditional response [n_rec, n_t]: Gaussian smearing of the quenched energy, a low tail, noise."""
    d = "cuda"
    te = torch.tensor(t_edges, dtype=torch.float64, device=d)
    x = torch.tensor(rec_edges, dtype=torch.float64, device=d)[:, None]
    tc = 0.5 * (te[1:] + te[:-1])
    m = (tc * tc / (tc + 0.01))[None, :]
    sig = torch.clamp(res * torch.sqrt(m), min=1e-9)
    r = torch.diff(0.5 * (1.0 + torch.erf((x - m) / (math.sqrt(2.0) * sig))), dim=0)
    if tail > 0.0:
        low = torch.where(x < m, torch.exp((torch.minimum(x, m) - m) / (2.0 * sig)), torch.ones_like(m))
        r = (1.0 - tail) * r + tail * torch.diff(low, dim=0)
    if noise > 0.0:
        r = r * (1.0 - noise + 2.0 * noise * torch.rand(r.shape, generator=gen, dtype=torch.float64, device=d))
    return r.to(torch.float32).contiguous()


def _backgrounds(rec_edges, kind, exposure):
    """Background templates in expected counts (peaks, beta-like shapes, flat, falling)."""
    lo, hi = rec_edges[:-1], rec_edges[1:]
    c, w = 0.5 * (lo + hi), hi - lo
    if kind == "line":
        return np.full((1, c.size), 0.1 * exposure / c.size)

    def beta(q, off=0.0):
        k = np.clip(c - off, 0.0, q)
        return np.sqrt(k * k + 2 * k * M_E) * (k + M_E) * (q - k) ** 2

    shapes = [(np.exp(-0.5 * ((c - 0.40) / 0.03) ** 2), 0.2), (beta(0.687), 0.05), (beta(1.16), 0.1),
              (beta(0.96, 1.02), 0.04), (np.ones_like(c), 0.02), (np.exp(-c / 0.8), 0.03), (beta(0.156), 0.5),
              (np.exp(-0.5 * ((c - 2.61) / 0.08) ** 2), 0.005)]
    return np.stack([s * w * (f * exposure / max((s * w).sum(), 1e-300)) for s, f in shapes])


def _couplings(theta):
    """The monomials that multiply the coefficient spectra, [P, 8], 64 bits."""
    t = theta.double()
    gle, gre = 0.5 + SIN2W + t[:, 0], SIN2W + t[:, 1]
    glt, grt = -0.5 + SIN2W + t[:, 2], SIN2W + t[:, 3]
    return torch.stack([gle * gle, gre * gre, -gle * gre, glt * glt, grt * grt, -glt * grt, torch.ones_like(gle),
                        t[:, 4] ** 2], dim=1)


def _basis(sources, t_edges):
    """Recoil spectra per monomial, [8, n_t]: bin integrals clipped to [T_MIN, T_max(E)], 64 bits."""
    te = torch.tensor(t_edges, dtype=torch.float64, device="cuda")
    lo, hi = torch.clamp(te[:-1], min=T_MIN)[None, :], te[1:][None, :]
    out = torch.zeros(8, te.numel() - 1, dtype=torch.float64, device="cuda")
    gl, gr = -0.5 + SIN2W, SIN2W
    for e_all, w_all, p_all in sources:
        for k in range(0, e_all.size, 250):
            e, w, p = (torch.tensor(v[k:k + 250], dtype=torch.float64, device="cuda")[:, None]
                       for v in (e_all, w_all, p_all))
            nb = int(np.searchsorted(t_edges[:-1], float((2 * e * e / (M_E + 2 * e)).max())))
            if nb == 0:
                continue
            a = lo[:, :nb]
            b = torch.minimum(hi[:, :nb], 2 * e * e / (M_E + 2 * e))
            ok = b > a
            b = torch.where(ok, b, a)
            one = b - a
            rr = (e / 3) * ((1 - a / e) ** 3 - (1 - b / e) ** 3)
            lr = M_E * (b * b - a * a) / (2 * e * e)
            mm = torch.log(b / a) - (b - a) / e
            pe, pm, pt = p, (1 - p) * (1 - F_TAU), (1 - p) * F_TAU
            for q, v in enumerate((pe * one, pe * rr, pe * lr, pt * one, pt * rr, pt * lr,
                                   pm * (gl * gl * one + gr * gr * rr - gl * gr * lr), KAPPA * mm)):
                out[q, :nb] += (w * v).sum(0)
    return out


class _Model:
    """One detector configuration in plain arrays, and its quantities in 64 bits."""

    def __init__(self, case, seed):
        gen = torch.Generator("cuda").manual_seed(seed)
        line = case["sources"] == "line"
        top = 1.0 if line else 16.0
        self.exposure = float(case["exposure"])
        self.t_edges = np.linspace(0.0, top, case["n_t"] + 1)
        rec_edges = np.linspace(0.0, top, case["n_rec"] + 1)
        self.sources = _sources(case["sources"])
        self.R = _response(self.t_edges, rec_edges, case["res"], 0.0 if line else 1e-3, 0.01 if line else 0.0, gen)
        self.bkg = _backgrounds(rec_edges, case["sources"], self.exposure)
        self.mask = None
        if case["mask"]:  # one bin in fifty is dead
            self.mask = (torch.rand(case["n_rec"], generator=gen, device="cuda") > 0.02).to(torch.uint8)
        self.basis = _basis(self.sources, self.t_edges)
        sm = torch.zeros(1, 5, device="cuda")
        self.s_sm = (_couplings(sm) @ self.basis)[0]
        R = self.R.double()
        self.e_sm = self.s_sm * (self.exposure / float((R.sum(0) * self.s_sm).sum()))
        # where the standard spectrum vanishes the weight is 1
        safe = torch.where(self.s_sm != 0, self.s_sm, torch.ones_like(self.s_sm))
        shat = torch.where(self.s_sm != 0, self.basis * (self.e_sm / safe), torch.zeros_like(self.basis))
        shat[6] = torch.where(self.s_sm != 0, shat[6], self.e_sm)
        self.shat = shat
        self.M = shat @ R.T  # [8, n_rec]
        self.b = torch.tensor(self.bkg.sum(0), device="cuda")
        self.counts = torch.poisson(self.mu(sm)[0], generator=gen)
        self.gen = gen

    def signal(self, theta):
        return _couplings(theta) @ self.M

    def mu(self, theta):
        return self.signal(theta) + self.b

    def value_of(self, mu):
        """-2 ln L of expected counts [P, n_rec]."""
        n = self.counts
        t = 2.0 * (mu - torch.xlogy(n, mu) + torch.lgamma(n + 1.0))
        return (t if self.mask is None else t * self.mask).sum(1)

    def value(self, theta):
        return torch.cat([self.value_of(self.mu(c)) for c in theta.split(4096)])

    def gradient(self, theta):
        out = []
        for c in theta.split(4096):
            t = c.double().requires_grad_(True)
            self.value_of(self.mu(t)).sum().backward()
            out.append(t.grad)
        return torch.cat(out)

    def points(self, n, near):
        """Points of the parameter box, or near the data (where a fit or an interval is decided)."""
        u = torch.rand(n, 5, generator=self.gen, device="cuda")
        s = math.sqrt(1e5 / self.exposure)
        eps, mu = (0.02 * s, 0.5 * math.sqrt(s)) if near else (0.3, 3.0)
        return torch.cat([(2 * u[:, :4] - 1) * eps, u[:, 4:] * mu], 1).contiguous()

    def likelihood(self):
        h = srw.Likelihood({"t_edges": self.t_edges, "sources": [dict(zip(("e", "w", "pee"), s)) for s in self.sources],
                            "R": self.R.cpu().numpy(), "exposure": self.exposure, "t_min": T_MIN, "sin2w": SIN2W,
                            "f_tau": F_TAU, "bkg": self.bkg}, self.counts.cpu().numpy(),
                           mask=None if self.mask is None else self.mask.cpu().numpy())
        return h


def _group_sizes(case):
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["n"]):
        out.append({"sources": "solar", "n_t": max(64, int(rng.randint(512, 8192) * case["scale"])),
                    "n_rec": max(32, int(rng.randint(256, 4096) * case["scale"])),
                    "exposure": 10.0 ** rng.uniform(4, 7), "res": rng.uniform(0.03, 0.08), "mask": False,
                    "points": max(1, int(rng.randint(256, 4096) * case["scale"]))})
    return out


def _network(model, seed):
    """Weights of a network whose outputs scatter around the logarithm of the standard expectation."""
    rng = np.random.default_rng(seed)
    n_rec = model.R.shape[0]
    params = []
    for out, fan_in in ((HIDDEN, 5), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN)):
        params.append((rng.normal(0.0, math.sqrt(2.0 / fan_in), (out, fan_in)).astype(np.float32),
                       rng.normal(0.0, 0.1, out).astype(np.float32)))
    w = rng.normal(0.0, 0.1 / math.sqrt(HIDDEN), (n_rec, HIDDEN)).astype(np.float32)
    b = torch.log(model.mu(torch.zeros(1, 5, device="cuda"))[0]).cpu().numpy().astype(np.float32)
    return params + [(w, b)]


def _start_weights(n_rec, seed):
    rng = np.random.default_rng(seed)
    shapes = [(HIDDEN, 5), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (n_rec, HIDDEN)]
    return [(rng.normal(0.0, math.sqrt(2.0 / i), (o, i)).astype(np.float32), np.zeros(o, np.float32))
            for o, i in shapes]


def _inputs(case, seed):
    """(model, points) of every kind but the group."""
    m = _Model(case, seed)
    n = 1 if case["kind"] in ("call", "spectrum") else case["points"]
    return m, m.points(n, near=case["kind"] in ("call", "spectrum", "rank8", "profiled"))


# ------------------------------------------------------------------ what a program keeps, and one pass
def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case, "stream": _stream()}
    if kind == "group":
        members, theta = [], []
        for k, c in enumerate(_group_sizes(case)):
            m = _Model(c, seed + 1000 * k)
            members.append(m.likelihood())
            theta.append(m.points(c["points"], near=False))
        s["theta"] = torch.cat(theta)
        s["group"] = srw.GroupedLikelihood(members, [t.shape[0] for t in theta])
        s["out"] = torch.empty(s["theta"].shape[0], dtype=torch.float64, device="cuda")
        return s
    m, theta = _inputs(case, seed)
    s["lk"] = m.likelihood()
    n_rec, n_t = m.R.shape
    if kind == "spectrum":
        s["theta"] = theta.reshape(5).contiguous()
        s["out"] = torch.empty(n_t if case["stage"] <= 1 else n_rec, dtype=torch.float32, device="cuda")
    elif kind == "profiled" or (kind == "call" and case["where"] == "host"):
        s["theta"] = theta.cpu().numpy()
    elif kind == "fit":
        s["theta"] = theta.cpu().numpy()
        s["params"] = _start_weights(n_rec, seed)
        s["net"] = srw.Surrogate(s["lk"], s["params"], np.float32(BOX_CENTRE), np.float32(BOX_HALF))
    else:
        s["theta"] = theta
        s["out"] = torch.empty(theta.shape[0], dtype=torch.float64, device="cuda")
        if kind == "rank8" and case["grad"]:
            s["grad"] = torch.empty(theta.shape[0], 5, dtype=torch.float64, device="cuda")
        if kind == "surrogate":
            s["net"] = srw.Surrogate(s["lk"], _network(m, seed), np.float32(BOX_CENTRE), np.float32(BOX_HALF))
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "call":
        if case["where"] == "host":
            return s["lk"].loglik(s["theta"], srw.SRW_FP32)
        return s["lk"].loglik(s["theta"], srw.SRW_FP32, out=s["out"], stream=s["stream"])
    if kind == "spectrum":
        return s["lk"].spectrum(s["theta"], case["stage"], out=s["out"], stream=s["stream"])
    if kind == "scan":
        return s["lk"].loglik(s["theta"], PRECISION[case["precision"]], out=s["out"], stream=s["stream"])
    if kind == "group":
        return s["group"].loglik(s["theta"], PRECISION[case["precision"]], out=s["out"], stream=s["stream"])
    if kind == "rank8":
        return s["lk"].loglik_linear(s["theta"], out=s["out"], grad_out=s.get("grad"), stream=s["stream"])
    if kind == "profiled":
        return s["lk"].loglik_profiled(s["theta"], case["sigma"])
    if kind == "surrogate":
        return s["net"].loglik(s["theta"], out=s["out"], stream=s["stream"])
    net = s["net"]  # a training run from the same start
    net.set_weights(s["params"])
    losses = net.fit(s["theta"], case["epochs"], batch=case["batch"], lr=2e-3, lr_final=2e-5)
    return {"losses": losses, "weights": net.weights(), "standardization": net.standardization()}


# ------------------------------------------------------------------ the work, and the values in 64 bits
def work(case):
    """Bytes: the response, the points and the results once.  Operations: the fold 2 n_rec n_t a point (the rank-8
    forms 16 n_rec plus about 20 a bin; the direct spectrum about 20 a reachable (node, bin) pair; the network 2 a
    weight)."""
    if case["kind"] == "group":
        cs = _group_sizes(case)
        return {"bytes": float(sum(4 * c["n_t"] * c["n_rec"] + 28 * c["points"] for c in cs)),
                "flops": float(sum(2 * c["n_t"] * c["n_rec"] * c["points"] for c in cs))}
    n_t, n_rec = case["n_t"], case["n_rec"]
    fold = 2.0 * n_t * n_rec
    if case["kind"] in ("call", "spectrum"):
        pairs = n_t if case["sources"] == "line" else 1200.0 * n_t  # nodes reach a share of the bins
        folds = case["kind"] == "call" or case["stage"] >= 2
        return {"bytes": 4.0 * n_t * n_rec * folds + 64.0 * n_t + 24 * n_rec,
                "flops": fold * folds + (20 * pairs if case["kind"] == "spectrum" else 16 * n_t)}
    p = float(case["points"])
    if case["kind"] == "scan":
        return {"bytes": 4.0 * n_t * n_rec + 28 * p, "flops": fold * p}
    if case["kind"] in ("rank8", "profiled"):
        passes = 9 if case["kind"] == "profiled" else 1
        grad = case["kind"] == "rank8" and case["grad"]
        return {"bytes": 48.0 * n_rec + (28 + 40 * grad) * p, "flops": p * n_rec * (36 * passes + 14 * grad)}
    weights = 5 * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN * n_rec
    if case["kind"] == "surrogate":
        return {"bytes": 2.0 * weights + 28 * p, "flops": p * (2.0 * weights + 8 * n_rec)}
    # training: the exact spectra once, then three products per weight, point and epoch
    e = case["epochs"]
    return {"bytes": 4.0 * n_t * n_rec + 4 * p * n_rec * e + 20 * p, "flops": p * fold + 6.0 * weights * p * e}


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _forward(params, x):
    for k, (w, b) in enumerate(params):
        z = x @ w.T + b
        x = _gelu(z) if k < 3 else z
    return x


def _normalised(theta):
    c = torch.tensor(BOX_CENTRE, dtype=torch.float64, device="cuda")
    return (theta.double() - c) / torch.tensor(np.float32(BOX_HALF), device="cuda").double()


def _profiled(m, theta, sigma):
    sig, n = m.signal(theta), m.counts
    live = torch.ones_like(n) if m.mask is None else m.mask.double()
    iv = 1.0 / sigma**2 if sigma > 0 else 0.0
    a = torch.ones(theta.shape[0], 1, dtype=torch.float64, device="cuda")
    for _ in range(30):
        mu = a * sig + m.b
        g = (2 * live * sig * (1 - n / mu)).sum(1, keepdim=True) + 2 * (a - 1) * iv
        h = (2 * live * n * (sig / mu) ** 2).sum(1, keepdim=True) + 2 * iv
        a = torch.clamp(a - g / h, min=0.0)
    return (m.value_of(a * sig + m.b) + iv * (a[:, 0] - 1) ** 2), a[:, 0]


def _trained(m, theta, case, seed):
    """The training run in 64 bits."""
    n, batch, epochs = case["points"], case["batch"], case["epochs"]
    t = torch.cat([torch.log(m.mu(c)) for c in theta.split(4096)])
    mean = t.mean(0)
    std = torch.sqrt(torch.clamp((t * t).mean(0) - mean**2, min=0.0))
    std = torch.where(std > 1e-12, std, torch.ones_like(std))
    t = (t - mean) / std
    x = _normalised(theta)
    params = [torch.tensor(a, device="cuda").double().requires_grad_(True)
              for layer in _start_weights(m.R.shape[0], seed) for a in layer]
    m1, m2 = [torch.zeros_like(a) for a in params], [torch.zeros_like(a) for a in params]
    steps = -(-n // batch)
    losses, k = [], 0
    for _ in range(epochs):
        sse = 0.0
        for b in range(steps):
            xb, tb = x[b * batch:(b + 1) * batch], t[b * batch:(b + 1) * batch]
            e2 = (_forward(list(zip(params[::2], params[1::2])), xb) - tb).square().sum()
            grads = torch.autograd.grad(e2 / tb.numel(), params)
            sse += float(e2.detach())
            frac = k / (steps * epochs - 1) if steps * epochs > 1 else 0.0
            lr = 2e-5 + 0.5 * (2e-3 - 2e-5) * (1.0 + math.cos(math.pi * frac))
            k += 1
            with torch.no_grad():
                for a, g, u, v in zip(params, grads, m1, m2):
                    u.mul_(0.9).add_(g, alpha=0.1)
                    v.mul_(0.999).addcmul_(g, g, value=0.001)
                    a -= lr * (u / (1 - 0.9**k)) / ((v / (1 - 0.999**k)).sqrt() + 1e-8)
        losses.append(sse / (n * m.R.shape[0]))
    w = [a.detach() for a in params]
    return {"losses": np.array(losses), "weights": list(zip(w[::2], w[1::2])), "standardization": (mean, std)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "group":
        out = []
        for k, c in enumerate(_group_sizes(case)):
            m = _Model(c, seed + 1000 * k)
            out.append(m.value(m.points(c["points"], near=False)))
        return torch.cat(out)
    m, theta = _inputs(case, seed)
    if kind == "spectrum":
        c = _couplings(theta)
        stage = case["stage"]
        if stage == 0:
            return (c @ m.basis)[0]
        if stage == 1:
            return (c @ m.shat)[0]
        mu = m.signal(theta)[0] if stage == 2 else m.mu(theta)[0]
        return mu * m.mask if stage == 3 and m.mask is not None else mu
    if kind == "rank8":
        return (m.value(theta), m.gradient(theta)) if case["grad"] else m.value(theta)
    if kind == "profiled":
        parts = [_profiled(m, c, case["sigma"]) for c in theta.split(2048)]
        return tuple(torch.cat(v) for v in zip(*parts))
    if kind == "surrogate":
        params = [tuple(torch.tensor(a, device="cuda").double() for a in layer) for layer in _network(m, seed)]
        return torch.cat([m.value_of(torch.exp(_forward(params, _normalised(c)))) for c in theta.split(16384)])
    if kind == "fit":
        return _trained(m, theta, case, seed)
    return m.value(theta)
