"""What a user has this library do, as timed cases: likelihood evaluations with their gradients.

A fit is a long run of goo_nll_grad calls on one dataset (a few hundred gradients per fit, FP32
first and FP64 for the last Newton steps), a toy study is many such fits side by side, and a scan
over a lineshape parameter rebuilds the amplitude caches between evaluations.  The cases cover each
model family in the precisions and forms that fits use, from a one-dimensional dataset whose
evaluation is bound by latency to the ten-million-event three-dimensional one.

listed() names the cases, draw() gives further ones of the same ranges, prepare() makes a case's
dataset, model and parameter point on the GPU, run() is one evaluation through the public calls,
work() counts what it cannot do without, and exact() is the same result in 64 bits from plain torch.
"""
import math
import random

import numpy as np
import torch

from paper_1710_08826_gb300 import goo

CHUNK = 1 << 19  # events per step of the 64-bit evaluation


def listed():
    return [
        # a one-dimensional mass or time fit: a small dataset that stays in L2, bound by latency
        dict(name="fit1d_f32", kind="1d", precision="f32", n=100_000),
        # the three-dimensional signal + background fit on ten million events, separable grid norm
        dict(name="fit3d_f32", kind="3d", precision="f32", n=10_000_000, bins=128),
        # its FP64 evaluation: the library's default precision, and the last Newton steps of a fit
        dict(name="fit3d_f64", kind="3d", precision="f64", n=3_000_001, bins=128),
        # the same model on weighted events (efficiency weights, or the centres of filled bins)
        dict(name="fit3d_weighted_f32", kind="3d_weighted", precision="f32", n=2_000_003, bins=128),
        # three-body amplitude fit, lineshapes fixed: the cached amplitudes are read once per call
        dict(name="dalitz_f32", kind="dalitz", precision="f32", n=5_000_000, n_mc=1_000_000, n_res=8),
        dict(name="dalitz_f64", kind="dalitz", precision="f64", n=2_000_000, n_mc=1_000_000, n_res=8),
        # the same with masses and widths free: every amplitude is evaluated on every call
        dict(name="dalitz_floating_f32", kind="dalitz_floating", precision="f32", n=5_000_000, n_mc=1_000_000,
             n_res=8),
        # a scan over a resonance mass with fixed lineshapes: three points, each rebuilding the
        # amplitude caches of the events and of the normalisation sample and the Gram matrix
        dict(name="dalitz_scan_f32", kind="dalitz_scan", precision="f32", n=2_000_000, n_mc=1_000_000, n_res=8),
        # the batched evaluation of a toy study: 64 toys of 1e3 to 1e6 events
        dict(name="toys_f32", kind="toys", precision="f32", n_toys=64, n_lo=1_000, n_hi=1_000_000, n_mc=1_000_000,
             n_res=8),
        # time-dependent four-body mixing fit
        dict(name="td4_f32", kind="td4", precision="f32", n=2_000_000, n_mc=3_000_000),
        dict(name="td4_f64", kind="td4", precision="f64", n=1_000_000, n_mc=1_000_000),
        # time-dependent three-body mixing fit
        dict(name="td3_f32", kind="td3", precision="f32", n=2_000_000, n_mc=1_000_000),
    ]


# kind -> fewest events, most in FP32, most in FP64 (None: the form is FP32 only)
RANGES = {"1d": (10_000, 2_000_000, 500_000), "3d": (50_000, 10_000_000, 3_000_000),
          "3d_weighted": (30_000, 3_000_000, 1_000_000), "dalitz": (50_000, 5_000_000, 2_000_000),
          "dalitz_floating": (50_000, 4_000_000, None), "dalitz_scan": (50_000, 2_000_000, None),
          "toys": (0, 0, None), "td4": (50_000, 2_000_000, 1_000_000), "td3": (50_000, 2_000_000, 800_000)}


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    lo, most32, most64 = RANGES[kind]
    case = dict(kind=kind, precision=rng.choice(("f32", "f64")) if most64 else "f32")
    if kind == "toys":
        case.update(n_toys=rng.randint(4, 96), n_lo=rng.randint(1_000, 5_000), n_hi=rng.randint(50_000, 500_000))
    else:
        hi = most64 if case["precision"] == "f64" else most32
        case["n"] = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    if kind in ("3d", "3d_weighted"):
        case["bins"] = rng.choice((32, 64, 100, 128, 200))
    if kind not in ("1d", "3d", "3d_weighted"):
        case["n_mc"] = rng.randint(200_000, 1_000_000)
    if kind in ("dalitz", "dalitz_floating", "dalitz_scan", "toys"):
        case["n_res"] = rng.randint(3, 8)
    return case


def toy_sizes(case):
    """The toys' event counts: log-uniform over [n_lo, n_hi], at the quantiles (i + 1/2) / n."""
    k, lo, hi = case["n_toys"], case["n_lo"], case["n_hi"]
    return [int(lo * (hi / lo) ** ((i + 0.5) / k)) for i in range(k)]


# ---------------------------------------------------------------------------------------
# models: parameters are (name, value, fixed, step)
# ---------------------------------------------------------------------------------------
def spec_1d():
    return dict(name="fit1d", observables=[("x", 0.0, 10.0)],
                params=[("mu", 5.0, False, 0.01), ("sigma", 0.4, False, 0.01), ("lam", -0.3, False, 0.005),
                        ("frac", 0.3, False, 0.005)],
                pdf=("add", ["frac"], [("gauss", "x", "mu", "sigma"), ("expo", "x", "lam")]), norm=("analytic",))


def spec_3d(bins):
    return dict(name="fit3d", observables=[("m", 5.2, 5.3), ("dE", -0.2, 0.2), ("t", 0.0, 10.0)],
                params=[("mu_m", 5.279, False, 1e-4), ("sig_m", 0.003, False, 1e-4), ("mu_de", 0.0, False, 1e-3),
                        ("sig_de", 0.02, False, 1e-3), ("lam_s", -1.0 / 1.5, False, 1e-2), ("m0", 5.29, False, 1e-4),
                        ("c", -20.0, False, 0.5), ("p", 0.5, False, 0.02), ("a1", -1.0, False, 0.05),
                        ("a2", 0.5, False, 0.2), ("lam_b", -1.0 / 0.8, False, 1e-2), ("frac", 0.2, False, 1e-3)],
                pdf=("add", ["frac"], [
                    ("prod", [("gauss", "m", "mu_m", "sig_m"), ("gauss", "dE", "mu_de", "sig_de"),
                              ("expo", "t", "lam_s")]),
                    ("prod", [("argus", "m", "m0", "c", "p"), ("poly2", "dE", "a1", "a2"), ("expo", "t", "lam_b")])]),
                norm=("grid", [bins] * 3))


KPIPI0 = dict(M=1.865, m1=0.494, m2=0.140, m3=0.135, r_res=1.5, r_par=5.0)
# pair, spin, mass, width, coefficient of the three-body resonances (the constant term is the reference)
DALITZ = [("12", 1, 0.8955, 0.0473, 0.913, 0.303), ("13", 1, 0.8955, 0.0473, -0.456, 0.580),
          ("23", 1, 0.7753, 0.1491, 0.999, -0.447), ("12", 0, 1.425, 0.270, 0.585, 0.400),
          ("13", 0, 1.425, 0.270, -0.411, 0.366), ("12", 2, 1.4324, 0.109, 1.252, -0.293),
          ("12", 1, 1.718, 0.322, 1.726, 1.725), ("23", 1, 1.465, 0.400, -0.918, 1.725)]
PIPIPI0 = dict(M=1.865, m1=0.1350, m2=0.1396, m3=0.1396, r_res=1.5, r_par=5.0)
TD3 = [("12", 1, 0.7753, 0.1491, 1.0, 0.0), ("13", 1, 0.7753, 0.1491, 0.55, 0.45), ("23", 1, 0.7753, 0.1491, 0.52, 0.28),
       ("12", 1, 1.465, 0.400, 0.35, -0.25), ("13", 1, 1.465, 0.400, 0.30, 0.35), ("23", 1, 1.465, 0.400, 0.20, 0.10),
       ("12", 1, 1.720, 0.250, 0.25, 0.30), ("13", 1, 1.720, 0.250, -0.20, 0.30), ("23", 1, 1.720, 0.250, 0.15, -0.20),
       ("23", 0, 0.990, 0.070, 0.12, 0.05), ("23", 2, 1.2755, 0.1867, 0.25, 0.15), ("23", 0, 1.350, 0.350, 0.20, -0.10),
       ("23", 0, 1.505, 0.109, 0.10, 0.08), ("23", 0, 0.500, 0.400, 0.30, 0.20), ("23", 0, 1.720, 0.135, 0.06, -0.04)]
KPIPIPI = dict(M=1.865, m1=0.494, m2=0.140, m3=0.140, m4=0.140, r_res=1.5)
KST, K0ST, K2ST, KST14 = (0.8955, 0.0473), (1.425, 0.270), (1.4324, 0.109), (1.414, 0.232)
RHO, F0, RHO14 = (0.7753, 0.1491), (0.990, 0.070), (1.465, 0.400)
# angular structure, resonance in pair 12, in pair 34, free coefficient, fixed coefficient
TD4 = [("VV0", KST, RHO, (1.0, 0.0), (0.9, 0.3)), ("VVpar", KST, RHO, (0.45, 0.2), (0.3, -0.1)),
       ("VVperp", KST, RHO, (-0.3, 0.25), (0.2, 0.3)), ("VS0", KST, F0, (0.35, -0.15), (-0.4, 0.2)),
       ("SV0", K0ST, RHO, (0.5, 0.3), (0.45, 0.1)), ("SS", K0ST, F0, (0.25, -0.4), (0.3, 0.25)),
       ("TV0", K2ST, RHO, (0.3, 0.1), (-0.25, 0.2)), ("TS0", K2ST, F0, (-0.2, 0.15), (0.2, -0.1)),
       ("VV0", KST14, RHO, (0.4, -0.25), (0.35, 0.2)), ("VV0", KST, RHO14, (0.3, 0.35), (0.25, -0.3))]
SPINS = {"SS": (0, 0), "VS0": (1, 0), "SV0": (0, 1), "VV0": (1, 1), "VVpar": (1, 1), "VVperp": (1, 1), "TS0": (2, 0),
         "TV0": (2, 1)}
TIME = [("x", 0.004, False, 0.002), ("y", 0.006, False, 0.002), ("tau", 0.41, False, 0.002),
        ("sigma_t", 0.05, False, 0.001)]
T_LIMITS = ("t", -0.5, 10.0)


def dalitz_limits(kin):
    M, m1, m2, m3 = (kin[k] for k in ("M", "m1", "m2", "m3"))
    return [("s12", (m1 + m2) ** 2, (M - m3) ** 2), ("s13", (m1 + m3) ** 2, (M - m2) ** 2)]


def spec_three_body(kin, res, nr, time=False, floating=False):
    """Resonances with (mass, width, re, im) each and the constant amplitude; time: the mixing model."""
    params, amps = [], []
    for k, (pair, spin, m0, w, re, im) in enumerate(res):
        fixed = time and k == 0
        params += [(f"m0_{k}", m0, not floating, 0.001 if floating else 0.0),
                   (f"w_{k}", w, not floating, 0.001 if floating else 0.0),
                   (f"re_{k}", re, fixed, 0.02), (f"im_{k}", im, fixed, 0.02)]
        amps.append(("bw", pair, spin, f"m0_{k}", f"w_{k}", f"re_{k}", f"im_{k}"))
    params += [("re_nr", nr[0], not time, 0.02), ("im_nr", nr[1], not time, 0.02)]
    amps.append(("nr", "re_nr", "im_nr"))
    obs = dalitz_limits(kin)
    if not time:
        return dict(name="dalitz", observables=obs, params=params, pdf=("coherent", kin, amps), norm=("mc",))
    return dict(name="td3", observables=obs + [T_LIMITS], params=params + TIME,
                pdf=("td3", kin, amps, ("x", "y", "tau", "sigma_t")), norm=("mc",))


def spec_td4():
    kin = KPIPIPI
    M, m1, m2, m3, m4 = (kin[k] for k in ("M", "m1", "m2", "m3", "m4"))
    params, amps = [], []
    for k, (ang, r12, r34, (re, im), cf) in enumerate(TD4):
        params += [(f"re_{k}", re, False, 0.02), (f"im_{k}", im, False, 0.02)]
        amps.append((ang, r12, r34, f"re_{k}", f"im_{k}", cf))
    return dict(name="td4",
                observables=[("m12", m1 + m2, M - m3 - m4), ("m34", m3 + m4, M - m1 - m2), ("c12", -1.0, 1.0),
                             ("c34", -1.0, 1.0), ("phi", -math.pi, math.pi), T_LIMITS],
                params=params + TIME, pdf=("td4", kin, amps, ("x", "y", "tau", "sigma_t")), norm=("mc",))


def spec_of(case):
    kind = case["kind"]
    if kind == "1d":
        return spec_1d()
    if kind in ("3d", "3d_weighted"):
        return spec_3d(case["bins"])
    if kind == "td4":
        return spec_td4()
    if kind == "td3":
        return spec_three_body(PIPIPI0, TD3, (0.5, 0.2), time=True)
    return spec_three_body(KPIPI0, DALITZ[:case["n_res"]], (1.0, 0.0), floating=kind == "dalitz_floating")


def point(spec, seed, steps=3.0):
    """A parameter point as a fit meets it on its way: each free parameter a few steps off its true value."""
    rng = random.Random(seed)
    return np.array([v if fixed else v + steps * step * rng.uniform(-1.0, 1.0) for _, v, fixed, step in spec["params"]])


# ---------------------------------------------------------------------------------------
# events, made on the GPU
# ---------------------------------------------------------------------------------------
class Sampler:
    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))
        self.dtype = dtype

    def uniform(self, n, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(n, generator=self.g, device="cuda", dtype=self.dtype)

    def normal(self, n, mean=0.0, sigma=1.0):
        return mean + sigma * torch.randn(n, generator=self.g, device="cuda", dtype=self.dtype)

    def exponential(self, n, mean=1.0):
        return -mean * torch.log1p(-self.uniform(n))

    def kept(self, n, trial, batch=None):
        """n rows of what trial(k) keeps of k candidates: a list of equally long columns."""
        parts, have = [], 0
        while have < n:
            cols = trial(batch or max(4096, int(1.3 * (n - have))))
            parts.append(cols)
            have += cols[0].numel()
        return [torch.cat(c)[:n] for c in zip(*parts)]

    def inside(self, n, make, lo, hi):
        def trial(k):
            v = make(k)
            return [v[(v > lo) & (v < hi)]]
        return self.kept(n, trial)[0]


def events_1d(s, n):
    n_sig = int(0.3 * n)
    x = torch.cat([s.inside(n_sig, lambda k: s.normal(k, 5.0, 0.4), 0.0, 10.0),
                   s.inside(n - n_sig, lambda k: s.exponential(k, 1.0 / 0.3), 0.0, 10.0)])
    return [x[torch.randperm(n, generator=s.g, device="cuda")]]


def events_3d(s, n):
    n_sig = int(0.2 * n)
    n_bkg = n - n_sig

    def argus(k):  # u = 1 - m^2 / m0^2 ~ Gamma(3/2, 1/20)
        u = (s.exponential(k) + 0.5 * s.normal(k) ** 2) / 20.0
        return 5.29 * torch.sqrt((1.0 - u).clamp_min(0.0))

    def poly(k):
        x = s.uniform(k, -0.2, 0.2)
        return [x[(s.uniform(k, 0.0, 1.22) < 1.0 - x + 0.5 * x * x) & (x > -0.2) & (x < 0.2)]]

    m = torch.cat([s.inside(n_sig, lambda k: s.normal(k, 5.279, 0.003), 5.2, 5.2999),
                   s.inside(n_bkg, argus, 5.2001, 5.29)])
    de = torch.cat([s.inside(n_sig, lambda k: s.normal(k, 0.0, 0.02), -0.2, 0.2), s.kept(n_bkg, poly)[0]])
    t = torch.cat([s.inside(n_sig, lambda k: s.exponential(k, 1.5), 0.0, 10.0),
                   s.inside(n_bkg, lambda k: s.exponential(k, 0.8), 0.0, 10.0)])
    perm = torch.randperm(n, generator=s.g, device="cuda")
    return [m[perm], de[perm], t[perm]]


def dalitz_uniform(s, k, kin):
    """k candidates of the Dalitz box, those inside the kinematic region."""
    M, m1, m2, m3 = (kin[q] for q in ("M", "m1", "m2", "m3"))
    (_, a0, a1), (_, b0, b1) = dalitz_limits(kin)
    a, b = s.uniform(k, a0, a1), s.uniform(k, b0, b1)
    r = torch.sqrt(a)
    e1, e3 = (a + m1 * m1 - m2 * m2) / (2 * r), (M * M - a - m3 * m3) / (2 * r)
    p1, p3 = torch.sqrt((e1 * e1 - m1 * m1).clamp_min(0)), torch.sqrt((e3 * e3 - m3 * m3).clamp_min(0))
    es = (e1 + e3) ** 2
    ok = (b > es - (p1 + p3) ** 2) & (b < es - (p1 - p3) ** 2) & (e3 > m3) & (a > a0) & (a < a1) & (b > b0) & (b < b1)
    return [a[ok], b[ok]]


def dalitz_model_events(s, n, kin, res, nr):
    """n events of |sum c_k A_k|^2 by accept-reject from uniform candidates."""
    top = None

    def trial(k):
        nonlocal top
        a, b = dalitz_uniform(s, k, kin)
        sr, si = torch.full_like(a, nr[0]), torch.full_like(a, nr[1])
        for pair, spin, m0, w, re, im in res:
            ar, ai = breit_wigner(kin, pair, spin, m0, w, a, b)
            sr, si = sr + re * ar - im * ai, si + re * ai + im * ar
        f = sr * sr + si * si
        top = 1.1 * float(f.max()) if top is None else top
        keep = s.uniform(f.numel(), 0.0, top) < f
        return [a[keep], b[keep]]

    return s.kept(n, trial, batch=1 << 22)


def decay_times(s, n):
    def trial(k):
        t = s.exponential(k, 0.41) + s.normal(k, 0.0, 0.05)
        return [t[(t > T_LIMITS[1]) & (t < T_LIMITS[2])]]
    return s.kept(n, trial)[0]


def four_body(s, n, kin):
    """n points of four-body phase space: (m12, m34) by accept-reject on p q12 q34, uniform angles."""
    M, m1, m2, m3, m4 = (kin[q] for q in ("M", "m1", "m2", "m3", "m4"))

    def momentum(m, a, b):
        lam = (m * m - (a + b) ** 2) * (m * m - (a - b) ** 2)
        return torch.sqrt(lam.clamp_min(0)) / (2 * m)

    top = None

    def trial(k):
        nonlocal top
        a, b = s.uniform(k, m1 + m2, M - m3 - m4), s.uniform(k, m3 + m4, M - m1 - m2)
        w = momentum(torch.full_like(a, M), a, b) * momentum(a, m1, m2) * momentum(b, m3, m4)
        w = torch.where((a + b < M) & (a > m1 + m2) & (b > m3 + m4) & (a < M - m3 - m4) & (b < M - m1 - m2), w, 0.0 * w)
        top = 1.1 * float(w.max()) if top is None else top
        keep = s.uniform(k, 0.0, top) < w
        return [a[keep], b[keep]]

    lim = 1.0 - 1e-6
    return s.kept(n, trial, batch=1 << 21) + [s.uniform(n, -lim, lim), s.uniform(n, -lim, lim),
                                              s.uniform(n, -math.pi * lim, math.pi * lim)]


def make_events(case, seed):
    """The case's event columns (a list of them for the toys), and its normalisation sample's."""
    s = Sampler(seed, torch.float64 if case["precision"] == "f64" else torch.float32)
    kind, mc = case["kind"], None
    if kind == "1d":
        return events_1d(s, case["n"]), None
    if kind in ("3d", "3d_weighted"):
        return events_3d(s, case["n"]), None
    if kind == "td4":
        mc = four_body(s, case["n_mc"], KPIPIPI)
        mc.append(torch.zeros_like(mc[0]))
        return four_body(s, case["n"], KPIPIPI) + [decay_times(s, case["n"])], mc
    kin, res, nr = (PIPIPI0, TD3, (0.5, 0.2)) if kind == "td3" else (KPIPI0, DALITZ[:case["n_res"]], (1.0, 0.0))
    mc = s.kept(case["n_mc"], lambda k: dalitz_uniform(s, k, kin))
    if kind == "td3":
        mc.append(torch.zeros_like(mc[0]))
        return dalitz_model_events(s, case["n"], kin, res, nr) + [decay_times(s, case["n"])], mc
    if kind == "toys":
        sizes = toy_sizes(case)
        pool = dalitz_model_events(s, sum(sizes), kin, res, nr)
        parts = [torch.split(c, sizes) for c in pool]
        return [[c.clone() for c in toy] for toy in zip(*parts)], mc
    return dalitz_model_events(s, case["n"], kin, res, nr), mc


def make_weights(case, seed):
    """Per-event weights: efficiency corrections around 1, one event in ten left out (an empty bin)."""
    if case["kind"] != "3d_weighted":
        return None
    s = Sampler(seed + 1, torch.float32)
    w = s.uniform(case["n"], 0.5, 1.5)
    return torch.where(s.uniform(case["n"]) < 0.1, torch.zeros_like(w), w)


def make_thetas(case, seed, spec):
    """The parameter points of one pass: one, one per toy, or the points of the mass scan."""
    if case["kind"] == "toys":
        return [point(spec, seed * 1000 + i) for i in range(case["n_toys"])]
    theta = point(spec, seed)
    if case["kind"] != "dalitz_scan":
        return [theta]
    points = [theta.copy() for _ in range(3)]
    for p, shift in zip(points, (-0.002, 0.0, 0.002)):
        p[0] += shift  # the first resonance's mass
    return points


# ---------------------------------------------------------------------------------------
# the framework's side
# ---------------------------------------------------------------------------------------
_ctx = None


def prepare(case, seed):
    global _ctx
    if _ctx is None:
        _ctx = goo.Context(0)
    spec = spec_of(case)
    cols, mc = make_events(case, seed)
    torch.cuda.synchronize()  # the library reads the columns on its own stream
    lo, hi = [o[1] for o in spec["observables"]], [o[2] for o in spec["observables"]]

    def dataset(c):
        return goo.Dataset(_ctx, c, lo[:len(c)], hi[:len(c)], dtype=case["precision"])

    state = dict(kind=case["kind"], precision=case["precision"], thetas=make_thetas(case, seed, spec))
    state["data"] = [dataset(c) for c in cols] if case["kind"] == "toys" else dataset(cols)
    state["model"] = goo.Model(_ctx, spec, mc=dataset(mc) if mc else None)
    w = make_weights(case, seed)
    if w is not None:
        state["data"].set_weights(w.double().cpu().numpy())
    if case["kind"] == "dalitz_floating":
        state["model"].set_lineshapes("floating")
    return state


def given(precision, nll, grad):
    """An evaluation's results in the type their precision stands for."""
    t = np.float32 if precision == "f32" else np.float64
    return dict(nll=np.asarray(nll, dtype=t), grad=np.asarray(grad, dtype=t))


def run(state):
    model, data, precision, thetas = state["model"], state["data"], state["precision"], state["thetas"]
    if state["kind"] == "toys":
        return given(precision, *goo.nll_grad_batch(model, data, thetas, precision))
    if state["kind"] == "dalitz_scan":
        found = [model.nll_grad(data, th, precision) for th in thetas]
        return given(precision, [f[0] for f in found], [f[1] for f in found])
    return given(precision, *model.nll_grad(data, thetas[0], precision))


def work(case):
    """Events (or their cached amplitudes, where the lineshapes are fixed) read once; the arithmetic of
    the densities, their logarithms and the gradient lanes, a transcendental function counted as 10."""
    kind, size = case["kind"], 8 if case["precision"] == "f64" else 4
    n = sum(toy_sizes(case)) if kind == "toys" else case["n"]
    if kind == "1d":
        return dict(bytes=n * size, flops=n * 60)
    if kind in ("3d", "3d_weighted"):
        return dict(bytes=n * size * (4 if kind == "3d_weighted" else 3), flops=n * 150)
    if kind == "td4":
        return dict(bytes=n * size * (2 * len(TD4) + 1), flops=n * (24 * len(TD4) + 250))
    if kind == "td3":
        return dict(bytes=n * size * (4 * len(TD3) + 1), flops=n * (32 * len(TD3) + 270))
    k = case["n_res"]
    if kind == "dalitz_floating":
        return dict(bytes=(n + case["n_mc"]) * 2 * size, flops=(n + case["n_mc"]) * (120 * k + 30))
    if kind == "dalitz_scan":
        both = n + case["n_mc"]
        return dict(bytes=3 * both * 2 * size, flops=3 * (both * 80 * k + n * (16 * k + 30) + case["n_mc"] * 4 * k * k))
    return dict(bytes=n * size * 2 * k, flops=n * (16 * k + 30))


# ---------------------------------------------------------------------------------------
# the same results in 64 bits, by plain torch and its automatic differentiation
# ---------------------------------------------------------------------------------------
def breit_wigner(kin, pair, spin, m0, w, s12, s13):
    """Relativistic Breit-Wigner with running width, barrier factors and the spin factor, as (re, im)."""
    M, m1, m2, m3 = (kin[q] for q in ("M", "m1", "m2", "m3"))
    s23 = M * M + m1 * m1 + m2 * m2 + m3 * m3 - s12 - s13
    mA, mB, mC, s, sac, sbc = {"12": (m1, m2, m3, s12, s13, s23), "13": (m1, m3, m2, s13, s12, s23),
                               "23": (m2, m3, m1, s23, s12, s13)}[pair]
    lam = (s - (mA + mB) ** 2) * (s - (mA - mB) ** 2)
    lam_p = (s - (M + mC) ** 2) * (s - (M - mC) ** 2)
    q2 = (lam / (4 * s)).clamp_min(0)
    u = m0 * m0
    q02 = (u - (mA + mB) ** 2) * (u - (mA - mB) ** 2) / (4 * u)
    r2, z_p = kin["r_res"] ** 2, (kin["r_par"] ** 2 * lam_p / (4 * M * M)).clamp_min(0)
    z, z0 = r2 * q2, r2 * q02
    if spin == 0:
        ratio2, parent, factor = 1.0, 1.0, 1.0
    else:
        z1 = sac - sbc - (mA * mA - mB * mB) * (M * M - mC * mC) / s
        if spin == 1:
            ratio2, parent, factor = (1 + z0) / (1 + z), 1 / torch.sqrt(1 + z_p), z1
        else:
            ratio2 = (9 + 3 * z0 + z0 * z0) / (9 + 3 * z + z * z)
            parent, factor = 3 / torch.sqrt(9 + 3 * z_p + z_p * z_p), z1 * z1 - lam * lam_p / (3 * s * s)
    rho = q2 / q02
    di = m0 * w * torch.sqrt(rho) * rho ** spin * m0 / torch.sqrt(s) * ratio2
    dr = u - s
    scale = (ratio2 ** 0.5 if spin else 1.0) * parent * factor / (dr * dr + di * di)
    return dr * scale, di * scale


def three_body_sum(kin, res, coef, s12, s13):
    """sum_k c_k A_k as (re, im); coef: (mass, width, re, im) per resonance and the constant's (re, im)."""
    sr, si = coef[-1][0] + torch.zeros_like(s12), coef[-1][1] + torch.zeros_like(s12)
    for (pair, spin, *_), (m0, w, re, im) in zip(res, coef):
        ar, ai = breit_wigner(kin, pair, spin, m0, w, s12, s13)
        sr, si = sr + re * ar - im * ai, si + re * ai + im * ar
    return sr, si


def four_body_amplitudes(kin, m12, m34, c12, c34, phi):
    def barrier(L, z):
        return 1.0 if L == 0 else (1 / (1 + z)) ** 0.5 if L == 1 else (9 / (9 + 3 * z + z * z)) ** 0.5

    def shape(m, m0, g0, L, a, b):
        q = torch.sqrt(((m * m - (a + b) ** 2) * (m * m - (a - b) ** 2)).clamp_min(0)) / (2 * m)
        q0 = math.sqrt((m0 * m0 - (a + b) ** 2) * (m0 * m0 - (a - b) ** 2)) / (2 * m0)
        ratio = barrier(L, (kin["r_res"] * q) ** 2) / barrier(L, (kin["r_res"] * q0) ** 2)
        width = g0 * (q / q0) ** (2 * L + 1) * (m0 / m) * ratio ** 2
        return (q / q0) ** L * ratio / torch.complex(m0 * m0 - m * m, -m0 * width)

    st = torch.sqrt(((1 - c12 * c12) * (1 - c34 * c34)).clamp_min(0))
    p2 = 0.5 * (3 * c12 * c12 - 1)
    angle = {"SS": torch.ones_like(c12), "VS0": c12, "SV0": c34, "VV0": c12 * c34, "VVpar": st * torch.cos(phi),
             "VVperp": 1j * st * torch.sin(phi), "TS0": p2, "TV0": p2 * c34}
    out = []
    for ang, r12, r34, _, _ in TD4:
        L1, L2 = SPINS[ang]
        out.append(shape(m12, *r12, L1, kin["m1"], kin["m2"]) * shape(m34, *r34, L2, kin["m3"], kin["m4"]) * angle[ang])
    return torch.stack(out)


def time_terms(t, x, y, tau, s):
    """(T_ch, T_sh, T_c, T_s): cosh, sinh(y t / tau) and cos, sin(x t / tau) times e^(-t / tau), convolved with
    a Gaussian of width s, by the Taylor series in the moments of the convolved exponential."""
    G = 1 / tau
    u = (G * s * s - t) / (s * math.sqrt(2.0))
    gauss = torch.exp(-0.5 * (t / s) ** 2)
    h = 0.5 * gauss * torch.special.erfcx(u.abs())
    m0 = torch.where(u >= 0, h, torch.exp(0.5 * G * G * s * s - G * t) - h)
    v = t - G * s * s
    m = [m0, G * (v * m0 + s * gauss / math.sqrt(2 * math.pi))]
    for n in range(1, 15):
        m.append((G * v * m[n] + (G * s) ** 2 * m[n - 1]) / (n + 1))
    ch = sum(y ** k * m[k] for k in range(0, 16, 2))
    sh = sum(y ** k * m[k] for k in range(1, 16, 2))
    c = sum((-1) ** (k // 2) * x ** k * m[k] for k in range(0, 16, 2))
    sn = sum((-1) ** (k // 2) * x ** k * m[k] for k in range(1, 16, 2))
    return ch, sh, c, sn


def rate(A, B, terms):
    ch, sh, c, sn = terms
    aa, bb = (A * A.conj()).real, (B * B.conj()).real
    ab = A * B.conj()
    return 0.5 * (aa + bb) * ch + 0.5 * (aa - bb) * c + ab.real * sh + ab.imag * sn


def exact_density(case, spec):
    """log of the unnormalised density over a chunk of event columns, and the chunk's share of the
    normalisation integral over the phase-space sample, both as functions of theta."""
    kind = case["kind"]
    at = {p[0]: i for i, p in enumerate(spec["params"])}

    def integrals(th):
        x, y, tau = (th[at[q]] for q in ("x", "y", "tau"))
        return tau / (1 - y * y), y * tau / (1 - y * y), tau / (1 + x * x), x * tau / (1 + x * x)

    def terms(th, t):
        return time_terms(t, *(th[at[q]] for q in ("x", "y", "tau", "sigma_t")))

    if kind == "td4":
        fixed = torch.tensor([complex(*a[4]) for a in TD4], dtype=torch.complex128, device="cuda")

        def sums(th, cols):
            a = four_body_amplitudes(KPIPIPI, *cols[:5])
            c = torch.complex(th[0:2 * len(TD4):2], th[1:2 * len(TD4):2])
            return c @ a, fixed @ a
    else:
        kin, res = (PIPIPI0, TD3) if kind == "td3" else (KPIPI0, DALITZ[:case["n_res"]])

        def coefs(th):
            free = kind == "dalitz_floating"
            shapes = th if free else th.detach()
            return [(shapes[4 * k], shapes[4 * k + 1], th[4 * k + 2], th[4 * k + 3]) for k in range(len(res))] + \
                [(th[4 * len(res)], th[4 * len(res) + 1])]

        def sums(th, cols):
            c = coefs(th)
            a = torch.complex(*three_body_sum(kin, res, c, cols[0], cols[1]))
            return (a, torch.complex(*three_body_sum(kin, res, c, cols[1], cols[0]))) if kind == "td3" else (a, None)

    def logf(th, cols):
        A, B = sums(th, cols)
        return torch.log(A.real ** 2 + A.imag ** 2 if B is None else rate(A, B, terms(th, cols[-1])))

    def norm(th, cols):
        A, B = sums(th, cols)
        return A.real ** 2 + A.imag ** 2 if B is None else rate(A, B, integrals(th))

    return logf, norm


def exact_leaf(node, th, at, x):
    """log of a leaf's shape at x."""
    p = [th[at[q]] for q in node[2:]]
    if node[0] == "gauss":
        return -0.5 * ((x - p[0]) / p[1]) ** 2
    if node[0] == "expo":
        return p[0] * x
    if node[0] == "poly2":
        return torch.log(1 + p[0] * x + p[1] * x * x)
    u = 1 - (x / p[0]) ** 2
    ok = u > 0
    u = torch.where(ok, u, torch.ones_like(u))
    return torch.where(ok, torch.log(x) + p[2] * torch.log(u) + p[1] * u, torch.full_like(x, -math.inf))


def exact_sop(case, spec):
    """log of the density, normalised by closed forms (1d) or the midpoint grid (3d), over a chunk."""
    at = {p[0]: i for i, p in enumerate(spec["params"])}
    obs = {o[0]: i for i, o in enumerate(spec["observables"])}
    lim = {o[0]: o[1:] for o in spec["observables"]}

    def log_norm(node, th):
        lo, hi = lim[node[1]]
        if spec["norm"][0] == "grid":
            b = spec["norm"][1][obs[node[1]]]
            step = (hi - lo) / b
            mid = lo + (torch.arange(b, dtype=torch.float64, device="cuda") + 0.5) * step
            return torch.logsumexp(exact_leaf(node, th, at, mid), 0) + math.log(step)
        p = [th[at[q]] for q in node[2:]]
        if node[0] == "gauss":
            a, b = ((v - p[0]) / (p[1] * math.sqrt(2.0)) for v in (lo, hi))
            return torch.log(p[1] * math.sqrt(math.pi / 2) * (torch.erf(b) - torch.erf(a)))
        return torch.log((torch.exp(p[0] * hi) - torch.exp(p[0] * lo)) / p[0])

    _, (frac,), products = spec["pdf"]

    def logf(th, cols):
        f = th[at[frac]]
        found = []
        for weight, node in zip((f, 1 - f), products):
            leaves = node[1] if node[0] == "prod" else [node]
            found.append(torch.log(weight) + sum(exact_leaf(q, th, at, cols[obs[q[1]]]) - log_norm(q, th) for q in leaves))
        return torch.logsumexp(torch.stack(found), 0)

    return logf


def exact_point(case, spec, theta, cols, mc, weights):
    """(NLL, its gradient) at theta in 64 bits."""
    th = torch.tensor(theta, dtype=torch.float64, device="cuda", requires_grad=True)
    n = cols[0].numel()

    def over(columns, of):
        total, grad = torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(th)
        for i in range(0, columns[0].numel(), CHUNK):
            v = of(th, [c[i:i + CHUNK].double() for c in columns], i)
            g, = torch.autograd.grad(v, th)
            total, grad = total + v.detach(), grad + g
        return total, grad

    if mc is None:
        logf, norm = exact_sop(case, spec), None
    else:
        logf, norm = exact_density(case, spec)

    def summed(th, c, i):
        v = logf(th, c)
        if weights is None:
            return v.sum()
        w = weights[i:i + CHUNK].double()
        return torch.where(w > 0, w * v, torch.zeros_like(v)).sum()

    s, g = over(cols, summed)
    if norm is None:
        return float(-s), (-g).cpu().numpy()
    total, dn = over(mc, lambda th, c, i: norm(th, c).sum())
    return float(-s + n * torch.log(total / mc[0].numel())), (-g + n * dn / total).cpu().numpy()


def exact(case, seed):
    spec = spec_of(case)
    cols, mc = make_events(case, seed)
    thetas, weights = make_thetas(case, seed, spec), make_weights(case, seed)
    if case["kind"] == "toys":
        found = [exact_point(case, spec, th, c, mc, None) for th, c in zip(thetas, cols)]
    else:
        found = [exact_point(case, spec, th, cols, mc, weights) for th in thetas]
    nll, grad = np.array([f[0] for f in found]), np.array([f[1] for f in found])
    if case["kind"] not in ("toys", "dalitz_scan"):
        nll, grad = nll[0], grad[0]
    return dict(nll=np.float64(nll) if np.ndim(nll) == 0 else nll, grad=grad)
