"""The work a user of this package has it do, as cases that can be timed and checked.

Each case is one call (or the few calls that belong together) through the
public binding: operators, whole MAP solves, the differentiable MAP, the batch,
the comparison filters, the linear-bias model and the diagnostics.  Inputs are
synthetic lognormal-Poisson grids with the P(k) shape, boxes, amplitudes,
densities and selections of `mocks.WORKLOADS` and `mocks.batch_specs`, drawn on
the GPU from the seed.  `exact` is the same mathematics in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_0911_1407_gb300 import Batch, Context, mocks
from paper_0911_1407_gb300.autograd import map_field, neg_log_posterior

F64 = torch.float64

# Grid sides the library accepts (even, prime factors 2 and 3), by what users
# of the cases below run them at.
SIDES = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384,
         432, 512]


def listed():
    return [
        # The Hessian-vector product of the production workload (256^3, FP32
        # fields): the operator inside every CG iteration, and the call of a
        # user who brings an iteration of their own.
        {"name": "hv_mixed_256", "call": "hessvec", "precision": "mixed", "n": 256,
         "box": 500.0, "sigma": 1.8, "nbar": 1.0, "selection": False},
        # The same product in double precision with a survey selection, at the
        # side of the `selection128` workload.
        {"name": "hv_fp64_128", "call": "hessvec", "precision": "fp64", "n": 128,
         "box": 500.0, "sigma": 1.5, "nbar": 0.5, "selection": True},
        # The largest grid the library takes.
        {"name": "hv_mixed_512", "call": "hessvec", "precision": "mixed", "n": 512,
         "box": 1000.0, "sigma": 1.8, "nbar": 1.0, "selection": False},
        # -ln P and its gradient through torch autograd, forward and backward:
        # what a sampler or an outer optimiser calls, in double precision.
        {"name": "grad_fp64_192", "call": "grad", "precision": "fp64", "n": 192,
         "box": 500.0, "sigma": 1.5, "nbar": 0.5, "selection": True},
        # A whole reconstruction at production size and default options.
        {"name": "map_mixed_256", "call": "map", "precision": "mixed", "n": 256,
         "box": 500.0, "sigma": 1.8, "nbar": 1.0, "selection": False, "tol": 1e-6},
        # A whole reconstruction in double precision with a survey selection.
        {"name": "map_fp64_128", "call": "map", "precision": "fp64", "n": 128,
         "box": 500.0, "sigma": 1.5, "nbar": 0.5, "selection": True, "tol": 1e-6},
        # The smallest whole solve in use (`plain32`): all launches and latency.
        {"name": "map_fp64_32", "call": "map", "precision": "fp64", "n": 32,
         "box": 200.0, "sigma": 1.0, "nbar": 2.0, "selection": False, "tol": 1e-6},
        # The MAP as a differentiable function of counts and amplitude, forward
        # and backward (`adjoint128`).
        {"name": "adjoint_mixed_128", "call": "adjoint", "precision": "mixed", "n": 128,
         "box": 500.0, "sigma": 1.2, "nbar": 1.0, "selection": False, "tol": 1e-6},
        # 64 independent mocks of uneven size in one launch (`batch_specs`).
        {"name": "batch_64", "call": "batch", "precision": "mixed", "n": 128, "count": 64,
         "tol": 1e-6},
        # The estimators a reconstruction is compared with: LSQ-Wiener filter
        # and Gaussian-prior MAP, on a survey grid of a batch side.
        {"name": "filters_mixed_96", "call": "filters", "precision": "mixed", "n": 96,
         "box": 375.0, "sigma": 1.0, "nbar": 2.0, "selection": True, "tol": 1e-6},
        # The linear-bias model's objective, gradient and Hessian-vector
        # product at a side that is not a power of two: small and ragged.
        {"name": "bias_mixed_54", "call": "bias", "precision": "mixed", "n": 54,
         "box": 210.9375, "sigma": 0.6, "nbar": 2.0, "selection": False},
        # What follows a reconstruction: smoothing, the histogram and moments
        # of ln(1 + delta), and the comparison with a reference field.
        {"name": "diagnostics_256", "call": "diagnostics", "precision": "fp64", "n": 256,
         "box": 500.0, "sigma": 1.0, "nbar": 1.0, "selection": False},
    ]


def draw(rng):
    call = rng.choice(["hessvec", "hessvec", "grad", "map", "map", "adjoint", "batch", "filters",
                       "bias", "diagnostics"])
    precision = rng.choice(["mixed", "fp64"])
    most = {"hessvec": 512 if precision == "mixed" else 256, "grad": 256, "batch": 128,
            "map": 256 if precision == "mixed" else 128, "adjoint": 128, "filters": 128,
            "bias": 128, "diagnostics": 256}[call]
    # sides spread over their logarithm
    want = math.exp(rng.uniform(math.log(16), math.log(most)))
    n = min((s for s in SIDES if s <= most), key=lambda s: abs(math.log(s / want)))
    case = {"call": call, "precision": precision, "n": n,
            "box": round(n * rng.uniform(1.9, 6.3), 3),
            "sigma": round(rng.uniform(0.8, 1.8) if call not in ("bias", "filters")
                           else rng.uniform(0.4, 0.8), 3),
            "nbar": round(math.exp(rng.uniform(math.log(0.2), math.log(2.0))), 3),
            "selection": rng.random() < 0.5}
    if call in ("bias", "filters"):
        case["nbar"] = round(rng.uniform(1.0, 3.0), 3)
    if call in ("map", "adjoint", "batch", "filters"):
        case["tol"] = 1e-6
    if call == "batch":
        case = {"call": call, "precision": "mixed", "n": n, "count": rng.randint(2, 48),
                "tol": 1e-6}
    if call == "diagnostics":
        case["precision"] = "fp64"
        case["selection"] = False
    return case


# ------------------------------- inputs ------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _m2(n):
    """|m|^2 on the half spectrum [z][y][kx]."""
    m = torch.fft.fftfreq(n, 1.0 / n, dtype=F64, device="cuda") ** 2
    mx = torch.arange(n // 2 + 1, dtype=F64, device="cuda") ** 2
    return m[:, None, None] + m[None, :, None] + mx[None, None, :]


def _amplitude(n, box, sigma):
    """A such that the per-cell variance of the Gaussian field is sigma^2."""
    m2 = _m2(n)
    k = (2.0 * math.pi / box) * m2.sqrt()
    p = k / (1.0 + (k / 0.02) ** 2) ** 1.4
    twice = torch.full((n // 2 + 1,), 2.0, dtype=F64, device="cuda")
    twice[0] = twice[-1] = 1.0
    return sigma ** 2 * box ** 3 / float((p * twice).sum())


def _gaussian(n, box, A, gen):
    k = (2.0 * math.pi / box) * _m2(n).sqrt()
    lam = A * k / (1.0 + (k / 0.02) ** 2) ** 1.4 * (n / box) ** 3
    E = torch.fft.rfftn(torch.randn((n, n, n), dtype=F64, device="cuda", generator=gen))
    return torch.fft.irfftn(E.mul_(lam.sqrt_()), s=(n, n, n))


def _selection(n, box):
    """Radial selection with masked patches of sky (as mocks.radial_masked_selection)."""
    c = (torch.arange(n, dtype=F64, device="cuda") + 0.5) * (box / n) - 0.5 * box
    z, y, x = c[:, None, None], c[None, :, None], c[None, None, :]
    r = (x * x + y * y + z * z).sqrt()
    w = torch.exp(-(r / (0.4 * box)) ** 2)
    ic = ((z / r + 1.0) * 8.0).floor().clamp(0, 15).long()
    ip = ((torch.atan2(y, x).expand(1, n, n) / (2 * math.pi) % 1.0) * 32.0).floor().clamp(0, 31).long()
    patch = ic * 32 + ip
    masked = np.random.RandomState(7).permutation(512)[:102]
    keep = torch.ones(512, dtype=F64, device="cuda")
    keep[torch.from_numpy(masked).cuda()] = 0.0
    return w * keep[patch]


def _mock(case, gen):
    n, box, sigma = case["n"], case["box"], case["sigma"]
    A = _amplitude(n, box, sigma)
    G = _gaussian(n, box, A, gen)
    s_true = G - 0.5 * sigma ** 2
    w = _selection(n, box) if case["selection"] else None
    rate = case["nbar"] * torch.exp(s_true)
    N = torch.poisson(rate if w is None else rate * w, generator=gen).to(torch.int32)
    k, P = mocks.pk_table(n, box, A)
    return {"N": N, "w": w, "s": s_true, "k": k, "P": P, "mu": -0.5 * sigma ** 2,
            "nbar": case["nbar"]}


def _batch_cases(case, seed):
    """The uneven mix of mocks.batch_specs (1/4 half side, 1/2 three quarters,
    1/4 full), or `count` mocks of it."""
    n, count = case["n"], case["count"]
    sides = [min(SIDES, key=lambda s: abs(math.log(s / (f * n)))) for f in (0.5, 0.75, 0.75, 1.0)]
    r = np.random.RandomState(int(seed) % (1 << 31))
    return [{"n": m, "box": 3.90625 * m, "sigma": 0.8 + float(r.rand()),
             "nbar": math.exp(math.log(0.2) + math.log(10.0) * float(r.rand())),
             "selection": False}
            for m in (sides[i % 4] for i in range(count))]


def _context(case, d):
    c = Context(case["n"], case["box"], case["precision"])
    c.set_prior(d["k"], d["P"], d["mu"])
    return c


def _inputs(case, seed):
    """The inputs alone (no library object): what `prepare` and `exact` share."""
    gen = _gen(seed)
    call, n = case["call"], case.get("n")
    real = F64 if case["precision"] == "fp64" else torch.float32
    if call == "batch":
        return [_mock(dict(c), gen) for c in _batch_cases(case, seed)]
    d = _mock(case, gen)
    if call in ("hessvec", "grad", "bias"):
        d["s"] = d["s"].to(real)
        if call != "bias" and d["w"] is not None:
            d["w"] = d["w"].to(real)
        d["v"] = torch.randn((n, n, n), dtype=real, device="cuda", generator=gen)
    if call == "bias":
        d["s"] *= 0.25          # inside the domain u > 0, where a solve starts
        d["kb"], d["b"] = mocks.bias_table(n, case["box"], 1.2, 0.1)
    if call == "adjoint":
        d["u"] = torch.randn((n, n, n), dtype=F64, device="cuda", generator=gen)
        d["counts"] = d["N"].to(F64)
    if call == "diagnostics":
        # an estimate of the density and the density itself
        d["truth"] = torch.expm1(d["s"])
        d["estimate"] = torch.expm1(d["s"] + 0.1 * torch.randn((n, n, n), dtype=F64, device="cuda",
                                                               generator=gen))
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["call"] == "batch":
        cs = _batch_cases(case, seed)
        ctxs = [_context(dict(c, precision="mixed"), m) for c, m in zip(cs, d)]
        return {"call": "batch", "ctxs": ctxs, "batch": Batch(ctxs), "N": [m["N"] for m in d],
                "nbar": [m["nbar"] for m in d], "tol": case["tol"],
                "s": [torch.empty((c["n"],) * 3, dtype=F64, device="cuda") for c in cs]}
    d["call"], d["tol"], d["box"] = case["call"], case.get("tol"), case["box"]
    d["ctx"] = _context(case, d)
    if case["call"] == "bias":
        d["ctx"].set_bias(d["kb"], d["b"], 1.2)
    if case["call"] == "adjoint":
        d["counts"].requires_grad_(True)
        d["lnA"] = torch.zeros((), dtype=F64, device="cuda", requires_grad=True)
    if case["call"] == "grad":
        d["s"].requires_grad_(True)
    return d


def run(d):
    call = d["call"]
    if call == "hessvec":
        return d["ctx"].hessvec(d["s"], d["w"], d["nbar"], d["v"])
    if call == "grad":
        f = neg_log_posterior(d["s"], d["ctx"], d["N"], d["w"], d["nbar"])
        (g,) = torch.autograd.grad(f, d["s"])
        return {"f": f, "grad": g}
    if call == "map":
        return d["ctx"].newton_krylov_map(d["N"], d["w"], d["nbar"], tol=d["tol"]).s
    if call == "adjoint":
        s = map_field(d["counts"], d["lnA"], d["ctx"], d["k"], d["P"], d["mu"], d["w"], d["nbar"],
                      tol=d["tol"])
        gN, gA = torch.autograd.grad(s, (d["counts"], d["lnA"]), grad_outputs=d["u"])
        return {"s": s.detach(), "grad_N": gN, "grad_lnA": gA}
    if call == "batch":
        d["batch"].map(d["N"], None, d["nbar"], d["s"], tol=d["tol"], start=2)
        return d["s"]
    if call == "filters":
        wiener, _, _ = d["ctx"].wiener_lsq(d["N"], d["w"], d["nbar"], tol=d["tol"])
        return {"wiener": wiener,
                "gauss": d["ctx"].gauss_map(d["N"], d["w"], d["nbar"], tol=d["tol"]).s}
    if call == "bias":
        f, g = d["ctx"].bias_logpost_grad(d["s"], d["N"], d["w"], d["nbar"])
        return {"f": f, "grad": g,
                "hv": d["ctx"].bias_hessvec(d["s"], d["N"], d["w"], d["nbar"], d["v"])}
    y = d["ctx"].smooth(d["estimate"], 0.02 * d["box"])
    counts, outside, moments = d["ctx"].log_stats(d["estimate"], -6.0, 0.05, 240)
    r, dist = d["ctx"].compare(d["estimate"], d["truth"])
    return {"smooth": y, "counts": counts, "outside": list(outside), "moments": list(moments),
            "r": r, "distance": dist}


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the transforms a
    call cannot do without (2.5 n^3 log2 n^3 each way for real fields); for an
    iterative solve, of one gradient and of 8 Hessian-vector products per
    system, fewer than any of these problems takes."""
    if case["call"] == "batch":
        sides = [c["n"] for c in _batch_cases(case, 1)]
        return {"bytes": sum(12 * m ** 3 for m in sides),
                "flops": sum(9 * 15.0 * m ** 3 * math.log2(m) for m in sides)}
    n3, real = case["n"] ** 3, 8 if case["precision"] == "fp64" else 4
    pair = 15.0 * n3 * math.log2(case["n"])
    w = 1 if case["selection"] else 0
    b, f = {
        "hessvec": ((3 + w) * real, 1),
        "grad": ((2 + w) * real + 4, 1),
        "map": (12 + 8 * w, 9),
        "adjoint": (8 + 8 + 8 + 8 + 8 * w, 17),
        "filters": (2 * (4 + 8 * w + 8), 17),
        "bias": (4 * real + 4 + 8 * w, 8),
        "diagnostics": (16 + 8 + 16, 1),
    }[case["call"]]
    return {"bytes": b * n3, "flops": f * pair}


# ------------------------------ exact values --------------------------------

class _Reference:
    """S^-1, the MAP and its adjoint in plain FP64 torch."""

    def __init__(self, n, box, d):
        self.n, self.mu = n, d["mu"]
        self.inv = self.table(n, box, d["k"], d["P"])
        self.inv[0, 0, 0] = 1.0
        self.inv = (box / n) ** 3 / self.inv
        self.inv[0, 0, 0] = 0.0
        full = torch.full((n // 2 + 1,), 2.0, dtype=F64, device="cuda")
        full[0] = full[-1] = 1.0
        self.diag = float((self.inv * full).sum()) / n ** 3
        self.N = d["N"].to(F64)
        self.w = torch.ones((), dtype=F64, device="cuda") if d["w"] is None else d["w"].to(F64)
        self.rate = d["nbar"] * self.w

    @staticmethod
    def table(n, box, k, f):
        """f(|k|), linear in (ln k, ln f) between the table's points."""
        lk = torch.from_numpy(np.log(np.asarray(k))).cuda()
        lf = torch.from_numpy(np.log(np.asarray(f))).cuda()
        q = math.log(2.0 * math.pi / box) + 0.5 * torch.log(_m2(n).clamp_(min=1.0))
        j = (torch.searchsorted(lk, q, right=True) - 1).clamp_(0, lk.numel() - 2)
        t = (q - lk[j]) / (lk[j + 1] - lk[j])
        return torch.exp(lf[j] + t * (lf[j + 1] - lf[j]))

    def conv(self, x, mult):
        n = self.n
        return torch.fft.irfftn(torch.fft.rfftn(x).mul_(mult), s=(n, n, n))

    def prior(self, x):
        return self.conv(x, self.inv)

    def cg(self, D, b, tol, most=2000):
        """(S^-1 + D) x = b by Jacobi-preconditioned CG."""
        M = 1.0 / (D + self.diag)
        x, r = torch.zeros_like(b), b.clone()
        z = M * r
        p, rz, stop = z, (r * z).sum(), tol * tol * float((b * b).sum())
        for _ in range(most):
            q = self.prior(p) + D * p
            a = rz / (p * q).sum()
            x, r = x + a * p, r - a * q
            if float((r * r).sum()) <= stop:
                break
            z = M * r
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
        return x

    def solve(self, s, objective, curvature, cap, tol=1e-11):
        """Newton with backtracking; objective(s) -> (f, g)."""
        f, g = objective(s)
        g0 = float(g.norm())
        for _ in range(60):
            rel = float(g.norm()) / g0
            if rel < tol:
                break
            x = self.cg(curvature(s), -g, max(min(0.1, rel), 1e-6))
            t, slope = cap(s, x), float((g * x).sum())
            for _ in range(40):
                f2, g2 = objective(s + t * x)
                if f2 <= f + 1e-4 * t * slope or -t * slope < 1e-12 * abs(f):
                    break
                t *= 0.5
            s, f, g = s + t * x, f2, g2
        return s

    def map(self):
        def objective(s):
            y, D = self.prior(s - self.mu), self.rate * torch.exp(s)
            return float(0.5 * ((s - self.mu) * y).sum() + (D - self.N * s).sum()), y + D - self.N
        return self.solve(torch.full_like(self.N, self.mu), objective,
                          lambda s: self.rate * torch.exp(s),
                          lambda s, x: min(1.0, 2.0 / float(x.abs().max())))

    def gauss(self):
        occ = self.N > 0

        def objective(d):
            y, u = self.prior(d), torch.where(occ, 1.0 + d, torch.ones_like(d))
            f = 0.5 * (d * y).sum() + (self.rate * (1.0 + d) - self.N * torch.log(u)).sum()
            return float(f), y + self.rate - self.N / u

        def cap(d, x):
            frac = torch.where(occ, -x / (1.0 + d), torch.zeros_like(d)).max()
            return min(1.0, 0.99 / float(frac)) if float(frac) > 0 else 1.0
        return self.solve(torch.zeros_like(self.N), objective,
                          lambda d: torch.where(occ, self.N / (1.0 + d) ** 2,
                                                torch.zeros_like(d)), cap)


def exact(case, seed):
    d = _inputs(case, seed)
    call, n, box = case["call"], case["n"], case.get("box")
    if call == "batch":
        return [_Reference(c["n"], c["box"], m).map() for c, m in zip(_batch_cases(case, seed), d)]
    if call == "diagnostics":
        e, t = d["estimate"], d["truth"]
        kr2 = (2.0 * math.pi / box * 0.02 * box) ** 2
        x = torch.log1p(e)
        c = x - x.mean()
        var = (c * c).mean()
        return {"smooth": torch.fft.irfftn(torch.fft.rfftn(e) * torch.exp(-0.5 * kr2 * _m2(n)),
                                           s=(n, n, n)),
                "counts": None, "outside": None,
                "moments": [float(x.mean()), float(var), float((c ** 3).mean() / var ** 1.5),
                            float((c ** 4).mean() / var ** 2 - 3.0)],
                "r": float((e * t).sum() / ((e * e).sum().sqrt() * (t * t).sum().sqrt())),
                "distance": float(((e - t) ** 2).mean().sqrt())}
    R = _Reference(n, box, d)
    if call == "hessvec":
        v = d["v"].to(F64)
        return R.prior(v) + R.rate * torch.exp(d["s"].to(F64)) * v
    if call == "grad":
        s = d["s"].to(F64)
        y, D = R.prior(s - R.mu), R.rate * torch.exp(s)
        return {"f": 0.5 * ((s - R.mu) * y).sum() + (D - R.N * s).sum(), "grad": y + D - R.N}
    if call == "map":
        return R.map()
    if call == "adjoint":
        s = R.map()
        lam = R.cg(R.rate * torch.exp(s), d["u"], 1e-11)
        return {"s": s, "grad_N": lam, "grad_lnA": float((lam * R.prior(s - R.mu)).sum())}
    if call == "filters":
        rate = R.rate.expand_as(R.N)
        return {"wiener": R.cg(rate, R.N - rate, 1e-11), "gauss": R.gauss()}
    # linear bias
    B = R.table(n, box, d["kb"], d["b"])
    B[0, 0, 0] = 1.2
    s, v = d["s"].to(F64), d["v"].to(F64)
    e, y = torch.exp(s), R.prior(s - R.mu)
    u = 1.0 + R.conv(torch.expm1(s), B)
    d1 = e * R.conv(R.rate - R.N / u, B)
    f = 0.5 * ((s - R.mu) * y).sum() + (R.rate * u - R.N * torch.log(u)).sum()
    return {"f": float(f), "grad": y + d1,
            "hv": R.prior(v) + d1 * v + e * R.conv(R.N / u ** 2 * R.conv(e * v, B), B)}
