"""What a user of the library has it do, as timed cases.

The work is the grouped Fourier transform of a node set and its adjoint, the
solvers that call both in every iteration, many problems at once, and the
evaluation of a solved model at new nodes.  Sizes are those of the workloads in
`paper_2010_10199_gb300/inputs.py`, of the tests and of the benchmark:

* pair_small         d = 6, 2000 nodes, |u| <= 2: the smallest problem a user
                     solves; one forward and one adjoint transform, bound by
                     launches and latency
* trafo_d20          the benchmark's size, one million nodes, 211 terms:
* adjoint_d20        predictions of a model, and the gradient of its data term
* trafo_third        third-order terms (|u| <= 3, d = 10, half a million nodes,
* adjoint_third      Beta-distributed): the Tikhonov path's transforms
* pair_d30           the group-lasso workload, 466 terms and two million nodes:
                     the largest problem
* pair_cosine        the half-period cosine system at the application's size
                     (36 160 nodes in the unit cube, 79 terms)
* pair_f64           an FP64 plan: reference solutions
* batch_pair         many independent problems of uneven size, one call per
                     direction for all of them
* lsqr_third         a Tikhonov solve with Sobolev weights, ten thousand nodes,
                     |u| <= 3 (the paper's experiments)
* fista_path         a group-lasso path over five lambda values at the same size
* predict_new_nodes  a model's coefficients evaluated once at nodes that have not
                     been seen before: plan, one forward transform, release

Node counts and bandwidths of drawn cases spread over the ranges between these,
odd node counts among them.  FP16 and BF16 grid storage exist for a precision
study and save nothing over FP32, so no case uses them.

`exact` sums the definitions directly in FP64 (one table of the one-dimensional
basis per coordinate, contracted term by term) and runs the solvers' published
iterations on those sums.
"""
import itertools
import math

import torch

from paper_2010_10199_gb300 import gft

CHUNK = 1 << 16          # nodes per step of the FP64 sums
ITERS_PER_LAMBDA = 20    # FISTA iterations per lambda value, as a capped path runs


def listed():
    return [
        {"name": "pair_small", "kind": "pair", "d": 6, "order": 2, "M": 2000, "N1": 16, "N2": 8},
        {"name": "trafo_d20", "kind": "trafo", "d": 20, "order": 2, "M": 1000000, "N1": 64, "N2": 32},
        {"name": "adjoint_d20", "kind": "adjoint", "d": 20, "order": 2, "M": 1000000, "N1": 64, "N2": 32},
        {"name": "trafo_third", "kind": "trafo", "d": 10, "order": 3, "M": 500000, "N1": 100, "N2": 24, "N3": 10,
         "points": "beta"},
        {"name": "adjoint_third", "kind": "adjoint", "d": 10, "order": 3, "M": 500000, "N1": 100, "N2": 24, "N3": 10,
         "points": "beta"},
        {"name": "pair_d30", "kind": "pair", "d": 30, "order": 2, "M": 2000000, "N1": 32, "N2": 16},
        {"name": "pair_cosine", "kind": "pair", "basis": "cos", "d": 12, "order": 2, "M": 36160, "N1": 82, "N2": 10},
        {"name": "pair_f64", "kind": "pair", "f64": True, "d": 20, "order": 2, "M": 30011, "N1": 64, "N2": 32},
        {"name": "batch_pair", "kind": "batch", "problems": 32, "Mlo": 10000, "Mhi": 200000, "N1": 32, "N2": 16},
        {"name": "lsqr_third", "kind": "lsqr", "d": 9, "order": 3, "M": 10000, "N1": 26, "N2": 6, "N3": 4,
         "lam": 7.389, "iters": 50},
        {"name": "fista_path", "kind": "fista", "d": 9, "order": 3, "M": 10000, "N1": 26, "N2": 6, "N3": 4,
         "lambdas": 5},
        {"name": "predict_new_nodes", "kind": "predict", "d": 20, "order": 2, "M": 100003, "N1": 64, "N2": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return 2 * rng.randint(lo // 2, hi // 2)


def draw(rng):
    """One case of the same ranges: |u| <= 2 with d up to 30 and up to a million
    nodes, |u| <= 3 with d up to 10, the cosine system, FP64 plans, batches and
    solves of up to thirty thousand nodes."""
    kind = rng.choice(["pair", "pair", "trafo", "adjoint", "third", "cosine", "f64", "batch", "lsqr", "fista",
                       "predict"])
    if kind == "batch":
        lo = _log_int(rng, 500, 20000)
        return {"kind": "batch", "problems": rng.randint(4, 32), "Mlo": lo, "Mhi": lo * rng.randint(2, 10),
                "N1": _even(rng, 16, 64), "N2": _even(rng, 8, 24)}
    if kind == "third":
        return {"kind": rng.choice(["trafo", "adjoint"]), "d": rng.randint(4, 10), "order": 3,
                "M": _log_int(rng, 2000, 400000), "N1": _even(rng, 16, 100), "N2": _even(rng, 8, 32),
                "N3": _even(rng, 4, 10), "points": rng.choice(["beta", "uniform"])}
    if kind == "cosine":
        return {"kind": "pair", "basis": "cos", "d": rng.randint(4, 16), "order": 2, "M": _log_int(rng, 2000, 300000),
                "N1": rng.randint(16, 100), "N2": rng.randint(4, 18)}
    if kind in ("lsqr", "fista"):
        c = {"kind": kind, "d": rng.randint(5, 9), "order": rng.choice([2, 3]), "M": _log_int(rng, 2000, 30000),
             "N1": _even(rng, 16, 32), "N2": _even(rng, 4, 10), "N3": 4}
        c.update({"lam": rng.choice([1.0, 2.718, 7.389]), "iters": rng.randint(20, 50)} if kind == "lsqr"
                 else {"lambdas": rng.randint(2, 5)})
        return c
    c = {"kind": "pair" if kind == "f64" else kind, "d": rng.randint(6, 30 if kind == "pair" else 20), "order": 2,
         "M": _log_int(rng, 2000, {"f64": 60000, "predict": 300000}.get(kind, 1000000)),
         "N1": _even(rng, 16, 100), "N2": _even(rng, 8, 40)}
    if kind == "f64":
        c["f64"] = True
    return c


# ------------------------------------------------------------------ inputs --

def _terms(case, d=None):
    """All terms with |u| <= order, the empty set first, and their bandwidths."""
    d = case["d"] if d is None else d
    terms = [u for s in range(case.get("order", 2) + 1) for u in itertools.combinations(range(d), s)]
    return terms, [case["N%d" % len(u)] if u else 0 for u in terms]


def _cosine(case):
    return case.get("basis") == "cos"


def _freqs(case, N, dev):
    k = torch.arange(1, N, device=dev) if _cosine(case) else torch.tensor(
        [q for q in range(-N // 2, N // 2) if q], device=dev)
    return k.to(torch.float64)


def _count(case, terms, bw):
    return sum((N - 1) ** len(u) for u, N in zip(terms, bw))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _nodes(case, g, d, M):
    """Uniform or Beta(2,2) nodes on the torus, or in the unit cube."""
    real = torch.float64 if case.get("f64") else torch.float32
    if case.get("points") == "beta":
        x = torch.rand(3, d, M, generator=g, device="cuda", dtype=real).median(0).values - 0.5
    else:
        x = torch.rand(d, M, generator=g, device="cuda", dtype=real)
        if not _cosine(case):
            x -= 0.5
    return x.contiguous()


def _normal(g, n, case):
    cplx = torch.complex128 if case.get("f64") else torch.complex64
    return torch.randn(n, generator=g, device="cuda", dtype=cplx)


def _coefficients(case, g, terms, bw):
    """N(0, 1) / (1 + |k|^2): the decay of a smooth function's coefficients."""
    c = _normal(g, _count(case, terms, bw), case)
    scale, at, by = torch.ones(c.numel(), device="cuda", dtype=torch.float64), 0, {}
    for u, N in zip(terms, bw):
        if u and (len(u), N) not in by:
            k2, total = _freqs(case, N, "cuda") ** 2, 0.0
            for t in range(len(u)):
                total = total + k2.reshape([-1 if q == t else 1 for q in range(len(u))])
            by[len(u), N] = (1.0 / (1.0 + total)).reshape(-1)
        m = (N - 1) ** len(u)
        if u:
            scale[at:at + m] = by[len(u), N]
        at += m
    return (c * scale).to(c.dtype)


def _data(case, g, x):
    """Values of a sum of low-order bumps at the nodes, with one percent noise."""
    y = torch.exp(-8 * (x[0] ** 2 + x[1] ** 2)) + torch.exp(-8 * (x[2] ** 2 + x[3] ** 2 + x[4] ** 2))
    y = y + torch.sin(2 * math.pi * x[3])
    y = y + 0.01 * torch.randn(x.shape[1], generator=g, device="cuda", dtype=x.dtype)
    return y.to(torch.complex64)


def _sobolev(case, terms, bw):
    """Weights 1 + |k|^2 / 4 per coefficient."""
    w = []
    for u, N in zip(terms, bw):
        k2, total = _freqs(case, max(N, 2), "cuda") ** 2, torch.ones(1, device="cuda", dtype=torch.float64)
        for t in range(len(u)):
            total = total + 0.25 * k2.reshape([-1 if q == t else 1 for q in range(len(u))])
        w.append(total.reshape(-1))
    return torch.cat(w).contiguous()


def _batch_sizes(case, seed):
    """Uneven (dimension, nodes) of the problems: the same for every seed."""
    rng = torch.Generator().manual_seed(17 * case["problems"] + case["Mlo"])
    u = torch.rand(case["problems"], 2, generator=rng, dtype=torch.float64).tolist()
    return [(5 + int(v * 11), int(round(case["Mlo"] * (case["Mhi"] / case["Mlo"]) ** t))) for t, v in u]


def _inputs(case, seed):
    """The host program's data, the plan aside."""
    g, s = _gen(seed), {"case": case}
    if case["kind"] == "batch":
        s["xs"], s["terms"], s["bw"], fh, ys = [], [], [], [], []
        for d, M in _batch_sizes(case, seed):
            terms, bw = _terms(case, d)
            s["xs"].append(_nodes(case, g, d, M))
            s["terms"].append(terms)
            s["bw"].append(bw)
            fh.append(_coefficients(case, g, terms, bw))
            ys.append(_normal(g, M, case))
        s["fhat"], s["y"] = torch.cat(fh), torch.cat(ys)
        return s
    s["terms"], s["bw"] = _terms(case)
    s["x"] = _nodes(case, g, case["d"], case["M"])
    if case["kind"] in ("pair", "trafo", "predict"):
        s["fhat"] = _coefficients(case, g, s["terms"], s["bw"])
    if case["kind"] in ("pair", "adjoint"):
        s["y"] = _normal(g, case["M"], case)
    if case["kind"] in ("lsqr", "fista"):
        s["y"] = _data(case, g, s["x"])
    if case["kind"] == "lsqr":
        s["w"] = _sobolev(case, s["terms"], s["bw"])
    if case["kind"] == "fista":
        # the step constant and the lambda scale such a program keeps: 1.1 times
        # ||F||^2 by power iteration, lambdas from half the largest useful one
        F = _Sums(case, s["x"], s["terms"], s["bw"])
        v = torch.ones(F.n, device="cuda", dtype=torch.complex128)
        for _ in range(12):
            v = F.adjoint(F.trafo(v / v.norm()))
        s["L"] = 1.1 * float(v.norm())
        q = F.adjoint(s["y"].to(torch.complex128))
        top = max(float(b.norm()) for b in q.split(F.sizes) if b.numel() > 1)
        s["lambdas"] = [0.5 * top * 4.0 ** -i for i in range(case["lambdas"])]
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "batch":
        s["batch"] = gft.Batch(s["xs"], s["terms"], s["bw"])
    elif case["kind"] != "predict":
        s["plan"] = gft.Plan(s["x"], s["terms"], s["bw"], **_options(case))
    return s


def _options(case):
    return {"precision": gft.PREC_F64 if case.get("f64") else gft.PREC_F32,
            "basis": gft.BASIS_COS if _cosine(case) else gft.BASIS_EXP}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pair":
        return {"f": state["plan"].trafo(state["fhat"]), "g": state["plan"].adjoint(state["y"])}
    if kind == "trafo":
        return {"f": state["plan"].trafo(state["fhat"])}
    if kind == "adjoint":
        return {"g": state["plan"].adjoint(state["y"])}
    if kind == "batch":
        return {"f": state["batch"].trafo(state["fhat"]), "g": state["batch"].adjoint(state["y"])}
    if kind == "lsqr":
        return {"fhat": state["plan"].lsqr(state["y"], case["lam"], max_it=case["iters"], w=state["w"])[0]}
    if kind == "fista":
        return {"path": state["plan"].fista(state["y"], state["lambdas"], max_it=ITERS_PER_LAMBDA, tol=0.0,
                                            L0=state["L"])[0]}
    plan = gft.Plan(state["x"], state["terms"], state["bw"], **_options(case))
    f = plan.trafo(state["fhat"])
    plan.close()
    return {"f": f}


# ------------------------------------------------------------------- work --

def _one_way(case, d, M):
    """(bytes, flops) of one transform: nodes, coefficients and values once, and
    per node and term the 8 window weights of each coordinate (degree 7) and the
    window's weighted complex sum."""
    terms, bw = _terms(case, d)
    real = 8 if case.get("f64") else 4
    per = {0: 2, 1: 2 * (8 * 7 + 8 * 2), 2: 2 * (16 * 7 + 64 * 3), 3: 2 * (24 * 7 + 512 * 2 + 64 * 3)}
    return real * d * M + 2 * real * (M + _count(case, terms, bw)), M * sum(per[len(u)] for u in terms)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_one_way(case, d, M) for d, M in _batch_sizes(case, 0)]
        return {"bytes": 2 * sum(b for b, _ in each), "flops": 2 * sum(f for _, f in each)}
    b, f = _one_way(case, case["d"], case["M"])
    ways = {"pair": 2, "lsqr": 2 * case.get("iters", 0) + 1,
            "fista": 2 * ITERS_PER_LAMBDA * case.get("lambdas", 0)}.get(kind, 1)
    return {"bytes": b * (2 if kind == "pair" else 1), "flops": ways * f}


# ------------------------------------------------------------------ exact --

class _Sums:
    """The direct sums of one node set in FP64."""

    def __init__(self, case, x, terms, bw):
        self.case, self.x, self.terms, self.bw = case, x.to(torch.float64), terms, bw
        self.sizes = [(N - 1) ** len(u) for u, N in zip(terms, bw)]
        self.n, self.M = sum(self.sizes), x.shape[1]

    def _tables(self, a, b):
        made = {}

        def table(t, N):
            if (t, N) not in made:
                k, x = _freqs(self.case, N, self.x.device), self.x[t, a:b, None]
                if _cosine(self.case):
                    made[t, N] = (math.sqrt(2.0) * torch.cos(math.pi * k * x)).to(torch.complex128)
                else:
                    p = k * x
                    p = 2 * math.pi * (p - p.round())
                    made[t, N] = torch.complex(torch.cos(p), torch.sin(p))
            return made[t, N]
        return table

    def trafo(self, c):
        blocks = c.to(torch.complex128).split(self.sizes)
        out = torch.empty(self.M, device=self.x.device, dtype=torch.complex128)
        for a in range(0, self.M, CHUNK):
            b = min(self.M, a + CHUNK)
            E, f = self._tables(a, b), torch.zeros(b - a, device=self.x.device, dtype=torch.complex128)
            for u, N, v in zip(self.terms, self.bw, blocks):
                if not u:
                    f += v
                    continue
                t = E(u[0], N) @ v.reshape(N - 1, -1)
                for q in u[1:]:
                    t = torch.einsum("jk,jkr->jr", E(q, N), t.reshape(b - a, N - 1, -1))
                f += t[:, 0]
            out[a:b] = f
        return out

    def adjoint(self, y):
        y = y.to(torch.complex128)
        out = [torch.zeros(m, device=self.x.device, dtype=torch.complex128) for m in self.sizes]
        for a in range(0, self.M, CHUNK):
            b = min(self.M, a + CHUNK)
            E = self._tables(a, b)
            for u, N, o in zip(self.terms, self.bw, out):
                t = y[a:b, None]
                if not u:
                    o += t.sum()
                    continue
                for q in u[1:]:
                    t = (t[:, :, None] * E(q, N).conj()[:, None, :]).reshape(b - a, -1)
                o += (E(u[0], N).conj().T @ t).reshape(-1)
        return torch.cat(out)


def _lsqr(F, y, w, lam, iters):
    """LSQR (Paige and Saunders) on F W^{-1/2} with damping sqrt(2 lam)."""
    s, damp = w.rsqrt(), math.sqrt(2.0 * lam)
    beta = float(y.norm())
    u = y / beta
    v = s * F.adjoint(u)
    alpha = float(v.norm())
    v, x = v / alpha, torch.zeros_like(v)
    p, phibar, rhobar = v.clone(), beta, alpha
    for _ in range(iters):
        u = F.trafo(s * v) - alpha * u
        beta = float(u.norm())
        u = u / beta
        v = s * F.adjoint(u) - beta * v
        alpha = float(v.norm())
        v = v / alpha
        hat = math.hypot(rhobar, damp)
        phibar *= rhobar / hat
        rho = math.hypot(hat, beta)
        c, sn = hat / rho, beta / rho
        theta, rhobar, phi, phibar = sn * alpha, -c * alpha, c * phibar, sn * phibar
        x = x + (phi / rho) * p
        p = v - (theta / rho) * p
    return s * x


def _fista(F, y, lambdas, L):
    """FISTA for the group lasso with step 1 / L, warm started along the path."""
    f, path = torch.zeros(F.n, device=y.device, dtype=torch.complex128), []
    for lam in lambdas:
        h, t = f, 1.0
        for _ in range(ITERS_PER_LAMBDA):
            z = h - F.adjoint(F.trafo(h) - y) / L
            new = []
            for b in z.split(F.sizes):
                nb = float(b.norm())
                new.append(b * (1.0 - lam / L / nb) if nb > lam / L else torch.zeros_like(b))
            new = torch.cat(new)
            tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
            h, f, t = new + (t - 1.0) / tn * (new - f), new, tn
        path.append(f)
    return torch.stack(path)


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    if kind == "batch":
        f, g, i, j = [], [], 0, 0
        for x, terms, bw in zip(s["xs"], s["terms"], s["bw"]):
            F = _Sums(case, x, terms, bw)
            f.append(F.trafo(s["fhat"][i:i + F.n]))
            g.append(F.adjoint(s["y"][j:j + F.M]))
            i, j = i + F.n, j + F.M
        return {"f": torch.cat(f), "g": torch.cat(g)}
    F = _Sums(case, s["x"], s["terms"], s["bw"])
    if kind == "lsqr":
        return {"fhat": _lsqr(F, s["y"].to(torch.complex128), s["w"], case["lam"], case["iters"])}
    if kind == "fista":
        return {"path": _fista(F, s["y"].to(torch.complex128), s["lambdas"], s["L"])}
    return {**({"f": F.trafo(s["fhat"])} if "fhat" in s else {}), **({"g": F.adjoint(s["y"])} if "y" in s else {})}
