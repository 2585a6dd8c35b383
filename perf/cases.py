"""The work whose speed this repository is judged by, as calls through its public entry points.

A case names one call: `prepare` makes what a program has in hand before it (the problem, a
handle, the starting point), `run` makes the call, `work` gives the bytes and operations that the
call cannot do without, and `exact` gives the call's result in plain 64-bit torch arithmetic.

Calls that solve run under a fixed step budget: a solve to convergence takes thousands of steps of
a nonconvex iteration, whose single steps are what can be compared between two versions.  They
start from a multiplier of the size that the later outer iterations (and the learned warm start)
have, at the default penalty, where the preconditioner's diagonal is positive and a step does not
amplify rounding.  An
eigenvector's sign is arbitrary, so returned eigenvectors (and the factor columns grown along
them) are given the sign that makes their largest entry positive.  A handle in the FP32 form
returns its multipliers, constraint values and quartic coefficients in FP64 words that carry the
accuracy of its FP32 factor: they are returned here in the handle's precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import sdp_instances as si
from paper_2505_15775_gb300 import alm

RANK = 32          # columns of a batch factor and of the network's head
HID, FEAT, LAYERS = 64, 8, 3


# ------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------
def listed():
    return [
        # the benchmark: MaxCut on the 1000 x 1000 torus, full rank, FP32 form; 32 inner steps of
        # the ~18,000 that the whole solve takes
        dict(name="solve-torus-1e6-fp32", op="solve", graph="torus", n=1_000_000, r=32, r_max=32,
             precision="fp32", sigma=1.0, outer=1, inner=32),
        # the same problem class in plain FP64 (the form the benchmark compares with), odd sizes
        dict(name="solve-torus-449x449-fp64", op="solve", graph="torus", n=201_601, r=32, r_max=32,
             precision="fp64", sigma=1.0, outer=1, inner=16),
        # the ER(800, 0.06) configuration: plain FP64, rank-adaptive from 8, the first three outer
        # iterations with their eigensolves and growth steps; small, so bound by latency
        dict(name="solve-er800-adaptive-fp64", op="solve", graph="er", n=800, deg=48.0, r=8, r_max=32,
             precision="fp64", sigma=1.0, outer=3, inner=5000),
        # matrix completion (the paper's second experiment) at its smallest table size: entry
        # constraints, S moves with y, rank 3
        dict(name="solve-mc-10000-fp32", op="solve", graph="mc", n=10_000, r=3, r_max=3,
             precision="fp32", sigma=1.0, outer=1, inner=32),
        # a ragged batch of small MaxCut SDPs in one persistent launch (n 64..4096, degree 3..30)
        dict(name="batch-300-fp32", op="batch", count=300, n_lo=64, n_hi=4096, d_lo=3.0, d_hi=30.0, r=32,
             sigma=1.0, outer=2, inner=16),
        # the learned warm start for the benchmark torus (BF16 activations, as it is deployed)
        dict(name="warm-start-torus-1e6-bf16", op="warm", graph="torus", n=1_000_000, storage="bf16"),
        # one training step's loss and gradient on a ragged batch of ER instances
        dict(name="train-grad-64-bf16", op="train", count=64, n_lo=64, n_hi=4096, d_lo=3.0, d_hi=30.0,
             storage="bf16"),
        # the eigensolve of a growth step on a torus (long vectors, FP32 basis)
        dict(name="lambda-torus-501x501-fp32", op="lambda", graph="torus", n=251_001, r=32, precision="fp32", sigma=10.0),
        # the gradient on a random 3-regular graph: neighbour rows are random gathers from memory
        dict(name="grad-regular3-1e6-fp32", op="grad", graph="regular3", n=1_000_000, r=32, precision="fp32", sigma=1.0),
        # the gradient on a Kronecker graph: heavy-tailed degrees, rows of thousands of entries
        dict(name="grad-kron-65536-fp32", op="grad", graph="kron", n=65_536, r=32, precision="fp32", sigma=1.0),
        # the exact line search of a Lovasz theta SDP (low-rank objective, 200,000 edge
        # constraints), odd rank
        dict(name="linesearch-theta-20000-fp32", op="linesearch", graph="theta", n=20_000, deg=20.0, r=29,
             precision="fp32", sigma=100.0),
        # the smallest call: the constraint map and augmented Lagrangian on ER(800), FP64
        dict(name="eval-er800-fp64", op="eval", graph="er", n=800, deg=48.0, r=8, precision="fp64", sigma=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "batch", "warm", "train", "lambda", "grad", "grad", "linesearch", "eval"])
    if op in ("batch", "train"):
        n_hi = _log_int(rng, 200, 4096)
        c = dict(op=op, count=rng.randint(1, 64 if op == "train" else 300), n_lo=64, n_hi=n_hi,
                 d_lo=3.0, d_hi=round(rng.uniform(4.0, 30.0), 2))
        if op == "batch":
            return dict(c, r=rng.choice([8, 13, 24, 32, 32]), sigma=1.0, outer=rng.randint(1, 2), inner=rng.randint(4, 16))
        return dict(c, storage=rng.choice(["bf16", "bf16", "fp32"]))
    if op == "warm":
        return dict(op=op, graph=rng.choice(["torus", "er"]), n=_log_int(rng, 500, 300_000),
                    deg=round(rng.uniform(3.0, 24.0), 2), storage=rng.choice(["bf16", "bf16", "fp32"]))
    precision = rng.choice(["fp32", "fp32", "fp64"])
    r = rng.choice([1, 3, 5, 8, 12, 13, 16, 24, 29, 32, 32])
    if op == "lambda":
        n = _log_int(rng, 20_000, 250_000) if precision == "fp32" else _log_int(rng, 500, 20_000)
        return dict(op=op, graph="torus" if precision == "fp32" else rng.choice(["torus", "er"]), n=n, r=r,
                    deg=round(rng.uniform(4.0, 24.0), 2), precision=precision, sigma=10.0)
    graph = rng.choice(["torus", "torus", "er", "regular3", "kron", "theta", "mc"])
    if op == "solve" and graph in ("kron", "theta"):
        graph = "torus"
    top = {"torus": 500_000, "er": 60_000, "regular3": 500_000, "kron": 65_536, "theta": 20_000, "mc": 10_000}[graph]
    if precision == "fp64":
        top = min(top, 100_000)
    n = _log_int(rng, 400, top)
    if graph == "kron":
        n = 1 << rng.randint(9, 16)
    if graph == "mc":
        r = rng.choice([1, 2, 3, 4, 5])
    c = dict(op=op, graph=graph, n=n, r=r, deg=round(rng.uniform(4.0, 48.0 if n < 5000 else 24.0), 2),
             precision=precision, sigma=rng.choice([1.0, 10.0]))
    if op == "solve":  # at full rank no eigensolve follows the inner solve's step budget
        return dict(c, sigma=1.0, r_max=r, outer=1, inner=rng.randint(4, 24))
    return c


# ------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------
def _instance(case, seed):
    """The problem data of a case (host arrays), from the seed alone."""
    n, graph = case["n"], case["graph"]
    if graph == "torus":
        n1 = max(3, math.isqrt(n))
        return si.torus_maxcut(n1, max(3, n // n1), seed=seed)
    if graph == "er":
        return si.er_maxcut(n, min(1.0, case["deg"] / (n - 1)), seed=seed)
    if graph == "regular3":
        return si.regular3_maxcut(n + n % 2, seed=seed)
    if graph == "kron":
        return si.kron_maxcut(n.bit_length() - 1, seed=seed)
    if graph == "theta":
        return si.theta_er(n, case["deg"], seed=seed)
    if graph == "mc":
        return si.matrix_completion(n // 2, n - n // 2, 3, seed=seed)
    raise ValueError(graph)


def _batch_instances(case, seed):
    """A ragged batch: the sizes are the case's, the graphs the seed's."""
    specs = si.batch_specs(case["count"], seed=6, n_lo=case["n_lo"], n_hi=case["n_hi"], d_lo=case["d_lo"], d_hi=case["d_hi"])
    return [si.er_maxcut(n, p, seed=(seed, k)) for k, (n, p, _) in enumerate(specs)]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _normal(shape, seed, stream, dtype):
    g = torch.Generator(device=_device()).manual_seed(seed * 16 + stream)
    return torch.randn(shape, generator=g, device=_device(), dtype=dtype)


def _dtype(case):
    return torch.float64 if case.get("precision") == "fp64" else torch.float32


def _factor(case, inst, seed):
    """A starting factor: rows near the unit sphere for MaxCut (as every iterate but the first is),
    unit trace on average for theta."""
    if inst.kind == "maxcut":
        return _near_unit(inst.n, case["r"], seed, _dtype(case))
    scale = 0.3 if inst.kind == "mc" else 1.0 / math.sqrt(case["r"] * inst.n)
    return _normal((inst.n, case["r"]), seed, 1, _dtype(case)) * scale


def _near_unit(n, r, seed, dtype):
    x = _normal((n, r), seed, 1, dtype)
    return x / x.norm(dim=1, keepdim=True) * (1.0 + 0.02 * _normal((n, 1), seed, 4, dtype))


def _dual(case, inst, seed):
    return _normal((inst.m,), seed, 2, torch.float64) * 0.1


def _multiplier(inst, seed):
    """A multiplier to start a solve from: for MaxCut S_ii = C_ii - y_i ~ 2 (sum_j C_ij^2)^(1/2) + 1/2,
    a little above the spectral radius of a random graph's off-diagonal part."""
    if inst.kind != "maxcut":
        return np.random.default_rng(seed).standard_normal(inst.m) * 0.1
    d = inst.c_i == inst.c_j
    sq = inst.c_v[~d] ** 2
    row = np.bincount(inst.c_i[~d], sq, inst.n) + np.bincount(inst.c_j[~d], sq, inst.n)
    return np.bincount(inst.c_i[d], inst.c_v[d], inst.n) - 2.0 * np.sqrt(row) - 0.5


def _theta(seed):
    """Network parameters: uniform weights of variance 1 / fan-in, small biases."""
    rng = np.random.default_rng(seed)
    parts, din = [], FEAT
    for _ in range(LAYERS):
        for _ in range(2):
            parts.append(rng.uniform(-1, 1, HID * din) * math.sqrt(3.0 / din))
        parts.append(rng.uniform(-0.1, 0.1, HID))
        din = HID
    for rows in (RANK, 1):
        parts.append(rng.uniform(-1, 1, rows * HID) * math.sqrt(3.0 / HID))
    parts.append(rng.uniform(-0.1, 0.1, 1))
    return np.concatenate(parts).astype(np.float32)


class _State(dict):
    """What a program keeps between calls; its handles are destroyed with it."""

    def __del__(self):
        for destroy, key in ((alm.alm_destroy, "h"), (alm.alm_gnn_destroy, "g"), (alm.alm_batch_destroy, "hb")):
            if self.get(key) is not None:
                destroy(self[key])


def prepare(case, seed):
    op = case["op"]
    if op in ("batch", "train", "warm"):
        insts = [_instance(case, seed)] if op == "warm" else _batch_instances(case, seed)
        options = dict(sigma0=10.0, r_max=case.get("r", RANK))
        if op == "batch":
            options.update(sigma0=case["sigma"], max_outer=case["outer"], max_inner=case["inner"], inner_start=1e-6)
        s = _State(case=case, hb=alm.alm_batch_create(insts, **options))
        rows = s["hb"].rows
        if op == "batch":
            s["R0"] = torch.zeros((rows, RANK), device="cuda")
            s["R0"][:, : case["r"]] = _near_unit(rows, case["r"], seed, torch.float32)
            s["y0"] = torch.as_tensor(np.concatenate([_multiplier(x, seed) for x in insts]), device="cuda")
            s["R"], s["y"] = torch.empty_like(s["R0"]), torch.empty(rows, dtype=torch.float64, device="cuda")
            s["rank"] = torch.empty(case["count"], dtype=torch.int32, device="cuda")
            return s
        s["g"] = alm.alm_gnn_create(alm.ALM_GNN_BF16 if case["storage"] == "bf16" else alm.ALM_GNN_FP32, feat_seed=seed)
        alm.alm_gnn_set_params(s["g"], _theta(seed))
        if op == "train":
            s["Rs"], s["ys"] = _solution(rows, seed)
        return s
    inst = _instance(case, seed)
    options = dict(precision=alm.ALM_FP64 if case["precision"] == "fp64" else alm.ALM_FP32)
    if op == "solve":
        options.update(r_max=case["r_max"], sigma0=case["sigma"], max_outer=case["outer"], max_inner=case["inner"])
        if case["r"] == case["r_max"]:
            options.update(inner_start=1e-6)  # the step budget ends the inner solve, not its tolerance
    s = _State(case=case, h=alm.alm_create(inst, **options))
    s["R"], s["y"] = _factor(case, inst, seed), _dual(case, inst, seed)
    if op == "solve":
        s["y"] = torch.as_tensor(_multiplier(inst, seed), device="cuda")
    else:
        s["R"] = alm.factor_tensor(s["h"], s["R"])
    if op == "linesearch":
        s["D"] = alm.factor_tensor(s["h"], _direction(case, inst, seed))
    return s


def _direction(case, inst, seed):
    return 0.1 * float(_factor(case, inst, seed).std()) * _normal((inst.n, case["r"]), seed, 3, _dtype(case))


def _solution(rows, seed):
    """A solution to train on: unit rows of rank 12 and a negative multiplier."""
    R = torch.zeros((rows, RANK), device=_device())
    x = _normal((rows, 12), seed, 1, torch.float32)
    R[:, :12] = x / x.norm(dim=1, keepdim=True)
    return R, -1.0 - 0.2 * _normal((rows,), seed, 2, torch.float64).abs()


# ------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------
def _fix_sign(x):
    """Each column with its largest entry made positive."""
    top = x.gather(0, x.abs().argmax(dim=0, keepdim=True))
    return torch.where(top < 0, -x, x)


def run(s):
    case = s["case"]
    op, r = case["op"], case.get("r")
    if op == "solve":
        R, _, y, st = alm.alm_solve(s["h"], s["R"], s["y"])
        if case["r"] < case["r_max"]:
            R = _fix_sign(R)
        return dict(R=R, y=y.to(R.dtype), objective=st["objective"])
    if op == "batch":
        s["R"].copy_(s["R0"])
        s["rank"].fill_(r)
        s["y"].copy_(s["y0"])
        _, per = alm.alm_batch_solve(s["hb"], s["R"], s["rank"], s["y"])
        return dict(R=s["R"], y=s["y"].float(), rank=s["rank"],
                    objective=np.array([p["objective"] for p in per], np.float32))
    if op == "warm":
        R0, rank, y0 = alm.alm_gnn_warm_start(s["g"], s["hb"])
        return dict(R=R0, y=y0.float(), rank=rank)
    if op == "train":
        loss, grad = alm.alm_gnn_loss_grad(s["g"], s["hb"], s["Rs"], s["ys"], 0.01)
        return dict(loss=loss, grad=grad)
    h, R, y, sigma = s["h"], s["R"], s["y"], case["sigma"]
    if op == "lambda":
        lam, v, _ = alm.alm_lambda_min(h, R, r, y, sigma)
        return dict(lam=lam, v=_fix_sign(v[:, None]))
    if op == "grad":
        G, g2 = alm.alm_grad(h, R, r, y, sigma)
        return dict(G=G, g2=g2)
    if op == "linesearch":
        q, alpha = alm.alm_linesearch(h, R, s["D"], r, y, sigma)
        return dict(q=q if h.dtype == torch.float64 else q.astype(np.float32), alpha=alpha)
    if op == "eval":
        L, AX, CX = alm.alm_eval(h, R, r, y, sigma)
        return dict(L=L, AX=AX.to(h.dtype), CX=CX)
    raise ValueError(op)


# ------------------------------------------------------------------------------------
# what a call cannot do without
# ------------------------------------------------------------------------------------
def _mean_size(case):
    """(rows, off-diagonal entries of the upper triangle, constraints) of a case, on average."""
    if case["op"] in ("batch", "train"):
        n = 0.5 * (case["n_lo"] + case["n_hi"]) * case["count"]
        return n, 0.25 * (case["d_lo"] + case["d_hi"]) * n, n
    n, graph = case["n"], case["graph"]
    if graph == "mc":
        m = min(math.ceil(9 * math.log(n) * (n - 3)), (n // 2) * (n - n // 2))
        return n, m, m
    edges = {"torus": 2.0, "regular3": 1.5, "kron": 14.0}.get(graph, 0.5 * case.get("deg", 0.0)) * n
    return n, edges, edges if graph == "theta" else n


def work(case):
    n, nu, m = _mean_size(case)
    e = 8 if case.get("precision") == "fp64" else 4
    op, r = case["op"], case.get("r", RANK)
    pattern = nu * (8 + e) + n * 8            # each entry of the triangle once: indices, value, diagonal
    if op in ("solve", "batch"):
        steps = case["outer"] * (case["inner"] if case["inner"] < 1000 else 10)
        # a step reads R, Z, D and writes them; two products with S and about 20 operations an element
        by, fl = steps * (6 * n * r * e + pattern), steps * n * r * 20 + steps * 8 * nu * r
        if op == "solve" and case["r"] < case["r_max"]:  # one Lanczos cycle per outer iteration
            by += case["outer"] * 32 * (pattern + n * e * 16)
            fl += case["outer"] * 32 * (4 * nu + 4 * 2 * 16 * n)
        return dict(bytes=by, flops=fl)
    if op in ("warm", "train"):
        a = 2 if case["storage"] == "bf16" else 4
        acts = n * a * (FEAT + LAYERS * HID)
        fl = n * 2 * (2 * FEAT * HID + 4 * HID * HID + RANK * HID + HID) + 4 * nu * (FEAT + 2 * HID)
        if op == "warm":
            return dict(bytes=2 * acts + 8 * 2 * nu + n * (4 * RANK + 8), flops=fl)
        return dict(bytes=4 * acts + 16 * 2 * nu + n * (4 * RANK * 3 + 16), flops=3 * fl + 8 * nu * RANK)
    if op == "lambda":
        return dict(bytes=32 * (pattern + n * e * 16) + n * r * e, flops=32 * (4 * nu + 4 * 2 * 16 * n))
    blocks = {"eval": 1, "grad": 2, "linesearch": 2}[op]
    return dict(bytes=pattern + blocks * n * r * e + 16 * m, flops=(2 + 4 * (blocks - 1)) * (nu + n) * r)


# ------------------------------------------------------------------------------------
# the results in plain 64-bit arithmetic
# ------------------------------------------------------------------------------------
class _Problem:
    """The SDP data of one or several instances (block-diagonal) as 64-bit tensors."""

    def __init__(self, insts):
        off = np.concatenate([[0], np.cumsum([x.n for x in insts])])
        moff = np.concatenate([[0], np.cumsum([x.m for x in insts])])
        cat = lambda key, o: torch.as_tensor(np.concatenate(
            [np.asarray(getattr(x, key), np.int64) + k for x, k in zip(insts, o)]), device=_device())
        val = lambda key: torch.as_tensor(np.concatenate([getattr(x, key) for x in insts]), dtype=torch.float64, device=_device())
        self.n, self.m, self.count = int(off[-1]), int(moff[-1]), len(insts)
        self.ci, self.cj, self.cv = cat("c_i", off), cat("c_j", off), val("c_v")
        self.ak, self.ai, self.aj, self.av, self.b = cat("a_k", moff), cat("a_i", off), cat("a_j", off), val("a_v"), val("b")
        lr = insts[0].c_lr_k > 0
        self.u = torch.as_tensor(insts[0].c_lr_u.T, dtype=torch.float64, device=_device()) if lr else None
        self.s = torch.as_tensor(insts[0].c_lr_s, dtype=torch.float64, device=_device()) if lr else None
        rep = lambda sizes: torch.repeat_interleave(torch.arange(self.count, device=_device()), torch.as_tensor(sizes, device=_device()))
        self.seg, self.mseg = rep([x.n for x in insts]), rep([x.m for x in insts])
        d = self.ci == self.cj
        self.cd = torch.zeros(self.n, dtype=torch.float64, device=_device()).index_add_(0, self.ci[d], self.cv[d])
        w2 = torch.where(d, 1.0, 2.0) * self.cv ** 2
        self.norm_c = self.total(torch.zeros_like(self.cd).index_add_(0, self.ci, w2)).sqrt()
        self.norm_b = self.mtotal(self.b ** 2).sqrt()
        sel = (self.ai == self.aj) & (torch.bincount(self.ak, minlength=self.m)[self.ak] == 1)
        self.sel_a = torch.zeros_like(self.cd).index_add_(0, self.ai[sel], self.av[sel])

    def total(self, x):
        return torch.zeros(self.count, dtype=torch.float64, device=x.device).index_add_(0, self.seg, x)

    def mtotal(self, x):
        return torch.zeros(self.count, dtype=torch.float64, device=x.device).index_add_(0, self.mseg, x)

    def dot(self, x, y):
        return self.total((x * y).sum(1))

    @staticmethod
    def _pairs(i, j, v, x, y):
        xy = (x[i] * y[j]).sum(1) + (x[j] * y[i]).sum(1)
        return v * torch.where(i == j, 0.5 * xy, xy)

    def amap(self, x, y):
        """<A_k, (x y^T + y x^T) / 2> of every constraint."""
        return torch.zeros_like(self.b).index_add_(0, self.ak, self._pairs(self.ai, self.aj, self.av, x, y))

    def cost(self, x):
        c = self.total(torch.zeros_like(self.cd).index_add_(0, self.ci, self._pairs(self.ci, self.cj, self.cv, x, x)))
        return c if self.u is None else c + ((self.u.T @ x) ** 2).sum(1) @ self.s

    def slack(self, w, x):
        """(C - A^*(w)) x."""
        out = torch.zeros_like(x)
        for i, j, v in ((self.ci, self.cj, self.cv), (self.ai, self.aj, -self.av * w[self.ak])):
            out.index_add_(0, i, v[:, None] * x[j])
            o = i != j
            out.index_add_(0, j[o], v[o, None] * x[i[o]])
        return out if self.u is None else out + self.u @ (self.s[:, None] * (self.u.T @ x))

    def diagonal(self, w):
        d = self.ai == self.aj
        return self.cd.clone().index_add_(0, self.ai[d], -(self.av * w[self.ak])[d])

    def dual(self, x, y, sigma):
        res = self.amap(x, x) - self.b
        return y - sigma[self.mseg] * res, res

    def quartic(self, R, D, y, sigma):
        w, res = self.dual(R, y, sigma)
        a1, a2 = 2.0 * self.amap(R, D), self.amap(D, D)
        SD = self.slack(w, D)
        half = 0.5 * sigma
        q0 = self.cost(R) - self.mtotal(y * res) + half * self.mtotal(res ** 2)
        return torch.stack([q0, 2.0 * self.dot(SD, R), self.dot(SD, D) + half * self.mtotal(a1 ** 2),
                            sigma * self.mtotal(a1 * a2), half * self.mtotal(a2 ** 2)], 1)


def _argmin(q):
    """The smallest minimiser of the quartic on alpha >= 0 (0: no descent)."""
    roots = np.roots([4 * q[4], 3 * q[3], 2 * q[2], q[1]])
    best = (0.0, 0.0)
    for a in sorted(roots[np.abs(roots.imag) <= 1e-7 * (1 + np.abs(roots))].real):
        v = a * (q[1] + a * (q[2] + a * (q[3] + a * q[4])))
        if a > 0 and v < best[0]:
            best = (v, a)
    return best[1]


def _splitmix(seed, n):
    with np.errstate(over="ignore"):
        z = np.uint64(seed % (1 << 64)) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.as_tensor(2.0 * ((z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0) - 1.0, device=_device())


def _lanczos(product, n, seed, tol_rel, tol_abs, k=32, cycles=400):
    """Smallest eigenpair by restarted Lanczos with twice-applied Gram-Schmidt."""
    q = _splitmix(seed, n)
    q = q / q.norm()
    for _ in range(cycles):
        Q, a, b, norm = [q], [], [], 0.0
        for j in range(min(k, n)):
            B = torch.stack(Q, 1)
            w = product(Q[j][:, None])[:, 0]
            h1 = B.T @ w
            w = w - B @ h1
            h2 = B.T @ w
            w = w - B @ h2
            a.append(float(h1[j] + h2[j]))
            b.append(float(w.norm()))
            norm = max(norm, abs(a[j]) + b[j] + (b[j - 1] if j else 0.0))
            if not b[j] > 1e-13 * norm:
                break
            Q.append(w / b[j])
        m = len(a)
        val, vec = np.linalg.eigh(np.diag(a) + np.diag(b[: m - 1], 1) + np.diag(b[: m - 1], -1))
        q = torch.stack(Q[:m], 1) @ torch.as_tensor(vec[:, 0], device=_device())
        q = q / q.norm()
        if abs(b[m - 1] * vec[m - 1, 0]) <= max(tol_rel * norm, tol_abs) or not b[m - 1] > 1e-13 * norm:
            break
    return float(val[0]), q


def _inner(P, R, y, sigma, tau, budget):
    """Preconditioned Polak-Ribiere CG with exact steps on the augmented Lagrangian."""
    floor = (1e-2 * (1.0 + P.total(P.cd.abs()) / torch.bincount(P.seg, minlength=P.count)))[P.seg]
    ka = 4.0 * sigma[P.seg] * P.sel_a ** 2
    Z, D = torch.zeros_like(R), torch.zeros_like(R)
    zg_prev, run_on = torch.zeros_like(sigma), torch.ones_like(sigma, dtype=torch.bool)
    for _ in range(budget):
        w, _ = P.dual(R, y, sigma)
        G = 2.0 * P.slack(w, R)
        run_on &= P.dot(G, G).sqrt() > tau
        if not bool(run_on.any()):
            break
        sd = 2.0 * torch.maximum(P.diagonal(w), floor)
        coef = ka * (R * G).sum(1) / (sd + ka * (R * R).sum(1))
        Zn = (G - coef[:, None] * R) / sd[:, None]
        zg, go, gd = P.dot(Zn, G), P.dot(G, Z), P.dot(G, D)
        beta = torch.where(zg_prev > 0, ((zg - go) / zg_prev).clamp(min=0.0), 0.0)
        beta = torch.where(-zg + beta * gd >= 0, 0.0, beta)
        D, Z, zg_prev = beta[P.seg, None] * D - Zn, Zn, zg
        q = P.quartic(R, D, y, sigma)
        q[:, 1] = -zg + beta * gd
        alpha = torch.tensor([_argmin(x) if on else 0.0 for x, on in zip(q.cpu().numpy(), run_on.tolist())],
                             dtype=torch.float64, device=R.device)
        run_on &= alpha > 0
        R = R + alpha[P.seg, None] * D
    return R


def _solve(P, R, y, case, eps=1e-6):
    """The augmented-Lagrangian iterations of a solve under its step budget."""
    fp32 = case.get("precision") != "fp64"
    sigma = torch.full((P.count,), case["sigma"], dtype=torch.float64, device=R.device)
    adaptive = case.get("r_max", case["r"]) > case["r"]
    tau, prev = 0.1 if adaptive else 1e-6, None
    for outer in range(1, case["outer"] + 1):
        if outer > 1:
            tau = max(0.1 * eps, 0.7 * tau if prev is None else min(0.7 * tau, 0.1 * prev))
        R = _inner(P, R, y, sigma, tau * (1.0 + P.norm_c), case["inner"])
        w, res = P.dual(R, y, sigma)
        lam = 0.0
        if adaptive and R.shape[1] < case["r_max"]:
            lam, v = _lanczos(lambda x: P.slack(w, x), P.n, 0x5EED + outer * 0x100000001, 1e-5 if fp32 else 1e-10,
                              0.1 * eps * float(1.0 + P.norm_c))
            if lam < -eps * float(1.0 + P.norm_c):
                vv = v[:, None]
                grow = math.sqrt(-lam / (case["sigma"] * float((P.amap(vv, vv) ** 2).sum())))
                R = torch.cat([R, grow * vv], 1)
                y = P.dual(R, y, sigma)[0]
                continue
        y = w
        c0, bw = P.cost(R), P.mtotal(P.b * w)
        p = P.mtotal(res ** 2).sqrt() / (1.0 + P.norm_b)
        g = (c0 - bw).abs() / (1.0 + c0.abs() + bw.abs())
        prev = max(float(p.max()), abs(min(0.0, lam)) / float(1.0 + P.norm_c.min()), float(g.max()))
    return R, y, P.cost(R)


def _network(case, seed, insts, theta):
    """The network's heads (rhat, yhat) and each row's mean |C_ij| scale."""
    P = _Problem(insts)
    o = P.ci != P.cj
    i, j = torch.cat([P.ci[o], P.cj[o]]), torch.cat([P.cj[o], P.ci[o]])
    a = P.cv[o].repeat(2)
    rows = lambda x: torch.zeros(P.n, dtype=torch.float64, device=_device()).index_add_(0, i, x)
    deg, s = rows(torch.ones_like(a)), rows(a)
    cnt = torch.bincount(P.seg, minlength=P.count).double()
    nnz, asum = P.total(deg), P.total(rows(a.abs()))
    cbar = torch.where(nnz > 0, asum / nnz.clamp(min=1.0), 1.0)
    sbar = P.total(s.abs()) / cnt
    sbar = torch.where(sbar > 0, sbar, 1.0)
    x = [torch.ones_like(deg), deg / (nnz / cnt).clamp(min=1.0)[P.seg], s / sbar[P.seg], (cnt.log() / 8.0)[P.seg]]
    x += [torch.cat([_splitmix(seed + k, t.n) for t in insts]) for k in range(4)]
    h, at, din = torch.stack(x, 1), 0, FEAT

    def take(rows_, cols):
        nonlocal at
        at += rows_ * cols
        return theta[at - rows_ * cols: at].reshape(rows_, cols)

    for _ in range(LAYERS):
        Ws, Wn, bias = take(HID, din), take(HID, din), take(1, HID)
        agg = torch.zeros_like(h).index_add(0, i, (a / cbar[P.seg][i])[:, None] * h[j]) / deg.clamp(min=1.0)[:, None]
        h, din = torch.relu(h @ Ws.T + agg @ Wn.T + bias), HID
    return P, h @ take(RANK, HID).T, (h @ take(1, HID).T)[:, 0] + take(1, 1)[0, 0], cbar


def exact(case, seed):
    op = case["op"]
    if op in ("warm", "train"):
        insts = [_instance(case, seed)] if op == "warm" else _batch_instances(case, seed)
        theta = torch.as_tensor(_theta(seed), dtype=torch.float64, device=_device()).requires_grad_(op == "train")
        P, rhat, yhat, cbar = _network(case, seed, insts, theta)
        if op == "warm":
            u = torch.cat([_splitmix(seed ^ 0x3A1D, t.n * RANK).reshape(-1, RANK) for t in insts])
            w = torch.nn.functional.normalize(rhat, dim=1) + torch.nn.functional.normalize(u, dim=1)
            return dict(R=torch.nn.functional.normalize(w, dim=1), y=cbar[P.seg] * yhat, rank=None)
        Rs, ys = (t.double() for t in _solution(P.n, seed))
        o = P.ci != P.cj
        i, j = torch.cat([torch.arange(P.n, device=_device()), P.ci[o]]), torch.cat([torch.arange(P.n, device=_device()), P.cj[o]])
        e = (rhat[i] * rhat[j]).sum(1) - (Rs[i] * Rs[j]).sum(1)
        loss = (e ** 2).sum() / i.numel() + 0.01 * ((yhat - ys / cbar[P.seg]) ** 2).mean()
        loss.backward()
        return dict(loss=loss, grad=theta.grad)
    if op == "batch":
        insts = _batch_instances(case, seed)
        P = _Problem(insts)
        y = torch.as_tensor(np.concatenate([_multiplier(x, seed) for x in insts]), device=_device())
        R0 = _near_unit(P.n, case["r"], seed, torch.float32).double()
        R, y, objective = _solve(P, R0, y, case)
        return dict(R=torch.nn.functional.pad(R, (0, RANK - case["r"])), y=y, rank=None, objective=objective)
    inst = _instance(case, seed)
    P = _Problem([inst])
    R = _factor(case, inst, seed).double()
    sigma = torch.full((1,), case["sigma"], dtype=torch.float64, device=_device())
    if op == "solve":
        R, y, objective = _solve(P, R, torch.as_tensor(_multiplier(inst, seed), device=_device()), case)
        return dict(R=_fix_sign(R) if case["r"] < case["r_max"] else R, y=y, objective=objective[0])
    y = _dual(case, inst, seed)
    w, res = P.dual(R, y, sigma)
    if op == "lambda":
        lam, v = _lanczos(lambda x: P.slack(w, x), P.n, 0x5EED, 1e-10 if case["precision"] == "fp64" else 1e-5, 0.0)
        return dict(lam=lam, v=_fix_sign(v[:, None]))
    if op == "grad":
        G = 2.0 * P.slack(w, R)
        width = 2 if case["precision"] == "fp64" else 4  # elements of 16 bytes
        return dict(G=torch.nn.functional.pad(G, (0, -G.shape[1] % width)), g2=(G * G).sum())
    if op == "linesearch":
        q = P.quartic(R, _direction(case, inst, seed).double(), y, sigma)[0].cpu().numpy()
        return dict(q=q, alpha=_argmin(q))
    L = P.cost(R)[0] - (y * res).sum() + 0.5 * sigma[0] * (res ** 2).sum()
    return dict(L=L, AX=P.amap(R, R), CX=P.cost(R)[0])
