"""Performance cases of the butterfly completion library: what its users have it do,
from one small look-up to a full sweep at n = 65536, through the public entry points.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a
program holds before the call, run() is one pass, work() what a pass cannot do without,
exact() the same results in plain 64-bit torch.  Operations ("op"):

  eval      entries x_ij of a fitted operator (predictions)
  sweep     one ALS sweep from given factors, the loop body of a completion
  grad      the full gradient, the loop body of gradient-based completion
  matvec    the fitted operator applied to a block of vectors
  adam, adf a few iterations of a first-order completion
  complete  a whole completion from host arrays: context, low-rank start, sweeps, predictions

Data: the line-to-line Helmholtz kernel exp(i omega rho) / rho (or the phases of the
discretized Radon transform) at positions drawn without replacement, with relative noise
1e-4; factors: an embedded low-rank start, slightly perturbed (well-conditioned systems,
so that two runs that round differently can be compared).  Results of the complex64
precision form come back as complex64, the accuracy that they have.
"""
import math

import numpy as np
import torch

import paper_2510_17734_gb300 as bfc

RIDGE_C64 = 2.0 ** -20      # the precision form's documented ridge floor
CASES = [
    # a handful of predictions from a small operator, host arrays: call latency
    dict(name="eval_n256_few", op="eval", prec="fp64", n=256, L=4, r=4, m=61, host=True),
    # predictions at the test positions of the n = 65536 workload
    dict(name="eval_n65536", op="eval", prec="c64", n=65536, L=12, r=8, m=419430, host=False),
    # the sweep of the n = 256 workload: launches and short kernels
    dict(name="sweep_n256_r4", op="sweep", prec="c64", n=256, L=4, r=4, c=8.0, data="line"),
    # the n = 4096 workload in FP64 (the reference precision, refinement sweeps)
    dict(name="sweep_n4096_r6_fp64", op="sweep", prec="fp64", n=4096, L=8, r=6, c=6.0, data="line"),
    # an odd rank and a leaf size that is no power of two, at the sampling rule 6 r n log n
    dict(name="sweep_n3072_r5", op="sweep", prec="c64", n=3072, L=8, r=5, c=30.0, data="line"),
    # the n = 65536 workload, 3.8 M entries: the headline sweep
    dict(name="sweep_n65536_r8", op="sweep", prec="c64", n=65536, L=12, r=8, c=4.0, data="line"),
    # the Radon study's matrix, rank estimate and sampling (70 n log n) with leaves of 16
    dict(name="sweep_radon_n4096_r12", op="sweep", prec="c64", n=4096, L=8, r=12, c=77.0, data="radon"),
    # gradient of the n = 65536 workload
    dict(name="grad_n65536_r8", op="grad", prec="c64", n=65536, L=12, r=8, c=4.0, data="line"),
    # the fitted n = 65536 operator applied to 64 vectors
    dict(name="matvec_n65536_64", op="matvec", prec="c64", n=65536, L=12, r=8, m=64),
    # ADAM iterations on the n = 4096 workload in FP64
    dict(name="adam_n4096_r6_fp64", op="adam", prec="fp64", n=4096, L=8, r=6, c=6.0, data="line", iters=3),
    # ADF iterations on a rank-8, n = 16384 problem
    dict(name="adf_n16384_r8", op="adf", prec="c64", n=16384, L=10, r=8, c=6.0, data="line", iters=2),
    # a whole completion of a small problem from host arrays
    dict(name="complete_n1024_r6_fp64", op="complete", prec="fp64", n=1024, L=6, r=6, c=36.0, data="line", iters=3),
]


def listed():
    return [dict(c) for c in CASES]


def draw(rng):
    op = rng.choice(["eval", "sweep", "sweep", "sweep", "grad", "matvec", "adam", "adf", "complete"])
    prec = "fp64" if op == "complete" or op == "adam" or rng.random() < 0.3 else "c64"
    r = rng.randint(2, 12)
    b = rng.choice([x for x in (8, 11, 12, 16, 16, 20, 24) if 4 * r <= 3 * x])
    top = {"eval": 16, "matvec": 16, "complete": 12}.get(op, 16 if r <= 8 else 12)
    if prec == "fp64":
        top = min(top, 13 if r <= 6 else 12)
    L = rng.randint(4, max(4, int(math.log2(2.0 ** top / b))))
    n = b << L
    case = dict(op=op, prec=prec, n=n, L=L, r=r)
    if op == "eval":
        case.update(m=int(round(math.exp(rng.uniform(math.log(1), math.log(400000))))), host=rng.random() < 0.5)
    elif op == "matvec":
        case.update(m=int(round(math.exp(rng.uniform(0.0, math.log(min(256.0, 2.0 ** 22 / n)))))))
    else:
        # at least eight observations per unknown of a slice, four per unknown of a fiber; never most of the matrix
        low = max(16.0 * r * r / b, 5.0 * r) / math.log2(n)
        c = low * math.exp(rng.uniform(0.0, math.log(3.0)))
        most = min(3.5e6 if r <= 8 else 3.0e6, 0.5 * n * n) / (n * math.log2(n))
        case.update(c=round(min(c, most), 3), data=rng.choice(["line", "line", "radon"]))
        if op in ("adam", "adf"):
            case.update(iters=rng.randint(1, 3))
        if op == "complete":
            case.update(iters=rng.randint(1, 3))
    return case


# ------------------------------------------------------------------ inputs

def _counts(case):
    """(training entries, test entries) of a case with observations."""
    n_obs = int(case["c"] * case["n"] * math.log2(case["n"]))
    return n_obs - n_obs // 10, n_obs // 10


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _cnormal(shape, sigma, g):
    x = torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=g)
    return torch.view_as_complex(x * (sigma / math.sqrt(2.0)))


def _pairs(n, m, g):
    """m distinct (row, column) pairs in random order."""
    total = n * n
    if total <= 1 << 22:
        q = torch.randperm(total, device="cuda", generator=g)[:m]
    else:
        q = torch.unique(torch.randint(total, (2 * m + 1024,), device="cuda", generator=g))
        q = q[torch.randperm(q.numel(), device="cuda", generator=g)[:m]]
    return (q // n).to(torch.int32), (q % n).to(torch.int32)


def _values(kind, n, i, j, g):
    x, y = i.double(), j.double()
    if kind == "radon":
        x, y = (x + 1.0) / n, y + 1.0 - n / 2.0
        phi = x * y + (2.0 + torch.sin(2.0 * math.pi * x)) / 8.0 * y.abs()
        t = torch.polar(torch.ones_like(phi), 2.0 * math.pi * (phi - torch.floor(phi)))
    else:
        rho = torch.hypot((x - y) / n, torch.full_like(x, 1.5))
        t = torch.polar(1.0 / rho, math.pi * n / 16 * rho)
    return t + 1e-4 * t.abs().mean() * _cnormal(t.shape, 1.0, g)


def _factors(n, L, r, g):
    """An embedded low-rank pair with its slices slightly off the identity."""
    S = 2 << L
    z1, zL = _cnormal((n, r), 1.0, g), _cnormal((n, r), 1.0 / math.sqrt(r), g)
    Z = torch.eye(r, dtype=torch.complex128, device="cuda") + _cnormal((L, S, r, r), 0.2 / math.sqrt(r), g)
    return z1, Z, zL


def _inputs(case, seed):
    """Everything that a case's pass reads, on the GPU, from the seed alone."""
    g = _generator(seed)
    n, L, r = case["n"], case["L"], case["r"]
    d = {}
    if case["op"] in ("eval", "matvec"):
        d["i"], d["j"] = _pairs(n, 256, g)
        d["it"] = d["jt"] = d["tt"] = None
        d["t"] = _values("line", n, d["i"], d["j"], g)
        if case["op"] == "eval":
            d["pi"] = torch.randint(n, (case["m"],), dtype=torch.int32, device="cuda", generator=g)
            d["pj"] = torch.randint(n, (case["m"],), dtype=torch.int32, device="cuda", generator=g)
        else:
            d["V"] = _cnormal((n, case["m"]), 1.0, g)
    else:
        train, test = _counts(case)
        i, j = _pairs(n, train + test, g)
        t = _values(case["data"], n, i, j, g)
        d["i"], d["j"], d["t"] = i[:train].clone(), j[:train].clone(), t[:train].clone()
        d["it"], d["jt"], d["tt"] = i[train:].clone(), j[train:].clone(), t[train:].clone()
    if case["op"] == "complete":
        d["A"], d["B"] = _cnormal((n, r), 1.0, g), _cnormal((n, r), 1.0 / math.sqrt(r), g)
    else:
        d["z1"], d["Z"], d["zL"] = _factors(n, L, r, g)
    return d


LAMBDA = 1e-7
LR_SWEEPS = 4


class State:
    """A case's inputs, its context and the buffers that a program keeps between calls."""

    def __init__(self, case, seed):
        self.case, self.ctx, self.fit = case, None, None
        d = _inputs(case, seed)
        n, L, r = case["n"], case["L"], case["r"]
        self.c64 = case["prec"] == "c64"
        prec = bfc.PREC_C64 if self.c64 else bfc.PREC_FP64
        host = lambda x: x.cpu().numpy()  # noqa: E731
        if case["op"] == "complete":
            self.host = {k: host(v) for k, v in d.items()}
            return
        self.X = torch.cat([d["z1"].reshape(-1), d["Z"].reshape(-1), d["zL"].reshape(-1)])
        if case["op"] == "eval" and case["host"]:
            self.fit = bfc.Completion(n, L, n >> L, r, LAMBDA, host(d["i"]), host(d["j"]), host(d["t"]), prec=prec)
            self.fit.set_factors(host(self.X))
            self.pi, self.pj = host(d["pi"]), host(d["pj"])
            return
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        p = bfc.Params(n=n, L=L, b=n >> L, r=r, lam=LAMBDA, prec=prec, max_sweeps=20, tol=0.0, values_on_device=1)
        self.ctx = bfc.bfc_create(p, d["i"], d["j"], d["t"], d["it"], d["jt"], d["tt"])
        bfc.bfc_set_stream(self.ctx, self.stream.cuda_stream)
        bfc.bfc_set_factors(self.ctx, self.X)
        if case["op"] == "eval":
            self.pi, self.pj = d["pi"], d["pj"]
            self.out = torch.empty(case["m"], dtype=torch.complex128, device="cuda")
        elif case["op"] == "matvec":
            self.V = d["V"]
            self.out = torch.empty_like(self.V)
        else:
            self.out = torch.empty_like(self.X)

    def __del__(self):
        if self.ctx is not None:
            bfc.bfc_destroy(self.ctx)
        if self.fit is not None:
            self.fit.close()


def prepare(case, seed):
    return State(case, seed)


# -------------------------------------------------------------------- run

def run(s):
    op = s.case["op"]
    if op == "complete":
        return _complete(s)
    if s.fit is not None:
        x = s.fit.eval(s.pi, s.pj)
        return x.astype(np.complex64) if s.c64 else x
    got = {}
    with torch.cuda.stream(s.stream):
        if op == "eval":
            bfc.bfc_eval(s.ctx, s.pi, s.pj, s.out)
        elif op == "matvec":
            bfc.bfc_matvec(s.ctx, s.case["m"], s.V, s.out)
        elif op == "grad":
            got["objective"] = bfc.bfc_grad(s.ctx, True, s.out)
        else:
            bfc.bfc_set_factors(s.ctx, s.X)
            if op == "sweep":
                st = bfc.bfc_als_sweep(s.ctx)
            elif op == "adam":
                st = bfc.bfc_adam(s.ctx, s.case["iters"])[-1]
            else:
                st = bfc.bfc_adf(s.ctx, s.case["iters"])[-1]
            got.update(objective=st.objective, train=st.train_rel_err, test=st.test_rel_err,
                       singular=int(st.singular_slices))
            bfc.bfc_get_factors(s.ctx, s.out)
        got["out"] = s.out.to(torch.complex64) if s.c64 else s.out
    return got


def _complete(s):
    h, n, L = s.host, s.case["n"], s.case["L"]
    with bfc.Completion(n, L, n >> L, s.case["r"], LAMBDA, h["i"], h["j"], h["t"], h["it"], h["jt"], h["tt"],
                        max_sweeps=s.case["iters"], tol=0.0) as fit:
        fit.lowrank_init(h["A"], h["B"], LR_SWEEPS)
        hist = fit.complete()
        return {"train": np.array([st["train_rel_err"] for st in hist], dtype=np.float32),
                "test": np.array([st["test_rel_err"] for st in hist], dtype=np.float32),
                "out": fit.eval(h["it"], h["jt"]).astype(np.complex64)}


# ------------------------------------------------------------------- work

def _groups(case, N):
    """Expected sum over the middle levels of the smaller of the row and the column groups."""
    n, L = case["n"], case["L"]
    b, S, total = n >> L, 2 << L, 0.0
    for m in range(1, L + 1):
        cells = S * min(b << (m - 1), b << (L - m))
        total += cells * -math.expm1(-N / cells)
    return total


def work(case):
    n, L, r = case["n"], case["L"], case["r"]
    D, S, vs = r * r, 2 << L, 8 if case["prec"] == "c64" else 16
    P = 2 * n * r + L * S * D
    entry = 8.0 * (L * D + r)                       # one evaluation of x_ij
    if case["op"] == "eval":
        touched = min(P, case["m"] * (2 * r + L * D))
        return {"bytes": case["m"] * (8 + 16) + touched * vs, "flops": case["m"] * entry}
    if case["op"] == "matvec":
        return {"bytes": 2 * n * case["m"] * 16 + P * vs, "flops": 8.0 * P * case["m"]}
    N, NT = _counts(case)
    data = 24.0 * (N + NT)
    chain = 2.0 * 8.0 * N * L * D                   # left and right environments
    if case["op"] == "grad":
        return {"bytes": 24.0 * N + P * (vs + 16), "flops": chain + 8.0 * N * (L * D + 3 * r)}
    if case["op"] == "adam":
        return {"bytes": case["iters"] * (data + 6.0 * P * 16),
                "flops": case["iters"] * (chain + 8.0 * N * L * 2 * D + NT * entry)}
    if case["op"] == "adf":
        return {"bytes": case["iters"] * (data + 2.0 * P * 16),
                "flops": case["iters"] * (chain + 8.0 * N * L * 3 * D + NT * entry + 8.0 * L * S * 6 * r ** 3)}

    def sweep(L, groups):
        mid = 8.0 * (groups * (D * (D + 1) / 2 + D) + N * L * (D + r)) + 8.0 * L * S * (D ** 3 / 6 + D * D)
        outer = 8.0 * 2 * (N * (r * (r + 1) / 2 + r) + n * (r ** 3 / 6 + D))
        return 2.0 * 8.0 * N * L * D + (mid if L else 0.0) + outer + NT * entry

    if case["op"] == "sweep":
        return {"bytes": data + 2.0 * P * 16, "flops": sweep(L, _groups(case, N))}
    return {"bytes": data + 2.0 * P * 16, "flops": LR_SWEEPS * sweep(0, 0.0) + case["iters"] * sweep(L, _groups(case, N))}


# ------------------------------------------------------------------ exact

class _Net:
    """The network of a case in plain torch, 64 bits."""

    def __init__(self, case, i, j, t):
        self.n, self.L, self.r = case["n"], case["L"], case["r"]
        self.b, self.S = self.n >> self.L, 2 << self.L
        self.i, self.j, self.t = i.long(), j.long(), t
        self.keys = self.keys_of(self.i, self.j)
        self.ridge = RIDGE_C64 if case["prec"] == "c64" else 0.0

    def keys_of(self, i, j):
        pi, pj = torch.div(i, self.b, rounding_mode="floor"), torch.div(j, self.b, rounding_mode="floor")
        return [((pi >> (m - 1)) << m) | (pj >> (self.L - m)) for m in range(1, self.L + 1)]

    @staticmethod
    def apply(Z, k, v, left):
        """v^T Z[k] (left) or Z[k] v, entry by entry."""
        out = torch.empty_like(v)
        for a in range(0, len(k), 1 << 19):
            e = slice(a, a + (1 << 19))
            M, x = Z[k[e]], v[e]
            out[e] = torch.bmm(x[:, None, :], M)[:, 0] if left else torch.bmm(M, x[:, :, None])[:, :, 0]
        return out

    def right(self, Z, zL):
        w = [None] * (self.L + 1)
        w[self.L] = zL[self.j]
        for m in range(self.L, 0, -1):
            w[m - 1] = self.apply(Z[m - 1], self.keys[m - 1], w[m], False)
        return w

    def entries(self, z1, Z, zL, i, j):
        i, j = i.long(), j.long()
        h = z1[i]
        for m, k in enumerate(self.keys_of(i, j)):
            h = self.apply(Z[m], k, h, True)
        return (h * zL[j]).sum(1)

    def segsum(self, key, K, D, f):
        """sum over the entries of each key of the rows f(slice of entries)."""
        out = torch.zeros(K, 2 * D, dtype=torch.float64, device="cuda")
        for a in range(0, len(key), 1 << 19):
            e = slice(a, a + (1 << 19))
            out.index_add_(0, key[e], torch.view_as_real(f(e).contiguous()).reshape(-1, 2 * D))
        return torch.view_as_complex(out.reshape(K, D, 2))

    def design(self, m, h, w, e=slice(None)):
        """Rows of the least-squares systems of level m (0: S^1, L + 1: S^{L+2})."""
        if m == 0:
            return w[0][e]
        if m == self.L + 1:
            return h[e]
        return (h[e][:, :, None] * w[m][e][:, None, :]).reshape(-1, self.r * self.r)

    def key(self, m):
        return (self.i, self.n) if m == 0 else (self.j, self.n) if m > self.L else (self.keys[m - 1], self.S)

    def fit(self, m, h, w):
        """The regularized least-squares solutions of one factor."""
        key, K = self.key(m)
        order = torch.argsort(key, stable=True)
        count = torch.bincount(key, minlength=K)
        start = torch.cumsum(count, 0) - count
        D, wide = (self.r if m in (0, self.L + 1) else self.r ** 2), int(count.max())
        per = max(1, int(2 ** 31 // (wide * D * 16)))
        eye, out = torch.eye(D, dtype=torch.complex128, device="cuda"), []
        for k0 in range(0, K, per):
            k1 = min(K, k0 + per)
            e = order[int(start[k0]): int(start[k1 - 1] + count[k1 - 1])]
            at = (key[e] - k0) * wide + torch.arange(len(e), device="cuda") + int(start[k0]) - start[key[e]]
            A = torch.zeros((k1 - k0) * wide, D, dtype=torch.complex128, device="cuda")
            y = torch.zeros((k1 - k0) * wide, 1, dtype=torch.complex128, device="cuda")
            A[at], y[at] = self.design(m, h, w, e), self.t[e][:, None]
            A, y = A.reshape(k1 - k0, wide, D), y.reshape(k1 - k0, wide, 1)
            G, rhs = A.mH @ A, A.mH @ y
            lam = (G.diagonal(dim1=1, dim2=2).real.mean(1) * self.ridge).clamp_min(LAMBDA)
            out.append(torch.linalg.solve(G + lam[:, None, None] * eye, rhs)[:, :, 0])
        return torch.cat(out)

    def sweep(self, z1, Z, zL):
        """Alg. 1: S^1, the middle factors, S^{L+2}; the last entries of the training set."""
        Z = Z.clone()
        w = self.right(Z, zL)
        z1 = self.fit(0, None, w)
        h = z1[self.i]
        for m in range(1, self.L + 1):
            Z[m - 1] = self.fit(m, h, w).reshape(-1, self.r, self.r)
            h = self.apply(Z[m - 1], self.keys[m - 1], h, True)
        zL = self.fit(self.L + 1, h, w)
        return z1, Z, zL, (h * zL[self.j]).sum(1)

    def gradient(self, m, h, w, res, s):
        key, K = self.key(m)
        D = s.numel() // K
        return (self.segsum(key, K, D, lambda e: res[e][:, None] * self.design(m, h, w, e).conj())
                + LAMBDA * s.reshape(K, D)).reshape(s.shape)

    def product(self, m, h, w, s):
        """The design rows times each entry's vector of s."""
        if m == 0:
            return (s[self.i] * w[0]).sum(1)
        if m == self.L + 1:
            return (h * s[self.j]).sum(1)
        return (h * self.apply(s.reshape(-1, self.r, self.r), self.keys[m - 1], w[m], False)).sum(1)

    def sums(self, x, z1, Z, zL, it, jt, tt):
        """objective, training and test error."""
        fit, norm = (x - self.t).abs().square().sum(), sum(v.abs().square().sum() for v in (z1, Z, zL))
        xt = self.entries(z1, Z, zL, it, jt)
        return {"objective": float(0.5 * fit + 0.5 * LAMBDA * norm),
                "train": float((fit / self.t.abs().square().sum()).sqrt()),
                "test": float(((xt - tt).abs().square().sum() / tt.abs().square().sum()).sqrt())}


def _adam(net, z1, Z, zL, iters):
    F = [z1.clone()] + [z.clone() for z in Z] + [zL.clone()]
    M, V = [torch.zeros(*f.shape, 2, dtype=torch.float64, device="cuda") for f in F], None
    V = [torch.zeros_like(m) for m in M]
    x = None
    for it in range(1, iters + 1):
        w, h = net.right(F[1:-1], F[-1]), None
        for m in range(net.L + 2):
            g = torch.view_as_real(net.gradient(m, h, w, net.product(m, h, w, F[m]) - net.t, F[m]))
            M[m], V[m] = 0.9 * M[m] + (1.0 - 0.9) * g, 0.999 * V[m] + (1.0 - 0.999) * g * g
            step = 1e-3 * (M[m] / (1.0 - 0.9 ** it)) / ((V[m] / (1.0 - 0.999 ** it)).sqrt() + 1e-8)
            F[m] = F[m] - torch.view_as_complex(step)
            if m == net.L + 1:
                x = net.product(m, h, w, F[m])
            else:
                h = F[0][net.i] if m == 0 else net.apply(F[m], net.keys[m - 1], h, True)
    return F[0], torch.stack(F[1:-1]), F[-1], x


def _qr(M):
    """QR with a real positive diagonal of R, twice through the Gram matrix."""
    R = torch.linalg.cholesky(M.mH @ M).mH
    Q = torch.linalg.solve_triangular(R, M, upper=True, left=False)
    R2 = torch.linalg.cholesky(Q.mH @ Q).mH
    return torch.linalg.solve_triangular(R2, Q, upper=True, left=False), R2 @ R


def _adf(net, z1, Z, zL, iters):
    L, r, b = net.L, net.r, net.b
    z1, Z, zL, x = z1.clone(), Z.clone(), zL.clone(), None
    for _ in range(iters):
        # right-to-left: the leaf blocks of zL, then the slice pairs of each level
        Q, R = _qr(zL.reshape(-1, b, r))
        zL, up = Q.reshape(-1, r), R.mT
        Z[L - 1] = (Z[L - 1].reshape(2, 1 << L, r, r) @ up).reshape(-1, r, r)
        for m in range(L, 0, -1):
            pair = Z[m - 1].reshape(-1, 2, r, r)
            Q, R = _qr(torch.cat([pair[:, 0], pair[:, 1]], 2).mH)
            Z[m - 1] = torch.stack([Q[:, :r].mH, Q[:, r:].mH], 1).reshape(-1, r, r)
            if m > 1:
                left = Z[m - 2].reshape(-1, 2, 1 << (m - 1), r, r)
                Z[m - 2] = (left @ R.mH.reshape(-1, 1, 1 << (m - 1), r, r)).reshape(-1, r, r)
            else:
                z1 = (z1.reshape(-1, b, r) @ R.mH).reshape(-1, r)
        w, h = net.right(Z, zL), None
        res = net.t - net.product(0, h, w, z1)
        for m in range(L + 2):
            s = z1 if m == 0 else zL if m > L else Z[m - 1]
            key, K = net.key(m)
            N = -net.gradient(m, h, w, -res, s)
            z, nn = net.product(m, h, w, N), N.reshape(K, -1).abs().square().sum(1)
            zz = torch.zeros(K, dtype=torch.float64, device="cuda").index_add_(0, key, z.abs().square())
            a = nn / (zz + LAMBDA * nn)
            s = s + (a[:, None] * N.reshape(K, -1)).reshape(s.shape)
            res = res - a[key] * z
            if m == 0:
                Q, R = _qr(s.reshape(-1, b, r))
                z1 = Q.reshape(-1, r)
                Z[0] = (R[:, None] @ Z[0].reshape(-1, 2, r, r)).reshape(-1, r, r)
                h = z1[net.i]
            elif m <= L:
                two = s.reshape(-1, 2, 1 << m, r, r)
                Q, R = _qr(torch.cat([two[:, 0], two[:, 1]], 2).reshape(-1, 2 * r, r))
                Q = Q.reshape(-1, 1 << m, 2 * r, r)
                Z[m - 1] = torch.stack([Q[:, :, :r], Q[:, :, r:]], 1).reshape(-1, r, r)
                if m < L:
                    Z[m] = (R[:, None] @ Z[m].reshape(-1, 2, r, r)).reshape(-1, r, r)
                else:
                    zL = (zL.reshape(-1, b, r) @ R.mT).reshape(-1, r)
                h = net.apply(Z[m - 1], net.keys[m - 1], h, True)
            else:
                zL = s
        x = net.t - res
    return z1, Z, zL, x


def _matvec(net, z1, Z, zL, V):
    L, r, b, q = net.L, net.r, net.b, V.shape[1]
    T = zL.reshape(-1, b, r).mT @ V.reshape(-1, b, q)           # per column prefix
    Y = Z[L - 1].reshape(2, 1 << L, r, r) @ T                   # k = (i_0, column prefix)
    for m in range(L - 1, 0, -1):
        T = Y.reshape(-1, 1, 1 << m, 2, r, q).sum(3)            # sum out j_m
        Y = Z[m - 1].reshape(-1, 2, 1 << m, r, r) @ T
    T = Y.reshape(-1, 2, r, q).sum(1)
    return (z1.reshape(-1, b, r) @ T).reshape(-1, q)


def exact(case, seed):
    d = _inputs(case, seed)
    net = _Net(case, d["i"], d["j"], d["t"])
    op = case["op"]
    if op == "complete":
        low = _Net(dict(case, L=0), d["i"], d["j"], d["t"])
        z1, Z, zL = d["A"], torch.empty(0, 2, case["r"], case["r"], dtype=torch.complex128, device="cuda"), d["B"]
        for _ in range(LR_SWEEPS):
            z1, Z, zL, x = low.sweep(z1, Z, zL)
        Z = torch.eye(net.r, dtype=torch.complex128, device="cuda").expand(net.L, net.S, net.r, net.r)
        hist = []
        for _ in range(case["iters"]):
            z1, Z, zL, x = net.sweep(z1, Z, zL)
            hist.append(net.sums(x, z1, Z, zL, d["it"], d["jt"], d["tt"]))
        return {"train": np.array([s["train"] for s in hist]), "test": np.array([s["test"] for s in hist]),
                "out": net.entries(z1, Z, zL, d["it"], d["jt"])}
    z1, Z, zL = d["z1"], d["Z"], d["zL"]
    if op == "eval":
        x = net.entries(z1, Z, zL, d["pi"], d["pj"])
        return x if case["host"] else {"out": x}
    if op == "matvec":
        return {"out": _matvec(net, z1, Z, zL, d["V"])}
    if op == "grad":
        w, h = net.right(Z, zL), None
        res, g = net.product(0, h, w, z1) - net.t, []
        for m in range(net.L + 2):
            s = z1 if m == 0 else zL if m > net.L else Z[m - 1]
            g.append(net.gradient(m, h, w, res, s).reshape(-1))
            h = z1[net.i] if m == 0 else h if m > net.L else net.apply(Z[m - 1], net.keys[m - 1], h, True)
        norm = sum(v.abs().square().sum() for v in (z1, Z, zL))
        return {"objective": float(0.5 * res.abs().square().sum() + 0.5 * LAMBDA * norm), "out": torch.cat(g)}
    if op == "sweep":
        z1, Z, zL, x = net.sweep(z1, Z, zL)
    elif op == "adam":
        z1, Z, zL, x = _adam(net, z1, Z, zL, case["iters"])
    else:
        z1, Z, zL, x = _adf(net, z1, Z, zL, case["iters"])
    got = net.sums(x, z1, Z, zL, d["it"], d["jt"], d["tt"])
    return dict(got, singular=None, out=torch.cat([z1.reshape(-1), Z.reshape(-1), zL.reshape(-1)]))
