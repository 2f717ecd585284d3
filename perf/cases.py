"""Performance cases of the force-kernel solver: what a training or prediction program calls.

A program sets up one context per kernel system, builds a preconditioner, solves by PCG -- whose
time is the matvec and the Woodbury apply of every iteration -- and predicts forces.  So the cases
are single matvecs and applies, preconditioner builds, a solve, a whole training call and a
prediction, from a few dozen geometries (where launches and latency count) to n = 630,000.  The
sizes are the workloads of ``paper_2212_12737_gb300.synth`` (ethanol9_m200, aspirin21_m1000,
mol42_m5000), ragged members of its batched suite and generic small ones.  FP64 is the default
precision of a context, OZAKI the one that the benchmark's solves run in.  The TF32 and BF16 forms
cannot reach the method's target at its ridge and are left out.

Ridge: matvecs use the workloads' own 1e-10 .. 1e-8.  A preconditioner's output at such a ridge is
rounding in C amplified by |C| / lambda, so outputs of builds and applies are compared at 1e-2, the
strongly regularised setting of the refinement tests; their time does not depend on it.  Solves use
1e-4 and few columns, so that PCG runs some tens of iterations to a solution that is well determined.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2212_12737_gb300 import gdml, synth

RIDGE = 1e-2
RIDGE_SOLVE = 1e-4


def listed():
    return [
        # the smallest call: a matvec of a few geometries with no context (real-time loops, callers
        # that cannot allocate); launches and latency are all of it
        dict(name="noalloc_tiny", kind="noalloc", N=6, M=24, sigma=4.0, noise=0.1, lam=1e-8),
        # the matvec of every PCG iteration: ethanol-sized (latency), aspirin-sized, and the
        # 42-atom system of the benchmark's headline
        dict(name="matvec_ethanol", kind="matvec", N=9, M=200, sigma=10.0, noise=0.05, lam=1e-10),
        dict(name="matvec_aspirin", kind="matvec", N=21, M=1000, sigma=20.0, noise=0.05, lam=1e-10),
        dict(name="matvec_mol42", kind="matvec", N=42, M=5000, sigma=30.0, noise=0.1, lam=1e-9),
        # the symmetric (sGDML) kernel, six atom permutations, odd M
        dict(name="matvec_sym", kind="matvec_sym", N=15, M=777, sigma=10.0, noise=0.05, lam=1e-8),
        # the preconditioner's apply of every PCG iteration, at the aspirin workload's k
        dict(name="apply_aspirin", kind="apply", N=21, M=1000, k=2000, sigma=20.0, noise=0.05),
        # a ragged member of the batched suite: n = 34,965 is odd, k = M // 10
        dict(name="apply_ragged", kind="apply", N=15, M=777, k=77, sigma=10.0, noise=0.05),
        # preconditioner builds: Algorithm 1 as in the aspirin workload, leverage scores as in the
        # 42-atom workload (an odd M, a fifth of its geometries)
        dict(name="build_pivchol", kind="build", select="pivchol", N=21, M=1000, k=2000, sigma=20.0, noise=0.05),
        dict(name="build_rls", kind="build", select="rls", N=42, M=1001, k=1500, sigma=30.0, noise=0.1),
        # PCG on a prepared context: the call that training time is spent in
        dict(name="solve_aspirin", kind="solve", N=21, M=1000, k=100, sigma=20.0, noise=0.05),
        # a whole training call as the defaults give it (FP64): set-up, uniform columns, solve
        dict(name="train_ethanol", kind="train", N=9, M=200, k=100, sigma=10.0, noise=0.05),
        # forces for new geometries from a trained model
        dict(name="predict_aspirin", kind="predict", N=21, M=1000, Q=300, sigma=20.0, noise=0.05),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "matvec", "matvec", "matvec", "matvec_sym", "apply", "apply", "build", "build",
                       "solve", "train", "predict"])
    c = dict(kind=kind, N=rng.choice([9, 12, 15, 21, 42]), sigma=rng.choice([5.0, 10.0, 20.0, 40.0]), noise=0.05)
    if kind == "noalloc":
        c.update(N=rng.randint(4, 24), M=_log_int(rng, 8, 128), lam=1e-8, noise=0.1)
    elif kind == "matvec":
        c.update(M=_log_int(rng, 100, 4000), lam=rng.choice([1e-10, 1e-8]))
    elif kind == "matvec_sym":
        c.update(N=rng.choice([9, 12, 15]), M=_log_int(rng, 100, 1000), lam=1e-8)
    elif kind in ("apply", "solve"):
        c.update(M=_log_int(rng, 100, 1000), noise=0.05)
        c.update(N=rng.choice([9, 12, 15, 21]), k=_log_int(rng, 20, 800))
    elif kind == "build":
        c.update(N=rng.choice([9, 12, 15, 21]), M=_log_int(rng, 100, 1000), k=_log_int(rng, 50, 1200))
        c.update(select=rng.choice(["pivchol", "rls"]))
    elif kind == "train":
        c.update(N=rng.choice([6, 9]), M=_log_int(rng, 50, 200))
        c.update(k=max(1, c["M"] // 2))
    else:
        c.update(N=rng.choice([9, 12, 15, 21]), M=_log_int(rng, 100, 1000), Q=_log_int(rng, 1, 500))
    if "k" in c:
        c["k"] = min(c["k"], 3 * c["N"] * c["M"] // 4)
    return c


# ------------------------------------------------------------------------------ inputs
def _perms(N):
    """S3 on atoms 0, 1, 2: six permutations of the atoms, a group."""
    return [list(p) + list(range(3, N)) for p in itertools.permutations((0, 1, 2))]


def _inputs(case, seed):
    """Geometries R (M, N, 3), labels y and a search direction v (n) as CUDA tensors."""
    tmpl = synth.template(case["N"], 0)
    R = synth.geometries(tmpl, case["M"], case["noise"], seed)
    y = synth.morse_forces(R, tmpl).reshape(-1)
    v = np.random.default_rng([seed, 1]).standard_normal(y.size)
    return tuple(torch.from_numpy(x).cuda() for x in (R, y, v))


def _queries(case, seed):
    tmpl = synth.template(case["N"], 0)
    return torch.from_numpy(synth.geometries(tmpl, case["Q"], 2 * case["noise"], seed + 1_000_003)).cuda()


def prepare(case, seed):
    R, y, v = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case, R=R, y=y, v=v)
    if kind in ("matvec", "matvec_sym"):
        s["ctx"] = gdml.kernel_setup(R, case["sigma"], case["lam"], "ozaki",
                                     perms=_perms(case["N"]) if kind == "matvec_sym" else None)
    elif kind in ("apply", "solve", "build"):
        s["ctx"] = gdml.kernel_setup(R, case["sigma"], RIDGE_SOLVE if kind == "solve" else RIDGE, "ozaki")
        if kind != "build":
            s["ctx"].precond_build("pivchol", case["k"])
    elif kind == "predict":
        s["ctx"] = gdml.kernel_setup(R, case["sigma"], RIDGE)
        s["Rq"] = _queries(case, seed)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "noalloc":
        return gdml.matvec_noalloc(state["R"], case["sigma"], case["lam"], state["v"])
    if kind in ("matvec", "matvec_sym"):
        return gdml.matvec(state["ctx"], state["v"])
    if kind == "apply":
        return gdml.precond_apply(state["ctx"], state["v"])
    if kind == "build":
        # the selected columns, Algorithm 1's residual trace, and the built operator at work
        piv, trace = gdml.precond_build(state["ctx"], case["select"], case["k"], pivots=True, trace=True)
        return dict(pivots=piv, trace=trace, z=gdml.precond_apply(state["ctx"], state["v"]))
    if kind == "solve":
        return gdml.pcg_solve(state["ctx"], state["y"], rtol=1e-11)[0]
    if kind == "train":
        ctx = gdml.kernel_setup(state["R"], case["sigma"], RIDGE_SOLVE)
        gdml.precond_build(ctx, "uniform", case["k"])
        alpha = gdml.pcg_solve(ctx, state["y"], rtol=1e-11)[0]
        ctx.destroy()
        return alpha
    return state["ctx"].predict_forces(state["Rq"], state["v"])


def work(case):
    """Vectors, geometries and (for the apply) the stored factor once; the method's products."""
    M, N, kind = case["M"], case["N"], case["kind"]
    n, D = 3 * M * N, N * (N - 1) // 2
    S = 6 if kind == "matvec_sym" else 1
    mv = 6.0 * M * M * S * D
    if kind in ("noalloc", "matvec", "matvec_sym"):
        return dict(bytes=8.0 * 3 * n, flops=mv)
    k = case.get("k", 0)
    if kind == "apply":
        return dict(bytes=4.0 * n * k + 16.0 * n, flops=4.0 * n * k)
    if kind == "build":
        # the factor is written once; columns, triangular products and C = lambda I + L^T L
        f = {"pivchol": 2.0, "rls": 5.0}[case["select"]]
        return dict(bytes=4.0 * n * k + 16.0 * n, flops=f * n * k * k)
    if kind == "solve":
        return dict(bytes=4.0 * n * k + 24.0 * n, flops=20.0 * (mv + 4.0 * n * k))
    if kind == "train":
        return dict(bytes=24.0 * n, flops=2.0 * n * k * k + 20.0 * (mv + 4.0 * n * k))
    Q = case["Q"]
    return dict(bytes=8.0 * (2 * n + 6 * Q * N), flops=6.0 * Q * M * D)


# ------------------------------------------------------------- the same in plain FP64 torch
class _Kernel:
    """The force kernel of the training geometries, plain torch in FP64."""

    def __init__(self, R, sigma, perms=None):
        N = R.shape[1]
        self.N, self.c = N, math.sqrt(5.0) / sigma
        i, j = np.tril_indices(N, -1)
        self.i, self.j = torch.from_numpy(i).to(R.device), torch.from_numpy(j).to(R.device)
        self.x, self.g = self.desc(R)
        self.pi = None
        if perms is not None:  # (P_q x)_(i,j) = x_(s(i), s(j)) for the permutation s
            rows = []
            for s in perms:
                a, b = np.asarray(s)[i], np.asarray(s)[j]
                hi, lo = np.maximum(a, b), np.minimum(a, b)
                rows.append(hi * (hi - 1) // 2 + lo)
            self.pi = torch.from_numpy(np.stack(rows)).to(R.device)
        self.mean = self.x.mean(0)

    def desc(self, R):
        d = R[:, self.i] - R[:, self.j]
        r = d.norm(dim=2)
        return 1.0 / r, d / r.pow(3)[:, :, None]

    def jv(self, g, v):  # w_a = J_a v_a
        v = v.view(g.shape[0], self.N, 3)
        return -(g * (v[:, self.i] - v[:, self.j])).sum(2)

    def jtu(self, g, u):  # J_a^T u_a
        t = g * u[:, :, None]
        out = torch.zeros(g.shape[0], self.N, 3, dtype=torch.float64, device=g.device)
        out.index_add_(1, self.i, -t)
        out.index_add_(1, self.j, t)
        return out

    def times(self, xq, gq, v):
        """Rows of K for the geometries (xq, gq) against all training geometries, times v."""
        w, xb = self.jv(self.g, v), self.x
        if self.pi is not None:
            w, xb = w[:, self.pi].reshape(-1, w.shape[1]), xb[:, self.pi].reshape(-1, w.shape[1])
        xb, xq = xb - self.mean, xq - self.mean
        t = (xb * w).sum(1)
        c, out = self.c, []
        for a0 in range(0, xq.shape[0], 256):
            xa = xq[a0:a0 + 256]
            r = torch.cdist(xa, xb, compute_mode="donot_use_mm_for_euclid_dist")
            s = (c * c / 3.0) * torch.exp(-c * r)
            beta = c * c * s * (xa @ w.T - t)
            u = (s * (1.0 + c * r)) @ w + beta @ xb - beta.sum(1, keepdim=True) * xa
            out.append(self.jtu(gq[a0:a0 + 256], u))
        return torch.cat(out)

    def column(self, q):
        """K[:, q]."""
        b, l = divmod(q, 3 * self.N)
        v = torch.zeros(1, 3 * self.N, dtype=torch.float64, device=self.x.device)
        v[0, l] = 1.0
        w = self.jv(self.g[b:b + 1], v)
        d = self.x - self.x[b]
        r = d.norm(dim=1, keepdim=True)
        c = self.c
        s = (c * c / 3.0) * torch.exp(-c * r)
        u = s * ((1.0 + c * r) * w - c * c * d * (d * w).sum(1, keepdim=True))
        return self.jtu(self.g, u).reshape(-1)

    def diagonal(self):
        q = self.g.square()
        out = torch.zeros(q.shape[0], self.N, 3, dtype=torch.float64, device=q.device)
        out.index_add_(1, self.i, q)
        out.index_add_(1, self.j, q)
        return (self.c * self.c / 3.0) * out.reshape(-1)


def _pivoted(K, k):
    """Rows l_0 .. l_(k-1) of L^T by incomplete Cholesky with diagonal pivoting, and the trace of
    the residual after each step."""
    d = K.diagonal()
    L = torch.zeros(k, d.numel(), dtype=torch.float64, device=d.device)
    trace = []
    for m in range(k):
        p = int(torch.argmax(d))
        root = d[p].sqrt()
        L[m] = (K.column(p) - L[:m, p] @ L[:m]) / root
        L[m][torch.isinf(d)] = 0.0
        L[m, p] = root
        d = d - L[m].square()
        d[p] = -math.inf
        trace.append(d[~torch.isinf(d)].sum())
    return L, torch.stack(trace)


def _apply(L, lam, r):
    C = L @ L.T + lam * torch.eye(L.shape[0], dtype=torch.float64, device=L.device)
    return (r - torch.linalg.solve(C, L @ r) @ L) / lam


def _converged(K, L, lam, y):
    """The solution by preconditioned CG in FP64, to the rounding of the residual."""
    C = torch.linalg.cholesky(L @ L.T + lam * torch.eye(L.shape[0], dtype=torch.float64, device=L.device))

    def prec(r):
        return (r - torch.cholesky_solve((L @ r)[:, None], C)[:, 0] @ L) / lam

    def op(v):
        return K.times(K.x, K.g, v).reshape(-1) + lam * v

    a = torch.zeros_like(y)
    r = y.clone()
    z = prec(r)
    p, rho = z.clone(), r @ z
    for _ in range(400):
        q = op(p)
        step = rho / (p @ q)
        a += step * p
        r -= step * q
        if float(r.norm()) <= 1e-13 * float(y.norm()):
            break
        z = prec(r)
        rho, old = r @ z, rho
        p = z + (rho / old) * p
    return a


def exact(case, seed):
    kind = case["kind"]
    R, y, v = _inputs(case, seed)
    K = _Kernel(R, case["sigma"], _perms(case["N"]) if kind == "matvec_sym" else None)
    if kind in ("noalloc", "matvec", "matvec_sym"):
        return K.times(K.x, K.g, v).reshape(-1) + case["lam"] * v
    if kind == "predict":
        return K.times(*K.desc(_queries(case, seed)), v)
    if kind == "apply":
        return _apply(_pivoted(K, case["k"])[0], RIDGE, v)
    if kind == "build":
        if case["select"] != "pivchol":
            return None
        L, trace = _pivoted(K, case["k"])
        return dict(pivots=None, trace=trace, z=_apply(L, RIDGE, v))
    # the solution does not depend on the preconditioner
    return _converged(K, _pivoted(K, min(case["k"], 300))[0], RIDGE_SOLVE, y)
