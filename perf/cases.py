"""The work that users of the selected-inversion library have it do, as measurable cases.

Every case goes through the public entry points of
``paper_2309_05435_gb300.qsel``: the exact one-part selected inverse (the form
that the planner picks on one GPU), the plain and the mixed RBMC estimator,
the Krylov sampler, the hyperparameter gradient, the captured batch and the
control-variate network, in binary64 and in the mixed form, from the smallest
parity model to the block size of the benchmark workload.  A state is one
context (or batch, or network) with its model, as a program keeps it between
passes; a pass sets theta (or the seed) again and reads the results, which is
one step of a hyperparameter loop.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2309_05435_gb300 import qsel

LISTED = [
    # The benchmark's form (exact one part, mixed, tensor cores) at its own
    # block size, 96 x 96 grid: the largest factorisation blocks.
    dict(name="exact_mixed_96x96x16", kind="exact", precision="mixed", m=96, n_t=16, kappa=0.1, rho=0.98, obs=0.10),
    # The same form at the second workload's 64 x 64 grid.
    dict(name="exact_mixed_64x64x24", kind="exact", precision="mixed", m=64, n_t=24, kappa=0.2, rho=0.95, obs=0.25),
    # An ordinary small mesh whose size fits no tile (1369 nodes).
    dict(name="exact_mixed_37x37x21", kind="exact", precision="mixed", m=37, n_t=21, kappa=0.3, rho=0.9, obs=0.25),
    # Binary64 selected inverse: what weakly observed, ill-conditioned models
    # (here 5 % observed) need, since the mixed form is not for them.
    dict(name="exact_fp64_40x40x12", kind="exact", precision="fp64", m=40, n_t=12, kappa=0.2, rho=0.95, obs=0.05),
    # The plain method on the parity workload, the smallest call.
    dict(name="rbmc_fp64_16x16x8", kind="rbmc", precision="fp64", precond="jacobi", m=16, n_t=8, kappa=0.5, rho=0.9,
         obs=0.30, parts=2, overlap=1, k=64, tol=1e-10),
    # The plain method (block-Jacobi PCG, four parts) at an ordinary size.
    dict(name="rbmc_fp64_32x32x32", kind="rbmc", precision="fp64", precond="jacobi", m=32, n_t=32, kappa=0.3, rho=0.9,
         obs=0.25, parts=4, overlap=2, k=128, tol=1e-10),
    # The mixed estimator with the Kronecker preconditioner as the benchmark
    # runs it, many samples on the 64 x 64 grid.
    dict(name="rbmc_mixed_64x64x16", kind="rbmc", precision="mixed", precond="kron", m=64, n_t=16, kappa=0.2,
         rho=0.95, obs=0.25, parts=2, overlap=2, k=256, tol=1e-10),
    # The non-separable diffusion model, whose samples need the Krylov sampler.
    dict(name="lanczos_diffusion_24x24x16", kind="lanczos", precision="fp64", m=24, n_t=16, kappa=0.5, rho=0.9,
         obs=0.25, parts=2, overlap=1, k=64, steps=50),
    # One step of a hyperparameter fit: posterior mean and gradient.
    dict(name="hyper_mixed_48x48x16", kind="hyper", precision="mixed", precond="kron", m=48, n_t=16, kappa=0.2,
         rho=0.95, obs=0.25, parts=2, overlap=2, k=64, tol=1e-10),
    # Independent uneven models in one captured graph.
    dict(name="batch_mixed_8", kind="batch", precision="mixed", models=8, m_low=16, m_high=40, nt_low=8, nt_high=32,
         k=128, tol=1e-8),
    # Planning: features of every node and the network's forward pass.
    dict(name="network_forward_64x64x128", kind="forward", m=64, n_t=128, kappa=0.2, rho=0.95, obs=0.25, parts=8,
         overlap=2),
    # Training: loss and gradient of the network over a training set.
    dict(name="network_backward_65000", kind="backward", rows=65000),
]


def listed():
    return [dict(c) for c in LISTED]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["exact_mixed", "exact_mixed", "exact_fp64", "rbmc_fp64", "rbmc_mixed", "lanczos", "hyper",
                       "batch", "forward", "backward"])
    kappa, rho, obs = round(rng.uniform(0.15, 0.6), 3), round(rng.uniform(0.7, 0.97), 3), round(rng.uniform(0.1, 0.35), 3)
    model = dict(kappa=kappa, rho=rho, obs=obs)
    if kind == "exact_mixed":
        m = _log_int(rng, 12, 96)
        most = max(2, min(64, int(16 * (96 / m) ** 3)))
        return dict(kind="exact", precision="mixed", m=m, n_t=_log_int(rng, 2, most), **model)
    if kind == "exact_fp64":
        m = _log_int(rng, 8, 48)
        return dict(kind="exact", precision="fp64", m=m, n_t=_log_int(rng, 2, max(3, min(32, int(8 * (48 / m) ** 3)))), **model)
    if kind in ("rbmc_fp64", "rbmc_mixed", "hyper"):
        fp64 = kind == "rbmc_fp64"
        m = _log_int(rng, 8, 32) if fp64 else _log_int(rng, 16, 64)
        parts = rng.randint(2, 4)
        n_t = max(3 * parts, _log_int(rng, 6, 24))
        return dict(kind="hyper" if kind == "hyper" else "rbmc", precision="fp64" if fp64 else "mixed",
                    precond="jacobi" if fp64 else "kron", m=m, n_t=n_t, parts=parts, overlap=rng.randint(1, 3),
                    k=_log_int(rng, 16, 128 if fp64 else 256), tol=1e-10, **model)
    if kind == "lanczos":
        parts = rng.randint(2, 3)
        return dict(kind="lanczos", precision="fp64", m=_log_int(rng, 8, 24), n_t=rng.randint(3 * parts, 16), parts=parts,
                    overlap=1, k=_log_int(rng, 8, 64), steps=rng.randint(20, 50), **model)
    if kind == "batch":
        return dict(kind="batch", precision="mixed", models=rng.randint(2, 8), m_low=12, m_high=rng.randint(16, 40),
                    nt_low=6, nt_high=rng.randint(8, 32), k=_log_int(rng, 16, 128), tol=1e-8)
    if kind == "forward":
        parts = rng.randint(2, 8)
        return dict(kind="forward", m=_log_int(rng, 16, 64), n_t=rng.randint(3 * parts, 128), parts=parts,
                    overlap=rng.randint(1, 4), **model)
    return dict(kind="backward", rows=_log_int(rng, 500, 65000))


# --------------------------------------------------------------------------
# Models
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _mesh(m):
    """Linear elements on the unit m x m grid: lumped mass and stiffness (CSR)."""
    tri = np.zeros((m, m))
    for di, dj in ((0, 0), (1, 0), (1, 1), (0, 0), (1, 1), (0, 1)):
        tri[di:m - 1 + di, dj:m - 1 + dj] += 1.0
    i, j = np.divmod(np.arange(m * m), m)
    cols, vals, live = [], [], []
    for di, dj in ((-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)):
        a, b = i + di, j + dj
        edge = np.where(di != 0, (j == 0) | (j == m - 1), (i == 0) | (i == m - 1))
        cols.append(a * m + b)
        vals.append(np.where(edge, -0.5, -1.0))
        live.append((a >= 0) & (a < m) & (b >= 0) & (b < m))
    cols, vals, live = np.stack(cols, 1), np.stack(vals, 1), np.stack(live, 1)
    vals[:, 2] = 0.0
    vals[:, 2] = -(vals * live).sum(1)
    rowptr = np.concatenate([[0], np.cumsum(live.sum(1))]).astype(np.int32)
    return tri.reshape(-1) / 6.0, rowptr, cols[live].astype(np.int32), vals[live].copy()


def _theta(kappa, rho, rng):
    """(log kappa, log tau, logit rho), moved a little by the seed."""
    return (math.log(kappa) + rng.uniform(-0.1, 0.1), rng.uniform(-0.2, 0.2),
            math.log(rho / (1.0 - rho)) + rng.uniform(-0.1, 0.1))


def _mask(n, share, rng):
    mask = np.zeros(n, dtype=np.uint8)
    mask[rng.choice(n, size=max(1, int(round(share * n))), replace=False)] = 1
    return mask


def _inputs(case, seed):
    """The model of one context: host arrays, as a program hands them over."""
    rng = np.random.default_rng([seed, case["m"], case["n_t"]])
    return dict(theta=_theta(case["kappa"], case["rho"], rng),
                mask=_mask(case["m"] ** 2 * case["n_t"], case["obs"], rng), sigma=0.5, seed=int(rng.integers(1, 1 << 40)),
                rng=rng)


def _batch_inputs(case, seed):
    """Uneven models: grid side, slabs, parts, theta and mask of each."""
    size = np.random.default_rng([case["models"], case["m_high"], case["nt_high"]])
    rng = np.random.default_rng([seed, 77])
    out = []
    for _ in range(case["models"]):
        m = int(size.integers(case["m_low"], case["m_high"] + 1))
        n_t = int(size.integers(case["nt_low"], case["nt_high"] + 1))
        parts = int(size.integers(2, max(2, min(8, n_t // 3)) + 1))
        out.append(dict(m=m, n_t=n_t, parts=parts, theta=_theta(size.uniform(0.15, 0.8), size.uniform(0.5, 0.95), rng),
                        mask=_mask(m * m * n_t, 0.25, rng), sigma=0.5))
    return out, int(rng.integers(1, 1 << 40))


def _precision(case):
    return qsel.QSEL_MIXED if case["precision"] == "mixed" else qsel.QSEL_FP64


def _context(case, inp, **options):
    m = case["m"]
    return qsel.qsel_create(m * m, case["n_t"], *_mesh(m), inp["mask"], inp["sigma"], inp["theta"], **options)


def _network_params(rng, mean, scale):
    """Weights of a network in use: Glorot-uniform, small biases, standardised inputs."""
    def weight(fan_out, fan_in):
        a = math.sqrt(6.0 / (fan_in + fan_out))
        return rng.uniform(-a, a, fan_in * fan_out)
    return np.concatenate([weight(64, 14), rng.uniform(-0.1, 0.1, 64), weight(64, 64), rng.uniform(-0.1, 0.1, 64),
                           weight(1, 64), [-2.0], mean, scale]).astype(np.float32)


def _feature_rows(rows, seed):
    """Features as the library lays them out (logs of entries, distances, theta)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((rows, 14), generator=g, device="cuda")
    x[:, 0] = 1.5 + 0.7 * x[:, 0]
    x[:, 1:9] = (0.5 + x[:, 1:9]).sort(dim=1, descending=True).values
    x[:, 9:11] = torch.floor(x[:, 9:11].abs() * 4.0).clamp_(max=8.0)
    y = -3.0 - 0.3 * x[:, 9] + 0.2 * torch.randn(rows, generator=g, device="cuda")
    return x.contiguous(), y.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "backward":
        x, y = _feature_rows(case["rows"], seed)
        net = qsel.qsel_cv_create(seed)
        params = _network_params(np.random.default_rng([seed, 3]), x.mean(0).cpu().numpy(),
                                 x.std(0).clamp(min=1e-3).cpu().numpy())
        qsel.qsel_cv_set_params(net, params)
        return dict(kind=kind, net=net, x=x, y=y, params=params)
    if kind == "batch":
        models, key = _batch_inputs(case, seed)
        args = []
        for s in models:
            c, rowptr, col, val = _mesh(s["m"])
            args.append(dict(n_s=s["m"] ** 2, n_t=s["n_t"], c_diag=c, g_rowptr=rowptr, g_col=col, g_val=val,
                             obs_mask=s["mask"], sigma=s["sigma"]))
        b = qsel.qsel_create_batch(args, [s["theta"] for s in models], [(s["parts"], None) for s in models],
                                   [1] * len(models), n_samples=case["k"], seed=key, precision=_precision(case),
                                   pcg_tol=case["tol"], n_streams=8)
        out = [torch.empty(s["m"] ** 2 * s["n_t"], dtype=torch.float64, device="cuda") for s in models]
        return dict(kind=kind, batch=b, theta=[s["theta"] for s in models], out=out)
    inp = _inputs(case, seed)
    state = dict(kind=kind, theta=inp["theta"], seed=inp["seed"])
    n = case["m"] ** 2 * case["n_t"]
    if kind == "forward":
        state["ctx"] = _context(case, inp, n_parts=case["parts"], overlap=case["overlap"], n_samples=32,
                                precision=qsel.QSEL_MIXED)
        state["overlap"] = case["overlap"]
        state["features"] = torch.empty((n, qsel.QSEL_CV_FEATURES), dtype=torch.float32, device="cuda")
        state["y"] = torch.empty(n, dtype=torch.float32, device="cuda")
        rng = np.random.default_rng([seed, 3])
        net = qsel.qsel_cv_create(seed)
        qsel.qsel_cv_set_params(net, _network_params(rng, rng.normal(0.0, 1.0, 14), rng.uniform(1.0, 3.0, 14)))
        state["net"] = net
        return state
    state["out"] = torch.empty(n, dtype=torch.float64, device="cuda")
    if kind == "exact":
        state["ctx"] = _context(case, inp, n_parts=1, overlap=0, n_samples=2, precision=_precision(case))
        return state
    options = dict(n_parts=case["parts"], overlap=case["overlap"], n_samples=case["k"], seed=inp["seed"],
                   precision=_precision(case))
    if kind == "lanczos":
        options.update(sampler=qsel.QSEL_SAMPLER_LANCZOS, lanczos_steps=case["steps"],
                       model=qsel.QSEL_MODEL_DIFFUSION)
    else:
        options.update(pcg_tol=case["tol"], preconditioner=qsel.QSEL_PRECOND_KRON if case["precond"] == "kron"
                       else qsel.QSEL_PRECOND_BLOCK_JACOBI)
    state["ctx"] = _context(case, inp, **options)
    if kind == "hyper":
        qsel.qsel_set_data(state["ctx"], _data(inp))
    return state


def _data(inp):
    return np.random.default_rng([inp["seed"], 5]).normal(0.0, 1.0, int(inp["mask"].sum()))


def run(state):
    kind = state["kind"]
    if kind == "backward":
        grad, loss = qsel.qsel_cv_grad(state["net"], state["x"], state["y"], state["x"].shape[0])
        return {"grad": grad, "loss": np.float32(loss)}
    if kind == "batch":
        b = state["batch"]
        for i, theta in enumerate(state["theta"]):
            qsel.qsel_batch_set_theta(b, i, theta)
        qsel.qsel_batch_run(b)
        diag = [qsel.qsel_batch_diag_inv(b, i, out) for i, out in enumerate(state["out"])]
        return {"diag": diag, "traces": [qsel.qsel_batch_trace_grads(b, i) for i in range(len(diag))]}
    ctx = state["ctx"]
    qsel.qsel_set_theta(ctx, state["theta"])
    if kind == "forward":
        qsel.qsel_cv_features(ctx, state["overlap"], state["features"])
        qsel.qsel_cv_predict(state["net"], state["features"], state["y"], state["y"].numel())
        return {"features": state["features"], "y": state["y"]}
    if kind == "hyper":
        mean = qsel.qsel_posterior_mean(ctx, state["out"])
        grad, terms = qsel.qsel_loglik_grad(ctx, with_terms=True)
        return {"mean": mean, "grad": grad, "terms": list(terms)}
    if kind != "exact":
        qsel.qsel_set_seed(ctx, state["seed"])
    diag = qsel.qsel_diag_inv(ctx, state["out"])
    traces = qsel.qsel_trace_grads(ctx)
    if kind == "exact":
        return {"diag": diag, "traces": traces}
    parts, whole = qsel.qsel_error_estimate(ctx)
    return {"diag": diag, "traces": traces, "part_error": parts, "error": whole}


# --------------------------------------------------------------------------
# Work and the answer in 64 bits
# --------------------------------------------------------------------------
def _parts(n_t, count, overlap):
    """(own slabs, extended slabs) of the balanced partition."""
    base, extra = divmod(n_t, count)
    at, out = 0, []
    for p in range(count):
        end = at + base + (p < extra)
        out.append(((at, end), (max(0, at - overlap), min(n_t, end + overlap))))
        at = end
    return out


def _model_work(m, n_t, parts, overlap, k, precision):
    """Inverse of each pivot block, its two Takahashi products, the correction
    solves and one product with Q for the samples."""
    n_s = m * m
    slabs = sum(e1 - e0 for _, (e0, e1) in _parts(n_t, parts, overlap))
    flops = 4.0 * slabs * n_s ** 3
    size = 4 if precision == "mixed" else 8
    read = n_s * 13 * size + n_s * n_t
    if parts > 1:
        flops += 4.0 * slabs * n_s ** 2 * k + 2.0 * 39 * n_s * n_t * k
        read += n_s * n_t * k * size
    return read + 8.0 * n_s * n_t, flops


def work(case):
    kind = case["kind"]
    if kind == "backward":
        return {"bytes": 60.0 * case["rows"] + 4 * 5185, "flops": 3.0 * 10112 * case["rows"]}
    if kind == "forward":
        n = case["m"] ** 2 * case["n_t"]
        return {"bytes": 60.0 * n, "flops": 10112.0 * n}
    if kind == "batch":
        models, _ = _batch_inputs(case, 0)
        both = [_model_work(s["m"], s["n_t"], s["parts"], 1, case["k"], case["precision"]) for s in models]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    b, f = _model_work(case["m"], case["n_t"], case.get("parts", 1), case.get("overlap", 0), case.get("k", 0),
                       case["precision"])
    if kind == "lanczos":
        f += 2.0 * case["steps"] * 2 * 39 * case["m"] ** 2 * case["n_t"] * case["k"]
    return {"bytes": b, "flops": f}


class _Chain:
    """A block-tridiagonal Q in 64 bits: diagonal blocks, one coupling matrix
    with a scale per step, and dQ/dtheta_j in the same form."""

    def __init__(self, case, inp):
        m, n_t = case["m"], case["n_t"]
        n_s = m * m
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        c, rowptr, col, val = _mesh(m)
        self.n_s, self.n_t, self.dev = n_s, n_t, dev
        C = torch.diag(torch.tensor(c, device=dev))
        rows = np.repeat(np.arange(n_s), np.diff(rowptr))
        G = torch.zeros((n_s, n_s), dtype=torch.float64, device=dev)
        G[torch.tensor(rows, device=dev), torch.tensor(col, device=dev).long()] = torch.tensor(val, device=dev)
        self.obs = torch.tensor(inp["mask"], device=dev).double().reshape(n_t, n_s) / inp["sigma"] ** 2
        th = inp["theta"]
        if case["kind"] == "lanczos":
            gs, gt, ge = (math.exp(x) for x in th)
            K1 = gs ** 2 * C + G
            K2 = (K1 / C.diagonal()) @ K1
            K3 = (K2 / C.diagonal()) @ K1
            end = torch.zeros(n_t, dtype=torch.float64)
            end[0] = end[-1] = 1.0
            m0, m1, m2 = 1.0 - 0.5 * end, 0.5 * end, 2.0 - end
            powers, sets = [C, K1, K2, K3], [(m0, 3, 0), (2.0 * m1, 2, 1), (m2, 1, 2)]

            def diag(weight):
                return lambda t: sum(w * float(j[t]) * M for j, a, p in sets for w, M in [weight(a, p)])
            self.diag = diag(lambda a, p: (ge ** 2 * gt ** p, powers[a]))
            self.off, self.scale = K1, -(ge * gt) ** 2
            ds = diag(lambda a, p: (ge ** 2 * gt ** p * 2.0 * gs ** 2 * a, powers[a - 1]))
            dt = diag(lambda a, p: (ge ** 2 * p * gt ** p, powers[a]))
            self.deriv = [(ds, C, -(ge * gt) ** 2 * 2.0 * gs ** 2), (dt, K1, -2.0 * (ge * gt) ** 2),
                          (lambda t: 2.0 * self.diag(t), K1, -2.0 * (ge * gt) ** 2)]
        else:
            kappa, tau, rho = math.exp(th[0]), math.exp(th[1]), 1.0 / (1.0 + math.exp(-th[2]))
            self.kappa, self.tau, self.rho, self.c = kappa, tau, rho, C.diagonal()
            K = kappa ** 2 * C + G
            Qs = (K / C.diagonal()) @ K
            self.K = K

            def a(t, inner, end):
                return end if t in (0, n_t - 1) else inner
            r2 = 1.0 - rho ** 2
            d_inner = (2.0 * rho / r2 + (1.0 + rho ** 2) * 2.0 * rho / r2 ** 2) * rho * (1.0 - rho)
            d_end = 2.0 * rho / r2 ** 2 * rho * (1.0 - rho)
            d_off = (-1.0 / r2 - rho * 2.0 * rho / r2 ** 2) * rho * (1.0 - rho)
            self.diag = lambda t: tau * a(t, (1.0 + rho ** 2) / r2, 1.0 / r2) * Qs
            self.off, self.scale = Qs, -tau * rho / r2
            dK = 4.0 * kappa ** 2 * K
            self.deriv = [(lambda t: tau * a(t, (1.0 + rho ** 2) / r2, 1.0 / r2) * dK, dK, -tau * rho / r2),
                          (self.diag, Qs, self.scale), (lambda t: tau * a(t, d_inner, d_end) * Qs, Qs, tau * d_off)]
        self.off_sparse = self.off.to_sparse_csr()

    def block(self, t):
        return self.diag(t) + torch.diag(self.obs[t])

    def pivots(self, e0, e1):
        inv, schur = [], 0.0
        for t in range(e0, e1):
            inv.append(torch.cholesky_inverse(torch.linalg.cholesky(self.block(t) - schur)))
            if t + 1 < e1:
                schur = self.scale ** 2 * (self.off_sparse @ (self.off_sparse @ inv[-1]).T.contiguous())
        return inv

    def solve(self, inv, b):
        """Q x = b over the slabs of inv; b: slab -> rows, overwritten."""
        for t in range(1, len(inv)):
            b[t] = b[t] - self.scale * (self.off_sparse @ (inv[t - 1] @ b[t - 1]))
        b[-1] = inv[-1] @ b[-1]
        for t in range(len(inv) - 2, -1, -1):
            b[t] = inv[t] @ (b[t] - self.scale * (self.off_sparse @ b[t + 1]))
        return b

    def estimate(self, parts, X, k):
        """Diagonal, traces and error estimate of the overlapping estimator."""
        diag, err, traces = [], [], [0.0] * len(self.deriv)
        for (s0, s1), (e0, e1) in parts:
            inv = self.pivots(e0, e1)
            w = None
            if X is not None:
                b = [torch.zeros((self.n_s, k), dtype=torch.float64, device=self.dev) for _ in inv]
                if e0 > 0:
                    b[0] += self.scale * (self.off_sparse @ X[e0 - 1])
                if e1 < self.n_t:
                    b[-1] += self.scale * (self.off_sparse @ X[e1])
                w = self.solve(inv, b)
            sigma, below, rows = None, None, []
            for t in range(e1 - 1, max(e0, s0 - 1) - 1, -1):
                D = inv[t - e0]
                if sigma is None:
                    sigma = D
                else:
                    W = self.scale * (self.off_sparse @ D)
                    Y = sigma @ W
                    sigma, below = D + W.T @ Y, -Y
                u = t - e0
                for j, (dd, doff, dscale) in enumerate(self.deriv):
                    if s0 <= t < s1:
                        S = sigma if w is None else sigma + w[u] @ w[u].T / k
                        traces[j] += float((S * dd(t)).sum())
                    share = (s0 <= t < s1) + (s0 <= t + 1 < s1)
                    if below is not None and share and t + 1 < e1:
                        S = below if w is None else below + w[u + 1] @ w[u].T / k
                        traces[j] += share * dscale * float((S * doff).sum())
                if s0 <= t < s1:
                    v = sigma.diagonal().clone()
                    if w is not None:
                        m2, m4 = w[u].square().mean(1), w[u].square().square().mean(1)
                        v = v + m2
                        rows.append((m4 - m2 * m2).clamp(min=0.0) / (k - 1) / v.square())
                    diag.append((t, v))
            err.append(torch.cat(rows) if rows else torch.zeros(self.n_s * (s1 - s0), dtype=torch.float64, device=self.dev))
        diag = torch.cat([v for _, v in sorted(diag, key=lambda x: x[0])])
        parts_err = np.array([math.sqrt(float(e.mean())) for e in err])
        return diag, np.array(traces), parts_err, math.sqrt(float(torch.cat(err).mean()))


def _normals(seed, stream, rows, k, dev):
    """Philox4x32-10 normals: counter (row, column pair, stream, 0), key = seed."""
    low = 0xFFFFFFFF
    pairs = (k + 1) // 2
    c = [torch.arange(rows, device=dev).repeat_interleave(pairs), torch.arange(pairs, device=dev).repeat(rows)]
    c += [torch.full_like(c[0], stream), torch.zeros_like(c[0])]
    k0, k1 = seed & low, seed >> 32 & low
    for _ in range(10):
        p, q = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [(q >> 32 & low) ^ c[1] ^ k0, q & low, (p >> 32 & low) ^ c[3] ^ k1, p & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    u1 = ((c[0] << 21 | c[1] >> 11).double() + 1.0) * 2.0 ** -53
    u2 = (c[2] << 21 | c[3] >> 11).double() * 2.0 ** -53
    r = torch.sqrt(-2.0 * torch.log(u1))
    z = torch.stack([r * torch.cos(2.0 * math.pi * u2), r * torch.sin(2.0 * math.pi * u2)], 1)
    return z.reshape(rows, 2 * pairs)[:, :k]


def _exact_samples(chain, inp, k):
    """x = Q^-1 (F^T z1 + A^T z2 / sigma) by a block solve."""
    n_s, n_t = chain.n_s, chain.n_t
    z1 = _normals(inp["seed"], 0, n_s * n_t, k, chain.dev).reshape(n_t, n_s, k)
    observed = torch.tensor(np.flatnonzero(inp["mask"]), device=chain.dev)
    rho = chain.rho
    M = (chain.K / chain.c.sqrt()).to_sparse_csr()
    b = []
    for t in range(n_t):
        z = z1[t] * (math.sqrt(1.0 - rho ** 2) if t == 0 else 1.0)
        if t + 1 < n_t:
            z = z - rho * z1[t + 1]
        b.append(math.sqrt(chain.tau / (1.0 - rho ** 2)) * (M @ z.contiguous()))
    b = torch.cat(b)
    b[observed] += _normals(inp["seed"], 1, len(observed), k, chain.dev) / inp["sigma"]
    inv = chain.pivots(0, n_t)
    return chain.solve(inv, list(b.reshape(n_t, n_s, k))), inv


def _krylov_samples(chain, inp, k, steps):
    """Columns L^-T V f(T) |z| e1 of the preconditioned Lanczos process."""
    n = chain.n_s * chain.n_t
    Q = torch.zeros((n, n), dtype=torch.float64, device=chain.dev)
    for t in range(chain.n_t):
        a, b = t * chain.n_s, (t + 1) * chain.n_s
        Q[a:b, a:b] = chain.block(t)
        if t:
            Q[a:b, a - chain.n_s:a] = chain.scale * chain.off
            Q[a - chain.n_s:a, a:b] = chain.scale * chain.off.T
    Linv = torch.zeros_like(Q)
    for a in range(0, n, 64):
        b = min(n, a + 64)
        L = torch.linalg.cholesky(Q[a:b, a:b])
        Linv[a:b, a:b] = torch.linalg.solve_triangular(L, torch.eye(b - a, dtype=L.dtype, device=chain.dev), upper=False)
    Q, Linv = Q.to_sparse_csr(), Linv.to_sparse_csr()
    LinvT = Linv.to_dense().T.contiguous().to_sparse_csr()
    z = _normals(inp["seed"], 0, n, k, chain.dev).contiguous()
    eta = z.norm(dim=0)
    V, alpha, beta = [z / eta], [], []
    for j in range(steps):
        w = Linv @ (Q @ (LinvT @ V[j]))
        if j:
            w = w - beta[-1] * V[j - 1]
        alpha.append((V[j] * w).sum(0))
        w = w - alpha[-1] * V[j]
        beta.append(w.norm(dim=0))
        V.append(w / beta[-1])
    T = torch.diag_embed(torch.stack(alpha, 1))
    side = torch.diag_embed(torch.stack(beta[:-1], 1), offset=1) if steps > 1 else 0.0 * T
    lam, U = torch.linalg.eigh(T + side + (side.transpose(1, 2) if steps > 1 else 0.0))
    f = torch.einsum("sij,sj->si", U, lam.rsqrt() * U[:, 0, :]) * eta[:, None]
    x = LinvT @ sum(V[j] * f[:, j] for j in range(steps))
    return list(x.reshape(chain.n_t, chain.n_s, k))


def _features(chain, case, inp):
    """Logs of the diagonal and the eight largest entries of every row of Q, distances, theta."""
    n_s, n_t, m = chain.n_s, chain.n_t, case["m"]
    i, j = np.divmod(np.arange(n_s), m)
    edge = np.minimum(np.minimum(np.minimum(i, m - 1 - i), np.minimum(j, m - 1 - j)), 8)
    sep = np.zeros(n_t)
    for (s0, s1), (e0, e1) in _parts(n_t, case["parts"], case["overlap"]):
        for t in range(s0, s1):
            sep[t] = min([16.0] + ([t - e0 + 1] if e0 > 0 else []) + ([e1 - t] if e1 < n_t else []))
    out = torch.empty((n_t, n_s, 14), dtype=torch.float64, device=chain.dev)
    for t in range(n_t):
        near = []
        A = chain.diag(t)
        a = A - torch.diag(A.diagonal())
        near.append(torch.topk(a.abs(), min(8, n_s), dim=1).values)
        near += [torch.topk((chain.scale * chain.off).abs(), min(8, n_s), dim=1).values] * ((t > 0) + (t + 1 < n_t))
        top = torch.topk(torch.cat(near, 1), 8, dim=1).values
        out[t, :, 0] = torch.log(A.diagonal() + chain.obs[t])
        out[t, :, 1:9] = torch.log(torch.clamp(top, min=1e-30))
        out[t, :, 9] = float(sep[t])
        out[t, :, 10] = torch.tensor(edge, device=chain.dev).double()
        out[t, :, 11:] = torch.tensor(inp["theta"], dtype=torch.float64, device=chain.dev)
    return out.reshape(n_t * n_s, 14)


def _network(params, x):
    """The network in 64 bits on its BF16 weights: (output, cache for the gradient)."""
    p = torch.tensor(params, device=x.device)
    r = lambda a, *shape: a.bfloat16().double().reshape(*shape)  # noqa: E731
    W1, W2, W3 = r(p[:896], 64, 14), r(p[960:5056], 64, 64), r(p[5120:5184], 64)
    b1, b2, b3, mean, scale = (p[a:b].double() for a, b in ((896, 960), (5056, 5120), (5184, 5185), (5185, 5199), (5199, 5213)))
    xn = (x.double() - mean) / scale
    a1 = xn @ W1.T + b1
    h1 = torch.nn.functional.gelu(a1)
    a2 = h1 @ W2.T + b2
    h2 = torch.nn.functional.gelu(a2)
    return h2 @ W3 + b3, (xn, a1, h1, a2, h2, W2, W3)


def _gelu_slope(a):
    return 0.5 * (1.0 + torch.erf(a / math.sqrt(2.0))) + a * torch.exp(-0.5 * a * a) / math.sqrt(2.0 * math.pi)


def _exact_backward(case, seed):
    x, target = _feature_rows(case["rows"], seed)
    params = _network_params(np.random.default_rng([seed, 3]), x.mean(0).cpu().numpy(),
                             x.std(0).clamp(min=1e-3).cpu().numpy())
    y, (xn, a1, h1, a2, h2, W2, W3) = _network(params, x)
    n = case["rows"]
    dy = 2.0 * (y - target.double()) / n
    d2 = dy[:, None] * W3 * _gelu_slope(a2)
    d1 = (d2 @ W2) * _gelu_slope(a1)
    grad = torch.cat([(d1.T @ xn).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), dy @ h2, dy.sum()[None]])
    return {"grad": grad, "loss": float((y - target.double()).square().mean())}


def exact(case, seed):
    kind = case["kind"]
    if kind == "backward":
        return _exact_backward(case, seed)
    if kind == "batch":
        models, key = _batch_inputs(case, seed)
        got = []
        for i, s in enumerate(models):
            inp = dict(s, seed=key + i)
            chain = _Chain(dict(kind="rbmc", m=s["m"], n_t=s["n_t"]), inp)
            X, _ = _exact_samples(chain, inp, case["k"])
            got.append(chain.estimate(_parts(s["n_t"], s["parts"], 1), X, case["k"]))
        return {"diag": [g[0] for g in got], "traces": [g[1] for g in got]}
    if kind != "forward" and (case["m"] ** 2) ** 3 * case["n_t"] > 2.5e12:
        return None
    inp = _inputs(case, seed)
    chain = _Chain(case, inp)
    if kind == "forward":
        rng = np.random.default_rng([seed, 3])
        x = _features(chain, case, inp)
        params = _network_params(rng, rng.normal(0.0, 1.0, 14), rng.uniform(1.0, 3.0, 14))
        return {"features": x, "y": _network(params, x)[0]}
    if kind == "exact":
        diag, traces, _, _ = chain.estimate(_parts(case["n_t"], 1, 0), None, 0)
        return {"diag": diag, "traces": traces}
    k, parts = case["k"], _parts(case["n_t"], case["parts"], case["overlap"])
    if kind == "lanczos":
        X = _krylov_samples(chain, inp, k, case["steps"])
    else:
        X, inv = _exact_samples(chain, inp, k)
    diag, traces, part_error, error = chain.estimate(parts, X, k)
    if kind != "hyper":
        return {"diag": diag, "traces": traces, "part_error": part_error, "error": error}
    b = torch.zeros(chain.n_s * chain.n_t, dtype=torch.float64, device=chain.dev)
    b[torch.tensor(np.flatnonzero(inp["mask"]), device=chain.dev)] = torch.tensor(_data(inp), device=chain.dev) / inp["sigma"] ** 2
    mu = chain.solve(inv, list(b.reshape(chain.n_t, chain.n_s, 1)))
    rho, n_t = chain.rho, chain.n_t
    prior = np.array([4.0 * n_t * chain.kappa ** 2 * float((torch.linalg.inv(chain.K).diagonal() * chain.c).sum()),
                      float(chain.n_s * n_t), chain.n_s * 2.0 * rho ** 2 * (n_t - 1) / (1.0 + rho)])
    quad = np.zeros(3)
    for j, (dd, doff, dscale) in enumerate(chain.deriv):
        quad[j] = sum(float((mu[t].T @ dd(t) @ mu[t]).sum()) for t in range(n_t))
        quad[j] += 2.0 * dscale * sum(float((mu[t + 1].T @ doff @ mu[t]).sum()) for t in range(n_t - 1))
    return {"mean": torch.cat(mu).reshape(-1), "grad": 0.5 * (prior - traces - quad), "terms": [prior, traces, quad]}
