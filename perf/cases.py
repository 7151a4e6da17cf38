"""The calls this library is used for, as measurable cases: posterior means, residual
recomputes (plain and compensated), gradient quadratic forms, solves in both precisions,
a training step and a one-shot solve of host data.

Every case is one call (a training step: two) of the public Python binding on synthetic
inputs of the same recipes as `workloads/`, drawn on the GPU from the seed.  `exact`
computes the same results in 64 bits with plain torch: dense kernel rows in chunks,
LAPACK-style Cholesky solves, Alg. 1 step by step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2310_17137_gb300 as ap

RBF, M32, M52 = ap.AP_RBF, ap.AP_MATERN32, ap.AP_MATERN52

# Every case names what it calls (`do`), the kernel family, n training points of
# dimension d, and the noise; solves add the block size, the right-hand sides c, the
# precision and the epochs that the run is capped at.  Single products take lengthscales
# from [0.3, 3]; solves take them from [0.1, 0.3] sqrt(d / 3), shrunk with the spacing of
# the points as n grows: a few dozen steps in float32 then give the iterates of Alg. 1 to
# about 1e-6 (smoother kernels amplify every rounding of a step by the conditioning).
_BASE = dict(outputscale=1.0, noise=0.1, block=4096, c=1, precision=ap.AP_FP32, epochs=1, refine_every=4,
             tol=1e-3, points=0, uniform=True)


def _case(name, do, kernel, n, d, **kw):
    return dict(_BASE, name=name, do=do, kernel=kernel, n=n, d=d, **kw)


def listed():
    return [
        # one prediction of an interactive program: a few test points against a small model
        _case("mean_tiny", "mean", M52, 1024, 3, points=16, block=512),
        # a serving request's posterior mean: 1024 test points, a ragged training set
        _case("mean_serving", "mean", RBF, 100003, 11, points=1024, block=1000),
        # checking one solution's residual on an odd-sized set (label column only)
        _case("residual_ragged", "residual", M32, 20600, 8, block=2048),
        # the refinement / certification pass of a 16-column solve
        _case("residual_c16", "residual", M52, 131072, 3, c=16, noise=0.01, uniform=False, block=1000),
        # the same pass at tolerances that need the compensated sums
        _case("residual_compensated", "residual", RBF, 16384, 8, tol=1e-6, block=512),
        # the backward pass of hyperparameter training: 31 probes and the labels
        _case("quadforms_c32", "quadforms", M32, 131072, 8, c=32, block=1000),
        # a small model's solve: 4 epochs of 8 short steps, where launches and latency count
        _case("solve_small", "solve", RBF, 4096, 8, block=512, epochs=4),
        # the default (FP32) solve with probes, one epoch
        _case("solve_fp32_c32", "solve", M32, 65536, 8, c=32, uniform=False),
        # the low-precision solve at full size, one epoch (as between two refinements)
        _case("solve_tc_c16", "solve", M52, 262144, 3, c=16, noise=1.0, precision=ap.AP_BF16_REFINE, steps=64),
        # the low-precision solve on higher-dimensional data: four epochs and their refinement
        _case("solve_tc_d11", "solve", RBF, 131072, 11, c=16, noise=0.5, block=8192, precision=ap.AP_BF16_REFINE,
              epochs=4),
        # one step of hyperparameter training: new hyperparameters, factor, solve, gradient
        _case("train_step", "train", M32, 20000, 8, c=16, tol=1.0),
        # a whole call on host data: copies, factor, solve
        _case("solve_host", "host", M52, 50000, 5, epochs=4, uniform=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["mean", "mean", "residual", "residual", "quadforms", "solve", "solve", "solve_tc", "train", "host"])
    kernel = rng.choice([RBF, M32, M52])
    d = rng.randint(3, 20)
    noise = round(math.exp(rng.uniform(math.log(0.05), math.log(0.2))), 4)
    kw = dict(noise=noise, outputscale=round(rng.uniform(0.5, 2.0), 3), uniform=rng.random() < 0.7)
    if do == "mean":
        n = _log_int(rng, 1024, 262144)
        return _unnamed("mean", kernel, n, d, points=_log_int(rng, 1, 4096), block=min(n, 1000), **kw)
    if do == "residual":
        n = _log_int(rng, 1024, 65536)
        tol = 1e-6 if n <= 16384 and rng.random() < 0.3 else 1e-3
        return _unnamed("residual", kernel, n, d, c=rng.choice([1, 1, 3, 8, 16, 32]), tol=tol, block=min(n, 1000), **kw)
    if do == "quadforms":
        n = _log_int(rng, 1024, 65536)
        return _unnamed("quadforms", kernel, n, d, c=rng.choice([1, 4, 16, 32]), block=min(n, 1000), **kw)
    block = _log_int(rng, 256, 4096)
    if do == "solve":
        n = min(_log_int(rng, 1024, 65536), 24 * block)
        return _unnamed("solve", kernel, n, d, c=rng.choice([1, 1, 4, 16, 32]), block=block, **kw)
    if do == "solve_tc":
        n = min(_log_int(rng, 8192, 131072), 24 * block)
        kw.update(noise=round(rng.uniform(0.4, 1.0), 4), uniform=True)
        return _unnamed("solve", kernel, n, d, c=rng.choice([1, 16, 32]), block=block, precision=ap.AP_BF16_REFINE, **kw)
    n = min(_log_int(rng, 2048, 30000), 8 * block)
    if do == "train":
        return _unnamed("train", kernel, n, d, c=rng.choice([8, 16, 32]), block=block, tol=1.0, **kw)
    return _unnamed("host", kernel, n, d, block=block, epochs=rng.randint(1, 3), **kw)


def _unnamed(do, kernel, n, d, **kw):
    case = _case("", do, kernel, n, d, **kw)
    del case["name"]
    return case


def _inputs(case, seed):
    """Inputs on the GPU, float32, from the seed alone: X (n x d), lengthscales, right-hand
    sides [y, probes] (n x c), test points, and vectors that stand for solutions."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    n, d, c = case["n"], case["d"], case["c"]

    def points(m):
        if case["uniform"]:
            return torch.rand(m, d, generator=g, device="cuda")
        return torch.randn(m, d, generator=g, device="cuda")

    r = {"X": points(n)}
    u = torch.rand(d, generator=g, device="cuda").cpu()
    if case["do"] in ("mean", "residual", "quadforms"):
        lo, hi, f = 0.3, 3.0, 1.0
    else:
        lo, hi, f = 0.1, 0.3, math.sqrt(d / 3) * min(1.0, 2048 / n) ** (1 / d)
    r["ell"] = (f * torch.exp(math.log(lo) + u * math.log(hi / lo))).numpy().astype(np.float32)
    y = torch.sin(2 * math.pi * r["X"]).sum(1) + 0.1 * torch.randn(n, generator=g, device="cuda")
    y = (y - y.mean()) / y.std()
    Z = torch.randint(0, 2, (n, max(c - 1, 0)), generator=g, device="cuda").float() * 2 - 1
    r["B"] = torch.cat([y[:, None], Z], 1).contiguous()
    if case["do"] == "mean":
        r["Xt"] = points(case["points"])
    if case["do"] in ("mean", "residual", "quadforms"):
        # K_hat^{-1} B of these smooth kernels is (B less its smooth part) / noise
        r["W"] = (r["B"] + 0.1 * torch.randn(n, c, generator=g, device="cuda")) / (case["noise"] + 0.1)
    return r


def _hyper(case, r):
    return ap.Hyper(case["kernel"], r["ell"], case["outputscale"], case["noise"], 0.0)


def _opts(case):
    kw = dict(block=case["block"], tol=case["tol"], precision=case["precision"], refine_every=case["refine_every"])
    if case["do"] == "train":  # the defaults of training: mean rule, at least 11 epochs
        return ap.ap_opts_default(max_epochs=22, **kw)
    return ap.ap_opts_default(stop=ap.AP_STOP_MAX_REL, min_epochs=1, max_epochs=case["epochs"],
                              max_steps=case.get("steps", 0), **kw)


def _alpha(c):
    return np.array([-0.5] + [0.5 / (c - 1)] * (c - 1)) if c > 1 else np.array([-0.5])


def prepare(case, seed):
    r = _inputs(case, seed)
    s = {"case": case, "hyper": _hyper(case, r), "opts": _opts(case)}
    if case["do"] == "host":
        s["X"] = r["X"].cpu().pin_memory().numpy()
        s["B"] = r["B"].cpu().pin_memory().numpy()
        s["W"] = torch.empty(r["B"].shape).pin_memory().numpy()
        return s
    s["ctx"] = ap.ap_create(r["X"], s["hyper"], s["opts"])
    if case["do"] == "mean":
        s["w"], s["Xt"] = r["W"][:, 0].contiguous(), r["Xt"]
    elif case["do"] == "quadforms":
        s["U"], s["V"], s["alpha"] = r["W"], torch.cat([r["W"][:, :1], r["B"][:, 1:]], 1).contiguous(), _alpha(case["c"])
    elif case["do"] == "train":
        s["y"], s["Z"] = r["B"][:, 0].contiguous(), r["B"][:, 1:].contiguous()
    else:
        s["B"], s["W"] = r["B"], r.get("W")
    return s


def run(s):
    case = s["case"]
    do = case["do"]
    if do == "mean":
        return ap.ap_predict_mean(s["ctx"], s["w"], s["Xt"])
    if do == "residual":
        return ap.ap_residual(s["ctx"], s["B"], s["W"])
    if do == "quadforms":
        # the gradient of float32 hyperparameters
        return ap.ap_grad_quadforms(s["ctx"], s["U"], s["V"], s["alpha"]).astype(np.float32)
    if do == "solve":
        return ap.ap_solve(s["ctx"], s["B"])[1]
    if do == "train":
        ap.ap_set_hyper(s["ctx"], s["hyper"])
        return ap.ap_mll_grad(s["ctx"], s["y"], case["c"] - 1, s["Z"])[1]
    return ap.ap_solve_host(s["X"], s["B"], s["hyper"], s["opts"], s["W"])[1]


def _entry_flops(case):
    """Flops of one kernel entry: the squared distance (3 d) and phi (RBF 1, Matern 5)."""
    return 3 * case["d"] + (1 if case["kernel"] == RBF else 5)


def work(case):
    n, d, c, b = case["n"], case["d"], case["c"], min(case["block"], case["n"])
    m = -(-n // b)
    e = _entry_flops(case)
    do = case["do"]
    if do == "mean":
        M = case["points"]
        return {"bytes": 4 * (n * d + n + M * d + M), "flops": M * n * (e + 2)}
    if do == "residual":
        return {"bytes": 4 * (n * d + 3 * n * c), "flops": n * n * (e + 2 * c)}
    # a gradient entry: U_i . V_j, phi and psi, d + 1 weighted sums
    quad = n * n * (e + 2 * c + 2 * d + 3)
    if do == "quadforms":
        return {"bytes": 4 * (n * d + 2 * n * c) + 8 * (d + 2), "flops": quad}
    epochs = 11 if do == "train" else case["epochs"]
    steps = case.get("steps", 0) or epochs * m
    step_flops = n * b * (e + 2 * c) + 2 * b * b * c
    # a step reads the block's triangular factor (FP32), X and R, and writes R
    step_bytes = 4 * (b * b // 2 + n * d + 2 * n * c)
    flops, nbytes = steps * step_flops, steps * step_bytes
    if case["precision"] == ap.AP_BF16_REFINE and not case.get("steps", 0):
        flops += n * n * (e + 2 * c)
        nbytes += 4 * (n * d + 3 * n * c)
    if do in ("train", "host"):
        flops += m * (b ** 3 * 2 // 3 + b * b * e // 2)
        nbytes += 4 * m * b * b // 2
    if do == "train":
        flops += quad
        nbytes += 4 * (n * d + 2 * n * c)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------- 64-bit results
class _Exact:
    """Kernel rows in float64: phi of the squared ARD distance, by coordinate differences."""

    def __init__(self, case, r):
        self.case = case
        self.ell = torch.from_numpy(r["ell"].astype(np.float64)).cuda()
        self.X = r["X"].double()
        self.s = float(np.float32(case["outputscale"]))
        self.noise = float(np.float32(case["noise"]))

    def r2(self, A, B):
        A, B = A / self.ell, B / self.ell
        t = torch.zeros(A.shape[0], B.shape[0], dtype=torch.float64, device="cuda")
        for k in range(A.shape[1]):
            df = A[:, k, None] - B[None, :, k]
            t.addcmul_(df, df)
        return t

    def phi(self, t):
        k = self.case["kernel"]
        if k == RBF:
            return t.mul_(-0.5).exp_()
        u = t.mul_(3.0 if k == M32 else 5.0).sqrt_()
        p = u + 1.0 if k == M32 else (u / 3.0 + 1.0).mul_(u).add_(1.0)
        return p.mul_(u.neg_().exp_())

    def k(self, A, B):
        return self.phi(self.r2(A, B)).mul_(self.s)

    def times(self, A, W, diag=False):
        """K(A, X) W (+ noise W when A is X), rows in chunks."""
        out = torch.empty(A.shape[0], W.shape[1], dtype=torch.float64, device="cuda")
        step = max(1, (1 << 29) // self.X.shape[0])
        for i in range(0, A.shape[0], step):
            out[i:i + step] = self.k(A[i:i + step], self.X) @ W
        return out + self.noise * W if diag else out

    def solve(self, B):
        """Alg. 1 with the Gauss-Southwell rule, as many steps as the call takes."""
        case = self.case
        n, b = case["n"], min(case["block"], case["n"])
        m = -(-n // b)
        train = case["do"] == "train"
        W, R, chol = torch.zeros_like(B), B.clone(), {}
        bn = B.square().sum(0)
        epochs = 22 if train else case["epochs"]
        steps = case.get("steps", 0) or epochs * m
        for j in range(steps):
            norms = torch.stack([R[J * b:(J + 1) * b].square().sum() for J in range(m)])
            J = int(torch.argmax(norms))
            lo, hi = J * b, min((J + 1) * b, n)
            if J not in chol:
                K = self.k(self.X[lo:hi], self.X[lo:hi])
                K.diagonal().add_(self.noise)
                chol[J] = torch.linalg.cholesky(K)
            delta = torch.cholesky_solve(R[lo:hi], chol[J])
            W[lo:hi] += delta
            step = max(1, (1 << 29) // b)
            for i in range(0, n, step):
                R[i:i + step] -= self.k(self.X[i:i + step], self.X[lo:hi]) @ delta
            R[lo:hi] -= self.noise * delta
            if (j + 1) % m == 0:
                rel = (R.square().sum(0) / bn).sqrt()
                if train and (j + 1) // m >= 11 and float(rel.mean()) < case["tol"]:
                    break
                if not train and float(rel.max()) <= case["tol"]:
                    break
        return W

    def quadforms(self, U, V, alpha):
        """sum_c alpha_c U_c^T (dK_hat / dtheta) V_c for theta = (l_1.., s, noise)."""
        case = self.case
        n, d, k = case["n"], case["d"], case["kernel"]
        a = torch.from_numpy(np.asarray(alpha, np.float64)).cuda()
        out = torch.zeros(d + 2, dtype=torch.float64, device="cuda")
        Ua = U * a
        step = max(1, (1 << 29) // n)
        for i in range(0, n, step):
            A = self.X[i:i + step]
            G = Ua[i:i + step] @ V.T
            t = self.r2(A, self.X)
            out[d] += (G * self.phi(t.clone())).sum()
            # dK/dl_k = s psi (x_k - x'_k)^2 / l_k^3 with psi = phi, 3 e^-u, 5/3 (1 + u) e^-u
            if k == RBF:
                psi = t.mul_(-0.5).exp_()
            else:
                u = t.mul_(3.0 if k == M32 else 5.0).sqrt_()
                psi = torch.exp(-u).mul_(3.0) if k == M32 else torch.exp(-u).mul_(u.add_(1.0)).mul_(5.0 / 3.0)
            G *= psi
            for q in range(d):
                df = A[:, q, None] - self.X[None, :, q]
                out[q] += (G * df.square_()).sum() * self.s / self.ell[q] ** 3
        out[d + 1] = (Ua * V).sum()
        return out


def exact(case, seed):
    r = _inputs(case, seed)
    E = _Exact(case, r)
    B = r["B"].double()
    do = case["do"]
    if do == "mean":
        return E.times(r["Xt"].double(), r["W"][:, :1].double())[:, 0]
    if do == "residual":
        return B - E.times(E.X, r["W"].double(), diag=True)
    if do == "quadforms":
        W = r["W"].double()
        return E.quadforms(W, torch.cat([W[:, :1], B[:, 1:]], 1), _alpha(case["c"])).cpu().numpy()
    W = E.solve(B)
    if do != "train":
        return W if do == "solve" else W.cpu().numpy()
    g = E.quadforms(W, torch.cat([W[:, :1], B[:, 1:]], 1), _alpha(case["c"]))
    return torch.cat([g, -W[:, :1].sum(0)]).cpu().numpy()
