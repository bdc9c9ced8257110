"""Performance cases: the work a program gives this library, through its public entry points.

A case names a kind of call and its sizes.  Kinds:

* solve      Problem.solve to 1e-8 max|F| from a zero iterate (FP64 or a mixed form, 1D or 2D, the
             coarse correction recursing to one point or solved exactly on a `direct`-point level)
* batched    solve_batched over 1D instances of their own orders, meshes and sizes
* smooth     one red-black smoothing sweep in FP64 (Problem.smooth)
* residual   the FP64-accurate defect of an iterate, which decides a solve (Problem.residual)
* line       line solves on compact FP32 columns, the mixed forms' inner smoother (Problem.line_solve_s)
* product    the H-matrix product on compact FP64 columns with FP32 arithmetic (Problem.hmatvec_f32)
* predict    the learned warm start (WSNet.predict, BF16 inference)
* train      loss and parameter gradients of the warm-start network (WSNet.loss_grad)

Sources are constant in time: eight sine modes in 1D, a Gaussian random field drawn as a sine series
in 2D.  Sizes are those of the benchmark's and the tests' workloads: N from 63 to 4095 points per
dimension, M from 64 to 4096 time levels, alpha in [0.2, 0.9], gamma in [1, 3].
"""
import math

import numpy as np
import torch

import paper_1706_07632_gb300 as fh

DEV = "cuda"
LEAF, TOL, RTOL, MAX_CYCLES = 64, 1e-10, 1e-8, 60
PREC = {"fp64": fh.FP64, "fp32": fh.MIXED_FP32, "bf16": fh.MIXED_BF16}


def listed():
    return [
        # a small FP64 solve (the size of a 1D convergence table): launches and latency count
        dict(name="solve_1d_small", kind="solve", dim=1, N=255, M=256, alpha=0.5, gamma=2.0, prec="fp64", direct=0),
        # the long 1D workload of the benchmark: fine grid, long time axis, mixed precision
        dict(name="solve_1d_long", kind="solve", dim=1, N=4095, M=4096, alpha=0.5, gamma=2.0, prec="fp32", direct=255),
        # the benchmark's headline grid, from zero, BF16 products
        dict(name="solve_2d_large", kind="solve", dim=2, N=1023, M=512, alpha=0.55, gamma=2.0, prec="bf16", direct=31),
        # an ordinary 2D grid on a longer time axis with FP32 products, the plain recursion
        dict(name="solve_2d_fp32", kind="solve", dim=2, N=255, M=1024, alpha=0.4, gamma=2.0, prec="fp32", direct=0),
        # many moderate 1D problems at once (a parameter study)
        dict(name="batched_1d", kind="batched", count=16, pick=7, Nmax=1023, Mmax=1024, prec="fp32"),
        # one FP64 smoothing step in 2D
        dict(name="smooth_2d_fp64", kind="smooth", dim=2, N=127, M=256, alpha=0.5, gamma=2.0),
        # the defect of a mixed 2D solve, an ordinary grid
        dict(name="residual_2d", kind="residual", dim=2, N=511, M=512, alpha=0.55, gamma=2.0, prec="bf16"),
        # the defect of a mixed 1D solve on a long time axis
        dict(name="residual_1d", kind="residual", dim=1, N=4095, M=2048, alpha=0.6, gamma=1.5, prec="fp32"),
        # the inner smoother's line solves, a ragged panel
        dict(name="line_s_wide", kind="line", cols=100003, M=512, alpha=0.55, gamma=2.0, prec="bf16"),
        # FP32 products on a narrow panel, odd width, long time axis
        dict(name="product_narrow", kind="product", cols=1001, M=2048, alpha=0.5, gamma=2.0),
        # the warm start of a 2D solve
        dict(name="predict_2d", kind="predict", N=511, M=512, alpha=0.55, gamma=2.0, K=24),
        # one gradient of the warm-start network at the batch and width it is trained with
        dict(name="train_grad", kind="train", batch=4096, hidden=320, layers=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "residual", "residual", "line", "line", "product", "predict", "train", "train",
                       "smooth", "batched"])
    order = dict(alpha=round(rng.uniform(0.2, 0.9), 3), gamma=round(rng.uniform(1.0, 3.0), 2))
    if kind == "train":
        return dict(kind=kind, batch=_log_int(rng, 257, 16384), hidden=rng.choice([64, 128, 200, 256, 320, 512]),
                    layers=rng.choice([2, 3, 4]))
    if kind == "predict":
        return dict(kind=kind, N=rng.choice([127, 255, 511]), M=rng.choice([128, 256, 512, 1024]),
                    K=rng.randint(9, 32), **order)
    if kind == "batched":
        return dict(kind=kind, count=rng.randint(3, 24), pick=rng.randint(1, 1 << 20), Nmax=rng.choice([255, 1023]),
                    Mmax=rng.choice([256, 512, 1024]), prec=rng.choice(["fp64", "fp32"]))
    if kind == "line":
        return dict(kind=kind, cols=_log_int(rng, 501, 250000), M=rng.choice([128, 256, 512, 1024]),
                    prec=rng.choice(["fp32", "bf16", "bf16"]), **order)
    if kind == "product":
        return dict(kind=kind, cols=_log_int(rng, 101, 20000), M=rng.choice([256, 512, 1024, 2048, 4096]), **order)
    dim = rng.choice([1, 2])
    if kind == "smooth":
        N, M = (rng.choice([255, 1023, 4095]), rng.choice([256, 512, 1024])) if dim == 1 else \
               (rng.choice([63, 127]), rng.choice([64, 128, 256]))
        return dict(kind=kind, dim=dim, N=N, M=M, **order)
    if kind == "residual":
        N, M = (rng.choice([511, 1023, 2047, 4095]), rng.choice([256, 512, 1024, 2048])) if dim == 1 else \
               (rng.choice([127, 255, 511]), rng.choice([128, 256, 512]))
        return dict(kind=kind, dim=dim, N=N, M=M, prec=rng.choice(["fp64", "fp32", "bf16"]) if dim == 1 else
                    rng.choice(["fp32", "bf16"]), **order)
    prec = rng.choice(["fp64", "fp32", "bf16"])
    if dim == 1:
        N, M = rng.choice([127, 255, 511, 1023]), rng.choice([128, 256, 512, 1024])
        return dict(kind=kind, dim=1, N=N, M=M, prec=prec, direct=rng.choice([0, 63]), **order)
    N, M = rng.choice([63, 127, 255] if prec == "fp64" else [127, 255, 511]), rng.choice([64, 128, 256, 512])
    return dict(kind=kind, dim=2, N=N, M=min(M, 128) if prec == "fp64" else M, prec=prec, direct=rng.choice([0, 31]), **order)


# ---------------------------------------------------------------- inputs


def _coeffs(dim, N, seed):
    """Sine coefficients of a source: (8,) in 1D, (k, k) in 2D (length scale 0.1)."""
    rng = np.random.default_rng(seed)
    if dim == 1:
        return rng.standard_normal(8) / np.arange(1, 9) ** 2
    p = np.arange(1, min(N, 22) + 1)
    return rng.standard_normal((len(p), len(p))) * np.exp(-(0.1 * math.pi) ** 2 * (p[:, None] ** 2 + p[None] ** 2) / 4)


def _sines(N, k):
    return torch.as_tensor(np.sin(math.pi * np.outer(np.arange(1, k + 1), np.arange(1, N + 1)) / (N + 1)), device=DEV)


def _space(c, N):
    """The grid function of a coefficient array, (N,) or (N, N)."""
    S = _sines(N, c.shape[0])
    c = torch.as_tensor(c, device=DEV)
    return c @ S if c.dim() == 1 else S.T @ c @ S


def _times(M, gamma):
    return (torch.arange(1, M + 1, dtype=torch.float64, device=DEV) / M) ** gamma


def _source(dim, N, M, seed):
    s = _space(_coeffs(dim, N, seed), N)
    return s.expand(M, *s.shape).contiguous()


def _instances(case):
    rng = np.random.default_rng(case["pick"])
    Ns = [n for n in (255, 511, 1023) if n <= case["Nmax"]]
    Ms = [m for m in (128, 256, 512, 1024) if m <= case["Mmax"]]
    return [dict(alpha=float(rng.uniform(0.2, 0.9)), gamma=float(rng.uniform(1.0, 3.0)), N=int(rng.choice(Ns)),
                 M=int(rng.choice(Ms))) for _ in range(case["count"])]


def _iterate(case, seed):
    """An iterate of a solve: a smooth field growing like t^alpha with a small rough error."""
    s = _space(_coeffs(case["dim"], case["N"], seed + 1), case["N"])
    t = _times(case["M"], case["gamma"]) ** case["alpha"]
    g = torch.Generator(DEV).manual_seed(seed)
    u = torch.randn(case["M"], *s.shape, dtype=torch.float64, device=DEV, generator=g).mul_(1e-3)
    return u.add_(t.reshape(-1, *[1] * s.dim()) * s)


def _panel(case, seed, dtype):
    g = torch.Generator(DEV).manual_seed(seed)
    return torch.randn(case["M"], case["cols"], dtype=dtype, device=DEV, generator=g)


def _net_params(hidden, layers, seed):
    rng = np.random.default_rng(seed)
    w = [6] + [hidden] * layers + [1]
    out = []
    for i, o in zip(w[:-1], w[1:]):
        out += [rng.standard_normal(o * i) * math.sqrt(2.0 / i) * (0.1 if o == 1 else 1.0), 0.1 * rng.standard_normal(o)]
    return np.concatenate(out).astype(np.float32)


def _net(hidden, layers, seed):
    net = fh.WSNet(hidden, layers, 0)
    net.set_params(_net_params(hidden, layers, seed))
    return net


def _features(lam, alpha, t):
    s = lam * t ** alpha
    return torch.stack([torch.log10(lam) / 5, alpha + 0 * s, torch.log10(t) / 5, s / (1 + s), torch.log1p(s) / 10,
                        t ** alpha], dim=-1)


def _samples(case, seed):
    """Training rows: eigenvalues, orders and times over their ranges, targets near s / (1 + s)."""
    rng = np.random.default_rng(seed)
    n = case["batch"]
    lam = torch.as_tensor(10 ** rng.uniform(1.2, 4.2, n), device=DEV)
    alpha = torch.as_tensor(rng.uniform(0.3, 0.8, n), device=DEV)
    t = torch.as_tensor((rng.integers(1, 513, n) / 512.0) ** 2, device=DEV)
    X = _features(lam, alpha, t)
    Y = X[:, 3] * (1 - 0.1 * alpha * torch.exp(-t))
    return X.float().contiguous(), Y.float().contiguous()


# ---------------------------------------------------------------- the cases


def _problem(case, dim, N, prec):
    H = fh.HMatrix(case["alpha"], case["gamma"], 1.0, case["M"], LEAF, 0, TOL)
    return fh.Problem(H, dim, N, 1.0, PREC[prec])


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "train":
        st["net"] = _net(case["hidden"], case["layers"], seed)
        st["X"], st["Y"] = _samples(case, seed)
    elif kind == "batched":
        st["P"], st["u"], st["f"] = [], [], []
        for i, c in enumerate(_instances(case)):
            P = _problem(c, 1, c["N"], case["prec"])
            st["P"].append(P)
            st["f"].append(_source(1, c["N"], c["M"], seed * 64 + i))
            st["u"].append(torch.zeros_like(st["f"][-1]))
    elif kind in ("line", "product"):
        st["P"] = _problem(case, 2, 255, case["prec"]) if kind == "line" else _problem(case, 1, 255, "fp32")
        st["B"] = _panel(case, seed, torch.float32 if kind == "line" else torch.float64)
        st["out"] = torch.empty_like(st["B"])
    else:
        dim = case.get("dim", 2)
        st["P"] = _problem(case, dim, case["N"], case.get("prec", "bf16" if kind == "predict" else "fp64"))
        st["f"] = _source(dim, case["N"], case["M"], seed)
        if kind == "solve":
            if case["direct"]:
                st["P"].set_coarse_direct(case["direct"])
            st["P"].set_rtol_reference(1)
            st["u"] = torch.zeros_like(st["f"])
        elif kind == "predict":
            st["net"] = _net(320, 3, seed)
            st["u"] = torch.empty_like(st["f"])
        else:
            st["u"] = _iterate(case, seed)
            st["out"] = torch.empty_like(st["f"])
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "solve":
        st["u"].zero_()
        k, _ = st["P"].solve(st["u"], st["f"], None, 1, 1, RTOL, MAX_CYCLES, allow_notconv=True)
        return {"u": st["u"], "cycles": k}
    if kind == "batched":
        for u in st["u"]:
            u.zero_()
        k, _ = fh.solve_batched(st["P"], st["u"], st["f"], 1, 1, RTOL, MAX_CYCLES, allow_notconv=True)
        return {"u": st["u"], "cycles": k}
    if kind == "smooth":
        st["out"].copy_(st["u"])
        st["P"].smooth(st["out"], st["f"], 1)
        return st["out"]
    if kind == "residual":
        st["P"].residual(st["u"], st["f"], None, st["out"])
        return st["out"]
    if kind == "line":
        st["P"].line_solve_s(st["P"].levels - 1, st["out"], st["B"])
        return st["out"]
    if kind == "product":
        st["P"].hmatvec_f32(st["out"], st["B"])
        return st["out"]
    if kind == "predict":
        return st["net"].predict(st["P"], st["f"], case["alpha"], case["K"], True, st["u"])
    loss, grad = st["net"].loss_grad(st["X"], st["Y"])
    return {"loss": np.float32(loss), "grad": grad}


# ---------------------------------------------------------------- work


def _walk_flops(M):
    """Flops of one H-matrix product or solve over M time levels (leaf 64, ranks near 5): the near field
    and 59 flops per level of the block tree and row."""
    return M * (128 + 59 * math.log2(max(M // LEAF, 1)))


def work(case):
    kind = case["kind"]
    if kind == "train":
        h, n = case["hidden"], case["batch"]
        params = 7 * h + (case["layers"] - 1) * (h * h + h) + h + 1
        return {"bytes": 4 * (7 * n + 2 * params), "flops": 6.0 * n * params}
    if kind == "batched":
        its = _instances(case)
        return {"bytes": sum(16 * c["N"] * c["M"] for c in its),
                "flops": sum(8 * 6 * c["N"] * _walk_flops(c["M"]) for c in its)}
    M = case["M"]
    if kind in ("line", "product"):
        return {"bytes": (8 if kind == "line" else 16) * M * case["cols"], "flops": case["cols"] * _walk_flops(M)}
    n = case["N"] ** case.get("dim", 2)
    if kind == "predict":  # the source's last level in, the start values out; the network's rows and the synthesis
        N, K = case["N"], case["K"]
        return {"bytes": 8 * n * (M + 1), "flops": 2.0 * M * K * K * (6 * 320 + 2 * 320 * 320) + 2.0 * M * K * (K * N + n)}
    if kind == "solve":  # source in, solution out; about 8 cycles of two sweeps, transfers, coarser levels, defects
        return {"bytes": 16 * n * M, "flops": 8 * (6 if case["dim"] == 1 else 4) * n * _walk_flops(M)}
    return {"bytes": 24 * n * M, "flops": n * (_walk_flops(M) + 6 * M)}


# ---------------------------------------------------------------- reference values in 64 bits


def _l1(alpha, gamma, M):
    """The L1 matrix of the Caputo derivative on the graded mesh: closed form near the diagonal,
    integration by parts and Gauss-Legendre quadrature three or more steps below it."""
    t = (torch.arange(M + 1, dtype=torch.float64, device=DEV) / M) ** gamma
    tau = t[1:] - t[:-1]
    p = 1 - alpha
    b = (t[1:, None] - t[None, 1:]).clamp(min=0)
    d = torch.where(b > 0, b.clamp(min=1e-300) ** p * torch.expm1(p * torch.log1p(tau / b.clamp(min=1e-300))), tau ** p)
    d = torch.tril(d / (tau * math.gamma(2 - alpha)))
    R = d.clone()
    R[:, :-1] -= d[:, 1:]
    if M > 3:
        x, w = (torch.as_tensor(v, device=DEV) for v in np.polynomial.legendre.leggauss(24))
        up, down, w = (1 + x) / 2, (1 - x) / 2, w / 2
        tl, tr = tau[:-1, None] * up, tau[1:, None] * up  # hats j = 1..M-1, offsets of the nodes
        for r0 in range(3, M, 64):
            r1 = min(M, r0 + 64)
            nj = r1 - 3
            tm = t[r0 + 1:r1 + 1, None, None]
            dl = (tm - (t[:nj, None] + tl[:nj])).clamp(min=1e-300) ** (-1 - alpha)
            dr = (tm - (t[1:nj + 1, None] + tr[:nj])).clamp(min=1e-300) ** (-1 - alpha)
            far = tau[:nj] * (dl @ (up * w)) + tau[1:nj + 1] * (dr @ (down * w))
            far = far * (-alpha / math.gamma(1 - alpha))
            keep = torch.arange(nj, device=DEV)[None] <= torch.arange(r0, r1, device=DEV)[:, None] - 3
            R[r0:r1, :nj] = torch.where(keep, far, R[r0:r1, :nj])
    return R


def _eigs(N, k):
    return 4.0 * (N + 1) ** 2 * np.sin(math.pi * np.arange(1, k + 1) / (2 * (N + 1))) ** 2


def _solution(dim, N, R, c):
    """The discrete solution for a source with sine coefficients c: one time system per mode."""
    M = R.shape[0]
    lam = _eigs(N, c.shape[0])
    lam = (lam if dim == 1 else lam[:, None] + lam[None]).ravel()
    one = torch.ones(1, M, 1, dtype=torch.float64, device=DEV)
    eye = torch.eye(M, dtype=torch.float64, device=DEV)
    w = []
    step = max(1, (1 << 28) // (M * M))
    for l in torch.as_tensor(lam, device=DEV).split(step):
        w.append(torch.linalg.solve_triangular(R + l[:, None, None] * eye, one.expand(len(l), M, 1), upper=False)[..., 0])
    a = torch.cat(w).T * torch.as_tensor(c.ravel(), device=DEV)  # (M, modes)
    S = _sines(N, c.shape[0])
    return a @ S if dim == 1 else torch.matmul(S.T, torch.matmul(a.reshape(M, *c.shape), S))


def _neighbours(u):
    s = torch.zeros_like(u)
    for d in range(1, u.dim()):
        n = u.shape[d]
        s.narrow(d, 0, n - 1).add_(u.narrow(d, 1, n - 1))
        s.narrow(d, 1, n - 1).add_(u.narrow(d, 0, n - 1))
    return s


def _forward(case_net, params, X):
    hidden, layers = case_net
    w, at, a = [6] + [hidden] * layers + [1], 0, X
    for i, (n, m) in enumerate(zip(w[:-1], w[1:])):
        z = a @ params[at:at + n * m].reshape(m, n).T + params[at + n * m:at + n * m + m]
        at += n * m + m
        a = torch.nn.functional.silu(z) if i < layers else z
    return a[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, Y = _samples(case, seed)
        par = torch.as_tensor(_net_params(case["hidden"], case["layers"], seed), device=DEV).double().requires_grad_()
        loss = ((_forward((case["hidden"], case["layers"]), par, X.double()) - Y.double()) ** 2).mean()
        loss.backward()
        return {"loss": np.float64(loss.item()), "grad": par.grad.cpu().numpy()}
    if kind == "batched":
        return {"u": [_solution(1, c["N"], _l1(c["alpha"], c["gamma"], c["M"]), _coeffs(1, c["N"], seed * 64 + i))
                      for i, c in enumerate(_instances(case))], "cycles": None}
    M = case["M"]
    if kind == "predict":
        c = np.zeros((case["K"], case["K"]))
        co = _coeffs(2, case["N"], seed)[:case["K"], :case["K"]]
        c[:co.shape[0], :co.shape[1]] = co
        lam = _eigs(case["N"], case["K"])
        lam = torch.as_tensor((lam[:, None] + lam[None]).ravel(), device=DEV)
        t = _times(M, case["gamma"])
        X = _features(lam[:, None].expand(-1, M).reshape(-1), torch.tensor(case["alpha"], device=DEV, dtype=torch.float64),
                      t.repeat(len(lam)))
        par = torch.as_tensor(_net_params(320, 3, seed), device=DEV).double()
        y = torch.cat([_forward((320, 3), par, x) for x in X.split(1 << 16)]).reshape(len(lam), M)
        a = (y / lam[:, None]).T.reshape(M, case["K"], case["K"]) * torch.as_tensor(c, device=DEV)
        S = _sines(case["N"], case["K"])
        return torch.matmul(S.T, torch.matmul(a, S))
    R = _l1(case["alpha"], case["gamma"], M)
    if kind == "solve":
        return {"u": _solution(case["dim"], case["N"], R, _coeffs(case["dim"], case["N"], seed)), "cycles": None}
    if kind == "line":
        A = R + 4.0 * 256 ** 2 * torch.eye(M, dtype=torch.float64, device=DEV)
        return torch.linalg.solve_triangular(A, _panel(case, seed, torch.float32).double(), upper=False)
    if kind == "product":
        return R @ _panel(case, seed, torch.float64)
    dim, N = case["dim"], case["N"]
    u, f = _iterate(case, seed), _source(dim, N, M, seed)
    ih2 = float(N + 1) ** 2
    if kind == "residual":
        return f - ih2 * (2 * dim * u - _neighbours(u)) - (R @ u.reshape(M, -1)).reshape(u.shape)
    A = R + 2 * dim * ih2 * torch.eye(M, dtype=torch.float64, device=DEV)
    idx = torch.arange(N, device=DEV)
    parity = idx % 2 if dim == 1 else (idx[:, None] + idx[None]) % 2
    for colour in (0, 1):
        b = (f + ih2 * _neighbours(u))[:, parity == colour]
        u[:, parity == colour] = torch.linalg.solve_triangular(A, b, upper=False)
    return u
