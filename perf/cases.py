"""The calls that a user of the library makes, as measurable cases.

Every case is a plain dict with a ``kind`` (which entry points it goes
through) and its sizes. ``prepare`` makes seeded synthetic inputs on the GPU (a
planted nonnegative CP plus uniform noise, initial factors on (0, 1]), ``run`` is one
call as a program makes it, ``work`` the bytes and operations the call cannot do
without, and ``exact`` the same mathematics in plain float64 torch.

Fits update their factors in place, so ``run`` first copies the initial factors into the
working ones (a program that restarts a fit does the same). Sweep counts are shorter than
the 200 to 5000 of a full experiment: rounding differences grow with every sweep (the model does
not fix the scale between its factors), and the outputs of a short fit, as a program that
resumes a fit in pieces runs it, can still be compared to FP32 accuracy. What
single-precision fits report in FP64 (traces, errors, losses) is returned in their own
precision.
"""
from __future__ import annotations

import math

import torch

from paper_1909_07570_gb300 import autograd, native

EPS = 1e-12
L2_BYTES = 129 << 20
DEVICE = "cuda"


def _case(name, kind, dims, m, r, rank, iters, precision, **more):
    c = {"kind": kind, "dims": "x".join(map(str, dims)), "m": "x".join(map(str, m)), "r": r,
         "rank": rank, "iters": iters, "precision": precision, "dist": "uniform",
         "noise": 0.01}
    c.update(more)
    if name:
        c["name"] = name
    return c


def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def listed():
    return [
        # Alg. 1 end to end (nnTD, nnCPD of the core, lift, residual) on a small FP64 tensor: the
        # call of the synthetic experiments, where launches and latency count.
        _case("alg1_fp64_40cube", "alg1", (40, 40, 40), (5, 5, 5), 3, 3, 200, "fp64"),
        # The same on the shape of the fluorescence data (5 x 61 x 201, multirank 3): the smallest
        # real tensor, all modes ragged.
        _case("alg1_fp32_5x61x201", "alg1", (5, 61, 201), (3, 3, 3), 3, 3, 100, "fp32"),
        # nnTD of a mid-size FP32 tensor: the plain FP32 experiment.
        _case("ntd_fp32_256cube", "ntd", (256, 256, 256), (20, 20, 20), 0, 10, 30, "fp32",
              noise=0.02),
        # nnTD of measured data whose modes are no multiples of anything.
        _case("ntd_fp32_301x217x255", "ntd", (301, 217, 255), (24, 17, 12), 0, 10, 60, "fp32"),
        # nnTD of a large tensor with BF16 passes and final FP32 sweeps: the headline form.
        _case("ntd_bf16_512cube", "ntd", (512, 512, 512), (32, 32, 32), 0, 16, 100, "bf16",
              refine=10, dist="exponential"),
        # The same tensor with FP32 passes throughout: what the BF16 form is compared with.
        _case("ntd_fp32_512cube", "ntd", (512, 512, 512), (32, 32, 32), 0, 16, 15, "fp32",
              dist="exponential"),
        # nnTD of a 4-way tensor.
        _case("ntd_fp32_4way", "ntd", (128, 128, 128, 64), (24, 24, 24, 16), 0, 12, 30, "fp32"),
        # Loss and gradients of the lifted model as one layer of a differentiable pipeline
        # (autograd forward and backward).
        _case("grad_fp32_4way", "grad", (128, 128, 128, 64), (24, 24, 24, 16), 12, 12, 1, "fp32"),
        # Projected-gradient fit of the same model.
        _case("pg_fp32_4way", "pg", (128, 128, 128, 64), (24, 24, 24, 16), 12, 12, 20, "fp32"),
        # nnCPD of one large core (the second step of Alg. 1 on the 512^3 tensor).
        _case("core_fp32_32cube_r16", "core", (), (32, 32, 32), 16, 16, 300, "fp32"),
        # Model selection: the cores of many tensors (ranks 2..8, core sizes 4^3..16^3), each fitted at
        # ranks 2..8 from several random starts in one batched launch.
        _case("cores_fp32_64x7x8", "cores", (), (16, 16, 16), 8, 8, 200, "fp32", tensors=64,
              restarts=8),
        # The batch experiment: nnTD of 1000 small tensors in one batched launch.
        _case("batch_fp32_1000x40cube", "batch", (40, 40, 40), (3, 4, 5), 0, 5, 100, "fp32",
              jobs=1000, noise=0.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["alg1", "ntd", "ntd", "ntd", "ntd4", "grad", "pg", "core", "cores", "batch"])
    if kind == "alg1":
        dims = tuple(_log(rng, 5, 128) for _ in range(3))
        m = tuple(min(n, rng.randint(2, 8)) for n in dims)
        return _case("", "alg1", dims, m, rng.randint(2, 5), rng.randint(2, 5),
                     rng.randint(50, 100), rng.choice(["fp64", "fp32"]))
    if kind == "ntd":
        dims = tuple(_log(rng, 48, 512) for _ in range(3))
        if rng.random() < 0.5:
            dims = tuple(-(-n // 16) * 16 for n in dims)
        m = tuple(min(n, rng.randint(4, 32)) for n in dims)
        precision = rng.choice(["fp32", "fp32", "bf16"])
        more = {"refine": rng.randint(2, 8)} if precision == "bf16" else {}
        iters = rng.randint(30, 50) if precision == "bf16" else rng.randint(10, 15)
        return _case("", "ntd", dims, m, 0, rng.randint(4, 16), iters, precision,
                     dist=rng.choice(["uniform", "exponential"]), **more)
    if kind in ("ntd4", "grad", "pg"):
        d = 4 if kind == "ntd4" else rng.choice([3, 4])
        lo, hi = (24, 96) if d == 4 else (48, 320)
        dims = tuple(_log(rng, lo, hi) for _ in range(d))
        if rng.random() < 0.5:
            dims = dims[:-1] + (-(-dims[-1] // 4) * 4,)
        m = tuple(min(n, rng.randint(4, 24)) for n in dims)
        iters = {"ntd4": rng.randint(10, 20), "grad": 1, "pg": rng.randint(5, 20)}[kind]
        r = 0 if kind == "ntd4" else rng.randint(3, 16)
        return _case("", "ntd" if kind == "ntd4" else kind, dims, m, r, rng.randint(4, 12), iters,
                     "fp32")
    if kind == "core":
        m = tuple(_log(rng, 8, 40) for _ in range(3))
        return _case("", "core", (), m, rng.randint(3, 16), rng.randint(3, 16),
                     rng.randint(100, 300), "fp32")
    if kind == "cores":
        r = rng.randint(4, 8)
        return _case("", "cores", (), (2 * r,) * 3, r, r, rng.randint(100, 200), "fp32",
                     tensors=rng.randint(16, 64), restarts=rng.randint(2, 8))
    dims = tuple(_log(rng, 4, 40) for _ in range(3))
    m = tuple(min(n, rng.randint(2, 6)) for n in dims)
    return _case("", "batch", dims, m, 0, rng.randint(2, 5), rng.randint(50, 100),
                 rng.choice(["fp32", "fp32", "fp64"]), jobs=_log(rng, 64, 1000), noise=0.0)


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _planted(dims, rank, dist, noise, dtype, g, batch=()):
    """A planted nonnegative CP tensor (a batch of them) plus uniform noise of relative norm `noise`."""
    draw_ = (lambda n: torch.rand(*batch, n, rank, generator=g, device=DEVICE, dtype=dtype))
    A = [draw_(n) for n in dims]
    if dist == "exponential":
        A = [-torch.log1p(-a) for a in A]
    K = A[-1]
    for a in reversed(A[1:-1]):
        K = (a.unsqueeze(-2) * K.unsqueeze(-3)).reshape(*batch, -1, rank)
    X = (A[0] @ K.transpose(-1, -2)).reshape(*batch, *dims)
    if noise:
        E = torch.rand(X.shape, generator=g, device=DEVICE, dtype=dtype)
        X.add_(E, alpha=noise * float(X.norm() / E.norm()))
    return X


def _start(shape, dtype, g):
    return 1.0 - torch.rand(*shape, generator=g, device=DEVICE, dtype=dtype)


def _inputs(case, seed):
    """The tensors a program has in hand: data and initial factors."""
    dims, m, r = _ints(case["dims"]) if case["dims"] else (), _ints(case["m"]), case["r"]
    dtype, g, kind = _dtype(case), _gen(seed), case["kind"]
    if kind == "batch":
        n = case["jobs"]
        return {"X": _planted(dims, case["rank"], case["dist"], case["noise"], dtype, g, (n,)),
                "F": [_start((n, a, b), dtype, g) for a, b in zip(dims, m)],
                "G": _start((n, *m), dtype, g)}
    if kind == "core":
        return {"G": _planted(m, case["rank"], case["dist"], case["noise"], dtype, g),
                "B": [_start((a, r), dtype, g) for a in m]}
    if kind == "cores":
        cores = []
        for t in range(case["tensors"]):
            rk = 2 + t % (r - 1)
            G = _planted((2 * rk,) * 3, rk, case["dist"], case["noise"], dtype, g)
            for q in range(2, r + 1):
                cores += [(G, [_start((2 * rk, q), dtype, g) for _ in range(3)])
                          for _ in range(case["restarts"])]
        return {"cores": cores}
    s = {"X": _planted(dims, case["rank"], case["dist"], case["noise"], dtype, g),
         "F": [_start((a, b), dtype, g) for a, b in zip(dims, m)]}
    if kind in ("alg1", "ntd"):
        s["G"] = _start(m, dtype, g)
    if kind in ("alg1", "grad", "pg"):
        s["B"] = [_start((a, r), dtype, g) for a in m]
    if kind in ("grad", "pg"):
        # a model on the data's own scale, as a pipeline's initialisation gives it
        lifted = [(f.double() @ b.double()) for f, b in zip(s["F"], s["B"])]
        V = torch.ones(r, r, dtype=torch.float64, device=DEVICE)
        for a in lifted:
            V = V * (a.T @ a)
        scale = float(s["X"].double().norm() / V.sum().sqrt()) ** (0.5 / len(dims))
        s["F"] = [f * scale for f in s["F"]]
        s["B"] = [b * scale for b in s["B"]]
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.update(kind=case["kind"], iters=case["iters"], precision=case["precision"],
             refine=case.get("refine", 0))
    kind = case["kind"]
    if kind == "grad":
        for t in s["F"] + s["B"]:
            t.requires_grad_(True)
    elif kind == "cores":  # all starts in one buffer: one copy restarts every fit
        cores = s.pop("cores")
        flat = [b for _, B in cores for b in B]
        s["B0"] = torch.cat([b.reshape(-1) for b in flat])
        s["Bw"] = s["B0"].clone()
        views = [v.view(b.shape) for v, b in zip(s["Bw"].split([b.numel() for b in flat]), flat)]
        s["jobs"] = [(G, views[3 * i:3 * i + 3]) for i, (G, _) in enumerate(cores)]
    else:
        s["init"] = [t for key in ("F", "G", "B") if key in s and not (kind == "core" and key == "G")
                     for t in (s[key] if isinstance(s[key], list) else [s[key]])]
        s["work"] = [t.clone() for t in s["init"]]
        if kind == "batch":
            w = s["work"]
            s["jobs"] = [(s["X"][i], [w[0][i], w[1][i], w[2][i]], w[3][i])
                         for i in range(case["jobs"])]
    return s


def run(s):
    kind, it, prec = s["kind"], s["iters"], s["precision"]
    if kind == "grad":
        loss = autograd.lifted_loss(s["X"], s["F"], s["B"], precision=prec)
        grads = torch.autograd.grad(loss, s["F"] + s["B"])
        return {"loss": loss.detach().to(s["X"].dtype), "grads": list(grads)}
    if kind == "cores":
        s["Bw"].copy_(s["B0"])
        errs = native.nncp_core_fit_batched(s["jobs"], it, precision=prec)
        return {"B": s["Bw"], "errs": errs.to(s["Bw"].dtype)}
    torch._foreach_copy_(s["work"], s["init"])
    w = s["work"]
    if kind == "batch":
        errs = native.ntd_fit_small_batched(s["jobs"], it, precision=prec)
        return {"fit": w, "errs": errs.to(w[0].dtype)}
    if kind == "core":
        return {"B": w, "err": native.nncp_core_fit(s["G"], w, it, precision=prec)}
    X = s["X"]
    d = X.dim()
    F, rest = w[:d], w[d:]
    if kind == "pg":
        loss, trace = native.candelinc_pg_fit(X, F, rest, it, precision=prec)
        return {"fit": w, "loss": loss, "trace": trace.to(X.dtype)}
    G = rest[0]
    err, trace = native.ntd_fit(X, F, G, it, precision=prec, refine_iters=s["refine"])
    out = {"fit": w, "err": err, "trace": trace.to(X.dtype)}
    if kind == "alg1":
        B = rest[1:]
        out["core_err"] = native.nncp_core_fit(G, B, it, precision=prec)
        out["A"] = native.candelinc_lift(F, B)
        out["norms"] = list(native.recon_residual(X, out["A"]))
    return out


def _ntd_work(dims, m, iters, size):
    """Per sweep X is contracted with F_d and with F_1 (Gauss-Seidel needs both), and each result once
    more; X comes from memory at both unless the chip's cache holds it."""
    n = math.prod(dims)
    flops = 2 * n * (m[0] + m[-1])
    flops += 2 * (n // dims[-1]) * m[-1] * (m[0] + m[1]) + 2 * (n // dims[0]) * m[0] * m[1]
    reads = 2 * iters if n * size > L2_BYTES else 1
    small = 2 * size * (sum(a * b for a, b in zip(dims, m)) + math.prod(m))
    return reads * n * size + small, iters * flops


def work(case):
    dims, m, r = _ints(case["dims"]) if case["dims"] else (), _ints(case["m"]), case["r"]
    it, kind = case["iters"], case["kind"]
    size = 8 if case["precision"] == "fp64" else 4
    if kind in ("ntd", "alg1"):
        b, f = _ntd_work(dims, m, it, size)
        if case["precision"] == "bf16":
            # X once in FP32, its BF16 copy written once and read by the BF16 sweeps
            n, fp32 = math.prod(dims), case.get("refine", 0)
            half, _ = _ntd_work(dims, m, it - fp32, 2)
            full, _ = _ntd_work(dims, m, fp32, 4)
            b = half + full + 6 * n
        if kind == "alg1":
            f += it * 6 * math.prod(m) * r + 2 * r * sum(a * c for a, c in zip(dims, m))
            f += 2 * math.prod(dims) * r
            b += 2 * size * r * (sum(m) + sum(dims))
        return {"bytes": b, "flops": f}
    if kind == "batch":
        b, f = _ntd_work(dims, m, it, size)
        return {"bytes": case["jobs"] * b, "flops": case["jobs"] * f}
    if kind == "core":
        n = math.prod(m)
        return {"bytes": size * (n + 2 * r * sum(m)), "flops": it * 6 * n * r}
    if kind == "cores":
        b = f = 0
        for t in range(case["tensors"]):
            rk = 2 + t % (r - 1)
            n = (2 * rk) ** 3
            b += size * n
            for q in range(2, r + 1):
                b += case["restarts"] * size * 2 * 3 * 2 * rk * q
                f += case["restarts"] * it * 6 * n * q
        return {"bytes": b, "flops": f}
    # gradient and projected-gradient steps: two contractions of X each; the forward loss of a
    # gradient needs one more read of X
    b, f = _ntd_work(dims, m, it, size)
    n = math.prod(dims)
    if kind == "grad":
        b += n * size if n * size > L2_BYTES else 0
        f += 2 * n * m[-1]
    return {"bytes": b + 2 * size * r * sum(m), "flops": f}


# --- the same mathematics in plain float64 torch ---------------------------------------------


def _along(X, M, n):
    """X x_n M^T: mode n of X (length rows of M) becomes the columns of M."""
    return torch.movedim(torch.tensordot(X, M, dims=([n], [0])), -1, n)


def _chain(X, Ms, skip=None):
    """X contracted with M_k over every mode k but `skip`, the outer modes first."""
    d = X.dim()
    order = [k for k in ([d - 1] + list(range(d - 1)) if skip != d - 1 else range(d - 1)) if k != skip]
    for k in order:
        X = _along(X, Ms[k], k)
    return X


def _unfold(X, n):
    return torch.movedim(X, n, 0).reshape(X.shape[n], -1)


def _ratio(t, num, den):
    return torch.clamp(t * num / torch.clamp(den, min=EPS), min=0.0)


def _exact_ntd(X, F, G, iters):
    d, x2 = X.dim(), float((X * X).sum())
    trace = []
    for _ in range(iters):
        for n in range(d):
            S = [f.T @ f for f in F]
            num = _unfold(_chain(X, F, n), n) @ _unfold(G, n).T
            H = _unfold(_chain(G, S, n), n) @ _unfold(G, n).T
            F[n] = _ratio(F[n], num, F[n] @ H)
        S = [f.T @ f for f in F]
        M = _chain(X, F)
        G = _ratio(G, M, _chain(G, S))
        res = x2 - 2 * float((M * G).sum()) + float((G * _chain(G, S)).sum())
        trace.append(math.sqrt(max(res, 0.0) / x2))
    return F, G, trace


def _exact_cp(G, B, iters):
    """Batched over leading dimension: G (z, a, b, c), B three of (z, m, r)."""
    eq = ["zabc,zbr,zcr->zar", "zabc,zar,zcr->zbr", "zabc,zar,zbr->zcr"]
    for _ in range(iters):
        for n in range(3):
            o = [B[k] for k in range(3) if k != n]
            V = (o[0].transpose(1, 2) @ o[0]) * (o[1].transpose(1, 2) @ o[1])
            T = torch.einsum("zabc,zcr->zabr", G, o[1]) if n < 2 else torch.einsum(
                "zabc,zar->zbcr", G, o[0])
            num = (T * o[0].unsqueeze(1)).sum(2) if n == 0 else (
                (T * o[0].unsqueeze(2)).sum(1) if n == 1 else (T * o[1].unsqueeze(2)).sum(1))
            B[n] = _ratio(B[n], num, B[n] @ V)
    fit = torch.einsum("zar,zbr,zcr->zabc", *B)
    return B, ((G - fit).flatten(1).norm(dim=1) / G.flatten(1).norm(dim=1))


def _cp_full(A):
    K = A[-1]
    for a in reversed(A[1:-1]):
        K = (a.unsqueeze(-2) * K.unsqueeze(-3)).reshape(-1, K.shape[-1])
    return (A[0] @ K.T).reshape([a.shape[0] for a in A])


def _lifted_grad_A(X, F, B, n):
    """dL/dA_n and V_n of the lifted model."""
    d = len(F)
    A = [f @ b for f, b in zip(F, B)]
    V = torch.ones(B[0].shape[1], B[0].shape[1], dtype=torch.float64, device=X.device)
    for k in range(d):
        if k != n:
            V = V * (A[k].T @ A[k])
    T = torch.movedim(_chain(X, F, n), n, 0)
    rest = [B[k] for k in range(d) if k != n]
    K = rest[-1]
    for b in reversed(rest[:-1]):
        K = (b.unsqueeze(-2) * K.unsqueeze(-3)).reshape(-1, K.shape[-1])
    return A[n] @ V - T.reshape(T.shape[0], -1) @ K, V


def _lmax(M, iters=30):
    v = torch.ones(M.shape[0], dtype=M.dtype, device=M.device)
    for _ in range(iters):
        w = M @ v
        v = w / w.norm()
    return v @ (M @ v)


def _loss(X, F, B):
    return 0.5 * float((X - _cp_full([f @ b for f, b in zip(F, B)])).square().sum())


def _exact_pg(X, F, B, steps):
    trace = []
    for _ in range(steps):
        for n in range(len(F)):
            gA, V = _lifted_grad_A(X, F, B, n)
            F[n] = torch.clamp(F[n] - gA @ B[n].T / _lmax(B[n] @ V @ B[n].T), min=0.0)
            gA, V = _lifted_grad_A(X, F, B, n)
            L = _lmax(F[n].T @ F[n]) * _lmax(V)
            B[n] = torch.clamp(B[n] - F[n].T @ gA / L, min=0.0)
        trace.append(_loss(X, F, B))
    return F, B, trace


def exact(case, seed):
    s = _inputs(case, seed)
    kind, it = case["kind"], case["iters"]
    up = (lambda v: [t.double() for t in v])
    vec = (lambda v: torch.tensor(v, dtype=torch.float64))
    if kind == "cores":
        top, r, cores = 2 * case["r"], case["r"], s["cores"]
        n = len(cores)
        G = torch.zeros(n, top, top, top, dtype=torch.float64, device=DEVICE)
        B = [torch.zeros(n, top, r, dtype=torch.float64, device=DEVICE) for _ in range(3)]
        for i, (g, b) in enumerate(cores):  # zero rows and columns stay zero
            k = g.shape[0]
            G[i, :k, :k, :k] = g
            for q in range(3):
                B[q][i, :k, :b[q].shape[1]] = b[q]
        B, errs = _exact_cp(G, B, it)
        flat = [B[q][i, :b[q].shape[0], :b[q].shape[1]].reshape(-1)
                for i, (_, b) in enumerate(cores) for q in range(3)]
        return {"B": torch.cat(flat), "errs": errs}
    if kind == "core":
        B, errs = _exact_cp(s["G"].double()[None], [b.double()[None] for b in s["B"]], it)
        return {"B": [b[0] for b in B], "err": float(errs[0])}
    if kind == "batch":
        return _exact_batch(s, it)
    X, F = s["X"].double(), up(s["F"])
    if kind == "grad":
        B = up(s["B"])
        gA = [_lifted_grad_A(X, F, B, n)[0] for n in range(X.dim())]
        return {"loss": vec(_loss(X, F, B)), "grads": [a @ b.T for a, b in zip(gA, B)]
                + [f.T @ a for a, f in zip(gA, F)]}
    if kind == "pg":
        F, B, trace = _exact_pg(X, F, up(s["B"]), it)
        return {"fit": F + B, "loss": trace[-1], "trace": vec(trace)}
    F, G, trace = _exact_ntd(X, F, s["G"].double(), it)
    full = G
    for k, f in enumerate(F):
        full = _along(full, f.T, k)
    out = {"fit": F + [G], "err": float((X - full).norm() / X.norm()), "trace": vec(trace)}
    if kind == "alg1":
        B, errs = _exact_cp(G[None], [b.double()[None] for b in s["B"]], it)
        B = [b[0] for b in B]
        out["fit"] = F + [G] + B
        out["core_err"] = float(errs[0])
        out["A"] = [f @ b for f, b in zip(F, B)]
        out["norms"] = [float((X - _cp_full(out["A"])).norm()), float(X.norm())]
    return out


def _exact_batch(s, iters):
    X, G, F = s["X"].double(), s["G"].double(), [f.double() for f in s["F"]]

    def chain(T, Ms, skip=None):
        for k in (2, 1, 0) if skip != 2 else (0, 1):
            if k != skip:
                T = torch.movedim(torch.movedim(T, k + 1, -1).flatten(1, 2) @ Ms[k], -1, -1).reshape(
                    *torch.movedim(T, k + 1, -1).shape[:-1], Ms[k].shape[-1]).movedim(-1, k + 1)
        return T

    def unfold(T, n):
        return torch.movedim(T, n + 1, 1).flatten(2)

    for _ in range(iters):
        for n in range(3):
            S = [f.transpose(1, 2) @ f for f in F]
            num = unfold(chain(X, F, n), n) @ unfold(G, n).transpose(1, 2)
            H = unfold(chain(G, S, n), n) @ unfold(G, n).transpose(1, 2)
            F[n] = _ratio(F[n], num, F[n] @ H)
        S = [f.transpose(1, 2) @ f for f in F]
        G = _ratio(G, chain(X, F), chain(G, S))
    fit = chain(G, [f.transpose(1, 2) for f in F])
    err = (X - fit).flatten(1).norm(dim=1) / X.flatten(1).norm(dim=1)
    return {"fit": F + [G], "errs": err}
