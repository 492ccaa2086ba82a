"""Kernels and dispatch branches at the edges of their tiles, remainders and
ranges, against the oracle on the same inputs."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1909_07570_gb300 import inputs, native

pytestmark = pytest.mark.gpu


def _dev(a, dt):
    return torch.tensor(np.asarray(a), dtype=dt, device="cuda")


# FP64: a few sweeps amplify 1e-16 rounding by far less than 1e-9. FP32: sums of at
# most a few thousand positive terms, a few sweeps: 1e-4 (the one-sweep bound of the
# FP32 kernels).
_TOL = {torch.float64: 1e-9, torch.float32: 1e-4}


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("jobs", [
    [((1, 1, 1), (1, 1, 1)), ((5, 1, 3), (2, 1, 2))],
    [((4, 4, 4), (5, 5, 5)), ((40, 40, 40), (3, 4, 5)), ((7, 33, 18), (4, 8, 1))],
    [((9, 3, 31), (8, 3, 8)), ((3, 65, 4), (3, 7, 4))],
    [((17, 20, 24), (16, 9, 13)), ((33, 6, 7), (12, 6, 7))],
    [((64, 2, 64), (4, 2, 4))],
    [((120, 4, 120), (4, 4, 4))],      # X x_2 F2^T beyond a block: N2 far below N1 and N3
    [((10, 12, 11), (17, 4, 20))],     # a multirank beyond 16
])
def test_small_batched_edges(dt, jobs):
    probs = [inputs.small_problem(d, 3, m, 2, seed=31 + i) for i, (d, m) in enumerate(jobs)]
    dev = [(_dev(X, dt), [_dev(f, dt) for f in F0], _dev(G0, dt)) for X, _, F0, G0, _ in probs]
    errs = native.ntd_fit_small_batched(dev, 3).cpu().numpy()
    tol = _TOL[dt]
    for (X, _, F0, G0, _), (Xd, F, G), e in zip(probs, dev, errs):
        Xr = Xd.double().cpu().numpy()
        Fo, Go, _ = orc.ntd_fit(Xr, [f.astype(np.float32).astype(float) if dt == torch.float32 else f
                                     for f in F0],
                                G0.astype(np.float32).astype(float) if dt == torch.float32 else G0, 3)
        for a, b in zip(F + [G], Fo + [Go]):
            np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
        assert e == pytest.approx(orc.rel_err_tucker(Xr, Go, Fo), abs=tol)


# Few outputs with many partial sums (32 or more: the wide sum), and the weighted sums of
# the inner modes below, at and past one group of 16 terms.
@pytest.mark.parametrize("dims,m,r", [((6, 40, 21, 9), (2, 16, 16, 8), 3),
                                      ((33, 5, 40, 7), (3, 5, 24, 5), 2),
                                      ((9, 70, 13), (4, 17, 3), 5)])
def test_lifted_gradient_sums(dims, m, r):
    rng = np.random.default_rng(5)
    X = rng.random(dims)
    F = [1 - rng.random((n, k)) for n, k in zip(dims, m)]
    B = [1 - rng.random((k, r)) for k in m]
    dt = torch.float64
    loss, gF, gB = native.candelinc_lifted_grad(_dev(X, dt), [_dev(f, dt) for f in F],
                                                [_dev(b, dt) for b in B])
    gFo, gBo = orc.lifted_loss_grad(X, F, B)
    assert loss == pytest.approx(orc.lifted_loss(X, F, B), rel=1e-9)
    for a, b in zip(gF + gB, list(gFo) + list(gBo)):
        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=1e-9, atol=1e-9 * np.abs(b).max())


def test_scratch_is_kept_bounded_and_given_back():
    X = torch.rand(256, 256, 256, device="cuda")
    F = [torch.rand(256, 8, device="cuda") + 0.1 for _ in range(3)]
    G = torch.rand(8, 8, 8, device="cuda") + 0.1
    native.ntd_fit(X, F, G, 2)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    native.nnc_release_scratch()
    freed = torch.cuda.mem_get_info()[0] - held
    # The scratch of the call holds a copy of X (64 MiB) and more; 4 GiB is the most
    # the library keeps.
    assert 64 << 20 <= freed <= 4 << 30


# The FP16 pair passes through one nnTD sweep: K just past a 64-entry chunk and a group of
# two, tiles with a remainder, NP = 64, the fused contraction (N2 % 128 == 0), slices of very
# different magnitude and zero slices, and operands past what a block holds (TF32x3).
# One sweep of FP32-accurate arithmetic on sums of up to a few thousand positive terms:
# 1e-4 elementwise, as the other FP32 kernels.
@pytest.mark.parametrize("dims,m,scaled", [
    ((65, 33, 68), (5, 4, 3), False), ((130, 20, 132), (33, 5, 40), False),
    ((24, 128, 72), (6, 8, 32), True), ((3, 256, 4), (2, 3, 4), True),
    ((129, 7, 516), (8, 6, 20), True), ((800, 6, 20), (4, 4, 4), False),
    ((17, 9, 900), (4, 4, 4), False)])
def test_pair_passes_one_sweep(dims, m, scaled):
    X, _, F0, G0, _ = inputs.small_problem(dims, 3, m, 2, seed=91)
    if scaled:
        rng = np.random.default_rng(3)
        for n in range(3):
            s = 10.0 ** rng.uniform(-3, 3, dims[n])
            s[rng.integers(dims[n])] = 0.0
            X = X * s.reshape([-1 if k == n else 1 for k in range(3)])
    X = X.astype(np.float32).astype(np.float64)
    F0 = [f.astype(np.float32).astype(np.float64) for f in F0]
    G0 = G0.astype(np.float32).astype(np.float64)
    F, G = [_dev(f, torch.float32) for f in F0], _dev(G0, torch.float32)
    err, _ = native.ntd_fit(_dev(X, torch.float32), F, G, 1, precision="fp32")
    Fo, Go, _ = orc.ntd_fit(X, F0, G0, 1)
    for a, b in zip(F + [G], Fo + [Go]):
        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=1e-4, atol=1e-30)
    assert abs(err - orc.rel_err_tucker(X, Go, Fo)) <= 1e-5


# The residual pass: rows of X shorter and longer than a block's columns, one row tile and
# a remainder, every register tile (K = 16, 32, 64 entries), both models, d = 3 and 4. The sums
# are FP64 (FP32 terms for FP32 data: 1e-5 of the norm is 100 times their rounding).
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("dims,m", [((3, 5, 1), (2, 3, 1)), ((9, 15, 517), (4, 5, 17)),
                                    ((40, 33, 30), (33, 3, 33)), ((6, 7, 5, 70), (3, 2, 5, 16)),
                                    ((17, 70, 9, 3), (2, 17, 4, 3))])
def test_residual_edges(dt, dims, m):
    rng = np.random.default_rng(17)
    X = rng.random(dims)
    F = [rng.random((n, k)) / k for n, k in zip(dims, m)]
    G = rng.random(m)
    A = [rng.random((n, m[0])) for n in dims]
    tol = 1e-11 if dt == torch.float64 else 1e-5
    Xd = _dev(X, dt)
    rn, xn = native.recon_residual(Xd, [_dev(f, dt) for f in F], _dev(G, dt))
    Xr = Xd.double().cpu().numpy()
    assert xn == pytest.approx(np.linalg.norm(Xr), rel=tol)
    assert rn / xn == pytest.approx(orc.rel_err_tucker(Xr, G, F), rel=tol)
    rn, xn = native.recon_residual(Xd, [_dev(a, dt) for a in A])
    assert rn / xn == pytest.approx(orc.rel_err_cp(Xr, A), rel=tol)


# A mode past 65535 tiles of 16 entries, as the first and as a middle mode. Tolerances as above.
@pytest.mark.parametrize("dims", [(1048593, 2, 3), (2, 1048577, 1)])
def test_residual_of_a_long_mode(dims):
    rng = np.random.default_rng(19)
    m = (2, 2, 1)
    X = rng.random(dims)
    F = [rng.random((n, k)) for n, k in zip(dims, m)]
    G = rng.random(m)
    rn, xn = native.recon_residual(_dev(X, torch.float64), [_dev(f, torch.float64) for f in F],
                                   _dev(G, torch.float64))
    assert xn == pytest.approx(np.linalg.norm(X), rel=1e-11)
    assert rn / xn == pytest.approx(orc.rel_err_tucker(X, G, F), rel=1e-11)


# FP32 terms are added in chains of at most 64 before FP64: equal terms, whose roundings add up.
# The i-th rounding of a chain is at most 2^-24 of the i terms so far, 32.5 2^-24 of the chain in
# all, and half of that in a norm. (Values whose chains of 1024 and 256 would be off by 7.6e-6
# and 1.9e-6.)
@pytest.mark.parametrize("value,last,dims", [(1.9976487, 16, (1000, 480, 512)),
                                             (1.9550849, 32, (1000, 480, 256))])
def test_residual_chains_are_short(value, last, dims):
    v = float(np.float32(value))
    X = torch.full(dims, v, device="cuda")
    F = [torch.zeros(n, k, device="cuda") for n, k in zip(dims, (2, 2, last))]
    rn, xn = native.recon_residual(X, F, torch.zeros(2, 2, last, device="cuda"))
    want = v * np.sqrt(np.prod(dims, dtype=np.float64))
    assert xn == pytest.approx(want, rel=32.5 * 2.0 ** -25)
    assert rn == pytest.approx(want, rel=32.5 * 2.0 ** -25)


# Whole fits on one cluster: modes shorter than the cluster (CTAs without slices), slices
# with a remainder, 16-byte and single columns, every tile width, exact checkpoints; and the
# same fit in pieces. The trace and factors against the oracle: FP64 rounding over a few
# sweeps; FP32 1e-4 on factors after three sweeps, 1e-5 on the trace.
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("dims,m", [((1, 1, 1), (1, 1, 1)), ((5, 61, 201), (3, 3, 3)),
                                    ((40, 40, 40), (5, 5, 5)), ((17, 3, 33), (2, 3, 7)),
                                    ((20, 18, 22), (8, 7, 4)), ((33, 16, 8), (1, 6, 4))])
def test_cluster_fit_edges(dt, dims, m):
    X, _, F0, G0, _ = inputs.small_problem(dims, 2, m, 2, seed=57)
    X, F0, G0 = (_dev(X, dt).double().cpu().numpy(),
                 [_dev(f, dt).double().cpu().numpy() for f in F0],
                 _dev(G0, dt).double().cpu().numpy())
    F, G = [_dev(f, dt) for f in F0], _dev(G0, dt)
    err, tr = native.ntd_fit(_dev(X, dt), F, G, 3)
    Fo, Go, tro = orc.ntd_fit(X, F0, G0, 3)
    tol = _TOL[dt]
    scale = max(1.0, float(np.max(tro)))
    np.testing.assert_allclose(tr.cpu().numpy(), tro, rtol=1e-8 if dt == torch.float64 else 0,
                               atol=(1e-8 if dt == torch.float64 else 1e-5) * scale)
    for a, b in zip(F + [G], Fo + [Go]):
        np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
    assert err == pytest.approx(orc.rel_err_tucker(X, Go, Fo), abs=tol)
    # In pieces, and with an exact checkpoint after every second sweep.
    F2, G2 = [_dev(f, dt) for f in F0], _dev(G0, dt)
    native.ntd_fit(_dev(X, dt), F2, G2, 1, trace=False, rel_err=False)
    err2, tr2 = native.ntd_fit(_dev(X, dt), F2, G2, 2, exact_every=2)
    for a, b in zip(F + [G], F2 + [G2]):
        assert torch.equal(a, b)
    assert tr2[1].item() == pytest.approx(err2, rel=1e-6)


# SIMT mode products: rows of every start modulo 16 bytes, K and Q at and past the tiles, one
# and two rows a thread, columns with a remainder and few enough rows j for one batch, and
# contractions split over blocks. FP64: 1e-12 of the largest sum; FP32: 1e-5 (sums of a
# few hundred positive terms in FP32).
@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-12), (torch.float32, 1e-5)])
@pytest.mark.parametrize("dims,Q", [((3, 5, 1), 1), ((2, 127, 33), 12), ((9, 43, 255), 13),
                                    ((513, 310, 17), 8), ((31, 9, 7), 64), ((17, 257, 65), 24),
                                    ((1, 129, 97), 9)])
def test_simt_mode_products(dt, tol, dims, Q):
    rng = np.random.default_rng(23)
    X = rng.random(dims)
    for mode in range(3):
        F = rng.random((dims[mode], Q))
        Y = native.mode_product(_dev(X, dt), _dev(F, dt), mode,
                                precision="fp64" if dt == torch.float64 else "fp32_simt")
        ref = np.moveaxis(np.tensordot(_dev(X, dt).double().cpu().numpy(),
                                       _dev(F, dt).double().cpu().numpy(), axes=([mode], [0])),
                          -1, mode)
        np.testing.assert_allclose(Y.double().cpu().numpy(), ref, rtol=0, atol=tol * ref.max())


# Core fits with the core in shared memory: modes of one entry, modes longer and shorter than
# a block, every row tile (r 1..4, 5..8, 9..16) in one batch, and a core that only the L1 form
# takes. Five sweeps: FP64 1e-9, FP32 1e-4.
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("jobs", [
    [((1, 1, 1), 1), ((4, 4, 4), 3), ((5, 1, 3), 4)],
    [((16, 16, 16), 8), ((2, 13, 7), 5), ((6, 5, 4), 2)],
    [((9, 12, 17), 16), ((3, 33, 2), 9), ((8, 8, 8), 7), ((2, 2, 2), 1)],
    [((40, 3, 64), 16), ((24, 24, 24), 12)],
    [((6, 7, 5), 17), ((3, 3, 3), 2)]])
def test_core_fits_in_shared_memory(dt, jobs):
    rng = np.random.default_rng(29)
    probs = [(rng.random(m), inputs.initial_cp(m, r, 7 + i)) for i, (m, r) in enumerate(jobs)]
    dev = [(_dev(G, dt), [_dev(b, dt) for b in B]) for G, B in probs]
    st = torch.full((len(jobs),), 9, dtype=torch.int32, device="cuda")
    errs = native.nncp_core_fit_batched(dev, 5, statuses=st).cpu().numpy()
    assert st.tolist() == [0] * len(jobs)
    tol = _TOL[dt]
    for (G, B0), (Gd, B), e in zip(probs, dev, errs):
        Gr = Gd.double().cpu().numpy()
        Bo, tro = orc.nncp_fit(Gr, [_dev(b, dt).double().cpu().numpy() for b in B0], 5)
        for a, b in zip(B, Bo):
            np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
        assert e == pytest.approx(tro[-1], abs=tol)


# Core fits of 16384 entries or more, one cluster each: modes shorter than the cluster (CTAs
# without rows of a factor), every row tile (4, 8, 12, 16), ranks that are not multiples of
# four, and fits of several ranks and shapes in one batch (each keeps the bits of its own fit).
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("jobs", [
    [((64, 5, 64), 4)],
    [((64, 5, 52), 12), ((64, 64, 4), 1), ((4, 64, 64), 4)],
    [((64, 4, 64), 16)],
    [((33, 9, 60), 11), ((26, 31, 27), 5), ((40, 17, 33), 13)]])
def test_core_fits_on_clusters(dt, jobs):
    rng = np.random.default_rng(37)
    probs = [(rng.random(m), inputs.initial_cp(m, r, 11 + i)) for i, (m, r) in enumerate(jobs)]
    dev = [(_dev(G, dt), [_dev(b, dt) for b in B]) for G, B in probs]
    errs = native.nncp_core_fit_batched(dev, 5).cpu().numpy()
    tol = _TOL[dt]
    for (G, B0), (Gd, B), e in zip(probs, dev, errs):
        Gr = Gd.double().cpu().numpy()
        Bo, tro = orc.nncp_fit(Gr, [_dev(b, dt).double().cpu().numpy() for b in B0], 5)
        for a, b in zip(B, Bo):
            np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
        assert e == pytest.approx(tro[-1], abs=tol)
        one = [_dev(b, dt) for b in B0]
        assert native.nncp_core_fit(Gd, one, 5) == e
        assert all(torch.equal(a, b) for a, b in zip(one, B))


# A core fit in shared memory has the bits of the form that reads the core through L1, which a
# zero column beyond rank 16 asks for: the column stays zero and adds exact zeros to every
# sum.
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("m,r", [((7, 8, 6), 3), ((4, 15, 9), 8), ((16, 3, 5), 5), ((2, 13, 7), 16),
                                 ((1, 1, 1), 1), ((9, 4, 33), 11)])
def test_core_fit_keeps_the_bits_of_the_general_form(dt, m, r):
    rng = np.random.default_rng(41)
    G = _dev(rng.random(m), dt)
    B = [_dev(b, dt) for b in inputs.initial_cp(m, r, 13)]
    wide = [torch.nn.functional.pad(b, (0, 17 - r)).contiguous() for b in B]
    e, ew = native.nncp_core_fit(G, B, 60), native.nncp_core_fit(G, wide, 60)
    assert e == ew
    for a, b in zip(B, wide):
        assert torch.equal(a, b[:, :r]) and not b[:, r:].any()


# Data and factors beyond the range of the FP16 pairs (28 powers of two below the largest entry
# of a slice or column): every sum is of nonnegative terms, so FP32-accurate arithmetic keeps the
# relative error of every entry: 1e-4 a sweep, as in the other one-sweep tests.
def _f32(a):
    return np.asarray(a).astype(np.float32).astype(np.float64)


def _entrywise(dev, ref, tol):
    for a, b in zip(dev, ref):
        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=tol, atol=1e-30)


@pytest.mark.parametrize("spike", [1e8, 1e12])
def test_pair_range_one_large_entry(spike):
    rng = np.random.default_rng(43)
    X = rng.random((64, 64, 64))
    X[11, 23, 42] = spike
    X, F0 = _f32(X), [_f32(1 - rng.random((64, 10))) for _ in range(3)]
    G0 = _f32(1 - rng.random((10, 10, 10)))
    F, G = [_dev(f, torch.float32) for f in F0], _dev(G0, torch.float32)
    native.ntd_fit(_dev(X, torch.float32), F, G, 3)
    Fo, Go, _ = orc.ntd_fit(X, F0, G0, 3)
    _entrywise(F + [G], list(Fo) + [Go], 3e-4)


# X in three blocks along its first and last mode, and a factor that is smaller by 1e12 on each
# block's slices than on the one's before: every term of a later block's numerators is tiny, and
# none may be lost beside the first block's.
def _three_blocks(dims, seed):
    rng = np.random.default_rng(seed)
    X = rng.random(dims)
    b = [np.arange(n) * 3 // n for n in dims]
    X *= (b[0][:, None] == b[-1][None, :]).reshape(dims[0], *[1] * (len(dims) - 2), dims[-1])
    return _f32(X), b, rng


@pytest.mark.parametrize("tiny", [0, -1])
@pytest.mark.parametrize("call,dims,m", [
    ("ntd", (48, 40, 68), (9, 10, 11)), ("ntd7", (48, 40, 68), (9, 10, 11)),
    ("ntd", (24, 128, 72), (9, 20, 32)),       # the fused contraction
    ("ntd", (130, 20, 132), (33, 5, 40)),      # columns of 64
    ("ntd4", (20, 12, 14, 36), (9, 10, 11, 12)), ("ntd4x3", (20, 12, 14, 36), (9, 10, 11, 12)),
    ("cp", (48, 40, 68), (9, 9, 9)), ("cp3", (48, 40, 68), (9, 9, 9))])
def test_pair_range_wide_factors(call, dims, m, tiny):
    X, b, rng = _three_blocks(dims, 47)
    iters = {"ntd7": 7, "ntd4x3": 3, "cp3": 3}.get(call, 1)
    F0 = [1 - rng.random((n, k)) for n, k in zip(dims, m)]
    F0[tiny] *= 10.0 ** (-12 * b[tiny])[:, None]
    F0, Xd = [_f32(f) for f in F0], _dev(X, torch.float32)
    F = [_dev(f, torch.float32) for f in F0]
    if call.startswith("cp"):
        err, tr = native.nncp_tensor_fit(Xd, F, iters)
        Fo, tro = orc.nncp_fit(X, F0, iters)
        out, ref = F, list(Fo)
    else:
        G0 = _f32(1 - rng.random(m))
        G = _dev(G0, torch.float32)
        err, tr = native.ntd_fit(Xd, F, G, iters)
        Fo, Go, tro = orc.ntd_fit(X, F0, G0, iters)
        out, ref = F + [G], list(Fo) + [Go]
    _entrywise(out, ref, 1e-4 * iters)
    np.testing.assert_allclose(tr.cpu().numpy(), tro, rtol=0, atol=1e-5)


def test_pair_range_lifted_gradient():
    dims, m, r = (48, 40, 68), (9, 10, 11), 5
    X, b, rng = _three_blocks(dims, 53)
    F = [1 - rng.random((n, k)) for n, k in zip(dims, m)]
    B = [_f32(1 - rng.random((k, r))) for k in m]
    F[0][b[0] > 0] = 0.0  # A^(1) is zero there and the gradient -MT B^T: nonnegative sums
    F[2] *= 10.0 ** (-12 * b[2])[:, None]
    F = [_f32(f) for f in F]
    _, gF, _ = native.candelinc_lifted_grad(_dev(X, torch.float32),
                                            [_dev(f, torch.float32) for f in F],
                                            [_dev(v, torch.float32) for v in B])
    gFo, _ = orc.lifted_loss_grad(X, F, B)
    np.testing.assert_allclose(gF[0].cpu().numpy()[b[0] > 0], gFo[0][b[0] > 0], rtol=1e-4)


# The same through the other pass, with slices and columns so small that the products of the two
# scales leave the normal floats: such a column is left whole for the second round.
def test_pair_range_small_columns():
    dims, m, r = (48, 40, 68), (9, 10, 11), 5
    X, b, rng = _three_blocks(dims, 79)
    X = _f32(X * 1e-15)
    F = [1 - rng.random((n, k)) for n, k in zip(dims, m)]
    B = [_f32(1 - rng.random((k, r))) for k in m]
    F[2][b[2] > 0] = 0.0
    F[0] *= 10.0 ** (-6 - 6 * b[0])[:, None]
    F = [_f32(f) for f in F]
    _, gF, _ = native.candelinc_lifted_grad(_dev(X, torch.float32),
                                            [_dev(f, torch.float32) for f in F],
                                            [_dev(v, torch.float32) for v in B])
    gFo, _ = orc.lifted_loss_grad(X, F, B)
    np.testing.assert_allclose(gF[2].cpu().numpy()[b[2] > 0], gFo[2][b[2] > 0], rtol=1e-4)


# The pairs are left after the first step (an X of wide range), and every step counts once: four
# steps have the bits of twice two.
@pytest.mark.parametrize("dims", [(48, 40, 68), (12, 10, 9, 16)])
def test_pair_range_projected_gradient(dims):
    rng = np.random.default_rng(59)
    m, r = (9, 10, 11, 7)[:len(dims)], 5
    X = rng.random(dims)
    X[(3,) * len(dims)] = 1e10
    X = _dev(X, torch.float32)
    F0 = [_dev(1 - rng.random((n, k)), torch.float32) for n, k in zip(dims, m)]
    B0 = [_dev(1 - rng.random((k, r)), torch.float32) for k in m]
    F, B = [f.clone() for f in F0], [b.clone() for b in B0]
    loss, tr = native.candelinc_pg_fit(X, F, B, 4)
    F2, B2 = [f.clone() for f in F0], [b.clone() for b in B0]
    _, tr2 = native.candelinc_pg_fit(X, F2, B2, 2)
    loss2, tr3 = native.candelinc_pg_fit(X, F2, B2, 2)
    assert loss == loss2 and torch.equal(tr, torch.cat([tr2, tr3]))
    for a, b in zip(F + B, F2 + B2):
        assert torch.equal(a, b)


# Factors that leave the range of one round late in a long fit (between sweeps 250 and 300 on
# these data), which then goes on with the other passes. The trace to 1e-5, as everywhere on the
# FP32 path.
def test_pair_range_left_late():
    dims, m, iters = (48, 40, 68), (9, 10, 11), 620
    rng = np.random.default_rng(7)
    X = np.zeros(dims)
    X[:24, :, :34] = rng.random((24, 40, 34))
    X[24:, :, 34:] = rng.random((24, 40, 34))
    X = _f32(X + 0.08 * rng.random(dims))
    F0, G0 = [_f32(1 - rng.random((n, k))) for n, k in zip(dims, m)], _f32(1 - rng.random(m))
    F, G = [_dev(f, torch.float32) for f in F0], _dev(G0, torch.float32)
    err, tr = native.ntd_fit(_dev(X, torch.float32), F, G, iters, exact_every=60)
    Fo, Go, tro = orc.ntd_fit(X, F0, G0, iters)
    least = min((np.where(f > 0, f, np.inf) / f.max(0)).min() for f in Fo)
    assert least < 2.0 ** -28
    np.testing.assert_allclose(tr.cpu().numpy(), tro, rtol=0, atol=1e-5)
    assert abs(err - orc.rel_err_tucker(X, Go, Fo)) <= 1e-5


# The tensor-core passes on shapes that no one-cluster fit takes (a multirank above 8): pairs with
# the fused contraction over two tiles a slab, on data whose magnitudes are no product of
# scales; and operands past what a block holds, which run as TF32x3: with the mode-3 shares formed
# by the pass (N2 % 128 == 0, N3 > 768 or N1 > 1024), without them, and with columns of 64
# (N1 > 512). One sweep to 1e-4 elementwise, as the pair passes above.
@pytest.mark.parametrize("dims,m,scaled", [
    ((3, 256, 4), (9, 3, 4), True), ((20, 128, 68), (10, 12, 9), True),
    ((17, 128, 900), (12, 10, 12), False), ((1100, 128, 8), (9, 6, 4), False),
    ((1030, 9, 20), (9, 4, 4), False), ((600, 9, 20), (40, 4, 4), True)])
def test_passes_past_the_cluster_and_the_pairs(dims, m, scaled):
    X, _, F0, G0, _ = inputs.small_problem(dims, 3, m, 2, seed=97)
    if scaled:
        X = X * 10.0 ** np.random.default_rng(61).uniform(-2, 2, dims)
    X, F0, G0 = _f32(X), [_f32(f) for f in F0], _f32(G0)
    F, G = [_dev(f, torch.float32) for f in F0], _dev(G0, torch.float32)
    err, _ = native.ntd_fit(_dev(X, torch.float32), F, G, 1, precision="fp32")
    Fo, Go, _ = orc.ntd_fit(X, F0, G0, 1)
    _entrywise(F + [G], list(Fo) + [Go], 1e-4)
    assert abs(err - orc.rel_err_tucker(X, Go, Fo)) <= 1e-5


# The sweep of separate kernels on small and degenerate shapes: a multirank above 8 keeps them off
# the cluster. Three sweeps, no sweep, and a fit whose residual overflows.
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("dims,m", [((1, 7, 12), (1, 2, 9)),
                                    ((12, 40, 1), (10, 3, 1)), ((37, 29, 23), (9, 6, 7)),
                                    ((5, 61, 201), (3, 9, 3))])
def test_separate_kernels_on_small_shapes(dt, dims, m):
    X, _, F0, G0, _ = inputs.small_problem(dims, 2, m, 2, seed=67)
    X, F0, G0 = (_dev(X, dt).double().cpu().numpy(),
                 [_dev(f, dt).double().cpu().numpy() for f in F0],
                 _dev(G0, dt).double().cpu().numpy())
    F, G = [_dev(f, dt) for f in F0], _dev(G0, dt)
    err, tr = native.ntd_fit(_dev(X, dt), F, G, 3)
    Fo, Go, tro = orc.ntd_fit(X, F0, G0, 3)
    tol = _TOL[dt]
    for a, b in zip(F + [G], Fo + [Go]):
        np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
    np.testing.assert_allclose(tr.cpu().numpy(), tro, rtol=0,
                               atol=(1e-8 if dt == torch.float64 else 1e-5) * max(1.0, tro.max()))
    F, G = [_dev(f, dt) for f in F0], _dev(G0, dt)
    err, _ = native.ntd_fit(_dev(X, dt), F, G, 0)
    assert err == pytest.approx(orc.rel_err_tucker(X, G0, F0), abs=tol)
    assert all(torch.equal(f, _dev(b, dt)) for f, b in zip(F + [G], F0 + [G0]))


def test_separate_kernels_report_an_overflow():
    X, _, F0, G0, _ = inputs.small_problem((24, 20, 16), 3, (9, 4, 4), 2, seed=21)
    with pytest.raises(native.NncError) as ei:
        native.ntd_fit(_dev(X * 1e30, torch.float32), [_dev(f, torch.float32) for f in F0],
                       _dev(G0, torch.float32), 10)
    assert ei.value.status == -3 and "sweep" in str(ei.value)


# Cluster core fits near and past the shared memory of a CTA: the slab of the second product
# there and, where it does not fit, read in place. Bounds as for the other cluster fits.
@pytest.mark.parametrize("dt,m,r", [(torch.float64, (38, 44, 53), 1), (torch.float64, (45, 33, 62), 1),
                                    (torch.float64, (59, 26, 56), 5), (torch.float64, (64, 17, 60), 13),
                                    (torch.float32, (61, 53, 52), 5), (torch.float32, (64, 63, 64), 4)])
def test_cluster_core_fits_at_the_shared_memory_limit(dt, m, r):
    rng = np.random.default_rng(71)
    G, B0 = rng.random(m), inputs.initial_cp(m, r, 17)
    B = [_dev(b, dt) for b in B0]
    err = native.nncp_core_fit(_dev(G, dt), B, 5)
    Bo, tro = orc.nncp_fit(_dev(G, dt).double().cpu().numpy(),
                           [_dev(b, dt).double().cpu().numpy() for b in B0], 5)
    tol = _TOL[dt]
    for a, b in zip(B, Bo):
        np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
    assert err == pytest.approx(tro[-1], abs=tol)


# Wide factors beside data without small entries: every sum has terms of the column's largest
# entry, and no more rounds are taken. Bounds as above.
@pytest.mark.parametrize("dims,m", [((48, 40, 68), (9, 10, 11)), ((24, 128, 72), (9, 20, 32)),
                                    ((12, 10, 14, 36), (9, 10, 11, 12))])
def test_pair_range_wide_factors_beside_dense_data(dims, m):
    rng = np.random.default_rng(73)
    X = _f32(0.25 + rng.random(dims))
    F0 = [_f32((1 - rng.random((n, k))) * 10.0 ** rng.uniform(-30, 0, (n, 1)))
          for n, k in zip(dims, m)]
    G0 = _f32(1 - rng.random(m))
    F, G = [_dev(f, torch.float32) for f in F0], _dev(G0, torch.float32)
    native.ntd_fit(_dev(X, torch.float32), F, G, 1)
    Fo, Go, _ = orc.ntd_fit(X, F0, G0, 1)
    for a, b in zip(F + [G], list(Fo) + [Go]):  # (FP32 ends at 1e-38)
        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=1e-4, atol=1e-30)
