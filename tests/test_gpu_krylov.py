"""GPU Krylov drivers (pjds_cg_solve, pjds_lanczos, pjds_ritz_refine) against
the fp64 oracles. Solvers run in the permuted basis; results are mapped back
to the original basis with the permutation before every comparison.

Tolerances:
  CG (fp64 or refined mixed precision): the fp64 residual ||b - A x|| / ||b||,
    evaluated by the oracle's CRS product, <= 1e-12, and x within 1e-11
    (relative, max norm) of the oracle's fp64 CG solution (both are converged:
    the stencil matrices here have condition numbers near 25).
  Lanczos fp64: alpha_j, beta_j within 1e-10 (relative) of the oracle for the
    first 15 steps (rounding differences grow once orthogonality is lost),
    the extreme Ritz value within 1e-12.
  Lanczos fp32/bf16 values with fp32 vectors: extreme Ritz value within 1e-5
    (relative) of the fp64 oracle run on the same rounded values; the
    fp64-refined Rayleigh quotient within 1e-6 (fp32) / 5e-3 (bf16) of the
    fp64 oracle on the exact matrix, and its residual equal to the oracle's
    recomputation within 1e-6.
"""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1112_5588_gb300 import build
    build.build()
    from paper_1112_5588_gb300 import krylov, pjds
    return torch, pjds, krylov


def _dev(pjds, A, dtype):
    H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype, permute_cols=True)
    perm = H.perm.copy()
    return H.to_device("cuda"), perm


@pytest.fixture(scope="module")
def stencil():
    return synth.stencil27(g=20, p_drop=0.1, seed=7)


def _true_rel_residual(oracle_lib, A, x, b):
    return float(np.linalg.norm(b - oracle_lib.crs_spmv(A, x)) / np.linalg.norm(b))


@pytest.mark.parametrize("lo,max_outer,inner", [(None, 1, 300), ("f32", 6, 50), ("bf16", 20, 25)])
@pytest.mark.parametrize("graph", [True, False])
def test_cg_matches_fp64_oracle(mods, oracle_lib, stencil, lo, max_outer, inner, graph):
    torch, pjds, krylov = mods
    from oracle import krylov as ok
    A = stencil
    b = synth.vector(A.n_rows, seed=3)
    D64, perm = _dev(pjds, A, "f64")
    Dlo = _dev(pjds, A, lo)[0] if lo else None
    bp = torch.from_numpy(b[perm]).cuda()
    xp = torch.zeros_like(bp)
    res = krylov.cg_solve(D64, Dlo, bp, xp, max_outer=max_outer, inner_iters=inner, use_graph=graph)
    x = np.empty(A.n_rows)
    x[perm] = xp.cpu().numpy()
    rel = _true_rel_residual(oracle_lib, A, x, b)
    assert rel <= 1e-12, (rel, res)
    assert res["rel_residual"] == pytest.approx(rel, rel=1e-3, abs=1e-15)
    x_ref, _ = ok.cg(A, b, 300)
    assert np.max(np.abs(x - x_ref)) <= 1e-11 * np.max(np.abs(x_ref))
    h = res["history"]
    assert h[0] == pytest.approx(1.0) and h[-1] < 1e-12


def test_cg_is_deterministic(mods, stencil):
    # also with use_graph, which is accepted and changes nothing
    torch, pjds, krylov = mods
    A = stencil
    b = synth.vector(A.n_rows, seed=5)
    D64, perm = _dev(pjds, A, "f64")
    D32, _ = _dev(pjds, A, "f32")
    bp = torch.from_numpy(b[perm]).cuda()
    outs = []
    for graph in (True, True, False):
        xp = torch.zeros_like(bp)
        krylov.cg_solve(D64, D32, bp, xp, max_outer=3, inner_iters=20, use_graph=graph)
        outs.append(xp.cpu().numpy())
    assert np.array_equal(outs[0].view(np.uint64), outs[1].view(np.uint64))
    assert np.array_equal(outs[0].view(np.uint64), outs[2].view(np.uint64))


def test_cg_rejects_bad_arguments(mods, stencil):
    torch, pjds, krylov = mods
    A = stencil
    H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype="f64")  # not permuted
    D = H.to_device("cuda")
    v = torch.zeros(A.n_rows, dtype=torch.float64, device="cuda")
    with pytest.raises(pjds.PjdsError):
        krylov.cg_solve(D, None, v, v.clone())
    D32, _ = _dev(pjds, A, "f32")
    with pytest.raises(pjds.PjdsError):  # A_hi must be fp64
        krylov.cg_solve(D32, None, v, v.clone())


def test_lanczos_fp64_matches_oracle(mods, oracle_lib):
    torch, pjds, krylov = mods
    from oracle import krylov as ok
    A = synth.stencil27(g=16, seed=4)
    v0 = synth.vector(A.n_rows, seed=8)
    D, perm = _dev(pjds, A, "f64")
    k = 60
    alpha, beta, V = krylov.lanczos(D, torch.from_numpy(v0[perm]).cuda(), k, keep_basis=True)
    ra, rb, _ = ok.lanczos(A, v0, k)
    assert np.allclose(alpha[:15], ra[:15], rtol=1e-10, atol=0)
    assert np.allclose(beta[1:16], rb[1:16], rtol=1e-10, atol=0)
    assert beta[0] == 0.0
    th, _ = krylov.tridiag_extreme(alpha, beta)
    assert th == pytest.approx(ok.tridiag_eigvals(ra, rb)[-1], rel=1e-12)
    Vh = V.cpu().numpy()[:10]
    assert np.allclose(Vh @ Vh.T, np.eye(10), atol=1e-10)


def test_lanczos_is_deterministic(mods):
    # also with use_graph, which is accepted and changes nothing
    torch, pjds, krylov = mods
    A = synth.stencil27(g=12, seed=4)
    D, perm = _dev(pjds, A, "f32")
    v0 = torch.from_numpy(synth.vector(A.n_rows, seed=2)[perm].astype(np.float32)).cuda()
    a1, b1, _ = krylov.lanczos(D, v0, 40, use_graph=True)
    a2, b2, _ = krylov.lanczos(D, v0, 40, use_graph=False)
    assert np.array_equal(a1, a2) and np.array_equal(b1, b2)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_lanczos_low_precision_with_fp64_ritz_refinement(mods, oracle_lib, dtype):
    torch, pjds, krylov = mods
    from oracle import krylov as ok
    A = synth.stencil27(g=16, seed=4)
    v0 = synth.vector(A.n_rows, seed=8)
    Dlo, perm = _dev(pjds, A, dtype)
    D64, _ = _dev(pjds, A, "f64")
    k = 80
    alpha, beta, V = krylov.lanczos(Dlo, torch.from_numpy(v0[perm].astype(np.float32)).cuda(), k, keep_basis=True)
    ra, rb, RV = ok.lanczos(A, v0, k, keep_basis=True)
    th_ref, y_ref = ok.ritz_pair(ra, rb, RV)
    th, s = krylov.tridiag_extreme(alpha, beta)
    # the fp32 recurrence sees the dtype-rounded matrix: compare against the
    # oracle on the same rounded values for the unrefined Ritz value
    Ar = A._replace(val=oracle_lib.round_f32(A.val) if dtype == "f32" else oracle_lib.round_bf16(A.val))
    ra_r, rb_r, _ = ok.lanczos(Ar, v0, k)
    th_r = ok.tridiag_eigvals(ra_r, rb_r)[-1]
    assert th == pytest.approx(th_r, rel=1e-5)
    y, th_ref64, resid = krylov.ritz_refine(D64, V, s)
    # the Ritz vector approximates an eigenvector of the rounded matrix; its
    # fp64 Rayleigh quotient errs by about (rounding * ||A|| / gap)^2 * ||A||:
    # ~1e-10 relative for fp32 values, ~1e-3 for bf16 on this spectrum
    assert th_ref64 == pytest.approx(th_ref, rel=1e-6 if dtype == "f32" else 5e-3)
    yo = np.empty(A.n_rows)
    yo[perm] = y.cpu().numpy()
    r_or = np.linalg.norm(oracle_lib.crs_spmv(A, yo) - th_ref64 * yo) / np.linalg.norm(yo) / abs(th_ref64)
    assert resid == pytest.approx(r_or, rel=1e-6, abs=1e-14)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_lanczos_basis_rows_of_odd_length(mods, oracle_lib, dtype):
    # n = 17^3 = 4913: basis row j starts j * n elements in, so most rows are
    # not 16-byte aligned and take the element-wise stores; keeping the basis
    # changes no arithmetic, and the stored rows are the Lanczos vectors
    torch, pjds, krylov = mods
    from oracle import krylov as ok
    A = synth.stencil27(g=17, seed=5)
    assert A.n_rows % 2 == 1
    v0 = synth.vector(A.n_rows, seed=9)
    D, perm = _dev(pjds, A, dtype)
    v0t = torch.from_numpy(v0[perm]).to("cuda", D.vec_dtype)
    k = 30
    a1, b1, V = krylov.lanczos(D, v0t, k, keep_basis=True)
    a2, b2, _ = krylov.lanczos(D, v0t, k, keep_basis=False)
    assert np.array_equal(a1, a2) and np.array_equal(b1, b2)
    Vh = V.double().cpu().numpy()
    v0n = v0t.double().cpu().numpy()
    assert np.allclose(Vh[0], v0n / np.linalg.norm(v0n), rtol=0, atol=1e-6 if dtype == "f32" else 1e-15)
    G = Vh[:8] @ Vh[:8].T
    assert np.allclose(G, np.eye(8), atol=1e-5 if dtype == "f32" else 1e-10)
    if dtype == "f64":
        ra, rb, _ = ok.lanczos(A, v0, k)
        assert np.allclose(a1[:10], ra[:10], rtol=1e-10, atol=0)


def _spd(name, n):
    """Symmetric, strictly diagonally dominant: `tri` three diagonals and empty
    couplings every 13 rows (rows of 1 to 3 entries), `arrow` a dense first row
    and column beside the diagonal (one row of n entries)."""
    i = np.arange(n)
    if name == "tri":
        off = np.where(np.arange(n - 1) % 13 == 5, 0.0, -1.0 / (1 + np.arange(n - 1) % 7))
        keep = np.nonzero(off)[0]
        r, c = np.concatenate([keep, keep + 1]), np.concatenate([keep + 1, keep])
        v = np.concatenate([off[keep], off[keep]])
        d = np.full(n, 3.0)
    else:
        r, c = np.concatenate([np.zeros(n - 1, int), i[1:]]), np.concatenate([i[1:], np.zeros(n - 1, int)])
        v = np.full(2 * (n - 1), 1.0 / n)
        d = np.full(n, 2.0)
    r, c, v = np.concatenate([r, i]), np.concatenate([c, i]), np.concatenate([v, d])
    o = np.lexsort((c, r))
    ptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    return synth.Crs(n, n, ptr, c[o].astype(np.int32), v[o])


# one launch for the solve: sizes at the edges of a warp's rows (32, 16, 8 for 1,
# 2, 4 threads per row) and of the rule that takes it (512 rows per SM without
# the matrix in shared memory: the arrow's long row); beyond it a launch a step
@pytest.mark.parametrize("lo,max_outer", [(None, 3), ("f32", 6), ("bf16", 12)])
@pytest.mark.parametrize("name,n", [("tri", 1), ("tri", 7), ("tri", 8), ("tri", 33), ("tri", 4097), ("tri", 40001),
                                    ("tri", 77857), ("arrow", 2), ("arrow", 3001), ("arrow", 77001),
                                    ("arrow", 78001)])
def test_cg_small_and_large_systems(mods, oracle_lib, name, n, lo, max_outer):
    torch, pjds, krylov = mods
    A = _spd(name, n)
    b = synth.vector(n, seed=n)
    D64, perm = _dev(pjds, A, "f64")
    Dlo = _dev(pjds, A, lo)[0] if lo else None
    bp = torch.from_numpy(b[perm]).cuda()
    x1, x2 = torch.zeros_like(bp), torch.zeros_like(bp)
    res = krylov.cg_solve(D64, Dlo, bp, x1, max_outer=max_outer, inner_iters=20, tol=1e-13)
    krylov.cg_solve(D64, Dlo, bp, x2, max_outer=max_outer, inner_iters=20, tol=1e-13)
    assert torch.equal(x1, x2)
    x = np.empty(n)
    x[perm] = x1.cpu().numpy()
    # kappa below 5: 20 steps reduce the error by ((sqrt 5 - 1) / (sqrt 5 + 1))^20 < 1e-8 or to the inner
    # type's rounding, and the outer steps repeat it until the residual is at 1e-13 (rounding of b - A x
    # in fp64: a few 1e-16 times (|A||x| + |b|) / |b| < 10)
    rel = _true_rel_residual(oracle_lib, A, x, b)
    assert rel <= 1e-12, (rel, res)
    assert res["rel_residual"] <= 1e-12 and res["inner_total"] == 20 * res["outer"]
    assert len(res["history"]) == res["outer"] + 1 and res["history"][-1] == res["rel_residual"]


# more rows than the one launch takes (512 per SM; the arrow's long row keeps the matrix out of shared memory) with
# every remainder of the vector kernels' 16-byte groups: a launch for every step, to the fp64 residual, twice the
# same bits
@pytest.mark.parametrize("lo,max_outer", [(None, 3), ("f32", 6), ("bf16", 12)])
@pytest.mark.parametrize("more", [1, 178, 1027])
def test_cg_larger_than_one_launch(mods, oracle_lib, more, lo, max_outer):
    torch, pjds, krylov = mods
    n = 512 * torch.cuda.get_device_properties(0).multi_processor_count + more
    A = _spd("arrow", n)
    b = synth.vector(n, seed=more)
    D64, perm = _dev(pjds, A, "f64")
    Dlo = _dev(pjds, A, lo)[0] if lo else None
    bp = torch.from_numpy(b[perm]).cuda()
    xs = [torch.zeros_like(bp) for _ in range(2)]
    for xp in xs:
        res = krylov.cg_solve(D64, Dlo, bp, xp, max_outer=max_outer, inner_iters=20, tol=1e-13)
    assert torch.equal(*xs)
    x = np.empty(n)
    x[perm] = xs[0].cpu().numpy()
    assert max(_true_rel_residual(oracle_lib, A, x, b), res["rel_residual"]) <= 1e-12  # (as above)


# vectors far outside the range in which fp32 holds a product and its rounding
# error: powers of two scale every step exactly, so the coefficients follow
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("power", [-70, 80])
def test_lanczos_scales_with_the_matrix(mods, dtype, power):
    torch, pjds, krylov = mods
    A = synth.stencil27(g=13, seed=6)  # 2197 rows: a remainder after the 16-byte groups
    v0 = synth.vector(A.n_rows, seed=3)
    D, perm = _dev(pjds, A, dtype)
    S, _ = _dev(pjds, A._replace(val=A.val * 2.0 ** power), dtype)
    v = torch.from_numpy(v0[perm]).to("cuda", D.vec_dtype)
    a1, b1, V1 = krylov.lanczos(D, v, 6, keep_basis=True)
    a2, b2, V2 = krylov.lanczos(S, v, 6, keep_basis=True)
    # in fp64 every operation scales exactly; with floats a sum is taken in another way, within its rounding
    # (2^-45) before the vectors' own (2^-24), which six steps amplify by less than 10
    tol = 1e-13 if dtype == "f64" else 1e-6
    assert np.allclose(a2 * 2.0 ** -power, a1, rtol=tol, atol=tol * np.abs(a1).max())
    assert np.allclose(b2 * 2.0 ** -power, b1, rtol=tol, atol=0)
    assert float((V1.double() - V2.double()).abs().max()) <= tol


def test_reduction_of_many_partial_sums_keeps_fp64(mods, oracle_lib):
    # 17,000 partial sums (1.1M rows, a group of rows per CTA) through the Ritz refinement, whose Rayleigh
    # quotient the oracle recomputes from the returned vector: y is one basis row, so theta = (v, A v) / (v, v)
    torch, pjds, krylov = mods
    A = synth.stencil27(g=103, seed=4)
    D, perm = _dev(pjds, A, "f64")
    v = synth.vector(A.n_rows, seed=12)
    y, theta, _ = krylov.ritz_refine(D, torch.from_numpy(v[perm]).cuda().reshape(1, -1), np.ones(1))
    assert torch.equal(y, torch.from_numpy(v[perm]).cuda())
    want = float(np.sum(v.astype(np.longdouble) * oracle_lib.crs_spmv(A, v)) / np.sum(v.astype(np.longdouble) ** 2))
    # two sums of 1.1M products, each in fp64 within a few ulps of the exact one (they are added in trees),
    # and the products' own rounding: 2^-53 on average over the rows, far below 1e-14
    assert theta == pytest.approx(want, rel=1e-14)


# a NaN or an infinity of a matrix row reaches the inner product that this row is part of, also where the other
# factor is zero (0 * inf is NaN), in every value type and on one CTA's rows as on many
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n", [5, 4097])
def test_lanczos_keeps_a_nan_beside_a_zero(mods, dtype, bad, n):
    torch, pjds, krylov = mods
    A = _spd("tri", n)
    row = 3
    val = A.val.copy()
    val[A.row_ptr[row]] = bad  # its coupling with row 2
    D, perm = _dev(pjds, A._replace(val=val), dtype)
    v0 = np.ones(n)
    v0[row] = 0.0
    alpha, beta, _ = krylov.lanczos(D, torch.from_numpy(v0[perm]).to("cuda", D.vec_dtype), 1)
    assert np.isnan(alpha[0]) and np.isnan(beta[1])


# a NaN in the start vector reaches every coefficient, and every element of the next vector
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_lanczos_from_a_nan(mods, dtype):
    torch, pjds, krylov = mods
    A = _spd("tri", 1029)
    D, perm = _dev(pjds, A, dtype)
    v0 = torch.ones(A.n_rows, dtype=D.vec_dtype, device="cuda")
    v0[::2] = 0.0
    v0[77] = float("nan")
    alpha, beta, V = krylov.lanczos(D, v0, 2, keep_basis=True)
    assert np.isnan(alpha).all() and np.isnan(beta[1:]).all()
    assert bool(torch.isnan(V[1]).all())


def _diagonal(pjds, d, dtype):
    n = len(d)
    A = synth.Crs(n, n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.asarray(d, np.float64))
    return _dev(pjds, A, dtype)[0]  # rows of one length: the sort keeps their order


# sums whose terms differ much in size are rounded to nearest at every level: a warp's, a CTA's and all CTAs' sums
# of one large term and many small negative ones, each below half of the large one's last bit (rounded down, 31 of
# them would take 4 of its last bits)
@pytest.mark.parametrize("n", [32, 250, 4096, 70_001])
@pytest.mark.parametrize("small", [2.0 ** -54, 2.0 ** -58, 2.0 ** -70, 2.0 ** -300])
def test_fp64_sums_of_terms_of_mixed_size(mods, n, small):
    torch, pjds, krylov = mods
    d = np.full(n, -small / n)
    d[n // 2] = 1.0
    alpha, _, V = krylov.lanczos(_diagonal(pjds, d, "f64"), torch.ones(n, dtype=torch.float64, device="cuda"), 1,
                                 keep_basis=True)
    v = V[0].cpu().numpy()
    terms = v * (d * v)
    # a few roundings of the sum itself at 2^-53 and of a warp's and the CTAs' terms below that
    assert abs(alpha[0] - math.fsum(terms)) <= 2 * 2.0 ** -53 * math.fsum(np.abs(terms))


# fp32 inner products are as good as sums in fp64: alpha = (v, A v) of a diagonal A, whose elements v_i (d_i v_i)
# are known to the last bit. Few rows (two products a thread, where a sum in twice fp32's precision alone errs by
# up to 2^-48 of the terms) and so many that a thread adds more than it keeps before it moves the sum to fp64
@pytest.mark.parametrize("n,runs", [(2, 200), (7, 100), (700, 20), (9_000_001, 1)])
def test_fp32_inner_products_keep_fp64_sums(mods, n, runs):
    torch, pjds, krylov = mods
    for seed in range(runs):
        rng = np.random.default_rng(seed)
        d = (rng.uniform(0.5, 1.5, n) * np.where(rng.random(n) < 0.5, -1, 1)).astype(np.float32)
        v0 = torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).cuda()
        alpha, _, V = krylov.lanczos(_diagonal(pjds, d, "f32"), v0, 1, keep_basis=True)
        v = V[0].cpu().numpy()
        terms = v.astype(np.float64) * (d * v).astype(np.float64)  # exact: 48 bits
        # roundings: a thread's three floats to a double, its warp's, CTA's and the launch's sums, each within
        # a few 2^-53 of the terms
        assert abs(alpha[0] - math.fsum(terms)) <= 8 * 2.0 ** -53 * math.fsum(np.abs(terms)), seed


# the Lanczos vectors of floats are the fp64 expressions rounded once, also where that rounding is decided by the
# last bits: with a diagonal A every element can be computed again (scaled, 1 / beta is near the end of fp32's range)
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 112])
def test_fp32_lanczos_vectors_are_rounded_once(mods, scale):
    torch, pjds, krylov = mods
    n = 4_200_001
    g = torch.Generator("cuda").manual_seed(5)
    d = (torch.rand(n, generator=g, device="cuda") + 0.5) * scale
    v0 = torch.rand(n, generator=g, device="cuda") - 0.5
    steps = 4
    alpha, beta, V = krylov.lanczos(_diagonal(pjds, d.cpu().numpy(), "f32"), v0, steps, keep_basis=True)
    off = 0
    for j in range(steps - 1):
        w = (d * V[j]).double() - alpha[j] * V[j].double()
        if j:
            w -= beta[j] * V[j - 1].double()
        nxt = (w.float().double() * (1.0 / beta[j + 1])).float()
        off += int((nxt != V[j + 1]).sum())
    # torch rounds the two products of the first expression, the kernel does not: that can decide about 2^-26 of
    # the 12.6 million roundings (a difference of 2^-52 of the terms at a boundary of 2^-24)
    assert off <= 1
