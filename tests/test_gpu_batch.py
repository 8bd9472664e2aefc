"""GPU batched products: pjds_spmm against the oracle's block product and,
column by column, bit for bit against pjds_spmv with one thread per row; the
persistent multi-matrix launch against the oracle and the single products."""
import numpy as np
import pytest

import synth
from synth import tiny
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1112_5588_gb300 import build
    build.build()
    from paper_1112_5588_gb300 import batch, pjds
    return torch, pjds, batch


SHAPES = [("dlr", lambda: synth.block_dense(n_brow=3000, bs=4, nb=36, frac=0.05, seed=3)),
          ("zipf", lambda: synth.zipf_rows(20_000, s=2.0, len_max=512, seed=4)),
          ("ragged", lambda: tiny.random_lengths(1037, 900, max_len=70, seed=5, p_empty=0.2))]


@pytest.mark.parametrize("dtype,k", [("f64", 2), ("f64", 8), ("f64", 32), ("f32", 4), ("f32", 16), ("f32", 32),
                                     ("f32", 128), ("bf16", 8)])
@pytest.mark.parametrize("name,make", SHAPES, ids=[s[0] for s in SHAPES])
def test_spmm_matches_oracle_and_columnwise_spmv(mods, oracle_lib, dtype, k, name, make):
    torch, pjds, batch = mods
    A = make()
    X = np.random.default_rng(k).uniform(-1, 1, (A.n_cols, k))
    if dtype != "f64":
        X = X.astype(np.float32).astype(np.float64)
    H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype)
    D = H.to_device("cuda")
    Xt = torch.from_numpy(X).to("cuda", D.vec_dtype).contiguous()
    Yt = torch.full((A.n_rows, k), float("nan"), dtype=D.vec_dtype, device="cuda")
    batch.spmm(D, Xt, Yt)
    torch.cuda.synchronize()
    Y = Yt.double().cpu().numpy()
    Ar = A if dtype == "f64" else A._replace(
        val=oracle_lib.round_f32(A.val) if dtype == "f32" else oracle_lib.round_bf16(A.val))
    Yr = oracle_lib.crs_spmm(Ar, X)
    S = oracle_lib.crs_spmm(Ar._replace(val=np.abs(Ar.val)), np.abs(X))
    lens = np.diff(A.row_ptr)
    check = parity.check_fp64 if dtype == "f64" else parity.check_fp32
    for c in range(k):
        r = check(Y[:, c], Yr[:, c], S[:, c], lens)
        assert r["ok"], (c, r)
    # same arithmetic as the single product, column by column
    for c in (0, k - 1):
        y1 = torch.empty(A.n_rows, dtype=D.vec_dtype, device="cuda")
        pjds.pjds_spmv_cfg(D, Xt[:, c].contiguous(), y1, threads_per_row=1, rows_per_thread=1)
        torch.cuda.synchronize()
        assert torch.equal(y1, Yt[:, c].contiguous())


def test_spmm_permuted_basis_and_k1(mods):
    torch, pjds, batch = mods
    A = synth.stencil27(g=16, seed=2)
    H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype="f32", permute_cols=True)
    D = H.to_device("cuda")
    X = torch.rand(A.n_rows, 8, device="cuda")
    Y = torch.empty_like(X)
    batch.spmm(D, X, Y)
    for c in range(8):
        y1 = torch.empty(A.n_rows, device="cuda")
        pjds.pjds_spmv_cfg(D, X[:, c].contiguous(), y1, threads_per_row=1)
        torch.cuda.synchronize()
        assert torch.equal(y1, Y[:, c].contiguous())
    X1 = X[:, :1].contiguous()
    Y1 = torch.empty(A.n_rows, 1, device="cuda")
    batch.spmm(D, X1, Y1)
    y1 = torch.empty(A.n_rows, device="cuda")
    pjds.pjds_spmv(D, X1.reshape(-1), y1)
    torch.cuda.synchronize()
    assert torch.equal(Y1.reshape(-1), y1)


def test_spmm_rejects_bad_k(mods):
    torch, pjds, batch = mods
    A = tiny.random_lengths(64, 64, max_len=8, seed=1)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, dtype="f32").to_device("cuda")
    for k in (3, 6, 132):
        with pytest.raises(pjds.PjdsError):
            batch.spmm(D, torch.zeros(64, k, device="cuda"), torch.zeros(64, k, device="cuda"))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("graph", [True, False])
def test_batch_uneven_matrices(mods, oracle_lib, dtype, graph):
    torch, pjds, batch = mods
    rng = np.random.default_rng(7)
    sizes = np.exp(rng.uniform(np.log(300), np.log(60_000), 24)).astype(int)
    mats, devs, xs, ys, xh = [], [], [], [], []
    for m, n in enumerate(sizes):
        A = synth.zipf_rows(int(n), s=2.0, len_max=512, seed=100 + m) if m % 3 else \
            tiny.random_lengths(int(n), int(n), max_len=min(40, int(n)), seed=m, p_empty=0.1)
        H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype,
                             permute_cols=(m % 4 == 1))
        D = H.to_device("cuda")
        x = synth.vector(A.n_cols, seed=m)
        if dtype == "f32":
            x = x.astype(np.float32).astype(np.float64)
        xin = x[H.perm] if m % 4 == 1 else x
        mats.append((A, H.perm.copy(), m % 4 == 1))
        devs.append(D)
        xs.append(torch.from_numpy(xin).to("cuda", D.vec_dtype))
        ys.append(torch.full((A.n_rows,), float("nan"), dtype=D.vec_dtype, device="cuda"))
        xh.append(x)
    B = batch.Batch(devs, xs, ys)
    info = B.info()
    # one-lane tiles hold 512 rows (two per thread), 8-lane tiles 32
    assert sum((A.n_rows + 511) // 512 for A, _, _ in mats) <= info["n_tiles"] <= sum(
        (A.n_rows + 31) // 32 for A, _, _ in mats)
    for _ in range(2):
        for y in ys:
            y.fill_(float("nan"))
        B.run(use_graph=graph)
        torch.cuda.synchronize()
        for (A, perm, permuted), x, y, D in zip(mats, xh, ys, devs):
            got = y.double().cpu().numpy()
            if permuted:
                g2 = np.empty_like(got)
                g2[perm] = got
                got = g2
            Ar = A if dtype == "f64" else A._replace(val=oracle_lib.round_f32(A.val))
            check = parity.check_fp64 if dtype == "f64" else parity.check_fp32
            r = check(got, oracle_lib.crs_spmv(Ar, x), oracle_lib.crs_absmv(Ar, x), np.diff(A.row_ptr))
            assert r["ok"], r
    # bit for bit the single product with the built-in rule's lanes: rows whose
    # block has >= 256 entries with 8 threads per row, >= 64 with 4, >= 16 with
    # 2, the others with one thread per row
    for m in (2, 5):
        A, perm, permuted = mats[m]
        H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype, permute_cols=permuted)
        bl = H.block_len[np.arange(A.n_rows) // 32]
        lanes = np.where(bl >= 256, 8, np.where(bl >= 64, 4, np.where(bl >= 16, 2, 1)))
        out_row = np.arange(A.n_rows) if permuted else H.perm  # output row of sorted row i
        want = np.full(A.n_rows, np.nan)
        for t in (1, 2, 4, 8):
            yt = torch.empty_like(ys[m])
            if t == 1:
                pjds.pjds_spmv_cfg(devs[m], xs[m], yt, threads_per_row=1, tile_order=-1)
            else:
                pjds.pjds_spmv_cfg(devs[m], xs[m], yt, threads_per_row=t, unroll=4, tile_order=-1)
            torch.cuda.synchronize()
            want[out_row[lanes == t]] = yt.double().cpu().numpy()[out_row[lanes == t]]
        assert np.array_equal(want, ys[m].double().cpu().numpy()), m
        assert (lanes > 1).any() or m == 2
    B.destroy()


@pytest.mark.parametrize("dtype,k", [("f32", 16), ("f32", 32), ("f64", 8), ("f64", 16)])
def test_spmm_two_chunk_lanes(mods, oracle_lib, dtype, k):
    # 160k rows of 144 entries: enough threads for lanes of two 16-byte chunks;
    # every column against the oracle, and bit for bit against pjds_spmv
    torch, pjds, batch = mods
    A = synth.block_dense(n_brow=40_000, bs=4, nb=36, frac=0.05, seed=11)
    X = np.random.default_rng(k).uniform(-1, 1, (A.n_cols, k))
    if dtype != "f64":
        X = X.astype(np.float32).astype(np.float64)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    Xt = torch.from_numpy(X).to("cuda", D.vec_dtype).contiguous()
    Yt = torch.full((A.n_rows, k), float("nan"), dtype=D.vec_dtype, device="cuda")
    batch.spmm(D, Xt, Yt)
    torch.cuda.synchronize()
    Ar = A if dtype == "f64" else A._replace(val=oracle_lib.round_f32(A.val))
    Yr = oracle_lib.crs_spmm(Ar, X)
    S = oracle_lib.crs_spmm(Ar._replace(val=np.abs(Ar.val)), np.abs(X))
    Y = Yt.double().cpu().numpy()
    check = parity.check_fp64 if dtype == "f64" else parity.check_fp32
    lens = np.diff(A.row_ptr)
    for c in range(k):
        r = check(Y[:, c], Yr[:, c], S[:, c], lens)
        assert r["ok"], (c, r)
    for c in range(k):
        y1 = torch.empty(A.n_rows, dtype=D.vec_dtype, device="cuda")
        pjds.pjds_spmv_cfg(D, Xt[:, c].contiguous(), y1, threads_per_row=1, rows_per_thread=1, tile_order=-1)
        torch.cuda.synchronize()
        assert torch.equal(y1, Yt[:, c].contiguous()), c


def test_batch_given_lanes(mods, oracle_lib):
    # lanes per row given per matrix (as an autotuner would): every row equals
    # the oracle, and bit for bit pjds_spmv_cfg with threads_per_row = lanes
    torch, pjds, batch = mods
    makes = [lambda: synth.zipf_rows(30_000, s=2.0, len_max=300, seed=31),
             lambda: synth.hmep_like(n=40_000, seed=32),
             lambda: tiny.random_lengths(1037, 1037, max_len=90, seed=33, p_empty=0.2),
             lambda: synth.zipf_rows(12_000, s=1.6, len_max=512, seed=34),
             lambda: synth.banded_uniform(n=20_000, seed=35),
             lambda: tiny.random_lengths(333, 500, max_len=40, seed=36)]
    lanes = [1, 2, 4, 8, 0, 2]
    mats, devs, xs, ys = [], [], [], []
    for k, make in enumerate(makes):
        A = make()
        D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32).to_device("cuda")
        mats.append(A)
        devs.append(D)
        xs.append(torch.from_numpy(synth.vector(A.n_cols, seed=k)).cuda())
        ys.append(torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda"))
    B = batch.Batch(devs, xs, ys, lanes=lanes)
    B.run(use_graph=True)
    torch.cuda.synchronize()
    for A, D, x, y, ln in zip(mats, devs, xs, ys, lanes):
        xh = x.cpu().numpy()
        r = parity.check_fp64(y.cpu().numpy(), oracle_lib.crs_spmv(A, xh), oracle_lib.crs_absmv(A, xh),
                              np.diff(A.row_ptr))
        assert r["ok"], (ln, r)
        if ln:
            y1 = torch.empty_like(y)
            pjds.pjds_spmv_cfg(D, x, y1, threads_per_row=ln, unroll=4, tile_order=-1)
            torch.cuda.synchronize()
            assert torch.equal(y1, y), ln
    B.destroy()
    with pytest.raises(pjds.PjdsError):
        batch.Batch(devs, xs, ys, lanes=[1, 2, 3, 8, 0, 2])


def test_batch_rule_and_rule_tuner(mods, oracle_lib):
    # tiles by a block-length rule: every rule gives oracle-exact rows; the
    # built-in rule given explicitly is bit for bit the default plan; the
    # tuner times each rule and picks the fastest
    torch, pjds, batch = mods
    mats, devs, xs, ys = [], [], [], []
    for k in range(10):
        A = synth.zipf_rows(int(5_000 + 7_000 * k), s=1.8 + 0.05 * k, len_max=400, seed=60 + k)
        devs.append(pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32).to_device("cuda"))
        xs.append(torch.from_numpy(synth.vector(A.n_cols, seed=k)).cuda())
        ys.append(torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda"))
        mats.append(A)
    B0 = batch.Batch(devs, xs, ys)
    B0.run(use_graph=False)
    torch.cuda.synchronize()
    y_default = [y.clone() for y in ys]
    B0.destroy()
    for rule in (batch.DEFAULT_RULES[0], (4, 16, 64), (2, 8, 32), (batch.NEVER, batch.NEVER, 1)):
        for y in ys:
            y.fill_(float("nan"))
        B = batch.Batch(devs, xs, ys, rule=rule)
        B.run(use_graph=True)
        torch.cuda.synchronize()
        for A, x, y in zip(mats, xs, ys):
            xh = x.cpu().numpy()
            r = parity.check_fp64(y.cpu().numpy(), oracle_lib.crs_spmv(A, xh), oracle_lib.crs_absmv(A, xh),
                                  np.diff(A.row_ptr))
            assert r["ok"], (rule, r)
        if rule == batch.DEFAULT_RULES[0]:
            assert all(torch.equal(a, b) for a, b in zip(y_default, ys))
        B.destroy()
    rules = batch.DEFAULT_RULES[:4]
    best, timings = batch.tune_rule(devs, xs, ys, rules=rules, reps=3, flush_bytes=0)
    assert len(timings) == 4 and all(us > 0 for _, us in timings)
    assert best == min(timings, key=lambda t: t[1])[0]


def test_batch_degenerate_matrices(mods, oracle_lib):
    # a matrix without rows, one whose rows are all empty, a one-row matrix
    # and two ordinary ones in one launch, with each way of choosing lanes
    torch, pjds, batch = mods
    makes = [lambda: tiny.from_lengths([], 5), lambda: tiny.from_lengths([0] * 77, 9),
             lambda: tiny.from_lengths([3], 4, seed=1), lambda: synth.zipf_rows(3_000, s=2.0, len_max=300, seed=71),
             lambda: tiny.random_lengths(515, 600, max_len=70, seed=72, p_empty=0.3)]
    mats, devs, xs = [], [], []
    for k, make in enumerate(makes):
        A = make()
        mats.append(A)
        devs.append(pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32).to_device("cuda"))
        xs.append(torch.from_numpy(synth.vector(A.n_cols, seed=k)).cuda())
    for kw in (dict(), dict(rule=(4, 16, 64)), dict(lanes=[1, 2, 4, 8, 0])):
        ys = [torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda") for A in mats]
        B = batch.Batch(devs, xs, ys, **kw)
        B.run(use_graph=True)
        torch.cuda.synchronize()
        for A, x, y in zip(mats, xs, ys):
            if A.n_rows == 0:
                continue
            xh = x.cpu().numpy()
            r = parity.check_fp64(y.cpu().numpy(), oracle_lib.crs_spmv(A, xh), oracle_lib.crs_absmv(A, xh),
                                  np.diff(A.row_ptr))
            assert r["ok"], (kw, r)
        B.destroy()


def _block_rows(n_rows, n_brows, bs, nb, mixed, seed):
    """CRS of n_rows rows in block rows of bs (their columns shared, nb blocks of
    bs columns each, drawn from n_brows); `mixed` of the rows get a column of
    their own, and the last rows are shorter."""
    rng = np.random.default_rng(seed)
    brow = np.arange(n_rows) // bs
    first = np.sort(rng.integers(0, n_brows, size=(brow[-1] + 1, nb)), axis=1)
    first += np.arange(nb)  # distinct: strictly ascending
    col = (first[brow][:, :, None] * bs + np.arange(bs)).reshape(n_rows, nb * bs)
    own = np.nonzero(rng.random(n_rows) < mixed)[0]
    n_cols = (n_brows + nb) * bs + 8
    col[own, -1] = n_cols - 1 - own % 8
    lens = np.full(n_rows, nb * bs)
    lens[-37:] = nb * bs - 3  # a kind of its own in the sorted order, and a remainder
    keep = np.arange(nb * bs) < lens[:, None]
    ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    val = rng.uniform(-1, 1, size=int(ptr[-1]))
    return synth.Crs(n_rows, n_cols, ptr, col[keep].astype(np.int32), val)


# four rows per thread (blocks of 4 and 8 rows, some rows with a column of their
# own), the fall back from it (blocks of 2 and 6), both depths (2^18 threads
# between k = 32 and 264 / 64 on 131,077 rows), row counts with every remainder
# of 4, and just below the size from which it is offered (n k = 2^20)
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,k,bs,nb,mixed", [(32768, 32, 4, 5, 0.0), (32769, 32, 4, 5, 0.02), (32767, 32, 4, 5, 0.02),
                                             (43691, 24, 8, 3, 0.02), (131074, 8, 4, 4, 0.02), (32771, 32, 2, 10, 0.0),
                                             (34950, 32, 6, 4, 0.01), (131077, 64, 4, 4, 0.02)])
def test_spmm_rows_sharing_their_columns_in_fours(mods, dtype, n, k, bs, nb, mixed):
    torch, pjds, batch = mods
    A = _block_rows(n, n // bs // 2, bs, nb, mixed, seed=n + k)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    assert D.pair_share >= 900
    X = torch.rand(A.n_cols, k, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) * 2 - 1
    Y = torch.full((A.n_rows, k), float("nan"), device="cuda")
    P = torch.full((A.n_rows, k), float("nan"), device="cuda")
    batch.spmm(D, X, Y)
    batch.spmm_pattern(D, X, P)
    assert not torch.isnan(Y).any() and not torch.isnan(P).any()
    # each column in the order and with the multiply-adds of the single product
    y1, p1 = (torch.empty(A.n_rows, device="cuda") for _ in range(2))
    for c in (0, 3, 4, 7, k - 1):
        x = X[:, c].contiguous()
        pjds.pjds_spmv_cfg(D, x, y1, threads_per_row=1, rows_per_thread=1)
        pjds.pjds_spmv_pattern(D, x, p1, threads_per_row=1, rows_per_thread=1)
        assert torch.equal(y1, Y[:, c].contiguous()) and torch.equal(p1, P[:, c].contiguous()), c


def test_spmm_in_fours_in_a_captured_graph(mods):
    # two launches and what follows them on the stream
    torch, pjds, batch = mods
    for bs, nb in ((4, 5), (2, 10)):
        A = _block_rows(33_000, 8_000, bs, nb, 0.0, seed=bs)
        D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype="f32").to_device("cuda")
        X = torch.rand(A.n_cols, 32, device="cuda")
        Y, Z = (torch.zeros(A.n_rows, 32, device="cuda") for _ in range(2))
        batch.spmm(D, X, Y)
        want = 2 * Y
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            batch.spmm(D, X, Y)
            torch.add(Y, Y, out=Z)
            Y.zero_()
        for _ in range(3):
            Z.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(Z, want)


# block products launched while the one before runs, each on what that one has
# written (one row, fours and the fall back from fours; pairs: test_spmm_pairs), in
# a row on a stream and in a graph: bit for bit the products one by one
@pytest.mark.parametrize("dtype,k,bs,nb", [("f64", 2, 4, 5), ("f32", 4, 2, 8), ("bf16", 8, 2, 8), ("f32", 32, 4, 5),
                                           ("f32", 32, 2, 10), ("bf16", 32, 6, 4)])
def test_spmm_one_after_another(mods, dtype, k, bs, nb):
    torch, pjds, batch = mods
    A = _block_rows(33_001, 33_001 // bs // 2, bs, nb, 0.01, seed=bs)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    one = torch.rand(A.n_rows, k, device="cuda", generator=torch.Generator("cuda").manual_seed(k)).to(D.vec_dtype) - 0.5
    v = [one] + [torch.full_like(one, float("nan")) for _ in range(5)]
    want = [one]
    for _ in range(5):
        want.append(torch.full_like(one, float("nan")))
        torch.cuda.synchronize()
        batch.spmm(D, want[-2][:A.n_cols], want[-1])
        torch.cuda.synchronize()
    assert torch.isfinite(want[-1]).all()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for i in range(5):
            batch.spmm(D, v[i][:A.n_cols], v[i + 1])
        stream.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(v, want))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for i in range(5):
                batch.spmm(D, v[i][:A.n_cols], v[i + 1])
    for _ in range(3):
        for a in v[1:]:
            a.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(v, want))


# long rows apart from the others (widely spread lengths, rows of 64 entries or more), in one launch (up to 2^21
# 16-byte chunks of Y) and in two ("two": 2,112,000 of them at k = 64 fp64 and 128 fp32): lengths at the edges of a
# round of 16, only long rows and a few, one long row; each column in the order and with the multiply-adds of the
# single product
@pytest.mark.parametrize("name,dtype,k", [(name, dtype, k) for name in ("edges", "one", "many") for dtype, k in
                                          (("f64", 2), ("f64", 6), ("f32", 4), ("bf16", 24), ("f32", 128))] +
                         [("two", "f64", 64), ("two", "f32", 128), ("two", "bf16", 128)])
def test_spmm_long_rows(mods, dtype, k, name):
    torch, pjds, batch = mods
    lens = {"edges": [64, 65, 79, 80, 81, 63, 95, 96, 97, 111, 112, 113, 128, 700] + [3] * 4001,
            "one": [64] + [1] * 900,
            "many": list(np.minimum(np.random.default_rng(3).zipf(1.5, size=9000), 600)),
            "two": list(np.minimum(np.random.default_rng(4).zipf(1.9, size=66_000), 300))}[name]
    A = tiny.from_lengths(np.array(lens), 9001, seed=k)
    rng = np.random.default_rng(5)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    assert D.n_max * A.n_rows > 4 * A.nnz
    X = torch.from_numpy(rng.uniform(-1, 1, size=(A.n_cols, k))).to("cuda", D.vec_dtype)
    Y, P = (torch.full((A.n_rows, k), float("nan"), dtype=D.vec_dtype, device="cuda") for _ in range(2))
    batch.spmm(D, X, Y)
    twice = 2 * Y  # (what follows on the stream sees all rows)
    batch.spmm_pattern(D, X, P)
    y1, p1 = (torch.empty(A.n_rows, dtype=D.vec_dtype, device="cuda") for _ in range(2))
    for c in (0, 1, k - 1):
        x = X[:, c].contiguous()
        pjds.pjds_spmv_cfg(D, x, y1, plan=-1, threads_per_row=1, rows_per_thread=1)
        pjds.pjds_spmv_pattern(D, x, p1, plan=-1, threads_per_row=1, rows_per_thread=1)
        assert torch.equal(y1, Y[:, c].contiguous()) and torch.equal(p1, P[:, c].contiguous()), c
        assert torch.equal(2 * y1, twice[:, c].contiguous()), c


# batches of which every tile has its CTA: run after run, each reading what the one
# before wrote (x and y change places), with and without use_graph and in a captured
# graph, bit for bit the single products of the same plan
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_small_batches_one_after_another(mods, dtype):
    torch, pjds, batch = mods
    mats = [synth.zipf_rows(n, s=2.0, len_max=300, seed=n) for n in (33, 1000, 2047)]
    devs = [pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
            for A in mats]
    a = [torch.from_numpy(synth.vector(A.n_cols, seed=2)).to("cuda", D.vec_dtype) for A, D in zip(mats, devs)]
    b = [torch.empty_like(v) for v in a]
    there, back = batch.Batch(devs, a, b), batch.Batch(devs, b, a)
    assert there.info()["n_ctas"] == there.info()["n_tiles"]
    first, want = [v.clone() for v in a], [v.clone() for v in a]
    for _ in range(6):
        for q, D in enumerate(devs):
            y = torch.empty_like(want[q])
            torch.cuda.synchronize()
            pjds.pjds_spmv_cfg(D, want[q], y, plan=1)
            torch.cuda.synchronize()
            want[q] = y
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for k in range(6):
            (back if k % 2 else there).run()

    def runs(use_graph):
        for k in range(6):
            (back if k % 2 else there).run(use_graph=use_graph)

    for go in (lambda: runs(True), lambda: runs(False), graph.replay, graph.replay):
        for v, u in zip(a, first):
            v.copy_(u)
        go()
        torch.cuda.synchronize()
        assert all(torch.equal(v, w) for v, w in zip(a, want))


# block products with X and Y changing places and new data before every run, so that an element left in a cache
# from an earlier product would show: one row a thread, long rows in one launch and in two, fours and the fall back
# from them, on a stream and in a graph
@pytest.mark.parametrize("name,dtype,k", [("rows", "f64", 2), ("rows", "f32", 8), ("spread", "f64", 4),
                                          ("spread", "bf16", 16), ("spread", "f32", 128), ("fours", "f32", 32),
                                          ("fours", "bf16", 32), ("twos", "f32", 32), ("sixes", "bf16", 32)])
def test_block_products_back_and_forth(mods, name, dtype, k):
    torch, pjds, batch = mods
    if name == "spread":
        n = 66_000 if k == 128 else 20_001  # two launches and one
        A = tiny.from_lengths(np.minimum(np.random.default_rng(2).zipf(1.9, size=n), 300), n, seed=6)
    elif name == "rows":
        n = 20_001
        A = tiny.from_lengths(np.full(n, 7), n, seed=6)
    else:
        bs, nb = {"fours": (4, 5), "twos": (2, 10), "sixes": (6, 4)}[name]
        n = 34_950
        A = _block_rows(n, n // bs // 2, bs, nb, 0.01, seed=bs)
    lens = np.maximum(np.diff(A.row_ptr), 1)
    A = A._replace(val=A.val / np.repeat(lens, np.diff(A.row_ptr)))  # row sums below 1: products stay in range
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    m = max(A.n_rows, A.n_cols)
    a, b, first, add = (torch.empty(m, k, dtype=D.vec_dtype, device="cuda") for _ in range(4))
    g = torch.Generator("cuda").manual_seed(k)
    add.uniform_(-1, 1, generator=g)

    def run(between=lambda: None):
        for i in range(6):
            x, y = (b, a) if i % 2 else (a, b)
            between()
            batch.spmm(D, x[:A.n_cols], y[:A.n_rows])
            between()
            if i == 2:
                b.add_(add)

    def check(go):
        for _ in range(4):
            first.uniform_(-1, 1, generator=g)
            a.copy_(first), b.zero_()
            run(torch.cuda.synchronize)
            want = a.clone(), b.clone()
            a.copy_(first), b.zero_()
            go()
            torch.cuda.synchronize()
            assert torch.equal(a, want[0]) and torch.equal(b, want[1])
        assert torch.isfinite(a).all() and a.abs().max() > 0

    check(run)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    check(graph.replay)


# two rows per thread (from 2^18 rows of 64 entries on): block rows of 2 and 6, which share no fours, so that
# spmm_quad_kernel leaves the work to spmm_pair_kernel, an odd number of rows and rows with a column of their own,
# every depth and width of a round, columns bit for bit the single products; products on one another's results, in
# a row on a stream and in a graph
@pytest.mark.parametrize("dtype,k,bs,nb", [("f32", 8, 2, 34), ("f32", 64, 6, 12), ("bf16", 8, 6, 12), ("bf16", 32, 2, 34)])
def test_spmm_pairs(mods, dtype, k, bs, nb):
    torch, pjds, batch = mods
    A = _block_rows(262_147, 262_147 // bs // 2, bs, nb, 0.01, seed=k + bs)
    assert A.nnz >= 64 * A.n_rows
    A = A._replace(val=A.val / (bs * nb))
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    assert D.pair_share >= 900
    g = torch.Generator("cuda").manual_seed(k)
    X = torch.rand(A.n_rows, k, device="cuda", generator=g) * 2 - 1
    Y, P, Z = (torch.full((A.n_rows, k), float("nan"), device="cuda") for _ in range(3))
    batch.spmm(D, X[:A.n_cols], Y)
    batch.spmm_pattern(D, X[:A.n_cols], P)
    y1, p1 = (torch.empty(A.n_rows, device="cuda") for _ in range(2))
    for c in (0, 3, k - 1):
        x = X[:A.n_cols, c].contiguous()
        pjds.pjds_spmv_cfg(D, x, y1, threads_per_row=1, rows_per_thread=1)
        pjds.pjds_spmv_pattern(D, x, p1, threads_per_row=1, rows_per_thread=1)
        assert torch.equal(y1, Y[:, c].contiguous()) and torch.equal(p1, P[:, c].contiguous()), c
    batch.spmm(D, Y[:A.n_cols], Z)
    torch.cuda.synchronize()
    a, b = X.clone(), torch.empty_like(X)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        batch.spmm(D, a[:A.n_cols], b)
        batch.spmm(D, b[:A.n_cols], a)
    for go in (lambda: (batch.spmm(D, a[:A.n_cols], b), batch.spmm(D, b[:A.n_cols], a)), graph.replay):
        a.copy_(X), b.fill_(float("nan"))
        go()
        torch.cuda.synchronize()
        assert torch.equal(b, Y) and torch.equal(a, Z)


# lanes of two chunks of one row on a matrix whose rows share nothing (spmm_kernel; on block matrices the fp32 and
# bf16 products of test_spmm_two_chunk_lanes take four rows per thread)
@pytest.mark.parametrize("dtype,k", [("f32", 64), ("bf16", 64), ("f64", 32)])
def test_spmm_two_chunk_lanes_of_single_rows(mods, dtype, k):
    torch, pjds, batch = mods
    A = tiny.from_lengths(np.tile([20, 19, 21, 3], 18_000)[:70_001], 30_000, seed=3)
    D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
    assert D.pair_share < 500
    X = torch.rand(A.n_cols, k, device="cuda", dtype=D.vec_dtype) * 2 - 1
    Y, P = (torch.full((A.n_rows, k), float("nan"), dtype=D.vec_dtype, device="cuda") for _ in range(2))
    batch.spmm(D, X, Y)
    batch.spmm_pattern(D, X, P)
    y1, p1 = (torch.empty(A.n_rows, dtype=D.vec_dtype, device="cuda") for _ in range(2))
    for c in range(k):
        x = X[:, c].contiguous()
        pjds.pjds_spmv_cfg(D, x, y1, threads_per_row=1, rows_per_thread=1)
        pjds.pjds_spmv_pattern(D, x, p1, threads_per_row=1, rows_per_thread=1)
        assert torch.equal(y1, Y[:, c].contiguous()) and torch.equal(p1, P[:, c].contiguous()), c


# batches of more tiles than CTAs, whose CTAs take tiles from the counter (all other batches of these tests are
# small): direct, by graph and as pattern, twice each, in the three value types, bit for bit the single products of
# the same plan
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_batches_of_more_tiles_than_ctas(mods, dtype):
    torch, pjds, batch = mods
    mats = [tiny.from_lengths(np.full(130_001, 17), 5_000, seed=1), synth.zipf_rows(200_003, s=1.8, len_max=400, seed=2),
            tiny.random_lengths(1037, 1037, max_len=90, seed=3, p_empty=0.2)]
    devs = [pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dtype).to_device("cuda")
            for A in mats]
    xs = [torch.from_numpy(synth.vector(A.n_cols, seed=4)).to("cuda", D.vec_dtype) for A, D in zip(mats, devs)]
    ys = [torch.empty(A.n_rows, dtype=D.vec_dtype, device="cuda") for A, D in zip(mats, devs)]
    want, ones = [torch.empty_like(y) for y in ys], [torch.empty_like(y) for y in ys]
    for D, x, y, p in zip(devs, xs, want, ones):
        pjds.pjds_spmv_cfg(D, x, y, plan=1)
        pjds.pjds_spmv_pattern(D, x, p, plan=1)
    B = batch.Batch(devs, xs, ys)
    assert B.info()["n_tiles"] > B.info()["n_ctas"]
    for go, expect in ((lambda: B.run(use_graph=False), want), (lambda: B.run(use_graph=True), want),
                       (B.run_pattern, ones)):
        for _ in range(2):
            for y in ys:
                y.fill_(float("nan"))
            go()
            torch.cuda.synchronize()
            assert all(torch.equal(y, w) for y, w in zip(ys, expect))
    B.destroy()
