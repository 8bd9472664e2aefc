"""Cases for the checked build (run by tests/test_gpu_checked.py in a process
with PJDS_LIBRARY=checked, which loads libpjds_checked.so).

Clean: every mapping of the product with device-side extent checks (one and
T threads per row, several rows per thread, tile order, per-tile mapping,
64-bit offsets), the pattern product, ELLPACK-R, the block product (also with
paired rows on a block-structured matrix) and the batched launch, on ragged,
spread, banded and block-dense matrices, must leave the check word at 0 and
match the oracle (fp64; fp32 bounds for the paired block product).

Planted: an index put out of range in a device copy of a matrix (a column
beyond n_cols, a perm entry beyond n_rows, a jagged-diagonal offset beyond
the stored entries, a block longer than the longest row; also in the block
product's launch for long rows) must be recorded with its code and skipped:
the kernels check each index before the access.

Refused: cooperative launches of more CTAs than a limit are refused, as in a
context of fewer SMs: their callers' other way must give the same results.

Prints one JSON line.
"""
import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

CFGS = [dict(), dict(threads_per_row=1), dict(rows_per_thread=2), dict(rows_per_thread=4), dict(threads_per_row=2),
        dict(threads_per_row=4), dict(threads_per_row=8), dict(tile_order=1), dict(plan=1), dict(index64=1),
        dict(plan=1, index64=1), dict(rows_per_thread=2, index64=1)]
CODE_SHIFT = 56


def split(w):
    return w >> CODE_SHIFT, w & ((1 << CODE_SHIFT) - 1)


def main():
    assert os.environ.get("PJDS_LIBRARY") == "checked"
    import torch

    import oracle
    import synth
    from paper_1112_5588_gb300 import batch, pjds
    from synth import tiny
    from tests import parity
    assert pjds.LIB_PATH.endswith("libpjds_checked.so")
    oracle.build()
    assert pjds.pjds_check_word(clear=True) == 0

    mats = {
        "ragged": tiny.random_lengths(1037, 1037, max_len=90, seed=61, p_empty=0.2),
        "zipf": synth.zipf_rows(70_000, s=1.8, len_max=600, seed=62),
        "hmep": synth.hmep_like(n=30_011, seed=63),
        "full_row": tiny.one_full_row(900, full_row=37),
    }
    res = {"clean": [], "planted": {}}

    def run(D, xt, cfg):
        y = torch.full((D.n_rows,), float("nan"), dtype=D.vec_dtype, device="cuda")
        pjds.pjds_spmv_cfg(D, xt, y, **cfg)
        torch.cuda.synchronize()
        return y

    for name, A in mats.items():
        x = synth.vector(A.n_cols, seed=64)
        yref, absax, lens = oracle.crs_spmv(A, x), oracle.crs_absmv(A, x), np.diff(A.row_ptr)
        for dt in ("f64", "f32", "bf16"):
            for b in (32, 128):
                H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=b, dtype=dt)
                D = H.to_device("cuda")
                H.destroy()
                xt = torch.from_numpy(x).to("cuda", D.vec_dtype)
                for cfg in CFGS:
                    y = run(D, xt, cfg)
                    w = pjds.pjds_check_word(clear=True)
                    ok = bool(torch.isfinite(y).all())
                    if dt == "f64":
                        ok = ok and parity.check_fp64(y.cpu().numpy(), yref, absax, lens)["ok"]
                    res["clean"].append([name, dt, b, cfg, w, ok])
                # the pattern product (the gather ceiling) with one and two rows per thread
                for cfg in (dict(threads_per_row=1), dict(rows_per_thread=2)):
                    y = torch.full((D.n_rows,), float("nan"), dtype=D.vec_dtype, device="cuda")
                    pjds.pjds_spmv_pattern(D, xt, y, **cfg)
                    torch.cuda.synchronize()
                    w = pjds.pjds_check_word(clear=True)
                    res["clean"].append([name, dt, b, dict(pattern=1, **cfg), w, bool(torch.isfinite(y).all())])
            E = pjds.ellr_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, dtype=dt).to_device("cuda")
            y = torch.full((A.n_rows,), float("nan"), dtype=E.vec_dtype, device="cuda")
            pjds.ellr_spmv(E, torch.from_numpy(x).to("cuda", E.vec_dtype), y)
            torch.cuda.synchronize()
            w = pjds.pjds_check_word(clear=True)
            ok = bool(torch.isfinite(y).all())
            if dt == "f64":
                ok = ok and parity.check_fp64(y.cpu().numpy(), yref, absax, lens)["ok"]
            res["clean"].append([name, dt, 0, "ellr", w, ok])

    # SpMM: k right-hand sides
    for name, A in mats.items():
        lens = np.diff(A.row_ptr)
        for dt, ks in (("f64", (2, 8)), ("f32", (4, 32))):
            D = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dt).to_device("cuda")
            for k in ks:
                X = np.stack([synth.vector(A.n_cols, seed=70 + c) for c in range(k)], axis=1)
                Y = torch.full((A.n_rows, k), float("nan"), dtype=D.vec_dtype, device="cuda")
                batch.spmm(D, torch.from_numpy(np.ascontiguousarray(X)).to("cuda", D.vec_dtype), Y)
                torch.cuda.synchronize()
                w = pjds.pjds_check_word(clear=True)
                ok = bool(torch.isfinite(Y).all())
                if dt == "f64":
                    Yr = oracle.crs_spmm(A, X)
                    S = np.abs(oracle.crs_spmm(A._replace(val=np.abs(A.val)), np.abs(X)))
                    Yg = Y.cpu().numpy()
                    ok = ok and all(parity.check_fp64(Yg[:, c], Yr[:, c], S[:, c], lens)["ok"] for c in range(k))
                res["clean"].append([name, dt, 32, f"spmm k={k}", w, ok])

    # the batched launch over all four matrices, with the built-in rule and given lanes
    devs = [pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32).to_device("cuda")
            for A in mats.values()]
    xs = [torch.from_numpy(synth.vector(A.n_cols, seed=65)).cuda() for A in mats.values()]
    for kw in (dict(), dict(lanes=[1, 8, 2, 4]), dict(rule=(4, 16, 64))):
        ys = [torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda") for A in mats.values()]
        B = batch.Batch(devs, xs, ys, **kw)
        B.run(use_graph=False)
        torch.cuda.synchronize()
        w = pjds.pjds_check_word(clear=True)
        ok = all(parity.check_fp64(y.cpu().numpy(), oracle.crs_spmv(A, xv.cpu().numpy()),
                                   oracle.crs_absmv(A, xv.cpu().numpy()), np.diff(A.row_ptr))["ok"]
                 for A, xv, y in zip(mats.values(), xs, ys))
        B.destroy()
        res["clean"].append(["batch", "f64", 32, kw.get("lanes") and "lanes" or kw.get("rule") and "rule" or "default",
                             w, ok])

    # a batch of more tiles than CTAs (the work counter; the one above has a CTA for every tile)
    many = [tiny.from_lengths(np.full(130_001, 17), 5_000, seed=1), mats["ragged"], mats["hmep"]]
    for dt in ("f64", "f32", "bf16"):
        devs = [pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32, dtype=dt).to_device("cuda")
                for A in many]
        xs = [torch.from_numpy(synth.vector(A.n_cols, seed=65)).to("cuda", D.vec_dtype) for A, D in zip(many, devs)]
        ys = [torch.full((A.n_rows,), float("nan"), dtype=D.vec_dtype, device="cuda") for A, D in zip(many, devs)]
        B = batch.Batch(devs, xs, ys)
        assert B.info()["n_tiles"] > B.info()["n_ctas"]
        B.run(use_graph=False)
        torch.cuda.synchronize()
        w = pjds.pjds_check_word(clear=True)
        ok = all(bool(torch.isfinite(y).all()) for y in ys)
        if dt == "f64":
            ok = ok and all(parity.check_fp64(y.cpu().numpy(), oracle.crs_spmv(A, xv.cpu().numpy()),
                                              oracle.crs_absmv(A, xv.cpu().numpy()), np.diff(A.row_ptr))["ok"]
                            for A, xv, y in zip(many, xs, ys))
        B.destroy()
        res["clean"].append(["batch", dt, 32, "counter", w, ok])

    # rows sharing their columns (2^18 rows of 64 or more: pair_share 1000), in 4x4 blocks and in blocks of 2: the
    # single product (two rows per thread), the block product with four rows per thread ("quad") and, where the
    # rows share in twos only, with two ("paired"), and their pattern products
    from tests.test_gpu_batch import _block_rows
    shared = {"quad": synth.block_dense(70_000, 4, 16, 0.05, seed=67),
              "paired": _block_rows(262_147, 60_000, 2, 34, 0.01, seed=5)}
    for name, dt, k in (("quad", "f32", 8), ("quad", "bf16", 16), ("paired", "f32", 8), ("paired", "bf16", 16)):
        Pm = shared[name]
        lens = np.diff(Pm.row_ptr)
        D = pjds.pjds_create(Pm.n_rows, Pm.n_cols, Pm.row_ptr, Pm.col, Pm.val, b=32, dtype=dt).to_device("cuda")
        assert D.pair_share >= 500 and pjds.pjds_spmv_resolve(D)["rows_per_thread"] == 2
        xt = torch.from_numpy(synth.vector(Pm.n_cols, seed=68)).to("cuda", D.vec_dtype)
        y = run(D, xt, {})
        res["clean"].append([name, dt, 32, "spmv", pjds.pjds_check_word(clear=True), bool(torch.isfinite(y).all())])
        X = np.stack([synth.vector(Pm.n_cols, seed=80 + c) for c in range(k)], axis=1).astype(np.float32)
        Xt = torch.from_numpy(np.ascontiguousarray(X)).cuda()
        for fn, tag in ((batch.spmm, "spmm"), (batch.spmm_pattern, "spmm_pattern")):
            Y = torch.full((Pm.n_rows, k), float("nan"), device="cuda")
            fn(D, Xt, Y)
            torch.cuda.synchronize()
            w = pjds.pjds_check_word(clear=True)
            ok = bool(torch.isfinite(Y).all())
            if tag == "spmm":
                Ar = Pm._replace(val=oracle.round_f32(Pm.val) if dt == "f32" else oracle.round_bf16(Pm.val))
                Xd = X.astype(np.float64)
                Yr, S = oracle.crs_spmm(Ar, Xd), oracle.crs_spmm(Ar._replace(val=np.abs(Ar.val)), np.abs(Xd))
                Yg = Y.double().cpu().numpy()
                ok = ok and all(parity.check_fp32(Yg[:, c], Yr[:, c], S[:, c], lens)["ok"] for c in (0, k - 1))
            res["clean"].append([name, dt, 32, f"{tag} k={k}", w, ok])
    # a column beyond n_cols in them: recorded and skipped
    for name, Pm in shared.items():
        D = pjds.pjds_create(Pm.n_rows, Pm.n_cols, Pm.row_ptr, Pm.col, Pm.val, b=32, dtype="f32").to_device("cuda")
        D.col[1] = Pm.n_cols + 11
        Y = torch.empty(Pm.n_rows, 8, device="cuda")
        batch.spmm(D, torch.rand(Pm.n_cols, 8, device="cuda"), Y)
        torch.cuda.synchronize()
        res["planted"][name + "_column"] = [[{}, *split(pjds.pjds_check_word(clear=True))]]
        res[name + "_n_cols"] = Pm.n_cols

    # planted indices (fp64, original basis)
    A = mats["ragged"]
    H = pjds.pjds_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val, b=32)
    x = synth.vector(A.n_cols, seed=66)
    mapping = [dict(threads_per_row=1), dict(rows_per_thread=2), dict(threads_per_row=4), dict(plan=1), dict()]

    def planted(mutate):
        out = []
        for cfg in mapping:
            D = H.to_device("cuda")
            mutate(D)
            xt = torch.from_numpy(x).cuda()
            pjds.pjds_check_word(clear=True)
            run(D, xt, cfg)
            out.append([cfg, *split(pjds.pjds_check_word(clear=True))])
        return out

    res["n"] = {"n_rows": A.n_rows, "n_cols": A.n_cols, "n_stored": H.n_stored, "n_max": H.n_max}
    res["planted"]["column"] = planted(lambda D: D.col.__setitem__(0, A.n_cols + 5))
    res["planted"]["perm"] = planted(lambda D: D.perm.__setitem__(3, A.n_rows + 7))
    res["planted"]["offset"] = planted(lambda D: D.col_start.__setitem__(1, H.n_stored + 1000))
    res["planted"]["block"] = planted(lambda D: D.block_len.__setitem__(0, H.n_max + 3))
    # a planted column changes at most the one row that holds it
    D = H.to_device("cuda")
    xt = torch.from_numpy(x).cuda()
    y0 = run(D, xt, dict(threads_per_row=1))
    D.col[0] = A.n_cols + 5
    y1 = run(D, xt, dict(threads_per_row=1))
    pjds.pjds_check_word(clear=True)
    res["column_rows_changed"] = int((y0 != y1).sum().item())
    # ELLPACK-R with a column beyond n_cols
    E = pjds.ellr_create(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val).to_device("cuda")
    k = int(np.argmax(np.diff(A.row_ptr) > 0))
    E.col[k] = A.n_cols + 9
    y = torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
    pjds.ellr_spmv(E, torch.from_numpy(x).cuda(), y)
    torch.cuda.synchronize()
    res["planted"]["ellr_column"] = [[{}, *split(pjds.pjds_check_word(clear=True))]]
    # SpMM with a column beyond n_cols
    D = H.to_device("cuda")
    D.col[0] = A.n_cols + 5
    Y = torch.empty(A.n_rows, 4, dtype=torch.float64, device="cuda")
    batch.spmm(D, torch.rand(A.n_cols, 4, dtype=torch.float64, device="cuda"), Y)
    torch.cuda.synchronize()
    res["planted"]["spmm_column"] = [[{}, *split(pjds.pjds_check_word(clear=True))]]
    # SpMM's launch for long rows (widely spread lengths): a column beyond n_cols, a block longer than the longest row
    Z = mats["zipf"]
    Hz = pjds.pjds_create(Z.n_rows, Z.n_cols, Z.row_ptr, Z.col, Z.val, b=32)
    assert Hz.n_max >= 64 and Hz.n_max * Z.n_rows > 4 * Z.nnz
    res["zipf"] = {"n_cols": Z.n_cols, "n_stored": Hz.n_stored, "n_max": Hz.n_max}
    for name, mutate in (("long_column", lambda D: D.col.__setitem__(0, Z.n_cols + 13)),
                         ("long_block", lambda D: D.block_len.__setitem__(0, Hz.n_max + 3))):
        D = Hz.to_device("cuda")
        mutate(D)
        Y = torch.empty(Z.n_rows, 4, dtype=torch.float64, device="cuda")
        batch.spmm(D, torch.rand(Z.n_cols, 4, dtype=torch.float64, device="cuda"), Y)
        torch.cuda.synchronize()
        res["planted"][name] = [[{}, *split(pjds.pjds_check_word(clear=True))]]
    # cooperative launches of more CTAs than a limit refused (0: all, -1: none): small CG systems
    from paper_1112_5588_gb300 import krylov
    from tests.test_gpu_krylov import _spd
    S = _spd("tri", 4097)
    rhs = synth.vector(S.n_rows, seed=3)
    low = {dt: pjds.pjds_create(S.n_rows, S.n_cols, S.row_ptr, S.col, S.val, b=32, dtype=dt, permute_cols=True)
           for dt in ("f64", "f32", "bf16")}
    perm = low["f64"].perm.copy()
    low = {dt: H.to_device("cuda") for dt, H in low.items()}
    bp = torch.from_numpy(rhs[perm]).cuda()
    res["refused_cg"] = []
    for limit in (0, 8, -1):
        pjds._lib.pjds_checked_cooperative_limit(limit)
        for dt in low:
            xp = torch.zeros_like(bp)
            out = krylov.cg_solve(low["f64"], None if dt == "f64" else low[dt], bp, xp, max_outer=12, inner_iters=20,
                                  tol=1e-13)
            xs = np.empty(S.n_rows)
            xs[perm] = xp.cpu().numpy()
            rel = float(np.linalg.norm(rhs - oracle.crs_spmv(S, xs)) / np.linalg.norm(rhs))
            res["refused_cg"].append([dt, limit, max(rel, out["rel_residual"]), out["outer"]])
    # and an epoch of the tuner's training, on fewer CTAs then
    from paper_1112_5588_gb300 import learned
    rng = np.random.default_rng(9)
    X = rng.standard_normal((2500, 15)).astype(np.float32)
    t = (np.sin(X[:, 0]) + 0.5 * X[:, 1] * X[:, 2] - X[:, 3]).astype(np.float32)
    res["refused_train"] = []
    for limit in (-1, 1, 40):
        pjds._lib.pjds_checked_cooperative_limit(limit)
        m = learned.init(4)
        hist = learned.train(m, X, t, epochs=3, batch=700, lr=1e-3, seed=2)
        res["refused_train"].append([limit, [float(v) for v in hist], [float(v) for v in m.w2]])
    pjds._lib.pjds_checked_cooperative_limit(0)
    try:
        learned.train(learned.init(4), X, t, epochs=1, batch=700, lr=1e-3)
        res["refused_train_error"] = 0
    except pjds.PjdsError as err:
        res["refused_train_error"] = err.code
    print(json.dumps(res))


if __name__ == "__main__":
    main()
