"""Hand-written MLP kernels (training and inference) against the fp64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1112_5588_gb300 import build
    build.build()
    from paper_1112_5588_gb300 import learned
    return learned


def _to_oracle(m):
    return {"w1": np.array(m.w1, np.float64).reshape(64, 15), "b1": np.array(m.b1, np.float64),
            "w2": np.array(m.w2, np.float64).reshape(64, 64), "b2": np.array(m.b2, np.float64),
            "w3": np.array(m.w3, np.float64), "b3": np.array([m.b3], np.float64)}


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 15)).astype(np.float32)
    y = (np.sin(X[:, 0]) + 0.5 * X[:, 1] * X[:, 2] - X[:, 3]).astype(np.float32)
    return X, y


def test_forward_matches_oracle(L):
    from oracle import mlp as om
    m = L.init(2)
    m.b1[:] = np.linspace(-0.1, 0.1, 64)
    X, _ = _data(333, 1)  # ragged: not a multiple of the 64-sample tile
    got = L.predict(m, X)
    want, _ = om.forward(_to_oracle(m), X.astype(np.float64))
    assert np.allclose(got, want, rtol=1e-5, atol=1e-5)


def test_one_full_batch_adam_step_matches_oracle(L):
    from oracle import mlp as om
    m = L.init(3)
    X, y = _data(200, 4)
    p = _to_oracle(m)
    g = om.grads(p, X.astype(np.float64), y.astype(np.float64))
    p1 = om.adam_step({k: v.copy() for k, v in p.items()}, g, {}, 1, lr=1e-3)
    L.train(m, X, y, epochs=1, batch=10_000, lr=1e-3)
    q = _to_oracle(m)
    for k in p:
        # the first Adam step is lr * g / (|g| + eps): compare where |g| is not tiny
        big = np.abs(g[k]) > 1e-4 * np.abs(g[k]).max()
        assert np.allclose(q[k][big], p1[k][big], rtol=0, atol=2e-6), k


def test_full_batch_training_tracks_oracle_loss(L):
    from oracle import mlp as om
    m = L.init(4)
    X, y = _data(256, 5)
    p, st = _to_oracle(m), {}
    Xd, yd = X.astype(np.float64), y.astype(np.float64)
    ref = []
    for t in range(1, 41):
        p = om.adam_step(p, om.grads(p, Xd, yd), st, t, lr=2e-3)
        ref.append(om.loss(p, Xd, yd))
    hist = L.train(m, X, y, epochs=40, batch=256, lr=2e-3)
    assert np.allclose(hist, ref, rtol=2e-3)


def test_minibatch_training_fits_and_is_deterministic(L):
    X, y = _data(4000, 6)
    m1, m2 = L.init(7), L.init(7)
    L.fit_scaling(m1, X, y)
    L.fit_scaling(m2, X, y)
    h1 = L.train(m1, X, y, epochs=60, batch=512, lr=3e-3, seed=11)
    h2 = L.train(m2, X, y, epochs=60, batch=512, lr=3e-3, seed=11)
    assert h1[-1] < 0.05 * h1[0]
    assert np.array_equal(np.array(m1.w2), np.array(m2.w2))
    assert np.array_equal(h1, h2)


# samples and batches around a tile of 16 and a CTA per SM, a batch larger than
# the data, more epochs than samples (losses are kept in n device slots)
@pytest.mark.parametrize("n,batch,epochs", [(1, 1, 3), (15, 4, 2), (16, 16, 2), (17, 16, 2), (33, 100, 4), (700, 17, 1),
                                            (2500, 2433, 2), (5000, 1000, 2)])
def test_training_in_batches_matches_oracle(L, n, batch, epochs):
    from oracle import mlp as om
    m = L.init(7)
    X, y = _data(n, 9)
    p, st = _to_oracle(m), {}
    hist = L.train(m, X, y, epochs=epochs, batch=batch, lr=1e-3, seed=3)

    def mix(z):
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9 % 2 ** 64
        z = (z ^ (z >> 27)) * 0x94D049BB133111EB % 2 ** 64
        return z ^ (z >> 31)

    t, want = 0, []
    for ep in range(epochs):
        o = list(range(n))
        if batch < n:
            base = mix((3 + 0x51ED2701 * (ep + 1)) % 2 ** 64)
            for i in range(n - 1, 0, -1):
                j = mix((base + i) % 2 ** 64) % (i + 1)
                o[i], o[j] = o[j], o[i]
        for b in range(0, n, batch):
            s = o[b:b + batch]
            t += 1
            p = om.adam_step(p, om.grads(p, X[s].astype(np.float64), y[s].astype(np.float64)), st, t, lr=1e-3)
        out, _ = om.forward(p, X.astype(np.float64))
        want.append(np.mean((out - y) ** 2))
    # a loss is a mean over fp32 outputs (sums of 64 products, relative 1e-5); the steps add lr times the
    # direction's rounding, in the first steps up to lr = 1e-3 where a gradient is at its rounding
    assert np.allclose(hist, want, rtol=2e-3, atol=1e-6), (hist, want)
    if t > 3:
        q = _to_oracle(m)
        for k in p:
            assert np.mean(np.abs(q[k] - p[k])) <= 2e-5, k


# the size that pjds_mlp_workspace_bytes gives for any batch serves pjds_mlp_predict on as many inputs, and no
# byte beyond it is written
@pytest.mark.parametrize("n,batch", [(1, 1), (17, 1), (100, 1000), (21600, 16), (21600, 21600), (200_000, 1024)])
def test_predict_in_a_training_workspace(L, n, batch):
    import ctypes

    import torch
    m = L.init(5)
    X, _ = _data(n, 8)
    need = ctypes.c_size_t()
    assert L._lib.pjds_mlp_workspace_bytes(n, batch, ctypes.byref(need)) == 0
    work = torch.full((need.value + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    out = np.full(n, np.nan, np.float32)
    rc = L._lib.pjds_mlp_predict(ctypes.byref(m), X.ctypes.data, n, out.ctypes.data, work.data_ptr(), need.value,
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == 0, L._p._lib.pjds_last_error()
    assert bool((work[need.value:] == 0x5A).all())
    assert np.array_equal(out, L.predict(m, X))
