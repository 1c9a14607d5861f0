"""The cost model's kernel at the edges of its tiles (16 rows a warp, 64 a CTA, features
padded to 16, several tiles per CTA) against the same model in FP64 with the kernel's BF16
roundings: features, weights, hidden layers and their gradients."""
import numpy as np
import pytest

from oracle import mlp_ref

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bf16(a):
    """FP64 -> FP32 -> BF16, as FP64."""
    return torch.tensor(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()


def _problem(K, n, seed):
    rng = np.random.default_rng(seed)
    T = rng.uniform(250.0, 3500.0, n)
    p = np.exp(rng.uniform(np.log(1e5), np.log(1e8), n))
    Y = 10.0 ** rng.uniform(-30.0, 0.0, (n, K))
    Y[rng.random((n, K)) < 0.2] = 0.0
    Y.ravel()[:: 97] = 5e-324
    sub = np.exp(rng.uniform(0.0, 6.0, n)).astype(np.int32)
    hf = np.exp(rng.uniform(-28.0, -14.0, n))
    D = K + 2
    f32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    # fixed normalisation of these ranges; one feature's is far off, so that its values cancel
    norm = [f32(np.r_[1.9, 15.0, np.full(K, -30.0)]), f32(np.r_[0.9, 2.0, rng.uniform(5.0, 20.0, K)]),
            f32([3.0, -21.0]), f32([1.7, 4.0])]
    params = {k: f32(v) for k, v in mlp_ref.init_params(D, seed=seed).items()}
    buf = np.concatenate(norm + [params[k].ravel() for k in mlp_ref.ORDER]).astype(np.float32)
    return T, p, Y, sub, hf, norm, params, buf


def _model(T, p, Y, norm, params):
    """Forward pass with the kernel's roundings; returns every layer."""
    X = _bf16((mlp_ref.features(T, p, Y) - norm[0]) / norm[1])
    W = {k: _bf16(params[k]) if k[0] == "W" else params[k] for k in mlp_ref.ORDER}
    Z1 = X @ W["W1"].T + W["b1"]
    H1 = _bf16(mlp_ref.gelu(Z1))
    Z2 = H1 @ W["W2"].T + W["b2"]
    H2 = _bf16(mlp_ref.gelu(Z2))
    return X, W, Z1, H1, Z2, H2, H2 @ W["W3"].T + W["b3"]


SIZES = [(1, 1), (1, 17), (14, 15), (15, 16), (54, 63), (54, 65), (54, 1000), (129, 130), (255, 257), (5, 20000)]


@pytest.mark.parametrize("K,n", SIZES)
def test_predict(K, n):
    import paper_2112_05834_gb300 as pkg

    T, p, Y, _, _, norm, params, buf = _problem(K, n, 100 + K)
    T[n // 2], Y[n // 2, 0] = np.nan, -1.0  # one cell outside the model's domain stays alone
    model = pkg.CostModel(K)
    model.set_params(buf)
    dev = lambda a: torch.tensor(a, device="cuda")
    got = torch.stack(model.predict(dev(T), dev(p), dev(Y)), 1).cpu().numpy().astype(np.float64)
    assert np.all(np.isnan(got[n // 2]))
    ok = np.arange(n) != n // 2
    with np.errstate(invalid="ignore"):
        *_, H2, out = _model(T, p, Y, norm, params)
    # FP32 sums may round a hidden value to the other BF16 neighbour: four of those at the
    # largest weight and value, and FP32's own rounding of the output's terms
    W3 = np.abs(params["W3"]).max()
    tol = 4 * 2.0 ** -8 * W3 * np.abs(H2[ok]).max(initial=0.0) + 1e-5
    err = np.abs((got - norm[2]) / norm[3] - out)[ok]
    print("max error", err.max(initial=0.0), "tolerance", tol)
    assert np.all(err <= tol)


@pytest.mark.parametrize("K,n", SIZES)
def test_gradient(K, n):
    import paper_2112_05834_gb300 as pkg

    T, p, Y, sub, hf, norm, params, buf = _problem(K, n, 200 + K)
    model = pkg.CostModel(K)
    model.set_params(buf)
    dev = lambda a: torch.tensor(a, device="cuda")
    loss, g = model.gradient(dev(T), dev(p), dev(Y), dev(sub), dev(hf))
    X, W, Z1, H1, Z2, H2, out = _model(T, p, Y, norm, params)
    r = out - (mlp_ref.targets(sub, hf) - norm[2]) / norm[3]
    d = r / n
    dZ2 = _bf16((d @ W["W3"]) * mlp_ref.gelu_grad(Z2))
    dZ1 = _bf16((dZ2 @ W["W2"]) * mlp_ref.gelu_grad(Z1))
    want = dict(W1=dZ1.T @ X, b1=dZ1.sum(0), W2=dZ2.T @ H1, b2=dZ2.sum(0), W3=d.T @ H2, b3=d.sum(0))
    assert abs(loss - 0.5 * (r * r).sum() / n) <= 1e-3 * 0.5 * (r * r).sum() / n
    got = mlp_ref.unflatten(g.astype(np.float64), K + 2)
    # a value that FP32 sums round to its other BF16 neighbour moves its row or column by 2^-8;
    # one in a thousand does, a single row's 128 columns hold none or one
    for k in mlp_ref.ORDER:
        e = np.linalg.norm(got[k] - want[k]) / np.linalg.norm(want[k])
        print(k, "relative error", e)
        assert e <= 2.0 ** -10, k
