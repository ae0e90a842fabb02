"""The training kernel at the edges of its tiles (16 samples) and grid (304
CTAs), against the oracle's backward pass with the tolerance of the gradient
test (1e-4 of a block's largest entry, float accumulation); samples with a
non-finite feature or target are skipped but count in the mean; unaligned
inputs; and training that repeats bit for bit."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


def _case(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((n, 12)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    return x, t, mlp.init(seed)


@pytest.mark.parametrize("n,bad", [(1, 0), (15, 0), (16, 0), (17, 3), (33, 0), (4864, 0), (4869, 7),
                                   (10007, 0)])
def test_gradient_at_tile_edges(orc, n, bad):
    import torch
    from paper_2211_12243_gb300 import hydro
    x, t, theta = _case(n, 7)
    rng = np.random.default_rng(1)
    skip = rng.choice(n, bad, replace=False)
    xb, tb = x.copy(), t.copy()
    for i, s in enumerate(skip):
        if i % 2:
            xb[s, i % 12] = np.nan if i % 3 else np.inf
        else:
            tb[s] = np.nan
    H = hydro.Hydro(hydro.default_config(precision="mixed"))
    H.mlp_load(theta)
    flat = torch.empty(12 * n + 1, dtype=torch.float32, device="cuda")
    xg = flat[1:].view(n, 12)   # (a base address that is only 4-byte aligned)
    xg.copy_(torch.as_tensor(xb))
    g, loss = H.mlp_gradient(xg, torch.as_tensor(tb, device="cuda"))
    g = g.cpu().numpy().astype(np.float64)
    keep = np.setdiff1d(np.arange(n), skip)
    x64, t64 = x[keep].astype(np.float64), t[keep].astype(np.float64)
    share = keep.size / n
    go = mlp.backward(theta, x64, t64) * share
    assert float(loss.item()) == pytest.approx(mlp.loss(theta, x64, t64) * share, rel=1e-4)
    y, _ = mlp.forward(theta, x64)
    k = 0
    for name, shp in mlp.SIZES:
        m = int(np.prod(shp))
        a, b = g[k:k + m], go[k:k + m]
        k += m
        if name in mlp.FIXED:
            assert np.all(a == 0.0)
            continue
        scale = np.mean(np.abs(y - t64)) if name == "b3" else np.max(np.abs(b))
        assert np.max(np.abs(a - b)) <= 1e-4 * scale + 1e-12, name
    H.close()


def test_training_repeats_bitwise():
    import torch
    from paper_2211_12243_gb300 import hydro
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    r = torch.rand((7, 5000), generator=g, device="cuda")
    faces = (0.1 + r).contiguous()
    faces[1] -= 0.6
    faces[4] -= 0.6
    out = []
    for _ in range(2):
        H = hydro.Hydro(hydro.default_config(precision="mixed"))
        loss = H.mlp_train(faces, 40, batch=777, seed=5)
        out.append((loss.cpu().numpy(), H.mlp_get()))
        H.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][0][-5:].mean() < out[0][0][:5].mean()


def test_gradients_on_two_streams():
    """Calls of one context on two streams at once, each with its own samples:
    the gradients of the calls alone (to the order of float sums)"""
    import torch
    from paper_2211_12243_gb300 import hydro
    H = hydro.Hydro(hydro.default_config(precision="mixed"))
    H.mlp_load(mlp.init(9))
    data, alone = [], []
    for seed in (1, 2):
        x, t, _ = _case(60000 + 17 * seed, seed)
        data.append((torch.as_tensor(x, device="cuda"), torch.as_tensor(t * seed, device="cuda")))
        g, loss = H.mlp_gradient(*data[-1])
        alone.append((g.clone(), loss.clone()))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in data]
    out = []
    for _ in range(10):
        for s, d in zip(streams, data):
            with torch.cuda.stream(s):
                out.append(H.mlp_gradient(*d, stream=s))
    torch.cuda.synchronize()
    for k, (g, loss) in enumerate(out):
        ga, la = alone[k % 2]
        assert float((g - ga).abs().max()) <= 1e-5 * float(ga.abs().max())
        assert float((loss - la).abs()) <= 1e-5 * float(la)
    H.close()
