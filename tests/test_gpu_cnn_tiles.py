"""The network at the edges of its tiles: strips of 128 columns, runs of rows per
CTA, pairs of rows in the weight gradient.  Forward and gradients against the
oracle's FP64 layers with the same BF16 roundings, at the tolerances derived
there (forward a quarter of BF16's unit 2^-8, gradients two flipped roundings)."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_cnn import bf16, random_params, reference_forward, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ny,nx,count", [(1, 1, 1), (1, 129, 2), (3, 128, 1), (2, 16, 5), (17, 130, 2), (9, 257, 1)])
def test_network_at_tile_edges_matches_oracle(ny, nx, count):
    import paper_1807_10151_gb300 as S
    rng = np.random.default_rng(ny * 1000 + nx)
    net = S.CNN(ny, nx, max_batch=count + 1, seed=3)      # more room than images
    p = random_params(net, rng)
    x = rng.uniform(0.5, 1.5, size=(count, ny, nx)).astype(np.float32)
    tb = rng.standard_normal((count, ny, nx)).astype(np.float32)
    tg = rng.standard_normal((count, ny, nx)).astype(np.float32)
    dev = [torch.tensor(a, device="cuda") for a in (x, tb, tg)]
    ref, acts, _ = reference_forward(p, x, tb)
    for _ in range(2):                                    # the second pass reuses the buffers
        assert rel_l2(net.forward(dev[0], dev[1]).cpu().numpy(), ref) <= 1e-3
    g, loss = net.gradients(*dev)
    n = ny * nx
    tgs = np.stack([t * np.float32(np.sqrt(n / np.sum(t.astype(np.float64) ** 2))) for t in tg])
    assert loss == pytest.approx(np.mean((ref - tgs) ** 2), rel=1e-2)
    layers = S.CNN.unflatten(p.astype(np.float64))
    want = [np.zeros_like(W) for W, _ in layers], [np.zeros_like(b) for _, b in layers]
    out = net.forward(dev[0], dev[1]).cpu().numpy().astype(np.float64)
    for k in range(count):
        G = bf16(2.0 * (out[k] - tgs[k]) / out.size)[None]
        for li in range(4, -1, -1):
            dx, dW, db = O.conv3x3_backward(acts[k][li], bf16(layers[li][0]), G, want_dx=li > 0)
            want[0][li] += dW
            want[1][li] += db
            if li > 0:
                G = bf16(dx * (acts[k][li] > 0))
    got = S.CNN.unflatten(g.astype(np.float64))
    for li in range(5):
        assert rel_l2(got[li][0], want[0][li]) <= 1e-2, li
        assert rel_l2(got[li][1], want[1][li]) <= 1e-2, li


def test_all_zero_and_very_large_images_keep_their_scales():
    """The unit-RMS factors: 0 for an all-zero image, and right where squares leave FP32's range."""
    import paper_1807_10151_gb300 as S
    rng = np.random.default_rng(5)
    net = S.CNN(24, 40, max_batch=3, seed=3)
    random_params(net, rng)
    x = rng.uniform(0.5, 1.5, size=(1, 24, 40)).astype(np.float32)
    tb = rng.standard_normal((1, 24, 40)).astype(np.float32)
    run = lambda a, t: net.forward(torch.tensor(a, device="cuda"), torch.tensor(t, device="cuda")).cpu().numpy()  # noqa: E731
    base = run(x, tb)
    for s in (2.0 ** 70, 2.0 ** -70):                     # powers of two: the scaled images are bit for bit the same
        np.testing.assert_array_equal(run(x * np.float32(s), tb * np.float32(s)), base)
    assert np.all(np.isfinite(run(0 * x, 0 * tb)))
