"""What a geometry's workspaces hold and share."""
import gc

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def used():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_a_batch_holds_a_geometrys_frequencies_once():
    """130 bytes per pixel and image of a batch without mirror pairs: twelve FP32 images (x, p and d in two
    layouts, g, z, h, tbar and the two low parts: 48), the backprojector's part sums (64), the transform's
    scratch and filter (18).  The frequencies, 4 bytes per pixel, depend on the geometry alone."""
    import paper_1807_10151_gb300 as S
    n, batch = 1024, 16
    G = S.Geometry(n, n_views=1, n_bins=8)
    x = torch.zeros(batch, n, n, device="cuda")
    y = torch.zeros(batch, 1, 8, device="cuda")
    G.project(x[:1], out=y[:1])                        # kernels loaded, one image's workspace
    before = used()
    G.project(x, out=y)
    grown = used() - before + 134 * n * n              # the first workspace is given back
    assert grown <= (130 * batch + 4) * n * n + (batch + 1) * (3 << 20)   # (an allocation per image, in units of 2 MB)


def test_frequencies_shared_by_batches_solves_and_streams():
    """Calls on other streams and other workspaces right behind the first use get the result of a
    geometry of their own."""
    import paper_1807_10151_gb300 as S
    n, V = 60, 20
    gen = torch.Generator(device="cuda").manual_seed(5)
    a = torch.randn(3, n, n, device="cuda", generator=gen)
    b = torch.rand(V, 86, device="cuda", generator=gen)
    new = lambda: S.Geometry(n, n_views=V, n_bins=86)  # noqa: E731
    want = [new().precondition(a[:k], 1e-4, 0.7).clone() for k in (1, 2, 3)]
    xs = new().solve(b, max_iter=3)[0].clone()
    G = new()
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for _ in range(2):
        got = [torch.empty_like(a[:k]) for k in (1, 2, 3)]
        torch.cuda.synchronize()
        for k, st in enumerate(streams):
            G.precondition(a[:k + 1], 1e-4, 0.7, out=got[k], stream=st)
        x = G.solve(b, max_iter=3)[0]
        torch.cuda.synchronize()
        assert all(torch.equal(g, w) for g, w in zip(got, want)) and torch.equal(x, xs)
