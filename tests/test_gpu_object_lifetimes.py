"""What a workspace keeps from one call to the next is matched by objects that may since have been destroyed,
and a new one may get a destroyed one's address."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_new_geometry_at_a_destroyed_ones_address():
    import paper_1807_10151_gb300 as S
    kw = dict(K=1, a=0.99, gamma=0.3, max_iter=3)
    gen = torch.Generator(device="cuda").manual_seed(2)
    b0 = torch.rand(30, 57, device="cuda", generator=gen)
    owner = S.Geometry(40, n_views=30, n_bins=57)
    seen = {}
    for n in (48, 33, 56, 41, 64, 37, 52, 45):
        G = S.Geometry(n, n_views=24, n_bins=92)
        b = torch.rand(24, 92, device="cuda", generator=gen)
        want, _, _ = G.solve(b, **kw)
        xs = [torch.zeros(40, 40, device="cuda"), torch.zeros(n, n, device="cuda")]
        S.solve_batched([owner, G], [b0, b], xs, **kw)
        np.testing.assert_array_equal(xs[1].cpu().numpy(), want.cpu().numpy())
        seen[G.handle.value] = seen.get(G.handle.value, 0) + 1
        G.close()
    if max(seen.values()) < 2:
        pytest.skip("the allocator gave every geometry an address of its own")


def test_a_new_network_at_a_destroyed_ones_address():
    """The solve's captured body is not taken over by a network that got a destroyed one's address; each
    network here has room for another number of images, so its buffers lie elsewhere."""
    import paper_1807_10151_gb300 as S
    n = 32
    kw = dict(K=4, a=0.97, gamma=0.3, max_iter=4)
    b = torch.rand(30, 46, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    owner = S.Geometry(n, n_views=30, n_bins=46)
    seen = {}
    for c, cap in enumerate((1, 9, 2, 30, 4, 1, 17)):
        net = S.CNN(n, n, max_batch=cap, seed=c + 1)
        p = net.get_params()
        S.CNN.unflatten(p)[4][0][...] = 0.05 * np.random.default_rng(c).standard_normal((1, 32, 3, 3))
        net.set_params(p)
        want, rw, _ = S.Geometry(n, n_views=30, n_bins=46).solve_learned(net, b, **kw)
        got, rg, _ = owner.solve_learned(net, b, **kw)
        np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())
        assert rw["ell"] == rg["ell"] and rw["n_learned"] == rg["n_learned"]
        seen[net.handle.value] = seen.get(net.handle.value, 0) + 1
        net.close()
    if max(seen.values()) < 2:
        pytest.skip("the allocator gave every network an address of its own")
