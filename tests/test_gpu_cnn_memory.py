"""The network's device memory, and a backward pass whose gradient buffers serve two layers each."""
import gc

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def used():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("ny,nx,count", [(64, 64, 512), (130, 100, 160), (90, 86, 300)])
def test_a_network_takes_the_memory_of_unpadded_layers(ny, nx, count):
    """584 bytes per pixel, the room of every layer's activations and gradients without padding (288
    BF16 channels) and two FP32 images; 64 MB for the parameters, their gradients' partial sums and the
    allocator's granularity."""
    import paper_1807_10151_gb300 as S
    S.CNN(8, 8, max_batch=1).close()
    before = used()
    net = S.CNN(ny, nx, max_batch=count)
    grown = used() - before
    net.close()
    assert grown <= 584 * ny * nx * count + (64 << 20)


def test_gradients_repeat_on_used_buffers():
    """Another batch in between leaves nothing behind in the buffers (their zero borders included)."""
    import paper_1807_10151_gb300 as S
    gen = torch.Generator(device="cuda").manual_seed(1)
    net = S.CNN(19, 37, max_batch=5, seed=2)
    p = net.get_params()
    S.CNN.unflatten(p)[4][0][...] = 0.1 * np.random.default_rng(0).standard_normal((1, 32, 3, 3))
    net.set_params(p)
    a = [torch.rand(3, 19, 37, device="cuda", generator=gen) + 0.1 for _ in range(3)]
    b = [torch.rand(5, 19, 37, device="cuda", generator=gen) + 0.1 for _ in range(3)]
    first, loss = net.gradients(*a)
    net.gradients(*b)
    again, loss2 = net.gradients(*a)
    np.testing.assert_array_equal(first, again)
    assert loss == loss2 and np.abs(first).max() > 0
