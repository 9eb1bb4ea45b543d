"""The training loss is an FP64 number: the mean of the FP32 differences' exact squares, summed in FP64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def unit_rms(rng, shape):
    """Random FP32 images whose unit-RMS factor rounds to exactly 1: the last pixel makes up the sum."""
    out = rng.standard_normal(shape).astype(np.float32)
    sq = lambda a: math.fsum(np.square(a.astype(np.float64)).ravel())  # noqa: E731
    for im in out:
        im[-1, -1] = 0.0
        im *= np.float32(math.sqrt((im.size - 1) / sq(im)))
        im[-1, -1] = math.sqrt(im.size - sq(im))
        assert abs(math.sqrt(im.size / sq(im)) - 1.0) < 2e-8    # (FP32's neighbours of 1: 6e-8 below, 1.2e-7 above)
    return out


@pytest.mark.parametrize("ny,nx,count", [(16, 16, 1), (24, 40, 3), (128, 128, 8)])
def test_loss_is_the_fp64_mean_of_the_squared_differences(ny, nx, count):
    """An untrained network returns the scaled tbar; with factors of 1 the differences are RN(tbar - target).
    Their squares are exact in FP64; a thread adds at most 2 of them, then 8 levels of a block's sum, and
    1024 blocks' sums in 12 more: 22 roundings and the quotient, 24 * 2^-53 of a sum of positive terms."""
    import paper_1807_10151_gb300 as S
    net = S.CNN(ny, nx, max_batch=count, seed=5)
    for seed in range(4):
        rng = np.random.default_rng(seed)
        tb, tg = unit_rms(rng, (count, ny, nx)), unit_rms(rng, (count, ny, nx))
        x = rng.uniform(0.5, 1.5, (count, ny, nx)).astype(np.float32)
        _, loss = net.gradients(*(torch.tensor(a, device="cuda") for a in (x, tb, tg)))
        d = (tb - tg).astype(np.float64)
        want = math.fsum(np.square(d).ravel()) / d.size
        assert abs(loss - want) <= 24 * 2.0 ** -53 * want
