"""S_TV by its two kernels: on tiles resident in shared memory where the launch's images fit the
device, in memory where they do not.  Which one a problem takes depends on how many problems share
its launch, so both have to give it the same steps."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1807_10151_gb300 import synth

from gpu_cases import gpu_geometry, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,a,gamma", [(1, 0.995, 0.5), (4, 0.99, 0.05)])
def test_a_problem_alone_equals_it_in_a_batch_that_does_not_fit(K, a, gamma):
    """26 images of 243^2 have 416 tiles of 128 rows, more than the device holds at two blocks per SM.
    l and the image are the same; TV(x_{k-1/2}) is the same terms added in another order: double-float
    sums of at most 40 terms (2^-47 each), then FP64, so within 1e-12."""
    import paper_1807_10151_gb300 as S
    og = O.Geometry(243, V=48, U=345)
    R = O.CSR(og)
    bs = [to_dev(np.asarray(synth.gaussian_noise(R.project(synth.ellipse_phantom(243, 12, 700 + c)), 0.01, 800 + c),
                            np.float32)) for c in range(2)]
    G = gpu_geometry(og)
    kw = dict(K=K, a=a, gamma=gamma, mu=1e-5, rho=0.8, max_iter=6)
    single = [G.solve(b, **kw) for b in bs]
    n = 26
    xs = [torch.zeros(243, 243, device="cuda") for _ in range(n)]
    reps = S.solve_batched([G] * n, [bs[c % 2] for c in range(n)], xs, **kw)
    for c in (0, 1, n - 1):
        x1, r1, _ = single[c % 2]
        assert reps[c]["status"] == 0 and reps[c]["ell"] == r1["ell"]
        assert reps[c]["tv_last"] == pytest.approx(r1["tv_last"], rel=1e-12, abs=0.0)
        np.testing.assert_array_equal(xs[c].cpu().numpy(), x1.cpu().numpy())


def test_one_step_on_an_image_whose_quotients_underflow():
    """The last row's tbar is a / T of the terms above it.  With a near FP32's least normal number and
    T = 1e-12 the quotient's residual a - q T is subnormal; the step must still take the rounded quotient,
    as tv_tbar does.  The last row is 0, so after one step it is c tbar by the pair step: the product's two
    parts added, the low one rounded to a subnormal number."""
    n = 1500
    og = O.Geometry(n, ny=2, V=4, U=8)
    G = gpu_geometry(og)
    rng = np.random.default_rng(4)
    x = np.zeros((2, n), np.float32)
    x[0, ::2] = rng.uniform(0.5e-37, 4e-37, n // 2)
    x[0, 1::2] = 1e-12 * rng.uniform(0.5, 1.5, n // 2)
    xd = to_dev(x)
    _, nn, t = G.tv_tbar(xd)
    gamma = 2e-13 * np.sqrt(nn)
    rc, ell, trials = G.superiorize(xd, 0, 0.9, gamma, 1)
    assert rc == 0 and trials == [1]
    ct = float(np.float32(gamma / np.sqrt(nn))) * t.double().cpu().numpy()[1]     # exact in FP64
    hi = ct.astype(np.float32)
    want = hi + (ct - hi).astype(np.float32)
    assert np.count_nonzero(want[::2]) > 700
    np.testing.assert_array_equal(xd.cpu().numpy()[1], want)


@pytest.mark.parametrize("nx", [4, 6, 12, 38, 107])
def test_step_length_is_rounded_from_fp64(nx):
    """Two rows of 1 and 0: tbar is -1 above and 1 below but for the last column, so ||tbar||^2 = 2 (nx - 1)
    exactly and the lower row is the step length c = RN(gamma / ||tbar||) itself.  gamma is taken so that
    the exact quotient is 2^-49 beside the middle of two FP32 numbers, four times FP64's error (a rounded
    reciprocal root and a product, 2^-51) and an eighth of a double-float product's."""
    from decimal import Decimal, getcontext
    getcontext().prec = 50
    og = O.Geometry(nx, ny=2, V=4, U=8)
    G = gpu_geometry(og)
    root = Decimal(2 * (nx - 1)).sqrt()
    rng = np.random.default_rng(nx)
    for k in range(48):
        lo = np.float32(rng.uniform(0.004, 0.016))
        hi = np.nextafter(lo, np.float32(1))
        mid = (Decimal(float(lo)) + Decimal(float(hi))) / 2
        up = k % 2 == 0
        gamma = float(mid * root * (1 + Decimal(2) ** -49 * (1 if up else -1)))
        off = Decimal(gamma) / root / mid - 1
        assert Decimal(2) ** -50 < abs(off) < Decimal(2) ** -48 and (off > 0) == up
        xd = to_dev(np.stack([np.ones(nx), np.zeros(nx)]))
        rc, ell, trials = G.superiorize(xd, 0, 0.9, gamma, 1)
        assert rc == 0 and trials == [1]
        want = np.full(nx, hi if up else lo)
        want[-1] = 0.0
        np.testing.assert_array_equal(xd.cpu().numpy()[1], want)
