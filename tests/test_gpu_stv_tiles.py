"""S_TV on resident tiles (32, 64 or 128 rows by 32 columns per block) at the sizes where a
tile, its ring or the choice of its height can go wrong, against the oracle's Algorithm 1."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1807_10151_gb300 import synth

from gpu_cases import gpu_geometry, rel_l2, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# below, at and above one tile; one row or column of a second tile; then images whose 32-row
# tiles do not fit the device at once (64 rows), whose 64-row tiles do not (128), and beyond
@pytest.mark.parametrize("ny,nx,K,a,gamma", [(31, 33, 4, 0.9, 0.1), (32, 32, 4, 0.9, 0.1), (33, 65, 4, 0.9, 0.1),
                                             (65, 31, 3, 0.5, 20.0), (1, 40, 3, 0.9, 0.05), (34, 2, 3, 0.9, 0.05),
                                             (600, 577, 3, 0.9, 2.0), (993, 801, 3, 0.9, 2.0), (1200, 1100, 2, 0.9, 2.0)])
def test_superiorize_at_tile_edges_matches_algorithm1(ny, nx, K, a, gamma):
    """l and the trials identical; the displacement within 2e-5: the image is rounded to FP32 when it
    is returned, at most 3e-8 per pixel of value < 1 (uniform: 1.7e-8 rms), so sqrt(n) 1.7e-8 against a
    displacement of norm about K gamma, 4e-6 at the largest size."""
    og = O.Geometry(nx, ny=ny, V=4, U=8)
    G = gpu_geometry(og)
    n = max(ny, nx)
    x = (synth.ellipse_phantom(n, 8, ny + nx)[:ny, :nx] * 0.9
         + 0.02 * np.random.default_rng(ny).standard_normal((ny, nx))).astype(np.float32)
    x[: min(ny, 4), : min(nx, 6)] = 0.25                     # a flat patch: undefined partials
    xd = to_dev(x)
    rc, ell, trials = G.superiorize(xd, 2, a, gamma, K)
    rrc, s, ell_o, tr_o = O.stv(x.astype(np.float64), 2, a, gamma, K)
    assert rc == 0 and rrc == 0 and ell == ell_o and trials == list(tr_o)
    assert rel_l2(xd.double().cpu().numpy() - x, s) <= 2e-5


def test_nan_image_backtracks_to_the_cap():
    """TV of an image with a NaN compares false: every trial is rejected and the image stays."""
    og = O.Geometry(40, ny=50, V=4, U=8)
    G = gpu_geometry(og)
    x = np.random.default_rng(3).uniform(size=(50, 40)).astype(np.float32)
    x[33, 35] = np.nan
    xd = to_dev(x)
    rc, ell, _ = G.superiorize(xd, 0, 0.9, 0.1, 2, max_trials=5)
    assert rc == -5 and ell == 5
    np.testing.assert_array_equal(xd.cpu().numpy(), x)
