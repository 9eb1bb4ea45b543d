"""ART on images whose rays have more rows than a block has threads, or than one group of a thread's
rows holds (2 or 4 per thread, by the image's sides), with several rays per block and class."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1807_10151_gb300 import synth

from gpu_cases import gpu_geometry, rel_l2, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,V,cycles", [(256, 30, 7, 2), (257, 40, 7, 2), (513, 513, 6, 2), (640, 600, 8, 1), (1100, 300, 5, 1),
                                            (1024, 513, 5, 1), (1100, 1030, 5, 1), (70, 1025, 6, 2)])
def test_art_matches_oracle_beyond_512(nx, ny, V, cycles):
    """The bound of the smaller sizes: sums in more than FP32, the image in FP32."""
    og = O.Geometry(nx, ny=ny, V=V, U=int(1.42 * max(nx, ny)) + 2)
    R = O.CSR(og)
    x = synth.ellipse_phantom(max(nx, ny), 6, nx)[:ny, :nx]
    b = np.asarray(R.project(x) + 0.01 * np.random.default_rng(nx).standard_normal((V, og.U)), np.float32).astype(np.float64)
    ref = O.art(R, b, r=5.0, lam=0.3, cycles=cycles)
    xg, rep = gpu_geometry(og).art(to_dev(b), r=5.0, lam=0.3, cycles=cycles)
    assert rep["status"] == 0
    assert rel_l2(xg.double().cpu().numpy(), ref["x"]) <= 2e-5
