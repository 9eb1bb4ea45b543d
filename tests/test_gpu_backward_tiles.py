"""Backprojector tiles of 8, 16 and 32 rows: a pixel sums its views in one order whatever the tile, so the
choice (by the number of blocks of the launch) shows in no bit, on images with ragged last tiles."""
import pytest

from oracle import oracle as O

from gpu_cases import gpu_geometry

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 4 blocks per tile of 32 x 32, on 152 SMs: a single call has 8 to 36 blocks (8 rows), 7 together 56 (8 rows),
# 84, 112 (16) or 252 (32), 40 together 320 and more (32)
@pytest.mark.parametrize("nx,ny,V,U", [(33, 37, 41, 59), (64, 40, 50, 92), (31, 65, 3, 80), (65, 72, 129, 101), (40, 8, 33, 150)])
def test_tile_rows_change_no_bit(nx, ny, V, U):
    og = O.Geometry(nx, ny=ny, V=V, U=U)
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    y = torch.randn(40, V, U, device="cuda", generator=g)
    many = gpu_geometry(og).backproject(y)
    some = gpu_geometry(og).backproject(y[:7].contiguous())
    G = gpu_geometry(og)
    torch.cuda.synchronize()
    assert torch.equal(many[:7], some)
    for c in (0, 6, 39):
        assert torch.equal(many[c], G.backproject(y[c].contiguous()))


def test_solver_pass_changes_no_bit():
    """The pass over two sinograms, from one problem (8 rows) and from 24 in one launch (32 rows)."""
    import paper_1807_10151_gb300 as S
    og = O.Geometry(37, ny=45, V=35, U=67)
    kw = dict(K=1, a=0.99, gamma=0.3, mu=1e-4, rho=0.8, max_iter=4)
    g = torch.Generator(device="cuda").manual_seed(5)
    bs = list(torch.rand(24, og.V, og.U, device="cuda", generator=g))
    xs = [torch.zeros(og.ny, og.nx, device="cuda") for _ in bs]
    reps = S.solve_batched([gpu_geometry(og) for _ in bs], bs, xs, **kw)
    for c in (0, 23):
        x, rep, _ = gpu_geometry(og).solve(bs[c], **kw)
        assert torch.equal(xs[c], x) and rep["f_last"] == reps[c]["f_last"]
