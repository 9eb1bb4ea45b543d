"""Backprojector tiles of 8, 16 and 32 rows: a pixel sums its views in one order whatever the tile, so the
choice (by the number of blocks of the launch) shows in no bit, on images with ragged last tiles.  And the
kernel over mirror pairs against the oracle."""
import math

import numpy as np
import pytest

from oracle import oracle as O

from gpu_cases import gpu_geometry, rel_l2, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 4 blocks per tile of 32 x 32, on 152 SMs: a single call has 8 to 36 blocks (8 rows), 7 together 56 (8 rows),
# 84, 112 (16) or 252 (32), 40 together 320 and more (32)
# (default angles: the kernel over mirror pairs, from V = 5 on; skewed ones: the general kernel)
@pytest.mark.parametrize("skew", [0.0, 0.01])
@pytest.mark.parametrize("nx,ny,V,U", [(33, 37, 41, 59), (64, 40, 50, 92), (31, 65, 3, 80), (65, 72, 129, 101), (40, 8, 33, 150)])
def test_tile_rows_change_no_bit(nx, ny, V, U, skew):
    og = O.Geometry(nx, ny=ny, V=V, U=U, theta=np.arange(V) * math.pi / V + skew)
    assert (gpu_geometry(og).mirror_pairs() == 0) == (skew > 0)
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


def test_batch_mixing_both_kernels_equals_single_solves():
    """Problems with and without mirror pairs in one schedule: each kernel's launch skips the other's problems."""
    import paper_1807_10151_gb300 as S
    kw = dict(K=1, a=0.99, gamma=0.3, mu=1e-4, rho=0.8, max_iter=5)
    ogs = [O.Geometry(n, ny=n + 3, V=V, U=U, theta=np.arange(V) * math.pi / V + skew)
           for n, V, U, skew in ((40, 33, 61, 0.01), (37, 35, 59, 0.0), (70, 20, 101, 0.0), (33, 21, 55, 0.02), (20, 30, 33, 0.0))]
    g = torch.Generator(device="cuda").manual_seed(6)
    bs = [torch.rand(og.V, og.U, device="cuda", generator=g) for og in ogs]
    xs = [torch.zeros(og.ny, og.nx, device="cuda") for og in ogs]
    reps = S.solve_batched([gpu_geometry(og) for og in ogs], bs, xs, **kw)
    for og, b, xb, rb in zip(ogs, bs, xs, reps):
        x, rep, _ = gpu_geometry(og).solve(b, **kw)
        assert torch.equal(xb, x) and rep["f_last"] == rb["f_last"]


# odd and even widths down to one column, half widths at and around a tile's 32 columns, bins finer (three
# candidates) and coarser than pixels, a shifted detector, and unpaired views among the pairs
@pytest.mark.parametrize("nx,ny,V,U,off,dsf,extra", [
    (1, 9, 8, 15, 0.0, 1.0, []), (2, 1, 12, 7, 0.0, 1.0, []), (63, 17, 30, 81, 0.0, 1.0, []), (64, 15, 31, 70, 0.01, 1.0, []),
    (65, 33, 32, 95, 0.0, 0.6, []), (66, 16, 90, 61, -0.02, 1.7, []), (47, 50, 26, 71, 0.0, 1.0, [0.2, 0.7, 2.0]),
    (130, 40, 47, 190, 0.003, 0.9, [1.0])])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_mirror_pairs_match_oracle(nx, ny, V, U, off, dsf, extra, storage):
    """The repository's bound for a backprojection, 1e-5 relative L2 (FP32 weights and sums); bf16 results are
    rounded once more, to 2^-9 of each value at most."""
    d = 1.0 / max(nx, ny)
    og = O.Geometry(nx, ny=ny, V=V + len(extra), U=U, off=off, ds=d * dsf, theta=np.array([v * math.pi / V for v in range(V)] + extra))
    y = torch.tensor(np.random.default_rng(nx * 100 + V).standard_normal((og.V, U)), dtype=torch.float32)
    if storage == "bf16":
        y = y.bfloat16()
    out = gpu_geometry(og, storage).backproject(y.cuda()).double().cpu().numpy()
    assert rel_l2(out, O.CSR(og).backproject(y.double().numpy())) <= (1e-5 if storage == "f32" else 1e-5 + 2.0 ** -9)
