"""Standalone operator calls in a row: different buffers, streams, options and an output that
overlaps the input, each against the same call on a geometry of its own."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def fresh(nx, ny, V, U, storage, op, a, **kw):
    import paper_1807_10151_gb300 as S
    out = getattr(S.Geometry(nx, ny, n_views=V, n_bins=U, storage=storage), op)(a, **kw)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("storage,batch", [("f32", 1), ("bf16", 1), ("f32", 3), ("bf16", 2)])
def test_calls_in_a_row_on_other_buffers_and_streams(storage, batch):
    """Each result equals (bit for bit) the same call on a new geometry, whatever was enqueued before it
    and on whichever stream, without a synchronisation between the calls."""
    import paper_1807_10151_gb300 as S
    nx, ny, V, U = 45, 38, 31, 67                                  # rows of odd length
    dt = torch.bfloat16 if storage == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(7)
    G = S.Geometry(nx, ny, n_views=V, n_bins=U, storage=storage)
    streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
    calls = []
    for k in range(12):
        x = torch.randn(batch, ny, nx, device="cuda", generator=g).to(dt)
        y = torch.randn(batch, V, U, device="cuda", generator=g).to(dt)
        p = torch.randn(batch, ny, nx, device="cuda", generator=g)
        torch.cuda.synchronize()
        op, a, kw = [("project", x, {}), ("backproject", y, {}), ("precondition", p, dict(mu=10.0 ** -(1 + k % 5)))][k % 3]
        with torch.cuda.stream(streams[k % 2 + k // 6]):
            calls.append((op, a, kw, getattr(G, op)(a, **kw)))
    torch.cuda.synchronize()
    for op, a, kw, out in calls:
        assert torch.equal(out, fresh(nx, ny, V, U, storage, op, a, **kw)), (op, kw)


def test_s_tv_and_art_between_operator_calls():
    """S_TV, TV and ART share the operators' scratch and descriptors (ART switches the low part of x off)."""
    import paper_1807_10151_gb300 as S
    nx, ny, V, U = 40, 33, 20, 59
    g = torch.Generator(device="cuda").manual_seed(3)
    G = S.Geometry(nx, ny, n_views=V, n_bins=U)
    x = torch.rand(ny, nx, device="cuda", generator=g)
    b = torch.rand(V, U, device="cuda", generator=g)
    first = G.project(x).clone()
    a1, rep1 = G.art(b, K=2, cycles=1, lam=0.05)
    y1 = x.clone()
    r1 = G.superiorize(y1, 0, 0.9, 0.05, 70)                       # more steps than are read back inline
    tv1 = G.tv_tbar(x)
    a2, rep2 = G.art(b, K=2, cycles=1, lam=0.05)
    y2 = x.clone()
    r2 = G.superiorize(y2, 0, 0.9, 0.05, 70)
    assert torch.equal(a1, a2) and rep1 == rep2
    assert torch.equal(y1, y2) and r1 == r2 and len(r1[2]) == 70 and r1[1] == sum(r1[2])
    tv2 = G.tv_tbar(x)
    assert tv1[:2] == tv2[:2] and torch.equal(tv1[2], tv2[2])
    assert torch.equal(first, G.project(x))


def test_backprojection_into_its_own_sinogram():
    """An output that overlaps the input gets the result of separate buffers."""
    n = 36
    y = torch.randn(n, n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = fresh(n, n, n, n, "f32", "backproject", y.clone())
    got = fresh(n, n, n, n, "f32", "backproject", y, out=y)
    assert torch.equal(got, want) and got.data_ptr() == y.data_ptr()


@pytest.mark.parametrize("ny,nx", [(64, 64), (5, 7), (48, 1)])
def test_preconditioner_in_place(ny, nx):
    g = torch.randn(2, ny, nx, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    want = fresh(nx, ny, 4, 2 * math.ceil(nx), "f32", "precondition", g.clone())
    got = fresh(nx, ny, 4, 2 * math.ceil(nx), "f32", "precondition", g, out=g)
    assert torch.equal(got, want)
    assert np.isfinite(got.cpu().numpy()).all()
