"""A call that is refused because its stream is under capture leaves the geometry usable."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("op", ["project", "precondition"])
def test_a_call_refused_under_capture_leaves_later_calls_as_they_were(op):
    import paper_1807_10151_gb300 as S
    cuda = C.CDLL("libcuda.so.1")                    # (torch's own capture also registers its random generator)
    G = S.Geometry(40, n_views=20, n_bins=57)
    x = torch.arange(1600, device="cuda", dtype=torch.float32).reshape(40, 40)
    y = torch.empty((20, 57) if op == "project" else (40, 40), device="cuda")
    call = getattr(G, op)
    want = call(x).clone()
    stream, graph = torch.cuda.Stream(), C.c_void_p()
    torch.cuda.synchronize()
    assert cuda.cuStreamBeginCapture_v2(C.c_void_p(stream.cuda_stream), 2) == 0      # 2: relaxed
    with pytest.raises(S.SupcgError):
        call(x, out=y, stream=stream)
    assert cuda.cuStreamEndCapture(C.c_void_p(stream.cuda_stream), C.byref(graph)) != 0   # the call ended the capture
    torch.cuda.synchronize()
    for st in (torch.cuda.current_stream(), stream):
        y.zero_()
        torch.cuda.synchronize()
        call(x, out=y, stream=st)
        torch.cuda.synchronize()
        assert torch.equal(y, want)
