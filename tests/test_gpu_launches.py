"""Kernels that a call queues, counted in a captured graph (needs a GB300)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _kernels(call, stream):
    """Kernel nodes of what `call` queues on `stream`."""
    rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    st, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(st, 1) == 0             # thread-local mode
    call()
    assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t()
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kind, kernels = ctypes.c_int(), 0
    for node in nodes:
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return kernels


# statistics, levels, pack, then the products: of a symmetric 128 x 128 target W = 2 with
# either rounding and each higher W with one, and the plain fallback
@pytest.mark.parametrize("form,W,kw,shape,kernels", [
    ("sym", 2, dict(target_snr_db=20.0), (4096, 4096, 512), 3 + 2 + 1),
    ("sym", 4, dict(target_snr_db=20.0), (4096, 4096, 512), 3 + 2 + 1 + 1 + 1),
    ("sym", 2, dict(bits=6), (4096, 4096, 512), 3),
    ("sym", 2, dict(target_snr_db=20.0), (700, 700, 512), 3 + 1),
    ("tc_fp8", 1, {}, (512, 512, 512), 2),
    ("tc_int", 1, dict(target_snr_db=20.0), (512, 512, 512), 3)])
def test_kernels_queued(form, W, kw, shape, kernels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = shape
    A, B = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda")
    C, st = torch.empty(M, N, device="cuda"), torch.cuda.Stream()
    torch.cuda.synchronize()
    with tdg.Plan(M, N, K, L=128, W=W, dtype="f32", form=form, **kw) as p:
        p.run(A, B, C, stream=st)
        st.synchronize()
        assert _kernels(lambda: p.run(A, B, C, stream=st), st) == kernels
