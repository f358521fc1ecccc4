"""The tensor-core code kernel at the edges of its tiles (64 and 128), for each
layout of the inputs, aligned and unaligned rows, with the statistics in the same
read and behind them: C against the oracle (needs a GB300)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 130, 129), (65, 200, 388), (300, 260, 64)])
@pytest.mark.parametrize("transA,transB", [("N", "N"), ("T", "T")])
@pytest.mark.parametrize("L,kw", [(64, dict(bits=8)), (128, dict(bits=8)), (64, dict(target=20.0)),
                                  (128, dict(target=20.0)), (256, dict(target=20.0))])
def test_codes_tile_edges(orc, M, N, K, transA, transB, L, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    A, B = synth.laplace((M, K), 71, np.float32), synth.gaussian((K, N), 72, np.float32)
    if M > 64:
        A[:64, :64] = 0.0                  # a zero block at L = 64
    ref = orc.tc_int_gemm(A, B, L=L, bits=kw.get("bits", 0))
    goal = dict(bits=8) if "bits" in kw else dict(target_snr_db=kw["target"])
    with tdg.Plan(M, N, K, L=L, W=1, dtype="f32", form="tc_int", transA=transA, transB=transB,
                  **goal) as p:
        As = torch.from_numpy(np.ascontiguousarray(A if transA == "N" else A.T)).cuda()
        Bs = torch.from_numpy(np.ascontiguousarray(B if transB == "N" else B.T)).cuda()
        C = p.run(As, Bs)
        i = p.info()
        assert (i["gamma_a"], i["gamma_b"]) == (ref.plan.gA, ref.plan.gB)
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 130, 129), (300, 260, 388)])
@pytest.mark.parametrize("L", [128, 256])
def test_fp8_codes_do_not_depend_on_the_layout(M, N, K, L):
    """E4M3 codes from k-contiguous and from x-contiguous inputs, 16-byte aligned
    rows and not: the same product bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    A = torch.from_numpy(synth.laplace((M, K), 73, np.float32)).cuda()
    B = torch.from_numpy(synth.gaussian((K, N), 74, np.float32)).cuda()
    out = []
    for tA, tB, pad in (("N", "N", 0), ("T", "T", 0), ("N", "T", 3), ("T", "N", 4)):
        As, Bs = A if tA == "N" else A.t(), B if tB == "N" else B.t()
        bufs = [torch.full((X.shape[0], X.shape[1] + pad), 7.0, device="cuda") for X in (As, Bs)]
        for buf, X in zip(bufs, (As, Bs)):
            buf[:, : X.shape[1]] = X
        with tdg.Plan(M, N, K, L=L, W=1, dtype="f32", form="tc_fp8", transA=tA, transB=tB,
                      lda=bufs[0].shape[1], ldb=bufs[1].shape[1]) as p:
            out.append(p.run(bufs[0], bufs[1]))
    assert all(torch.equal(c, out[0]) for c in out[1:])


@pytest.mark.parametrize("form,K", [("tc_int", 130), ("tc_fp8", 130), ("tc_int", 64 * 67)])
@pytest.mark.parametrize("M,N", [(256, 256), (2600, 2100), (3000, 3001), (5000, 4097)])
def test_tensor_core_last_wave(M, N, K, form):
    """Whole and half tiles (the last wave's) and factors beyond the first 32 slabs:
    every row block of a product equals the same rows multiplied alone, whose tiles
    fall differently (1, 99, 144 and 340 tile pairs for 76 clusters)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    L = 128 if form == "tc_fp8" else 64
    A = torch.from_numpy(synth.laplace((M, K), 75, np.float32)).cuda()
    B = torch.from_numpy(synth.gaussian((K, N), 76, np.float32)).cuda()
    kw = dict(L=L, W=1, dtype="f32", form=form, **({} if form == "tc_fp8" else dict(bits=6)))
    C = torch.full((M, N), 3.0, device="cuda")
    Cin = C.clone()
    with tdg.Plan(M, N, K, **kw) as p:
        p.run(A, B, C)
        p.run(A, B, Cin, alpha=1.0, beta=-1.0)
        assert p.info()["device_status"] == 0
    assert torch.equal(Cin, C - 3.0)
    for r0 in range(0, M, 1024):
        rows = min(1024, M - r0)
        with tdg.Plan(rows, N, K, **kw) as p:
            part = p.run(A[r0:r0 + rows], B)
            assert torch.equal(part, C[r0:r0 + rows]), r0
