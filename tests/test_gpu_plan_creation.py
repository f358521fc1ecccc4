"""A new plan's record and counters are cleared before its first call's kernels, on
whichever stream, and not by anything that comes later (needs a GB300)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("form,kw", [("sym", dict(W=2, target_snr_db=20.0)), ("tc_int", dict(W=1, bits=8))])
def test_plan_made_behind_queued_work_and_used_on_another_stream(form, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = 300, 260, 388
    A = torch.from_numpy(synth.laplace((M, K), 81, np.float32)).cuda()
    B = torch.from_numpy(synth.gaussian((K, N), 82, np.float32)).cuda()
    with tdg.Plan(M, N, K, L=128, dtype="f32", form=form, **kw) as p:
        ref = p.run(A, B)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.default_stream()):
        torch.cuda._sleep(100_000_000)             # some 50 ms on the default stream
    with tdg.Plan(M, N, K, L=128, dtype="f32", form=form, **kw) as p:
        C = torch.empty(M, N, device="cuda")
        p.quantize_pack(A, B, stream=side)
        side.synchronize()
        torch.cuda.synchronize()                   # the default stream's work is done too
        p.gemm(C, stream=side)
        side.synchronize()
        assert torch.equal(C, ref)
        p.run(A, B, C)                             # the counters stand at zero
        assert torch.equal(C, ref)


@pytest.mark.parametrize("goal", [dict(bits=7), dict(target_snr_db=20.0)])
def test_first_call_captured_and_the_graph_thrown_away(goal):
    """A capture queues the clearing and the upload of the noise table but may never
    run: an eager call after it, and a replay after that, find both done."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    A = torch.from_numpy(synth.laplace((300, 388), 83, np.float32)).cuda()
    B = torch.from_numpy(synth.gaussian((388, 260), 84, np.float32)).cuda()
    kw = dict(L=128, W=2, dtype="f32", form="sym", **goal)
    with tdg.Plan(300, 260, 388, **kw) as p:
        ref = p.run(A, B)
    with tdg.Plan(300, 260, 388, **kw) as p:
        C = torch.empty(300, 260, device="cuda")
        thrown, kept = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        for g in (thrown, kept):
            with torch.cuda.graph(g):
                p.run(A, B, C)
        del thrown
        for call in (lambda: p.run(A, B, C), kept.replay, lambda: p.run(A, B, C), kept.replay):
            C.zero_()
            call()
            assert torch.equal(C, ref)
