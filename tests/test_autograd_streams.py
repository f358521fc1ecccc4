"""Plans that the differentiation form shares never run on two streams at once."""
import contextlib

import pytest

torch = pytest.importorskip("torch")

OPTS = dict(L=64, W=2, form="sym", bits=6, dtype="f32")


class _Ctx:
    needs_input_grad = (True, True, False)
    opts = OPTS

    def __init__(self, A, B):
        self.saved_tensors = (A, B)


class _Stream:
    def __init__(self, n):
        self.cuda_stream, self.waited = n, []

    def wait_stream(self, other):
        self.waited.append(other.cuda_stream)


class _Plan:
    made = 0

    def __init__(self, *a, **kw):
        _Plan.made += 1
        self.streams = []

    def run(self, A, B, C, alpha=1.0, beta=0.0, stream=None):
        self.streams.append(stream.cuda_stream if stream is not None
                            else torch.cuda.current_stream().cuda_stream)


@pytest.fixture
def ag(monkeypatch):
    """autograd on CPU tensors: a fake plan, two fake streams, capture on demand."""
    from paper_1110_5765_gb300 import autograd as ag
    cur, side = _Stream(1), _Stream(2)
    state = {"stream": cur, "capturing": True}

    @contextlib.contextmanager
    def on(st):
        old, state["stream"] = state["stream"], st
        yield
        state["stream"] = old

    monkeypatch.setattr(ag, "Plan", _Plan)
    monkeypatch.setattr(ag, "_plans", {})
    monkeypatch.setattr(ag, "_side_stream", lambda d: side)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: state["stream"])
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: state["capturing"])
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda self, s: None, raising=False)
    return ag, state, cur, side, on


@pytest.mark.parametrize("square", [True, False])
def test_captured_adjoints_with_one_plan_stay_on_one_stream(ag, square):
    """dA = dC B^T and dB = A^T dC of a square layer whose A and B are transposed
    views have the same shape, layout and options, so the same plan."""
    ag, *_ = ag
    A = torch.randn(96, 96).t() if square else torch.randn(96, 96)
    B = torch.randn(96, 96).t()
    ag.TDGemmFn.backward(_Ctx(A, B), torch.randn(96, 96))
    assert len(ag._plans) == (1 if square else 2)
    for p in ag._plans.values():
        assert len(set(p.streams)) == 1, p.streams


def test_a_plan_waits_for_the_stream_that_used_it_last(ag):
    ag, state, cur, side, on = ag
    state["capturing"] = False
    A, B = torch.randn(64, 64), torch.randn(64, 64)
    ag.product(A, B, OPTS)
    with on(side):
        ag.product(A, B, OPTS)
        ag.product(A, B, OPTS)
    ag.product(A, B, OPTS)
    assert (side.waited, cur.waited) == ([1], [2])


@pytest.mark.gpu
def test_square_layer_of_transposed_views_captured():
    """Replays of a captured step, then an ordinary one: the eager gradients."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1110_5765_gb300 import autograd as ag
    g = torch.Generator(device="cuda").manual_seed(3)
    A, B, G = (torch.randn(512, 512, generator=g, device="cuda") for _ in range(3))
    A, B = A.t().requires_grad_(), B.t().requires_grad_()
    opts = dict(L=128, W=2, form="sym", target_snr_db=20.0)

    def step():
        return torch.autograd.grad(ag.tdg_matmul(A, B, **opts), (A, B), G)

    ref = [x.clone() for x in step()]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = step()
    for _ in range(3):
        for x in out:
            x.zero_()
        graph.replay()
        assert all(torch.equal(x, r) for x, r in zip(out, ref))
    assert all(torch.equal(x, r) for x, r in zip(step(), ref))
    ag.clear_plan_cache()


@pytest.mark.gpu
def test_one_shape_on_two_streams():
    """Products of one shape queued on two streams in turn, without the caller
    ordering them: each is the product that its own inputs give."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1110_5765_gb300 import autograd as ag
    g = torch.Generator(device="cuda").manual_seed(4)
    A = [torch.randn(700, 900, generator=g, device="cuda") for _ in range(6)]
    B = [torch.randn(900, 500, generator=g, device="cuda") for _ in range(6)]
    opts = dict(L=128, W=2, form="sym", target_snr_db=20.0, dtype="f32")
    ref = [ag.product(a, b, opts) for a, b in zip(A, B)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = []
    for i, (a, b) in enumerate(zip(A, B)):
        with torch.cuda.stream(streams[i % 2]):
            out.append(ag.product(a, b, opts))
    torch.cuda.synchronize()
    assert all(torch.equal(x, r) for x, r in zip(out, ref))
    ag.clear_plan_cache()
