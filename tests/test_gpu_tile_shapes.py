"""Every CTA tile that the packed GEMM chooses among, at the sizes where it can go
wrong: one tile and its remainders, just under and over the lines of the rule,
with and without slab splitting, against the oracle bit for bit (needs a GB300)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (M, N, K) for fp64 on 152 SMs: 16-tiles (one, ragged, split over slabs, two per
# SM), 32-tiles (143 of them; asymmetric 16), 16-tiles in many waves, 64-tiles (152 of
# them; then, for the asymmetric form, 297)
F64 = [(1, 1, 70), (17, 31, 130), (60, 70, 600), (257, 250, 130), (350, 410, 130),
       (600, 930, 66), (512, 1216, 66), (2048, 1728, 66)]


@pytest.mark.parametrize("shape", F64)
@pytest.mark.parametrize("form,W", [("sym", 2), ("sym", 3), ("asym", 3), ("plain", 1)])
def test_f64_tiles(orc, shape, form, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = shape
    A, B = synth.laplace((M, K), 61), synth.gaussian((K, N), 62)
    C0 = synth.gaussian((M, N), 63)
    kw = dict(L=64, W=W, dtype="f64", form=form, bits=0 if form == "plain" else 8)
    ref = orc.tdgemm(A, B, alpha=0.75, beta=-1.5, C_in=C0, **kw)
    with tdg.Plan(M, N, K, **kw) as p:
        C = torch.from_numpy(C0.copy()).cuda()
        p.run(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, 0.75, -1.5)
        assert p.info()["device_status"] == 0
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))


# fp32, symmetric: one ragged 64-tile, 64-tiles (up to one and two an SM), 128 x 64
# tiles, 128 x 128 tiles, slabs split over CTAs (asymmetric: 64-tiles; BY_RULE has the
# others)
F32 = [(60, 50, 130), (700, 690, 130), (1000, 777, 130), (1500, 1300, 130), (2000, 1900, 66),
       (129, 70, 1400)]


@pytest.mark.parametrize("shape", F32)
@pytest.mark.parametrize("form,W", [("sym", 1), ("sym", 2), ("sym", 3), ("asym", 2), ("asym", 4)])
def test_f32_tiles(orc, shape, form, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = shape
    A, B = synth.laplace((M, K), 64, np.float32), synth.gaussian((K, N), 65, np.float32)
    C0 = synth.gaussian((M, N), 66, np.float32)
    kw = dict(L=64, W=W, dtype="f32", form=form, bits=6)
    ref = orc.tdgemm(A, B, alpha=0.75, beta=-1.5, C_in=C0, **kw)
    with tdg.Plan(M, N, K, **kw) as p:
        C = torch.from_numpy(C0.copy()).cuda()
        p.run(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, 0.75, -1.5)
        assert p.info()["device_status"] == 0
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))


@pytest.mark.parametrize("shape", F32)
@pytest.mark.parametrize("form,W,target,used", [("sym", 2, 20.0, 2), ("sym", 2, 60.0, 1),
                                                ("sym", 4, 20.0, None), ("asym", 2, 20.0, 2),
                                                ("asym", 2, 60.0, 1)])
def test_f32_target_launches(orc, shape, form, W, target, used):
    """Targets met by packing and missed (plain fallback), in the launches that hold
    several candidates: the plan and C of the oracle."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = shape
    A, B = synth.uniform((M, K), 67, np.float32), synth.uniform((K, N), 68, np.float32)
    kw = dict(L=64, W=W, dtype="f32", form=form)
    ref = orc.tdgemm(A, B, target_db=target, s_table=orc.load_s_table(), **kw)
    assert used is None or ref.plan.W == used
    with tdg.Plan(M, N, K, target_snr_db=target, **kw) as p:
        C = p.run(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda())
        assert p.info()["W_used"] == ref.plan.W
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))


@pytest.mark.parametrize("dtype,shape,W,target,used", [
    ("f32", (1536, 1500, 130), 2, 20.0, 2), ("f32", (1536, 1500, 130), 2, 90.0, 1),
    ("f32", (1536, 1500, 130), 4, 90.0, 1), ("f32", (2500, 1200, 66), 3, 90.0, 1),
    ("f64", (512, 500, 130), 2, 20.0, 2), ("f64", (512, 500, 130), 3, 300.0, 1)])
def test_fallback_apart(orc, dtype, shape, W, target, used):
    """Asymmetric targets whose plain fallback has another tile than the packed
    product, and so a launch by itself: met and missed."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    npt = np.float32 if dtype == "f32" else np.float64
    M, N, K = shape
    A, B = synth.uniform((M, K), 77, npt), synth.uniform((K, N), 78, npt)
    C0 = synth.gaussian((M, N), 79, npt)
    kw = dict(L=128, W=W, dtype=dtype, form="asym")
    ref = orc.tdgemm(A, B, target_db=target, s_table=orc.load_s_table(), alpha=0.75, beta=-1.5,
                     C_in=C0, **kw)
    assert ref.plan.W == used
    with tdg.Plan(M, N, K, target_snr_db=target, **kw) as p:
        C = torch.from_numpy(C0.copy()).cuda()
        p.run(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, 0.75, -1.5)
        assert p.info()["W_used"] == used
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))


# the smallest products of a search that take each tile, whole and split (W of symmetric
# targets: decided on the device, tiled for 2); test_tile_rule.py checks the tiles
BY_RULE = [
    ("asym", 2, 64, (4200, 2000, 60), dict(bits=4), "big", False),
    ("asym", 2, 64, (130, 2000, 520), dict(bits=4), "big", True),
    ("asym", 3, 64, (2600, 2000, 66), dict(bits=4), "big", False),
    ("asym", 3, 64, (130, 2000, 520), dict(bits=4), "big", True),
    ("asym", 4, 64, (4200, 2000, 66), dict(bits=4), "big", False),
    ("asym", 4, 64, (260, 2000, 520), dict(bits=4), "big", True),
    ("asym", 4, 64, (700, 900, 130), dict(bits=4), "small", False),
    ("asym", 3, 64, (64, 40, 2000), dict(bits=4), "small", True),
    ("sym", 2, 64, (1300, 3300, 60), dict(bits=6), "big", False),
    ("sym", 2, 64, (260, 700, 3000), dict(bits=6), "big", True),
    ("sym", 2, 64, (4200, 400, 60), dict(bits=6), "mid", False),
    ("sym", 4, 64, (130, 130, 520), dict(bits=4), "small", True),
    ("sym", 4, 64, (130, 200, 2100), dict(target=15.0), "small", True),
    ("asym", 4, 64, (130, 200, 2100), dict(target=15.0), "small", True),
    ("asym", 3, 64, (1300, 900, 260), dict(target=15.0), "small", False),
]


@pytest.mark.parametrize("form,W,L,shape,kw", [c[:5] for c in BY_RULE])
def test_tiles_by_form_and_packing(orc, form, W, L, shape, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    M, N, K = shape
    A, B = synth.uniform((M, K), 84, np.float32), synth.uniform((K, N), 85, np.float32)
    goal = dict(bits=kw["bits"]) if "bits" in kw else dict(target_snr_db=kw["target"])
    okw = dict(bits=kw["bits"]) if "bits" in kw else dict(target_db=kw["target"],
                                                          s_table=orc.load_s_table())
    ref = orc.tdgemm(A, B, L=L, W=W, dtype="f32", form=form, **okw)
    with tdg.Plan(M, N, K, L=L, W=W, dtype="f32", form=form, **goal) as p:
        C = p.run(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda())
        assert p.info()["W_used"] == ref.plan.W
        assert np.array_equal(C.cpu().numpy().view(np.uint8), ref.C.view(np.uint8))
