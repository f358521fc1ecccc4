"""Distortion targets with up to four packings asked for: the packing, the level and
the companders that the device picks are the oracle's, whichever packing is the first to
meet the target, over the whole range of levels (81 to 145) and with noise tables that
leave levels out (needs a GB300)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _table(orc, dtype, form, L, measured):
    """A made-up s(R), at every third level only, or none at all."""
    tabs, dense = {}, {}
    for W in (2, 3, 4):
        d, arr = {}, np.full(192, -1.0)
        for t in range(W, orc.T_MAX[dtype] + 1, 3) if measured else ():
            arr[t] = 1e-4 * W * orc.r_level(t) ** 0.75
            d[str(t)] = {"s": arr[t]}
        tabs[orc.STable.key(dtype, form, W, L)] = d
        dense[W] = arr
    return orc.STable(tabs), dense


@pytest.mark.parametrize("dtype,L", [("f32", 16), ("f32", 128), ("f64", 16), ("f64", 64), ("f64", 1024)])
@pytest.mark.parametrize("rms", [False, True])
@pytest.mark.parametrize("measured", [False, True])
def test_every_packing(orc, dtype, L, rms, measured):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5765_gb300 as tdg
    T = np.float32 if dtype == "f32" else np.float64
    M, N, K = 70, 90, 130
    A, B = 3.0 * synth.uniform((M, K), 91, T), synth.laplace((K, N), 92, T)
    st, dense = _table(orc, dtype, "sym", L, measured)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    used = set()
    for W in (2, 3, 4):
        for target in (-20.0, 5.0, 12.0, 20.0, 30.0, 45.0, 60.0, 80.0, 250.0):
            for fallback in (True, False):
                ref = orc.tdgemm(A, B, L=L, W=W, dtype=dtype, form="sym", target_db=target,
                                 s_table=st, noise_rms=rms, allow_fallback=fallback).plan
                with tdg.Plan(M, N, K, L=L, W=W, dtype=dtype, form="sym", target_snr_db=target,
                              rep_noise=None, noise_rms=rms, allow_fallback=fallback) as p:
                    for w in (2, 3, 4):
                        p.set_rep_noise(w, dense[w], 0)
                    p.quantize_pack(dA, dB)
                    i = p.info()
                used.add(i["W_used"])
                assert i["W_used"] == ref.W, (W, target, fallback)
                if ref.W > 1:
                    assert (i["q"], i["gamma_a"], i["gamma_b"], i["level"]) == \
                        (ref.q, ref.gA, ref.gB, ref.t), (W, target, fallback)
                    if ref.t >= 0:
                        assert abs(i["pred_snr_db"] - ref.pred_snr_db) < 1e-6
                assert i["device_status"] == (0 if fallback or i["pred_snr_db"] >= target else 5)
    assert {1, 2} <= used
