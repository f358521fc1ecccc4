"""The fact that lets the kernels form fp32 companders by an fp32 division (CPU).  That
they do is tested on the GPU (test_gpu_compander_quotient.py)."""
import numpy as np


def test_fp32_quotient_is_the_rounded_fp64_quotient():
    """c = fl32(gamma / max) in fp32 division: the same bits as the fp64 quotient
    rounded to fp32, over normal, subnormal and overflowing quotients, for gamma up to
    2^24 (from there on gamma itself need not be an fp32 number)."""
    g = np.random.default_rng(5)
    m = np.abs(np.concatenate([g.standard_normal(200000) * 2.0 ** g.integers(-140, 127, 200000),
                               [1e-45, 1.4e-45, 3.4028235e38, 1.0, 3.0]])).astype(np.float32)
    m = m[(m > 0) & np.isfinite(m)]
    with np.errstate(over="ignore"):
        for gamma in (1, 3, 21, 127, 362, 448, 2047, 524287, 1 << 20, (1 << 24) - 1, 1 << 24):
            a = np.float32(gamma) / m
            b = (np.float64(gamma) / m.astype(np.float64)).astype(np.float32)
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
