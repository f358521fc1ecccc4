"""Companders of the pack and code kernels for block maxima whose quotient gamma / max is
hard to round, subnormal or near overflow: C against the oracle, whose companders are
fp64 quotients rounded to fp32, bit for bit (needs a GB300)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _near_ties(gamma, n, rng):
    """fp32 maxima in [1, 2) whose quotient lies nearest to the middle of two fp32
    numbers, of 400 n candidates."""
    m = (1.0 + rng.random(400 * n)).astype(np.float32)
    q = gamma / m.astype(np.float64)
    mant = np.frexp(q)[0] * 2.0 ** 24
    return m[np.argsort(np.abs(mant - np.floor(mant) - 0.5))[:n]].astype(np.float64)


def _blocks(rows, cols, L, maxima, rng):
    """Uniform values in blocks of L x L, the largest of each block one of the maxima."""
    X = rng.uniform(-0.99, 0.99, (rows, cols)).astype(np.float32)
    k = 0
    for i in range(0, rows, L):
        for j in range(0, cols, L):
            m = np.float32(maxima[k % len(maxima)])
            b = X[i:i + L, j:j + L] * m
            b[rng.integers(b.shape[0]), rng.integers(b.shape[1])] = m * rng.choice((-1.0, 1.0))
            X[i:i + L, j:j + L] = b
            k += 1
    return X


@pytest.mark.parametrize("transA,transB", [("N", "N"), ("T", "T")])
@pytest.mark.parametrize("form,W,bits,L", [("sym", 1, 20, 16), ("sym", 2, 8, 16), ("asym", 2, 20, 32),
                                           ("asym", 3, 5, 16), ("tc_int", 1, 9, 128),
                                           ("tc_int", 1, 10, 64)])
def test_hard_quotients(orc, form, W, bits, L, transA, transB):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(bits)
    gamma = 2 ** (bits - 1) - 1
    n = 256 if L < 64 else 16
    M = N = 16 * L if L < 64 else 4 * L
    K = 16 * L if L < 64 else 4 * L
    A = _blocks(M, K, L, _near_ties(gamma, n, rng), rng)
    B = _blocks(K, N, L, _near_ties(gamma, n, rng), rng)
    _compare(orc, A, B, form, W, bits, L, transA, transB)


@pytest.mark.parametrize("form,W,L", [("sym", 2, 16), ("asym", 2, 16), ("tc_int", 1, 64)])
def test_subnormal_and_huge_maxima(orc, form, W, L):
    """gamma = 1: maxima from the subnormal numbers whose quotient is still finite to
    those whose quotient is subnormal, in slabs whose other operand brings the product
    back to the middle of the range."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(3)
    scales = np.array([3.1e-39, 7e-39, 1.3e-38, 1e-30, 1.0, 1e30, 1.5e38, 2.9e38])
    A, B = np.empty((64, 8 * L), np.float32), np.empty((8 * L, 80), np.float32)
    for l, s in enumerate(scales):
        A[:, l * L:(l + 1) * L] = _blocks(64, L, L, [s, 1.01 * s], rng)
        B[l * L:(l + 1) * L] = _blocks(L, 80, L, [0.9 / s], rng)
    assert np.isfinite(A).all() and np.isfinite(B).all()
    _compare(orc, A, B, form, W, 2, L, "N", "N")


def _compare(orc, A, B, form, W, bits, L, transA, transB):
    import paper_1110_5765_gb300 as tdg
    if form == "tc_int":
        ref = orc.tc_int_gemm(A, B, L=L, bits=bits).C
    else:
        ref = orc.tdgemm(A, B, L=L, W=W, dtype="f32", form=form, bits=bits).C
    As = torch.from_numpy(np.ascontiguousarray(A if transA == "N" else A.T)).cuda()
    Bs = torch.from_numpy(np.ascontiguousarray(B if transB == "N" else B.T)).cuda()
    with tdg.Plan(A.shape[0], B.shape[1], A.shape[1], L=L, W=W, dtype="f32", form=form, bits=bits,
                  transA=transA, transB=transB) as p:
        C = p.run(As, Bs).cpu().numpy()
        assert p.info()["device_status"] == 0
    assert np.array_equal(C.view(np.uint32), ref.view(np.uint32))
