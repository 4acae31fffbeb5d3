"""Rounding of the 9 x 7 bit emulated GEMM's results on both sides of the
contraction length from which FP64 operations do it (112), over results that
are ordinary, zero by cancellation, subnormal or too large.  Bound as in the
GEMM's other tests: K 2^-57 max_k|A_rk| max_k|B_ck| and the rounding of the
result (half a unit in the last place, of the subnormals where it is one)."""
import numpy as np
import pytest

gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def ris_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18233_gb300 import build, ris
    build.build()
    return ris


@gpu
@pytest.mark.parametrize("K", [96, 111, 112, 113, 512])
def test_rounding(ris_mod, K):
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((130, K)), rng.standard_normal((50, K))
    A[1, 1::2], B[1] = -A[1, 0:K - K % 2:2], 1.0   # pairs that cancel against a row of ones
    if K % 2:
        A[1, -1] = 0.0
    A[2], B[2] = np.ldexp(A[2], -520), np.ldexp(B[2], -530)   # subnormal
    A[3], B[3] = np.ldexp(A[3], 515), np.ldexp(B[3], 515)     # overflow
    L = np.longdouble
    ref = A.astype(L) @ B.astype(L).T
    got = ris_mod.debug_gemm_f64emu(A, B, form="9x7")
    big = np.abs(ref) > L(np.finfo(np.float64).max)
    assert np.all(np.isinf(got[big])) and np.all(np.sign(got[big]) == np.sign(ref[big]))
    assert got[1, 1] == 0.0 and big[3, 3]
    bound = (K * L(2.0) ** -57 * np.abs(A).max(axis=1).astype(L)[:, None] * np.abs(B).max(axis=1).astype(L)[None, :]
             + L(2.0) ** -52 * np.abs(ref) + L(2.0) ** -1074)
    assert np.all((np.abs(got.astype(L) - ref) <= bound) | big)
