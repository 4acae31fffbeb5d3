"""FP64 GEMM with the finely split contractions of the FP64 form (slices down to
one step of 16), with few and with many rows, against an extended-precision
product.  A sum of k products in any order is within (k + 2) 2^-53 sum |a||b| of
the exact one; alpha, beta and the stored result add three roundings."""
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
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (1, 1, 17), (5, 22, 1455), (40, 18, 97), (41, 31, 300), (64, 64, 4096),
                                   (130, 17, 33), (3, 700, 129)])
def test_finely_split_contractions(ris_mod, m, n, k, ta, tb):
    rng = np.random.default_rng(m * 1000 + n * 10 + k)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    C = rng.standard_normal((m, n))
    got = ris_mod.debug_dgemm(A.T if ta else A, B.T if tb else B, C, transA=ta, transB=tb, alpha=-0.7, beta=0.3,
                              fine=True)
    L = np.longdouble
    ref = L(-0.7) * (A.astype(L) @ B.astype(L)) + L(0.3) * C.astype(L)
    bound = 2.0 ** -53 * ((k + 6) * 0.7 * (np.abs(A) @ np.abs(B)) + 4 * np.abs(C))
    assert np.all(np.abs(got - ref.astype(np.float64)) <= bound + 2.0 ** -53 * np.abs(ref.astype(np.float64)))
