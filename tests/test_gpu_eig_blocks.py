"""Subspace eigensolver on decoupled matrices: columns that are exactly zero
below the diagonal (their reflection is skipped) before, between and after
coupled ones, within one warp's rows (m <= 33) and beyond.  Fragments too far
apart to interact give such projected matrices.  Tolerances of the solver's
other tests: eigenvalues 1e-13, orthogonality and residuals 1e-10."""
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


def _blocks(m, size, rng):
    H = np.diag(0.3 + 2 * rng.permutation(m) / m + 1e-3 * rng.random(m))
    for a in range(0, m - 1, size):
        b = min(a + size, m)
        Q = 1e-2 * rng.standard_normal((b - a, b - a))
        H[a:b, a:b] += 0.5 * (Q + Q.T)
    return H


@gpu
@pytest.mark.parametrize("m", [3, 4, 12, 30, 33, 34, 60, 130])
@pytest.mark.parametrize("size", [1, 2, 3, 7])
def test_sym_eig_of_decoupled_blocks(ris_mod, m, size):
    rng = np.random.default_rng(100 * m + size)
    k = min(m, 10)
    H = _blocks(m, size, rng)
    for it in range(20):  # the same input: the same bits every time
        w, V = ris_mod.debug_sym_eig(H, k)
        first = (w, V) if it == 0 else first
        assert np.array_equal(w, first[0]) and np.array_equal(V, first[1])
    np.testing.assert_allclose(w, np.linalg.eigvalsh(H)[:k], rtol=0, atol=1e-13)
    np.testing.assert_allclose(V @ V.T, np.eye(k), atol=1e-10)
    assert np.max(np.abs(H @ V.T - V.T * w[None, :])) < 1e-10
