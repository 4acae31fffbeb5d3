"""The 9 x 7 bit form of the FP64-emulating GEMM at the edges of its tiles and
chunks, and the FP64 form's exchange products that run on it against the
same products on the FP64 pipe (emu_f64 = 0).

Bound of the GEMM per element: operands rounded to half a unit of a 62-bit
frame 2^E <= 2 max_k|x_k| (2^-61 max|A| max|B| per k together), products of
order p + q >= 9 dropped (eight of 64^2 2^-75 in the frames' product, 2^-58
max|A| max|B| with the lower orders), so K 2^-57 max_k|A_rk| max_k|B_ck| and
one rounding of the result (the reference has another).
"""
import numpy as np
import pytest

from paper_2511_18233_gb300 import synth

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
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 16, 15), (128, 48, 448), (129, 49, 449), (65, 33, 897),
                                   (40, 71, 5000), (300, 17, 2049), (257, 300, 42)])
def test_form_9x7_within_bound(ris_mod, M, N, K):
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    A = rng.standard_normal((M, K)) * 10.0 ** rng.uniform(-100, 100, size=(M, 1))
    B = rng.standard_normal((N, K)) * 10.0 ** rng.uniform(-3, 0, size=(1, K))
    if M > 3:
        A[1] = 0.0
        A[2] = np.abs(A[2]).max()          # constant row: every digit product of one sign
        A[3, 1:] *= 2.0 ** -60             # one element far above the rest
    if N > 1:
        B[1] = -1.0
    ref = (A.astype(np.longdouble) @ B.astype(np.longdouble).T).astype(np.float64)
    C = ris_mod.debug_gemm_f64emu(A, B, form="9x7")
    bound = (K * 2.0 ** -57 * np.abs(A).max(axis=1)[:, None] * np.abs(B).max(axis=1)[None, :]
             + 2.0 ** -52 * np.abs(ref))
    assert np.all(np.abs(C - ref) <= bound), float(np.max(np.abs(C - ref) / np.maximum(bound, 1e-300)))


@gpu
def test_form_9x7_non_finite_rows(ris_mod):
    rng = np.random.default_rng(4)
    A, B = rng.standard_normal((130, 500)), rng.standard_normal((50, 500))
    ref = ris_mod.debug_gemm_f64emu(A, B, form="9x7")
    A[5, 7], A[129, 0], B[49, 499] = np.inf, np.nan, -np.inf
    C = ris_mod.debug_gemm_f64emu(A, B, form="9x7")
    bad = np.zeros(C.shape, bool)
    bad[[5, 129]] = True
    bad[:, 49] = True
    assert np.all(np.isnan(C[bad])) and np.array_equal(C[~bad], ref[~bad])


def _ctx(ris_mod, mol, **opt):
    c = ris_mod.Context(**opt)
    c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
    c.build_B(mol.C, mol.mo_energy, mol.nocc)
    return c


@gpu
@pytest.mark.parametrize("n,nvec", [(8, 1), (9, 3), (13, 18)])
def test_emulated_exchange_equals_fp64_pipe(ris_mod, n, nvec):
    """Same inputs, same B^J: operator products, the Z-vector solution and
    gradients differ by the rounding of the exchange products alone (1e-15 of
    each product; 1e-12 and, with the fitting coefficients' cancellation in
    the derivatives, 1e-10 leave room)."""
    mol = synth.chain_molecule(n, 77 + n, True)
    X = synth.random_amplitudes(nvec, mol.nocc, mol.nvir, seed=n)
    Y = 0.1 * synth.random_amplitudes(nvec, mol.nocc, mol.nvir, seed=n + 1)

    def rel(a, b):
        return np.max(np.abs(a - b)) / np.max(np.abs(b))

    for rpa in (0, 1):
        emu, ref = (_ctx(ris_mod, mol, rpa=rpa, emu_f64=k) for k in (1, 0))
        for a, b in zip(np.atleast_1d(emu.apply(X)) if not rpa else emu.apply(X),
                        np.atleast_1d(ref.apply(X)) if not rpa else ref.apply(X)):
            assert rel(a, b) <= 1e-12
        st = range(min(nvec, 3))
        y = Y if rpa else None
        assert rel(emu.gradient(st, X=X, Y=y), ref.gradient(st, X=X, Y=y)) <= 1e-10
        if nvec > 1:
            om = np.linspace(0.3, 0.6, nvec)
            pr = [(0, 1), (2, 0)]
            assert rel(emu.nac(pr, X=X, Y=y, omega=om), ref.nac(pr, X=X, Y=y, omega=om)) <= 1e-10
        if not rpa:
            assert rel(emu.zvector(X[:2]), ref.zvector(X[:2])) <= 1e-8  # both stop at |r| <= 1e-10 |rhs|


@gpu
def test_emulated_exchange_keeps_vectors_apart(ris_mod):
    """A vector with a NaN gives NaN; its neighbours in the block do not change."""
    mol = synth.chain_molecule(9, 5, True)
    c = _ctx(ris_mod, mol)
    X = synth.random_amplitudes(3, mol.nocc, mol.nvir, seed=2)
    ref = c.apply(X)
    X[1, 3, 5] = np.nan
    got = c.apply(X)
    assert np.all(np.isnan(got[1]))
    assert np.allclose(got[[0, 2]], ref[[0, 2]], rtol=1e-13, atol=1e-15)
