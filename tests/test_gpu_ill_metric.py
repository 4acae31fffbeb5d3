"""FP64 couplings and gradients of auxiliary sets with a nearly singular metric.

The derivatives multiply the rounding of the MO transforms by the metric's
inflation (1e6 for the C54H18 flake), so the default form and the FP64 pipe
(emu_f64 = 0) agree there only if both sum those transforms alike.  What else
differs between the two (the exchange products and densities, the state
densities) enters with the square root of the metric's condition at most:
2.5e4 for a condition of 6e8, times 1e-16 and the root of the number of terms
of a sum (a few tens), 5e-11 to 1e-10.  Bar 2e-10 of the result's 2-norm, a
fifth of what FP64 results are held to.
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


def _states(mol, n, seed):
    """Amplitudes like a converged state's: large on the small orbital-energy differences."""
    rng = np.random.default_rng(seed)
    o = mol.nocc
    gap = mol.mo_energy[o:][None, :] - mol.mo_energy[:o][:, None]
    x = rng.standard_normal((n,) + gap.shape) / (gap[None] - 0.8 * gap.min())
    q = np.linalg.qr(x.reshape(n, -1).T)[0]
    return np.ascontiguousarray(q.T).reshape(x.shape)


@gpu
@pytest.mark.parametrize("radius,k_as_j", [(6.2, False), (5.7, True)])
def test_derivatives_of_ill_conditioned_metrics(ris_mod, radius, k_as_j):
    """k_as_j: the exchange set is the (nearly singular) Coulomb set too."""
    mol = synth.flake_molecule(radius, 3)
    X, omega = _states(mol, 5, 8), np.linspace(0.2, 0.3, 5)
    got = []
    for emu in (1, 0):
        c = ris_mod.Context(emu_f64=emu)
        c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_j if k_as_j else mol.aux_k)
        c.build_B(mol.C, mol.mo_energy, mol.nocc)
        got.append(c.nac([(0, 1), (1, 2), (2, 3), (3, 4)], X=X, omega=omega))
        got.append(c.gradient([1, 3], X=X))
        c.close()
    for a, b in zip(got[:2], got[2:]):
        off = np.linalg.norm(a - b) / np.linalg.norm(b)
        assert off <= 2e-10, off


@pytest.mark.parametrize("kind,size,low,high", [("chain", 12, 4e3, 6e3), ("chain", 40, 4e3, 6e3),
                                                ("flake", 4.0, 1.2e5, 1.4e5), ("flake", 6.2, 9e5, 1.1e6)])
def test_inflation_of_the_workloads(oracle, kind, size, low, high):
    """The figures that the library's line (2e5) was set by: max M_PP (M^-1)_PP of
    the Coulomb sets, on either side of it; the exchange sets are far below."""
    mol = (synth.chain_molecule(size, 1, True, False) if kind == "chain" else
           synth.flake_molecule(size, 1, False))
    for aux, lo, hi in ((mol.aux_j, low, high), (mol.aux_k, 1.0, 1e3)):
        M = oracle.int2c(mol.coords, aux)
        assert lo < np.max(np.diag(M) * np.diag(np.linalg.inv(M))) < hi
