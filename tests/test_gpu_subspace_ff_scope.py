"""What the mixed form's double-FP32 option covers: the Davidson alone.  At
given amplitudes its derivatives are FP64 where L_J^-1 amplifies rounding
(u = X B^J), so gradients and couplings are the same bits with it and without."""
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
@pytest.mark.parametrize("rpa", [0, 1])
def test_derivatives_do_not_depend_on_subspace_ff(ris_mod, rpa):
    mol = synth.chain_molecule(8, 21, True)
    X = synth.random_amplitudes(3, mol.nocc, mol.nvir, seed=4)
    Y = 0.1 * synth.random_amplitudes(3, mol.nocc, mol.nvir, seed=5) if rpa else None
    got = []
    for ff in (1, 0):
        c = ris_mod.Context(precision=ris_mod.MIXED, rpa=rpa, subspace_ff=ff)
        c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
        c.build_B(mol.C, mol.mo_energy, mol.nocc)
        got.append((c.gradient([0, 2], X=X, Y=Y), c.nac([(0, 1)], X=X, Y=Y, omega=np.array([0.2, 0.3, 0.4]))))
        c.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
