"""Derivatives at given Y amplitudes need the ov blocks that only an RPA context
builds: a TDA context refuses them and stays usable."""
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
@pytest.mark.parametrize("n,precision", [(4, "f64"), (8, "f64"), (4, "mixed")])
def test_tda_context_refuses_y(ris_mod, n, precision):
    mol = synth.chain_molecule(n, 2, n > 4)
    X = synth.random_amplitudes(2, mol.nocc, mol.nvir, seed=1)
    c = ris_mod.Context(precision=ris_mod.FP64 if precision == "f64" else ris_mod.MIXED)
    c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
    c.build_B(mol.C, mol.mo_energy, mol.nocc)
    g = c.gradient([0, 1], X=X)
    with pytest.raises(ris_mod.RisError, match="RPA"):
        c.gradient([0], X=X, Y=0.1 * X)
    with pytest.raises(ris_mod.RisError, match="RPA"):
        c.nac([(0, 1)], X=X, Y=0.1 * X, omega=np.array([0.2, 0.3]))
    assert np.array_equal(c.gradient([0, 1], X=X), g)
