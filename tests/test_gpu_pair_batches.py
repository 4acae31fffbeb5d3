"""Pairs of states that share the launches of a derivative call: any list of
pairs gives what each pair gives by itself.  The exchange parts are summed in
the same order; the Coulomb part's products over all states may be cut
differently, so the bound is FP64 rounding (1e-15) times the J metric's
condition (below 1e5 for this chain)."""
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
@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("size", [6, 8])  # FP64 exchange densities on the FP64 pipe / emulated
def test_lists_of_pairs(ris_mod, size, precision, rpa):
    mol = synth.chain_molecule(size, 31, True)
    n = 11
    X = synth.random_amplitudes(n, mol.nocc, mol.nvir, seed=3)
    Y = 0.1 * synth.random_amplitudes(n, mol.nocc, mol.nvir, seed=4) if rpa else None
    c = ris_mod.Context(precision=ris_mod.MIXED if precision == "mixed" else ris_mod.FP64, rpa=rpa)
    c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
    c.build_B(mol.C, mol.mo_energy, mol.nocc)
    om = np.linspace(0.2, 0.7, n)
    # runs, repeats, descending, far apart; nine and more pairs make two batches
    pairs = [(0, 1), (1, 2), (2, 3), (3, 4), (3, 5), (7, 2), (6, 1), (5, 0), (10, 9), (0, 10), (4, 8), (4, 9)]
    single = np.concatenate([c.nac([p], X=X, Y=Y, omega=om) for p in pairs])
    for k in (2, 5, 9, 12):
        got = c.nac(pairs[:k], X=X, Y=Y, omega=om)
        assert np.max(np.abs(got - single[:k])) <= 1e-10 * np.max(np.abs(single[:k]))
