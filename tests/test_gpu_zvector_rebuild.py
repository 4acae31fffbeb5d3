"""The Z-vector solve follows the context: after new MOs and after a new
geometry its result is that of a fresh context, bit for bit (also where that
is an error: MOs kept through a displacement can leave the mixed form's CG above
its tolerance)."""
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
@pytest.mark.parametrize("n,precision", [(4, "f64"), (10, "f64"), (8, "mixed")])
def test_zvector_after_new_mos_and_geometry(ris_mod, n, precision):
    prec = ris_mod.FP64 if precision == "f64" else ris_mod.MIXED
    mols = [synth.chain_molecule(n, seed, n > 4) for seed in (1, 2)]
    rhs = synth.random_amplitudes(2, mols[0].nocc, mols[0].nvir, seed=9)
    moved = synth.perturb(mols[0].coords, 0.05, np.random.default_rng(3))

    def solve(c, coords, mol):
        if coords is not None:
            c.build_aux(coords, mol.shells, mol.aux_j, mol.aux_k)
        c.build_B(mol.C, mol.mo_energy, mol.nocc)
        try:
            return c.zvector(rhs)
        except ris_mod.RisError as e:
            return e.code

    def fresh(coords, mol):
        c = ris_mod.Context(precision=prec)
        z = solve(c, coords, mol)
        c.close()
        return z

    c = ris_mod.Context(precision=prec)
    first = solve(c, mols[0].coords, mols[0])
    assert np.array_equal(solve(c, None, mols[1]), fresh(mols[0].coords, mols[1]))
    assert np.array_equal(solve(c, moved, mols[0]), fresh(moved, mols[0]))
    assert np.array_equal(solve(c, mols[0].coords, mols[0]), first)
