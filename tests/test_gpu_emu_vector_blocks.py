"""Emulated exchange products whose vectors run in several blocks (C40H42: blocks
of nine, the last one shorter) against the FP64 pipe, to the bar of the smaller
products (1e-12 of the largest element), and each vector as it is alone to the
same bar."""
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
def test_products_in_blocks_of_vectors(ris_mod, rpa):
    mol = synth.chain_molecule(40, 5, True)
    X = synth.random_amplitudes(17, mol.nocc, mol.nvir, seed=1)
    out = []
    for emu in (1, 0):
        c = ris_mod.Context(rpa=rpa, emu_f64=emu, deriv_prefetch=0)
        c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
        c.build_B(mol.C, mol.mo_energy, mol.nocc)
        r = c.apply(X)
        out.append(r if rpa else (r,))
        if emu:
            a = c.apply(np.ascontiguousarray(X[16:]))
            alone = a if rpa else (a,)
        c.close()
    for e, f, a in zip(out[0], out[1], alone):
        assert np.max(np.abs(e - f)) <= 1e-12 * np.max(np.abs(f))
        assert np.max(np.abs(e[16:] - a)) <= 1e-12 * np.max(np.abs(a))
