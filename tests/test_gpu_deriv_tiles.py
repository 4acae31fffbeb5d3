"""Derivative integrals at the edges of their tiling: auxiliary classes of one
shell, of a part of a warp, of more items than are held at a time, and of d
shells beside them.  FP64 gradients at given amplitudes against the oracle, at
the parity bar of the other FP64 tests (1e-9 of the largest element; the
even-tempered sets' metrics are conditioned to about 1e5, so that FP64
rounding reaches 1e-11), and the translation sum rule."""
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


def _aux(natm, counts):
    """counts[l] shells of angular momentum l, atoms in turn, exponents 0.15 3^k on each."""
    rows = []
    for l, n in enumerate(counts):
        rows += [((3 * i + l) % natm, l, 0.15 * (1 + 0.2 * l) * 3.0 ** (i // natm)) for i in range(n)]
    return np.array(rows, dtype=synth.SHELL_DTYPE)


@gpu
@pytest.mark.parametrize("counts", [(1, 0, 0), (2, 1, 0), (33, 0, 1), (10, 10, 3), (31, 2, 0)])
def test_gradient_of_odd_auxiliary_classes(ris_mod, oracle, counts):
    mol = synth.workload(0)
    aux = _aux(mol.natm, counts)
    orc = oracle.RisOracle(mol.coords, mol.shells, aux, aux[:1], mol.C, mol.mo_energy, mol.nocc)
    X = synth.random_amplitudes(2, mol.nocc, mol.nvir, seed=sum(counts))
    c = ris_mod.Context()
    c.build_aux(mol.coords, mol.shells, aux, aux[:1])
    c.build_B(mol.C, mol.mo_energy, mol.nocc)
    g = c.gradient([0, 1], X=X)
    ref = orc.gradients([0, 1], X)
    assert np.max(np.abs(g - ref)) <= 1e-9 * np.max(np.abs(ref))
    assert np.max(np.abs(g.sum(axis=1))) <= 1e-10 * np.max(np.abs(g))
