"""The serving footprint estimate bounds what an FP64 request holds at its peak
(the mixed form's is tested with the served stream): below, at and above the
line from which the FP64 form runs on digit slices."""
import pytest

from paper_2511_18233_gb300 import serve, synth

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
@pytest.mark.parametrize("kind,size,ns", [("chain", 4, 5), ("chain", 7, 5), ("chain", 20, 8), ("flake", 4.5, 5)])
def test_fp64_footprint_bounds_measured_peak(ris_mod, kind, size, ns):
    mol = synth.chain_molecule(size, 1, True) if kind == "chain" else synth.flake_molecule(size, 1)
    c = ris_mod.Context()
    c.build_aux(mol.coords, mol.shells, mol.aux_j, mol.aux_k)
    c.build_B(mol.C, mol.mo_energy, mol.nocc)
    c.excite(ns)
    c.gradient([1])
    c.nac([(0, 1), (1, 2)])
    peak = c.stats()["bytes_peak"]
    c.close()
    dm = serve.molecule_dims(mol)
    est = serve.footprint_bytes(dm["nao"], dm["nocc"], dm["nJ"], dm["nK"], dm["nU"], ns, 3, False)
    assert peak <= est <= 4 * peak + (64 << 20)
