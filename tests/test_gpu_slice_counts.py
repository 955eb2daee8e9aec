"""GPU tests of one handle used with several slice counts in turn."""
import pytest
import torch

from paper_2505_20375_gb300 import synth

from helpers import ENERGY_TOL, gpu_fci

pytestmark = pytest.mark.gpu


def _handle(n=8, ne=4, seed=45):
    h, g = synth.real_integrals(n, 6, seed)
    f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=n, na=ne, nb=ne))
    return f, torch.from_numpy(synth.random_vector(f.n_det, seed=7)).cuda()


def test_two_pass_sigma_after_a_fused_one_of_another_slice_count(fci_lib, monkeypatch):
    """Each operator image is scaled by its own power of two, whatever was prepared since."""
    f, c = _handle()
    out = []
    for path, s in (("gemm", 6), ("fused", 3), ("gemm", 6), ("fused", 6), ("gemm", 3)):
        monkeypatch.setenv("FCI_OZ_PATH", path)
        out.append(f.sigma(c, precision="oz_bf16", n_slices=s))
    f.sync_status()
    assert torch.equal(out[0], out[2]) and torch.equal(out[0], out[3]) and torch.equal(out[1], out[4])


def test_mixed_davidson_after_tuning_the_final_slice_count(fci_lib, monkeypatch):
    f, c = _handle(n=10, ne=5)
    f.tune(c, 6, reps=2)  # picks a path for 6 slices; 3 slices stay fused
    monkeypatch.setenv("FCI_OZ_PATH", "fused")
    r = f.davidson(tol_residual=1e-6, tol_energy=1e-10, precision="oz_bf16", n_slices=3, switch_residual=1e-4,
                   final_precision="oz_bf16", final_slices=6)
    r64 = f.davidson(tol_residual=1e-6, tol_energy=1e-10)
    assert r.converged and abs(r.energy - r64.energy) < ENERGY_TOL
