"""GPU tests of the rule that chooses between the two forms of the split FCI sigma."""
import pytest
import torch

from paper_2505_20375_gb300 import fci, synth

from helpers import gpu_fci

pytestmark = pytest.mark.gpu


def _handle(n, na, nb):
    h, g = synth.real_integrals(n, 4, 45 + n)
    f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=n, na=na, nb=nb))
    return f, torch.from_numpy(synth.random_vector(f.n_det, seed=7)).cuda()


# (1, 7) of 14 orbitals: 14 x 3,432 strings; the digit image of the two-pass form, one block per
# alpha string, would run on 14 SMs
@pytest.mark.parametrize("n,na,nb,form", [(8, 4, 4, "fused"), (9, 4, 3, "two-pass"), (14, 1, 7, "fused"),
                                          (14, 13, 7, "fused"), (12, 2, 6, "fused"), (10, 2, 5, "two-pass"),
                                          (14, 7, 1, "two-pass"), (12, 3, 6, "two-pass"), (14, 3, 7, "two-pass")])
def test_default_form_by_shape_of_the_space(fci_lib, monkeypatch, n, na, nb, form):
    """The form that is the faster one for the shape (the two-pass form times a gather phase,
    the fused one has none), with the bits of the other."""
    f, c = _handle(n, na, nb)
    f.set_phase_timing(True)
    out = f.sigma(c, precision="oz_bf16", n_slices=3)
    assert ("two-pass" if f.phase_times()["gather"]["launches"] else "fused") == form
    f.set_phase_timing(False)
    monkeypatch.setenv("FCI_OZ_PATH", "gemm" if form == "fused" else "fused")
    assert torch.equal(out, f.sigma(c, precision="oz_bf16", n_slices=3))
    f.sync_status()


@pytest.mark.parametrize("count,form", [(3, "two-pass"), (4, "fused")])
def test_medium_problems_of_a_large_group_share_a_launch(fci_lib, count, form):
    """10,584 and 44,100 determinants: the former fused in a group of four, the latter not."""
    fs, cs, outs, jobs, keep = [], [], [], [], []
    for i in range(count):
        f, c = _handle(*((10, 4, 4) if i == 0 else (9, 4, 3)))
        nb = f.sigma_workspace_bytes("oz_bf16", 3)
        keep.append(torch.empty(nb + 256, dtype=torch.uint8, device="cuda"))
        o = torch.full_like(c, float("nan"))
        fs, cs, outs = fs + [f], cs + [c], outs + [o]
        jobs.append((f, c, o, "oz_bf16", 3, (keep[-1].data_ptr() + 255) & ~255, nb))
        f.set_phase_timing(True)
    fci.sigma_grouped(jobs)
    forms = ["two-pass" if f.phase_times()["gather"]["launches"] else "fused" for f in fs]
    assert forms == ["two-pass"] + [form] * (count - 1)
    for f, c, o in zip(fs, cs, outs):
        f.set_phase_timing(False)
        assert torch.equal(o, f.sigma(c, precision="oz_bf16", n_slices=3))
        f.sync_status()
