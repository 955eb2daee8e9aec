"""GPU tests of calls repeated on a handle after one of their allocations failed on the host side."""
import pytest
import torch

from paper_2505_20375_gb300 import synth

from helpers import gpu_fci

pytestmark = pytest.mark.gpu


def _problem(kind):
    if kind == "spinor":
        h, g = synth.complex_integrals(10, 6, 46)
        return gpu_fci(dict(h=h, g=g, e_core=0.2, n=10, ne=4))
    h, g = synth.real_integrals(9, 6, 46)
    f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=9, na=3, nb=3))
    return f.build_das([3, 3, 3], [1, 1, 1], [1, 1, 1], 1) if kind.startswith("das") else f


@pytest.mark.parametrize("form", ["dense", "blocks"])
@pytest.mark.parametrize("kind,s", [("fci", 3), ("fci two-pass", 6), ("das", 3), ("das", 6), ("spinor", 4), ("das compressed", 0)])
def test_call_after_an_injected_allocation_failure(fci_lib, monkeypatch, kind, s, form):
    """The first sigma of a handle fails at its 1st, 2nd, .. device allocation; each next call on
    the same handle finds complete tables or builds them, and the result has the usual bits."""
    monkeypatch.setenv("FCI_SPLIT_FORM", form)
    monkeypatch.setenv("FCI_OZ_PATH", "gemm" if kind == "fci two-pass" else "fused")

    def call(f):
        if kind == "das compressed":
            n = min(f.n_det, 40)
            return torch.cat(f.sigma_compressed(torch.arange(n, device="cuda"), torch.linspace(1, 2, n, dtype=torch.float64, device="cuda")))
        c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()
        return f.sigma(c, precision="oz_bf16", n_slices=s)

    want = call(_problem(kind))
    f = _problem(kind)
    failed = 0
    for n in range(1, 40):
        # once per value: the count starts anew with the first call that sees it
        monkeypatch.setenv("FCI_FAULT_ALLOC_AT", str(n))
        try:
            got = call(f)
            break
        except fci_lib.FCIError as e:
            assert e.code == fci_lib.FCI_ERR_OOM
            failed += 1
        finally:
            monkeypatch.delenv("FCI_FAULT_ALLOC_AT")
    f.sync_status()
    assert failed >= 1 and torch.equal(got, want)
