"""GPU test of the launch counts that the phase timing reports."""
import pytest
import torch

from paper_2505_20375_gb300 import synth

from helpers import gpu_fci

pytestmark = pytest.mark.gpu


def _fci(n, na, nb):
    h, g = synth.real_integrals(n, 4, 45 + n)
    return gpu_fci(dict(h=h, g=g, e_core=0.2, n=n, na=na, nb=nb))


def _das():
    return _fci(9, 3, 3).build_das([3, 3, 3], [1, 1, 1], [1, 1, 1], 1)


def _spinor(n, ne):
    h, g = synth.complex_integrals(n, 4, 46)
    return gpu_fci(dict(h=h, g=g, e_core=0.2, n=n, ne=ne))


# kernels by phase (gather, contract, scatter, other); up to 2^14 values the fixed-point
# conversion is one kernel, above two
@pytest.mark.parametrize("make,s,form,want", [
    (lambda: _fci(8, 4, 4), 0, "dense", (0, 1, 1, 0)),
    (lambda: _fci(8, 4, 4), 3, "dense", (0, 1, 1, 1)),
    (lambda: _fci(9, 4, 4), 3, "dense", (2, 1, 1, 0)),   # two-pass, 15,876 determinants
    (lambda: _fci(10, 4, 4), 3, "dense", (3, 1, 1, 0)),  # two-pass, 44,100
    (_das, 0, "dense", (0, 1, 1, 0)),
    (_das, 3, "dense", (0, 1, 1, 1)),
    (_das, 6, "dense", (1, 1, 1, 1)),
    (_das, 6, "blocks", (1, 1, 1, 1)),                   # short rows: image by determinants
    (lambda: _fci(11, 4, 4).build_das([11], [4], [4], 0), 6, "blocks", (2, 1, 1, 2)),  # masks, image by rows
    (lambda: _spinor(10, 4), 0, "dense", (0, 1, 1, 0)),
    (lambda: _spinor(10, 4), 6, "blocks", (2, 1, 1, 0)),
    (lambda: _spinor(16, 6), 3, "dense", (2, 1, 1, 0)),  # 8,008 complex determinants: 16,016 values
    (lambda: _spinor(16, 7), 3, "dense", (3, 1, 1, 0)),  # 11,440: 22,880 values
])
def test_kernels_of_a_sigma_by_phase(fci_lib, monkeypatch, make, s, form, want):
    monkeypatch.setenv("FCI_SPLIT_FORM", form)
    f = make()
    c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()
    f.set_phase_timing(True)
    f.sigma(c, precision="oz_bf16" if s else "fp64", n_slices=s)
    f.sync_status()
    t = f.phase_times()
    assert tuple(t[k]["launches"] for k in ("gather", "contract", "scatter", "other")) == want


@pytest.mark.parametrize("form,gather,scatter", [("lists", 7, 3), ("walk", 4, 1)])
def test_kernels_of_a_compressed_sigma_by_phase(fci_lib, monkeypatch, form, gather, scatter):
    """Columns: expansion, category ranges, compaction, gather and, with lists, a scan of two kernels
    and the lists per string; support: emission, compaction and three kernels per 8 bits of the
    largest address; the sum in three forms or one."""
    monkeypatch.setenv("FCI_CS_FORM", form)
    f = _das()
    f.set_phase_timing(True)
    f.sigma_compressed(torch.arange(20, device="cuda"), torch.ones(20, dtype=torch.float64, device="cuda"))
    t = f.phase_times()
    bits = (f.n_det - 1).bit_length()
    assert tuple(t[k]["launches"] for k in ("gather", "contract", "scatter", "other")) == (gather, 1, scatter, 2 + 3 * -(-bits // 8))
