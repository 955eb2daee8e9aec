"""GPU tests of the block-sparse contraction on spaces where the default rule takes the dense
one: the edges of its blocks, pieces and digit images, selected by FCI_SPLIT_FORM."""
import pytest
import torch

from paper_2505_20375_gb300 import fci, synth

from helpers import gpu_fci, rel_inf, spinor_problem
from ozaki_model import das_sigma_model, spinor_sigma_model

pytestmark = pytest.mark.gpu


def _sigma(f, c, s):
    out = f.sigma(c, precision="oz_bf16", n_slices=s)
    f.sync_status()
    return out


def _das(spaces, ref, nel, T):
    n = sum(spaces)
    h, g = synth.real_integrals(n, 6, 50 + n)
    f = gpu_fci(dict(h=h, g=g, e_core=0.3, n=n, na=nel, nb=nel)).build_das(spaces, ref, ref, T)
    return h, g, f, torch.from_numpy(synth.random_vector(f.n_det, seed=7)).cuda()


@pytest.mark.parametrize("s", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("n,ne", [(2, 1), (8, 8), (9, 8), (10, 2), (16, 2), (17, 2), (18, 2), (11, 4)])
def test_spinor_blocks(fci_lib, monkeypatch, n, ne, s):
    """No upper spinors, one, a full block of 8 and one past it; even and odd block counts: the
    bits of the dense form, and up to 7 slices the exact integer model (at 8 the fixed-point G
    keeps 54 bits, so the last bit of the operator, which the library and the model assemble
    in different orders, reaches sigma)."""
    monkeypatch.setenv("FCI_SPLIT_FORM", "blocks")
    p = spinor_problem(n, ne, n_chol=4, seed=90 + n, e_core=0.3)
    f = gpu_fci(p)
    c = synth.random_vector(len(p["dets"]), seed=7, complex_=True)
    cd = torch.from_numpy(c).cuda()
    got = _sigma(f, cd, s)
    if s <= 7:
        assert rel_inf(got.cpu().numpy(), spinor_sigma_model(p["h"], p["g"], n, ne, c, s, e_core=0.3)) <= 1e-14
    monkeypatch.setenv("FCI_SPLIT_FORM", "dense")
    assert torch.equal(got, _sigma(f, cd, s))


LAYOUTS = [
    ([6, 3], [2, 1], 3, 1),                    # a diagonal class of 21 pairs: one full block and a rest
    ([5, 4], [2, 2], 4, 0),                    # 20 pairs between the spaces
    ([2, 2, 2, 2, 2], [1, 1, 0, 1, 0], 3, 1),  # 15 classes of 3 and 4 pairs sharing blocks
    ([9], [3], 3, 0),                          # one space: every block always active
    ([1, 4, 4], [1, 1, 1], 3, 2),
]


@pytest.mark.parametrize("image", ["rows", "determinants"])
@pytest.mark.parametrize("s", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("spaces,ref,nel,T", LAYOUTS)
def test_das_blocks(fci_lib, monkeypatch, spaces, ref, nel, T, s, image):
    """Both digit images of the block form: the bits of the dense form, and up to 7 slices the
    exact integer model (to the rounding of its inputs, as for the dense form)."""
    monkeypatch.setenv("FCI_SPLIT_FORM", "blocks")
    monkeypatch.setenv("FCI_DAS_ROW_BYTES", "1000000" if image == "rows" else "0")
    h, g, f, c = _das(spaces, ref, nel, T)
    got = _sigma(f, c, s)
    if s <= 7 and image == "rows":
        m = das_sigma_model(h, g, spaces, ref, nel, T, c.cpu().numpy(), s, e_core=0.3)
        assert rel_inf(got.cpu().numpy(), m) <= (1e-14 if s <= 5 else 1e-13)
    monkeypatch.setenv("FCI_SPLIT_FORM", "dense")
    assert torch.equal(got, _sigma(f, c, s))


@pytest.mark.parametrize("image", ["rows", "determinants"])
@pytest.mark.parametrize("s", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("spaces,ref,nel,T", [([3, 3, 2], [1, 2, 1], 4, 1), ([2, 2, 2, 2], [1, 1, 1, 0], 3, 2)])
def test_das_blocks_in_chunks_and_pieces(fci_lib, monkeypatch, spaces, ref, nel, T, s, image):
    """Digit image pieces that begin and end inside a row, E in several chunks: the bits of one
    dense pass."""
    _, _, f, c = _das(spaces, ref, nel, T)
    monkeypatch.setenv("FCI_SPLIT_FORM", "dense")
    want = _sigma(f, c, s)
    monkeypatch.setenv("FCI_SPLIT_FORM", "blocks")
    monkeypatch.setenv("FCI_DAS_ROW_BYTES", "1000000" if image == "rows" else "0")
    monkeypatch.setenv("FCI_DAS_IMAGE_DETS", "150")
    assert torch.equal(want, _sigma(f, c, s))
    monkeypatch.setenv("FCI_DAS_CHUNK_DETS", "700")
    assert f.info["n_det_intermediate"] > 2 * 704
    assert torch.equal(want, _sigma(f, c, s))


@pytest.mark.parametrize("s", [4, 6])
@pytest.mark.parametrize("kind", ["spinor", "das"])
def test_bounded_wait_of_the_block_form(fci_lib, monkeypatch, kind, s):
    """An MMA thread that never consumes a stage: the other roles' bounded waits expire, the
    kernel returns, the host reads FCI_ERR_TIMEOUT and the next call has the bits of the one
    before."""
    monkeypatch.setenv("FCI_SPLIT_FORM", "blocks")
    if kind == "spinor":
        f = gpu_fci(spinor_problem(10, 4, n_chol=6, seed=41))
    else:
        f = _das([3, 3, 2], [1, 2, 1], 4, 1)[2]
    c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()
    before = _sigma(f, c, s)
    monkeypatch.setenv("FCI_TEST_STALL_PRODUCER", "1")
    monkeypatch.setenv("FCI_WAIT_TIMEOUT_MS", "50")
    out = f.sigma(c, precision="oz_bf16", n_slices=s)
    with pytest.raises(fci.FCIError) as e:
        f.sync_status()
    assert e.value.code == fci.FCI_ERR_TIMEOUT
    assert torch.isnan(torch.view_as_real(out) if out.is_complex() else out).all()
    monkeypatch.delenv("FCI_TEST_STALL_PRODUCER")
    monkeypatch.delenv("FCI_WAIT_TIMEOUT_MS")
    assert torch.equal(before, _sigma(f, c, s))


@pytest.mark.parametrize("kind,s", [("spinor", 6), ("spinor", 4), ("das", 6)])
def test_default_rule_takes_the_blocks(fci_lib, monkeypatch, kind, s):
    """20 spinors, and 14 orbitals in three spaces with 2.5 M intermediate determinants in rows
    of more than 192: the block form (its workspace; its two kernels for the digit image), the bits
    of the dense one."""
    if kind == "spinor":
        h, g = synth.complex_integrals(20, 4, 71)
        f = gpu_fci(dict(h=h, g=g, e_core=0.3, n=20, ne=8))
        c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=True)).cuda()
    else:
        f, c = _das([6, 6, 2], [4, 3, 1], 8, 0)[2:]
    f.set_phase_timing(True)

    def run():
        out = _sigma(f, c, s)
        return out, (f.phase_times()["gather"]["launches"], f.sigma_workspace_bytes("oz_bf16", s))

    got, default = run()
    monkeypatch.setenv("FCI_SPLIT_FORM", "blocks")
    assert run()[1] == default
    monkeypatch.setenv("FCI_SPLIT_FORM", "dense")
    want, dense = run()
    assert dense != default and torch.equal(got, want)
