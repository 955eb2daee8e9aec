"""GPU tests of the contractions that cover active entries only: the edges of their blocks,
batches and lists."""
import numpy as np
import pytest
import torch

import oracle
from oracle import das as odas
from paper_2505_20375_gb300 import synth

from helpers import SIGMA_RTOL, fci_problem, gpu_fci, rel_inf, spinor_problem
from ozaki_model import das_sigma_model, spinor_sigma_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [(1, 1, 0), (1, 1, 1), (3, 3, 3), (5, 0, 2), (9, 1, 8), (20, 1, 1), (7, 3, 4)])
def test_fp64_active_lists_fci(fci_lib, n, na, nb):
    """Empty, full and one-determinant lists, a batch of one determinant, 210 pairs."""
    p = fci_problem(n, na, nb, n_chol=4, seed=60 + n, e_core=0.2)
    c = synth.random_vector(len(p["dets"]), seed=7)
    s = gpu_fci(p).sigma(torch.from_numpy(c).cuda()).cpu().numpy()
    assert rel_inf(s, oracle.sigma(p["hso"], p["gso"], p["dets"], c, e_core=0.2)) <= SIGMA_RTOL


@pytest.mark.parametrize("n,ne", [(1, 1), (3, 3), (5, 1), (12, 2), (13, 9), (18, 2)])
def test_fp64_active_lists_spinor(fci_lib, n, ne):
    p = spinor_problem(n, ne, n_chol=4, seed=70 + n, e_core=0.2)
    c = synth.random_vector(len(p["dets"]), seed=7, complex_=True)
    s = gpu_fci(p).sigma(torch.from_numpy(c).cuda()).cpu().numpy()
    assert rel_inf(s, oracle.sigma(p["hso"], p["gso"], p["dets"], c, e_core=0.2)) <= SIGMA_RTOL


@pytest.mark.parametrize("n,ne,s", [(2, 1, 3), (8, 8, 5), (9, 8, 3), (10, 2, 8), (16, 2, 4), (17, 2, 3), (18, 2, 2)])
def test_spinor_blocks_equal_exact_integer_model(fci_lib, n, ne, s):
    """No upper spinors, one, a full block of 8 and one past it; even and odd block counts."""
    p = spinor_problem(n, ne, n_chol=4, seed=90 + n, e_core=0.3)
    f = gpu_fci(p)
    c = synth.random_vector(len(p["dets"]), seed=7, complex_=True)
    sg = f.sigma(torch.from_numpy(c).cuda(), precision="oz_bf16", n_slices=s).cpu().numpy()
    f.sync_status()
    assert rel_inf(sg, spinor_sigma_model(p["h"], p["g"], n, ne, c, s, e_core=0.3)) <= 1e-14


@pytest.mark.parametrize("s", [4, 6])
@pytest.mark.parametrize("spaces,ref,nel,T", [
    ([6, 3], [2, 1], 3, 1),                    # a diagonal class of 21 pairs: one full block and a rest
    ([5, 4], [2, 2], 4, 0),                    # 20 pairs between the spaces
    ([2, 2, 2, 2, 2], [1, 1, 0, 1, 0], 3, 1),  # 15 classes of 3 and 4 pairs sharing blocks
    ([9], [3], 3, 0),                          # one space: every block always active
    ([1, 4, 4], [1, 1, 1], 3, 2),
])
def test_das_blocks_equal_exact_integer_model(fci_lib, spaces, ref, nel, T, s):
    n = sum(spaces)
    h, g = synth.real_integrals(n, 6, 50 + n)
    f = gpu_fci(dict(h=h, g=g, e_core=0.3, n=n, na=nel, nb=nel)).build_das(spaces, ref, ref, T)
    c = synth.random_vector(f.n_det, seed=7)
    sg = f.sigma(torch.from_numpy(c).cuda(), precision="oz_bf16", n_slices=s).cpu().numpy()
    f.sync_status()
    assert rel_inf(sg, das_sigma_model(h, g, spaces, ref, nel, T, c, s, e_core=0.3)) <= 1e-14
    dets, _ = odas.das_dets(spaces, ref, ref, nel, nel, T)
    hso, gso = oracle.spin_orbital_integrals(h, g)
    s64 = f.sigma(torch.from_numpy(c).cuda()).cpu().numpy()
    assert rel_inf(s64, oracle.sigma(hso, gso, dets, c, e_core=0.3)) <= SIGMA_RTOL


@pytest.mark.parametrize("ms", [3, 8, 17, 32])
@pytest.mark.parametrize("kind", ["real", "complex"])
def test_davidson_subspace_sizes(fci_lib, kind, ms):
    """The projected eigensolver and the reductions at every accumulator width, against the
    lowest eigenvalue of dense H.  tol_residual bounds the energy error by its square over
    the gap."""
    p = fci_problem(6, 3, 2, n_chol=8, seed=21, e_core=0.4) if kind == "real" else spinor_problem(8, 3, n_chol=8, seed=22, e_core=0.4)
    r = gpu_fci(p).davidson(max_iter=400, max_subspace=ms, tol_residual=1e-6, tol_energy=1e-12)
    w = np.linalg.eigvalsh(oracle.dense_h(p["hso"], p["gso"], p["dets"]))
    assert r.converged and abs(r.energy - (w[0] + 0.4)) <= max(1e-10, 1e-12 / (w[1] - w[0]))


@pytest.mark.parametrize("s", [3, 6])
@pytest.mark.parametrize("n,na,nb,path", [(6, 3, 3, "fused"), (10, 5, 5, "fused"), (9, 4, 4, "gemm"), (10, 5, 5, "gemm")])
def test_sigma_calls_back_to_back(fci_lib, monkeypatch, n, na, nb, path, s):
    """Kernels that start under the one before them: sigma builds queued without a wait, each on
    the result of the last or on another vector through the same workspace, on two streams in
    turn, give the bits of builds that are waited for one by one."""
    monkeypatch.setenv("FCI_OZ_PATH", path)
    h, g = synth.real_integrals(n, 6, 40 + n)
    f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=n, na=na, nb=nb))
    x = [torch.from_numpy(synth.random_vector(f.n_det, seed=k)).cuda() for k in (7, 8)]

    def chain(wait):
        out, y = [], x[0]
        for _ in range(12):
            y = f.sigma(y, precision="oz_bf16", n_slices=s)
            wait()
            out += [y, f.sigma(x[1], precision="oz_bf16", n_slices=s)]
            wait()
        torch.cuda.synchronize()
        return out

    ref = chain(torch.cuda.synchronize)
    f.sync_status()
    for st in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(st):
            got = chain(lambda: None)
        assert all(torch.equal(a, b) for a, b in zip(ref, got))


@pytest.mark.parametrize("s", [4, 6, 8])
@pytest.mark.parametrize("layout", ["spinor", "das one M-tile", "das two M-tiles"])
def test_dense_and_block_forms_agree(fci_lib, monkeypatch, layout, s):
    """The two forms of the contraction (every pair, or the blocks a tile uses) give the same
    bits, each with a workspace of its own size, also when one handle changes between them."""
    if layout == "spinor":
        h, g = synth.complex_integrals(11, 6, 71)
        f = gpu_fci(dict(h=h, g=g, e_core=0.3, n=11, ne=4))
    else:
        spaces, ref, nel = ([3, 3, 3], [1, 1, 1], 3) if layout == "das one M-tile" else ([6, 5, 5], [1, 1, 0], 2)
        h, g = synth.real_integrals(sum(spaces), 6, 72)  # 45 and 136 pairs
        f = gpu_fci(dict(h=h, g=g, e_core=0.3, n=sum(spaces), na=nel, nb=nel)).build_das(spaces, ref, ref, 1)
        if s * f.info["n_pair"] > 1023:
            pytest.skip("more slices than the level sums hold")
    c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()
    out = []
    for form in ("dense", "blocks", "dense"):
        monkeypatch.setenv("FCI_SPLIT_FORM", form)
        out.append(f.sigma(c, precision="oz_bf16", n_slices=s))
        f.sync_status()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
