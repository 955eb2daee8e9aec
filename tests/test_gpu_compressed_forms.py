"""GPU tests of the two ways in which the compressed sigma finds the columns of an entry: lists of
the columns per string, or a walk of the entry's replacements."""
import numpy as np
import pytest
import torch

from paper_2505_20375_gb300 import synth

from helpers import gpu_fci

pytestmark = pytest.mark.gpu


# random: columns of their own; first: neighbours share theirs; in the forced forms entries with
# more than 400 columns or 64 terms change from the lists to the walk, and more than 2^14
# entries from a walk by warps to one by threads
@pytest.mark.parametrize("spaces,ref,nel,T,count,which,form", [
    ([4, 4, 4], [2, 2, 2], 6, 2, 1, "random", "lists"),
    ([4, 4, 4], [2, 2, 2], 6, 2, 60, "random", "lists"),
    ([4, 4, 4], [2, 2, 2], 6, 2, 60, "first", "walk"),
    ([4, 4, 4], [2, 2, 2], 6, 2, 3000, "first", "walk"),
    ([5, 5], [2, 3], 5, 2, 20000, "first", "walk"),
    ([5, 5], [2, 3], 5, 2, 700, "random", "walk"),  # lists of more columns than pairs
    ([3, 3, 2], [1, 2, 1], 4, 1, 10 ** 6, "first", "walk"),  # every determinant
    ([2, 2], [1, 1], 2, 0, 1, "first", "lists"),
    ([1, 2], [1, 1], 2, 1, 3, "first", "walk"),
    ([6, 6], [1, 0], 1, 1, 40, "random", "walk"),
])
def test_lists_and_walk_agree(fci_lib, monkeypatch, spaces, ref, nel, T, count, which, form):
    n = sum(spaces)
    h, g = synth.real_integrals(n, 6, 31)
    f = gpu_fci(dict(h=h, g=g, e_core=0.4, n=n, na=nel, nb=nel)).build_das(spaces, ref, ref, T)
    count = min(count, f.n_det)
    addr = np.arange(count)
    if which == "random":
        addr = np.sort(np.random.default_rng(3).choice(f.n_det, count, replace=False))
    val = synth.random_vector(count, seed=5) if count > 1 else np.ones(1)
    addr, val = torch.from_numpy(addr).cuda(), torch.from_numpy(val).cuda()
    f.set_phase_timing(True)
    f.sigma_compressed(addr, val)
    assert f.phase_times()["scatter"]["launches"] == {"lists": 3, "walk": 1}[form]
    got = {}
    for force in ("lists", "walk"):
        monkeypatch.setenv("FCI_CS_FORM", force)
        got[force] = f.sigma_compressed(addr, val)
    c = torch.zeros(f.n_det, dtype=torch.float64, device="cuda")
    c[addr] = val
    dense = f.sigma(c)
    for a, v in got.values():
        assert torch.equal(a, got["lists"][0]) and torch.equal(v, dense[a])
