"""GPU tests of one handle used with several slice counts in turn."""
import pytest
import torch

from paper_2505_20375_gb300 import fci, synth

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


def _problem(kind):
    if kind == "spinor":
        h, g = synth.complex_integrals(10, 6, 46)
        f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=10, ne=4))
    else:
        h, g = synth.real_integrals(9, 6, 46)
        f = gpu_fci(dict(h=h, g=g, e_core=0.2, n=9, na=3, nb=3))
        if kind == "das":
            f.build_das([3, 3, 3], [1, 1, 1], [1, 1, 1], 1)
    return f, torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()


def _workspace(f, counts):
    nb = max(f.sigma_workspace_bytes("oz_bf16", s) for s in counts)
    buf = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    return buf, (buf.data_ptr() + 255) & ~255, nb


# (3, 2): the two images of one form; (3, 6): on the DAS layout the two forms; (6, 4): the
# one of the two-pass form
@pytest.mark.parametrize("counts", [(3, 2), (3, 6), (6, 4)])
@pytest.mark.parametrize("kind", ["fci", "das", "spinor"])
def test_graphs_of_two_slice_counts_replay_in_turn(fci_lib, kind, counts):
    """A captured sigma names the operator image of its slice count, which stays through
    builds with other counts, also for the grouped graph."""
    f, c = _problem(kind)
    want = {s: f.sigma(c, precision="oz_bf16", n_slices=s) for s in counts}
    buf, ws, nb = _workspace(f, counts)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    outs = {(how, s): torch.empty_like(c) for how in ("single", "grouped") for s in counts}
    with torch.cuda.stream(st):
        for _ in range(3):
            for (how, s), o in outs.items():
                o.fill_(float("nan"))
                if how == "single":
                    f.sigma_graph_into(c.data_ptr(), o.data_ptr(), "oz_bf16", s, ws, nb, stream=st)
                else:
                    fci.sigma_grouped([(f, c, o, "oz_bf16", s, ws, nb)], stream=st, graph=True)
                assert torch.equal(o, want[s])
    f.sync_status(st)
    f.clear_graphs()
    fci.clear_grouped_graphs()


def test_rebuilding_the_layout_drops_the_graphs(fci_lib):
    """das_build_categories frees the tables of the layout before; a graph of that layout with
    the same arguments must not replay."""
    f, c = _problem("das")
    buf, ws, nb = _workspace(f, (3,))
    big = torch.empty(8 * nb + 256, dtype=torch.uint8, device="cuda")
    ws, nb = (big.data_ptr() + 255) & ~255, 8 * nb
    out = torch.empty(4 * f.n_det, dtype=torch.float64, device="cuda")
    st = torch.cuda.Stream()
    x = torch.from_numpy(synth.random_vector(4 * f.n_det, seed=8)).cuda()
    torch.cuda.synchronize()
    for ref in ([1, 1, 1], [2, 1, 0], [1, 1, 1]):
        f.build_das([3, 3, 3], ref, ref, 1)
        n = f.n_det
        assert n <= x.numel() and f.sigma_workspace_bytes("oz_bf16", 3) <= nb
        for _ in range(2):
            f.sigma_graph_into(x.data_ptr(), out.data_ptr(), "oz_bf16", 3, ws, nb, stream=st)
            f.sync_status(st)
            assert torch.equal(out[:n], f.sigma(x[:n].contiguous(), precision="oz_bf16", n_slices=3))
            torch.cuda.synchronize()
