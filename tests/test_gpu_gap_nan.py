"""GPU test of a solve whose sigma turns NaN (a timed-out device wait) while the gap bound
converges the second Ritz pair."""
import pytest
import torch

from paper_2505_20375_gb300 import fci, synth

from helpers import gpu_fci

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["real", "complex"])
def test_nan_sigma_in_the_gap_phase_ends_the_solve(fci_lib, kind):
    """With every entry of the projected matrix NaN no diagonal entry has the rank of the second
    root; the eigensolver still takes an entry that exists, and the solve reports the value."""
    if kind == "real":
        h, g = synth.real_integrals(6, 8, 21)
        f = gpu_fci(dict(h=h, g=g, e_core=0.4, n=6, na=3, nb=3))
    else:
        h, g = synth.complex_integrals(8, 8, 22)
        f = gpu_fci(dict(h=h, g=g, e_core=0.4, n=8, ne=3))
    # from the ground state itself the subspace is small when the gap phase begins, so that phase
    # asks for further sigma builds
    c = f.davidson(tol_residual=1e-8, tol_energy=1e-12).vector
    ground = f.davidson(tol_residual=1e-6, tol_energy=1e-10, guess=c).n_sigma
    st = fci.DavidsonStepper(f, f.davidson_opts(tol_residual=1e-6, tol_energy=1e-10, gap_bound=True), guess=c)

    def vector(address):
        at = address - st._ws.data_ptr()
        return st._ws[at:at + f.n_det * (16 if f.is_complex else 8)].view(f.vector_dtype())

    for _ in range(ground):  # the ground state's solve, step by step
        x, y, *_ = st.request()
        vector(y).copy_(f.sigma(vector(x)))
        assert not st.advance()
    x, y, *_ = st.request()
    vector(y).fill_(float("nan"))
    with pytest.raises(fci.FCIError, match="non-finite"):
        st.advance()
    torch.cuda.synchronize()
    assert f.davidson(tol_residual=1e-6, tol_energy=1e-10).converged  # the handle stays usable
