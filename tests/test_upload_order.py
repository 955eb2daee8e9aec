"""Host-to-device uploads of the library are ordered before the kernels that read them."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_20375_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_no_upload_or_clear_leaves_the_callers_stream():
    """cudaMemcpy from pageable memory and cudaMemset may return before the device is done, on
    the default stream, and a non-blocking stream does not wait for that: uploads go through
    fci_upload (a copy on the stream), clears through cudaMemsetAsync."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = _code(path)
        assert not re.search(r"cudaMemset\s*\(", code), path
        for call in re.findall(r"cudaMemcpy\s*\([^;]*;", code):
            assert "cudaMemcpyHostToDevice" not in call, (path, call)
    body = re.search(r"int fci_upload\([^)]*\) \{.*?\n\}", _code(os.path.join(CSRC, "fci_api.cu")), re.S).group(0)
    assert re.search(r"cudaMemcpyAsync\([^;]*, s\)", body)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["fci", "das", "spinor"])
def test_handles_built_on_a_side_stream(fci_lib, kind):
    """Integrals, strings, layout and the first sigma of each precision on a non-blocking
    stream: the bits of a handle built on the default stream."""
    import torch

    from helpers import gpu_fci
    from paper_2505_20375_gb300 import synth

    if kind == "spinor":
        h, g = synth.complex_integrals(12, 6, 5)
        p = dict(h=h, g=g, e_core=0.3, n=12, ne=5)
    else:
        h, g = synth.real_integrals(12, 6, 5)
        p = dict(h=h, g=g, e_core=0.3, n=12, na=3, nb=3)

    def results():
        f = gpu_fci(p)
        if kind == "das":
            f.build_das([4, 4, 4], [1, 1, 1], [1, 1, 1], 1)
        c = torch.from_numpy(synth.random_vector(f.n_det, seed=7, complex_=f.is_complex)).cuda()
        out = [f.sigma(c)] + [f.sigma(c, precision="oz_bf16", n_slices=s) for s in (3, 6)]
        f.sync_status()
        return out

    ref = results()
    for _ in range(4):
        with torch.cuda.stream(torch.cuda.Stream()):
            got = results()
        assert all(torch.equal(a, b) for a, b in zip(ref, got))
