"""The adjoint's workspace of a handle made for many sources and times: the antenna
phases of the strip sweep are kept for as many sources as that sweep takes, so such a
handle works (for all of 2^20 sources they would be 412 GB) and gives the same bits as
one made for the call's own sources."""
import numpy as np
import pytest

from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import make_peeler  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grad_kernel", [0, 1], ids=["auto", "direct"])
def test_adjoint_of_a_large_handle(grad_kernel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()
    cad = Cadence(24, 1, 1024, 3, seed=311)
    rng = np.random.default_rng(311)
    J = torch.from_numpy(cad.jones().astype(np.complex64)).cuda()
    src = torch.from_numpy(cad.sources()).cuda()
    out = []
    for max_sources in (cad.n_src, 1 << 20):
        p = make_peeler(cad, "mixed", max_sources=max_sources, per_pass=1, grad_kernel=grad_kernel)
        if not out:
            v = rng.standard_normal(p.cube_shape + (2,)).astype(np.float32)
            vis = torch.view_as_complex(torch.from_numpy(v)).cuda()
        out.append(p.grad(vis, J, src))
        torch.cuda.synchronize()
        p.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
