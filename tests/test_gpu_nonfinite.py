"""Infinities in a cube (flagged or corrupt samples) stay what they are: an infinite
sample that a model is added to stays infinite, its neighbours are untouched, and the
loss of a cube that holds one is infinite, not no number."""
import numpy as np
import pytest

from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import make_peeler  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


@pytest.mark.parametrize("n_chan", [20, 130])
def test_prediction_onto_an_infinite_sample(n_chan):
    cad = Cadence(5, n_chan, 2, 1, seed=301)
    p = make_peeler(cad, "mixed")
    J = torch.from_numpy(cad.jones().astype(np.complex64)).cuda()
    base = torch.ones(p.cube_shape, dtype=torch.complex64, device="cuda")
    want = p.predict(cad.sources(), J, out=base.clone(), accumulate=True)
    at, values = (1, 3, n_chan - 1, 2), (complex(np.inf, 1.0), complex(1.0, -np.inf), complex(np.nan, 1.0))
    for v in values:
        cube = base.clone()
        cube[at] = v
        got = p.predict(cad.sources(), J, out=cube, accumulate=True)
        part = got[at].real if not np.isfinite(v.real) else got[at].imag
        bad = v.real if not np.isfinite(v.real) else v.imag
        assert part.item() == bad or (np.isnan(bad) and np.isnan(part.item()))
        got[at] = want[at]
        assert torch.equal(got, want)
    p.close()


@pytest.mark.parametrize("grad_kernel", [0, 1], ids=["auto", "direct"])
def test_loss_of_an_infinite_sample(grad_kernel):
    cad = Cadence(5, 40, 2, 3, seed=302)
    p = make_peeler(cad, "mixed", grad_kernel=grad_kernel)
    vis = torch.ones(p.cube_shape, dtype=torch.complex64, device="cuda")
    vis[1, 2, 39, 0] = complex(np.inf, 0.0)
    J = torch.from_numpy(cad.jones().astype(np.complex64)).cuda()
    loss, _, _ = p.grad(vis, J, torch.from_numpy(cad.sources()).cuda())
    assert loss.item() == np.inf
    p.close()
