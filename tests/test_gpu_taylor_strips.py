"""The Taylor pass on strips (k_taylor_pass_strip) at the edges of its geometry,
against the oracle's peel of the same cube: strips that do not fill a tile of 16
or a half warp's tiles, the widths at which the tiles a lane changes and the
longest strip, the first past it (tcgen05), one block and a ragged second, fewer
times than warps, as many, and more (running sums in shared memory).

Tolerances as test_gpu_taylor.py: G and H 1e-5 relative, residual 1e-5 x rms."""
import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import check_status, rms_of  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    ("17-chan", Cadence(10, 17, 5, 3, seed=271)),
    ("64-chan-2-blocks", Cadence(24, 64, 3, 22, seed=272)),
    ("65-chan", Cadence(16, 65, 8, 4, seed=279)),
    ("127-chan-9-times", Cadence(10, 127, 9, 4, seed=274)),
    ("128-chan-full-block", Cadence(24, 128, 4, 21, seed=275)),
    ("129-chan", Cadence(10, 129, 1, 3, seed=276)),
    ("256-chan-18-times", Cadence(9, 256, 18, 2, seed=277)),
    ("257-chan", Cadence(10, 257, 2, 3, seed=278)),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


def cube(cad):
    V = oracle.predict_taylor(cad.uvw(), cad.freqs(), cad.sources(), cad.jones(), cad.jones_slope(0.2))
    return (V + cad.noise().reshape(V.shape)).astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("name,cad", CASES, ids=[c[0] for c in CASES])
def test_taylor_strip_pass_matches_oracle(name, cad):
    from paper_1003_5575_gb300 import Peeler
    V = cube(cad)
    R_ref, G_ref, H_ref, st_ref, rel_ref = oracle.peel_taylor(cad.uvw(), cad.freqs(), V, cad.sources(), with_rel=True)
    p = Peeler(cad.uvw(), cad.freqs(), max_sources=cad.n_src)
    R, G, H, st = p.cadence_taylor(torch.from_numpy(V.astype(np.complex64)).cuda(), cad.sources())
    torch.cuda.synchronize()
    rel = p.rel(cad.n_src)
    p.close()
    assert np.abs(R.cpu().numpy() - R_ref).max() <= 1e-5 * rms_of(V)
    G, H = G.cpu().numpy(), H.cpu().numpy()
    for k in range(cad.n_src):
        X, X_ref = np.concatenate([G[k], H[k]], axis=1), np.concatenate([G_ref[k], H_ref[k]], axis=1)
        assert np.linalg.norm(X - X_ref) <= 1e-5 * np.linalg.norm(X_ref), k
    check_status(name, st, st_ref, rel, rel_ref, "taylor")
