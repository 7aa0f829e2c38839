"""The cluster solve of gains linear in frequency (k_cluster_taylor) at the edges
of its geometry, against the oracle's solve of the same cube: antenna counts with
ragged slots, the largest array it takes and the first past it (sweep launches),
sweep counts with and without a slope-rotation step, two channels (no step).

Tolerances as test_gpu_taylor.py: G and H 1e-5 relative, residual 1e-5 x rms."""
import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import check_status, rms_of  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    ("two-channels", Cadence(6, 2, 3, 1, seed=261), 20),
    ("three-channels", Cadence(9, 3, 4, 1, seed=262), 20),
    ("one-sweep", Cadence(17, 64, 2, 2, seed=263), 1),
    ("two-sweeps", Cadence(17, 64, 2, 2, seed=263), 2),
    ("three-sweeps", Cadence(17, 64, 2, 2, seed=263), 3),
    ("33-antennas", Cadence(33, 128, 2, 3, seed=264), 20),
    ("129-antennas", Cadence(129, 32, 2, 2, seed=265), 20),
    ("200-antennas", Cadence(200, 16, 1, 1, seed=266), 20),                  # past the cluster's shared memory
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


@pytest.mark.parametrize("name,cad,n_iter", CASES, ids=[c[0] for c in CASES])
def test_cluster_taylor_matches_oracle(name, cad, n_iter):
    from paper_1003_5575_gb300 import Peeler
    V = oracle.predict_taylor(cad.uvw(), cad.freqs(), cad.sources(), cad.jones(), cad.jones_slope(0.2))
    V = (V + cad.noise().reshape(V.shape)).astype(np.complex64).astype(np.complex128)
    R_ref, G_ref, H_ref, st_ref, rel_ref = oracle.peel_taylor(cad.uvw(), cad.freqs(), V, cad.sources(), n_iter=n_iter,
                                                              with_rel=True)
    p = Peeler(cad.uvw(), cad.freqs(), n_iter=n_iter, max_sources=cad.n_src)
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
