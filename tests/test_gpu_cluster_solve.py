"""The cluster solve of small arrays (k_cluster_solve) at the edges of its
geometry, against the oracle's sequential peel: one and two antennas' worth of
slots, cluster sizes 1 to 16, ragged last slots, the largest array it takes and the
first one past it (k_block_solve), sources in several groups with a short last one.

Tolerances as test_gpu_parity.py (residual and Jones 1e-5): the FP64 oracle moves
by at most 1.5e-7 (Jones) and 7e-8 x rms (residual) on these cases when its input
is perturbed by 1e-7 x rms."""
import numpy as np
import pytest

from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import TOL, check_status, jones_rel, make_peeler, oracle_case, rms_of, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    ("two-antennas", Cadence(2, 64, 4, 1, seed=201)),
    ("17-antennas", Cadence(17, 256, 2, 9, freq0_hz=167e6, seed=202)),        # 4 CTAs, 5 slots; groups 8 + 1
    ("33-antennas", Cadence(33, 192, 2, 17, freq0_hz=167e6, seed=203)),       # 8 CTAs, 5 slots; 8 + 8 + 1
    ("129-antennas", Cadence(129, 64, 2, 18, freq0_hz=167e6, seed=204)),      # 16 CTAs, 9 slots
    ("256-antennas", Cadence(256, 40, 2, 17, freq0_hz=167e6, seed=205)),      # 16 slots: the largest
    ("257-antennas", Cadence(257, 40, 2, 10, freq0_hz=167e6, seed=206)),      # past it: grid-wide solve
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


@pytest.mark.parametrize("name,cad", CASES, ids=[c[0] for c in CASES])
def test_cluster_solve_matches_oracle(name, cad):
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    p = make_peeler(cad, "mixed", per_pass=64)
    vis = to_dev(V, "mixed")
    resid, jones, st = p.cadence(vis, cad.sources())
    again, jones2, _ = p.cadence(vis, cad.sources())
    torch.cuda.synchronize()
    assert np.abs(resid.cpu().numpy() - R_ref).max() / rms_of(V) <= TOL["mixed"]
    assert jones_rel(jones.cpu().numpy(), J_ref) <= TOL["mixed"]
    check_status(name, st, st_ref, p.rel(cad.n_src), rel_ref)
    assert torch.equal(again, resid) and torch.equal(jones2, jones)          # deterministic
    p.close()


@pytest.mark.parametrize("n_iter", [1, 2, 5, 20])
@pytest.mark.parametrize("n_ant", [2, 3, 17, 129, 256, 300])
def test_single_solve_matches_oracle(n_ant, n_iter):
    """rts_peel_solve: one cluster up to 256 antennas (k_cluster_als), sweep launches
    past that, FP64 iterates both; tolerance 1e-5 as the other FP32 cases (the FP32
    products of each sweep's terms carry 1e-7)."""
    import oracle
    cad = Cadence(n_ant, 8, 1, 1, seed=251)
    rng = np.random.default_rng(n_ant)
    n_bl = n_ant * (n_ant - 1) // 2
    J = cad.jones()[0].reshape(n_ant, 2, 2)
    i, j = np.triu_indices(n_ant, k=1)
    S = 5.0
    avg = S * J[i] @ J[j].conj().transpose(0, 2, 1) + 0.1 * (rng.standard_normal((n_bl, 2, 2))
                                                             + 1j * rng.standard_normal((n_bl, 2, 2)))
    avg = avg.reshape(n_bl, 4).astype(np.complex64)
    J_ref, st_ref, rel_ref = oracle.als(avg.astype(np.complex128), S, n_ant, n_iter=n_iter)
    p = make_peeler(cad, "mixed", n_iter=n_iter)
    got, st = p.solve(torch.from_numpy(avg).cuda(), S)
    assert np.linalg.norm(got.cpu().numpy() - J_ref) / np.linalg.norm(J_ref) <= TOL["mixed"]
    check_status(f"solve-{n_ant}-{n_iter}", [st], [st_ref], p.rel(1), [rel_ref])
    p.close()
