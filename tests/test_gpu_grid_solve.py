"""Arrays past the cluster solve (257 antennas and more), as the benchmark's 512: the
cooperative block solve (k_block_solve) on full blocks beside the tcgen05 pass, and one
source's solve by sweep launches (k_als_sweep<float>), against the oracle at the
tolerances of test_gpu_parity.py.  The FP64 oracle moves by 3.1e-8 (gains) and
3.5e-8 x rms (residual) on the cadence when its input moves by 1e-7 x rms."""
import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import TOL, check_status, jones_rel, make_peeler, oracle_case, rms_of, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu

BLOCKS = Cadence(260, 257, 1, 130, freq0_hz=167e6, seed=321)       # blocks of 64, 64 and 2; 1.7 antennas a CTA


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import _abi, build
    build.build()
    return _abi


def test_block_solve_on_full_blocks_matches_oracle_and_launches(abi):
    cad = BLOCKS
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    out = []
    for kernel in (abi.RTS_SOLVE_AUTO, abi.RTS_SOLVE_LAUNCHES):
        p = make_peeler(cad, "mixed", solve_kernel=kernel)
        assert abi.rts_peel_kernels(p.h) == (abi.RTS_BLOCK_TCGEN05, kernel)
        resid, jones, st = p.cadence(to_dev(V, "mixed"), cad.sources())
        torch.cuda.synchronize()
        resid, jones, rel = resid.cpu().numpy(), jones.cpu().numpy(), p.rel(cad.n_src)
        p.close()
        assert np.abs(resid - R_ref).max() / rms_of(V) <= TOL["mixed"]
        assert jones_rel(jones, J_ref) <= TOL["mixed"]
        check_status(f"260x257x1x130, solve {kernel}", st, st_ref, rel, rel_ref)
        out.append((resid, jones, st, rel))
    # the same corrections, sweeps and models; the sums' grouping and the FP32 steps differ
    (r0, j0, s0, rel0), (r1, j1, s1, rel1) = out
    assert jones_rel(j0, j1) <= 3e-6
    assert np.abs(r0 - r1).max() <= 3e-6 * rms_of(V)
    check_status("block solve, launches", s0, s1, rel0, rel1)


@pytest.mark.parametrize("n_iter", [2, 20])
@pytest.mark.parametrize("n_ant", [257, 385, 512])
def test_single_solve_by_launches_matches_oracle(abi, n_ant, n_iter):
    cad = Cadence(n_ant, 8, 1, 1, seed=252)
    rng = np.random.default_rng(n_ant)
    n_bl = n_ant * (n_ant - 1) // 2
    J = cad.jones()[0].reshape(n_ant, 2, 2)
    i, j = np.triu_indices(n_ant, k=1)
    noise = 0.1 * (rng.standard_normal((n_bl, 2, 2)) + 1j * rng.standard_normal((n_bl, 2, 2)))
    avg = (5.0 * J[i] @ J[j].conj().transpose(0, 2, 1) + noise).reshape(n_bl, 4).astype(np.complex64)
    J_ref, st_ref, rel_ref = oracle.als(avg.astype(np.complex128), 5.0, n_ant, n_iter=n_iter)
    p = make_peeler(cad, "mixed", n_iter=n_iter)
    got, st = p.solve(torch.from_numpy(avg).cuda(), 5.0)
    assert np.linalg.norm(got.cpu().numpy() - J_ref) / np.linalg.norm(J_ref) <= TOL["mixed"]
    check_status(f"solve-{n_ant}-{n_iter}", [st], [st_ref], p.rel(1), [rel_ref])
    p.close()
