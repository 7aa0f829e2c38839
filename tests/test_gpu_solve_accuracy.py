"""Rounding of the cluster solve beside the per-step launches' on the same averages.

The launches solve every sweep's 2x2 systems in FP64 and subtract the in-block
corrections one by one; the cluster takes FP32 2x2 steps before the last sweep, which
moves the gains of the faintest sources by about 1e-7 of 3e-7.  Corrected averages are
small differences of large sums (61 sources within one block), so anything else that
is rounded carelessly shows: FP32 sums of 56 corrections alone double the error."""
import numpy as np
import pytest

from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import make_peeler, oracle_case, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def test_cluster_solve_rounds_like_the_per_step_launches():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()
    err = {0: [], 1: []}
    for seed in (281, 282, 283, 284):
        cad = Cadence(65, 203, 3, 61, freq0_hz=167e6, noise_sigma=12.0, seed=seed)
        V, _, J_ref, _, _ = oracle_case(cad)
        for kernel in err:
            p = make_peeler(cad, "mixed", per_pass=64, solve_kernel=kernel)
            _, jones, _ = p.cadence(to_dev(V, "mixed"), cad.sources())
            err[kernel].append(np.linalg.norm(jones.cpu().numpy() - J_ref) / np.linalg.norm(J_ref))
            p.close()
    cluster, launches = np.mean(err[0]), np.mean(err[1])
    print(f"gains: cluster {cluster:.2e}, per-step launches {launches:.2e}")
    assert cluster <= 1.5 * launches
