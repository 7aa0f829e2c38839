"""Cubes of many times: the prediction past the antenna-times whose phases a handle
keeps (k_predict_mixed, two sources a launch at 1024 times), and the FP64 stream whose
baseline tables do not hold all times at once."""
import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import TOL, check_status, jones_rel, make_peeler, oracle_case, rms_of, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


def test_prediction_without_kept_phases_matches_oracle():
    cad = Cadence(129, 1, 1024, 3, seed=331)                   # 132 096 antenna-times (131 072 are kept)
    J = cad.jones().astype(np.complex64)
    ref = oracle.predict(cad.uvw(), cad.freqs(), cad.sources(), J.astype(np.complex128))
    p = make_peeler(cad, "mixed", per_pass=1)
    got = p.predict(cad.sources(), torch.from_numpy(J).cuda())
    assert np.abs(got.cpu().numpy() - ref).max() <= TOL["mixed"] * rms_of(ref)
    base = torch.ones(p.cube_shape, dtype=torch.complex64, device="cuda")
    added = p.predict(cad.sources(), torch.from_numpy(J).cuda(), out=base, accumulate=True)
    assert np.abs(added.cpu().numpy() - (ref + 1.0)).max() <= TOL["mixed"] * rms_of(ref) + 1e-6
    p.close()


def test_fp64_tables_of_53_of_60_times():
    cad = Cadence(5, 600, 60, 2, precision="fp64", seed=332)    # 19 x 32 tables: 608 bytes a time, 32 KB hold 53
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    p = make_peeler(cad, "fp64")
    resid, jones, st = p.cadence(to_dev(V, "fp64"), cad.sources())
    torch.cuda.synchronize()
    assert np.abs(resid.cpu().numpy() - R_ref).max() / rms_of(V) <= TOL["fp64"]
    assert jones_rel(jones.cpu().numpy(), J_ref) <= TOL["fp64"]
    check_status("60-times", st, st_ref, p.rel(cad.n_src), rel_ref, "fp64")
    p.close()
