"""The tcgen05 pass (k_block_pass_tc05) at the edges of its geometry, against the
oracle: strips that fill one, two and three groups of 16 tiles or leave the last
ragged, the longest it takes, blocks that do not fill 64 sources, one time step
and odd counts (ring slots), and arrays whose CTAs take several baselines, with
one time step each (a flush every step) and more.

Tolerances as test_gpu_parity.py; the cases' responses to an input perturbation
of 1e-7 x rms are below 1.3e-7 (Jones) and 4e-7 x rms (residual) in the FP64 oracle."""
import numpy as np
import pytest

import oracle  # noqa: F401
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


CASES = [
    ("16-channels", Cadence(40, 16, 4, 3, freq0_hz=167e6, seed=281), 64),
    ("17-channels-blocks-of-8", Cadence(40, 17, 5, 9, freq0_hz=167e6, seed=282), 8),
    ("256-channels-65-sources", Cadence(40, 256, 3, 65, freq0_hz=167e6, seed=283), 64),   # one full block and one source
    ("257-channels", Cadence(24, 257, 2, 5, freq0_hz=167e6, seed=284), 64),
    ("512-channels-one-time", Cadence(24, 512, 1, 6, freq0_hz=167e6, seed=285), 64),
    ("513-channels-9-times", Cadence(16, 513, 9, 4, freq0_hz=167e6, seed=286), 64),
    ("768-channels-blocks-of-32", Cadence(30, 768, 3, 35, freq0_hz=167e6, seed=287), 32),
    ("2-baselines-a-cta-one-time", Cadence(72, 40, 1, 4, freq0_hz=167e6, seed=288), 64),
    ("3-baselines-a-cta", Cadence(87, 33, 2, 9, freq0_hz=167e6, seed=289), 8),
]


@pytest.mark.parametrize("name,cad,per_pass", CASES, ids=[c[0] for c in CASES])
def test_tc05_pass_matches_oracle(name, cad, per_pass):
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    p = make_peeler(cad, "mixed", per_pass=per_pass, block_kernel=3)
    vis = to_dev(V, "mixed")
    resid, jones, st = p.cadence(vis, cad.sources())
    work = vis.clone()
    r2, j2, _ = p.cadence(work, cad.sources(), resid=work)                   # in place: the same bits
    torch.cuda.synchronize()
    assert np.abs(resid.cpu().numpy() - R_ref).max() / rms_of(V) <= TOL["mixed"]
    assert jones_rel(jones.cpu().numpy(), J_ref) <= TOL["mixed"]
    check_status(name, st, st_ref, p.rel(cad.n_src), rel_ref)
    assert torch.equal(r2, resid) and torch.equal(j2, jones)
    p.close()
