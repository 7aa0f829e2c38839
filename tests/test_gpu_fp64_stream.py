"""The FP64 stream (k_stream_fp64) at the edges of its phasor tables, and on
channels that are uniform to 1e-9 only (one sincospi a sample instead of tables),
against the oracle; tolerance 1e-10 as the other FP64 cases."""
import numpy as np
import pytest

from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import TOL, check_status, jones_rel, make_peeler, oracle_case, rms_of, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


class Jittered(Cadence):
    """Channels off the uniform grid by up to 4e-10 of their frequency."""

    def freqs(self):
        f = super().freqs()
        return f * (1.0 + 4e-10 * np.sin(1.0 + np.arange(len(f))))


CASES = [
    ("one-channel", Cadence(6, 1, 5, 2, precision="fp64", seed=221)),               # tables of one entry each
    ("64-channels", Cadence(7, 64, 2, 2, precision="fp64", seed=222)),             # 8 x 8, full
    ("65-channels", Cadence(7, 65, 2, 2, precision="fp64", seed=223)),             # 16 x 5, a ragged last row
    ("many-times", Cadence(5, 600, 40, 2, precision="fp64", seed=224)),            # tables of 18 times at once, twice
    ("jittered", Jittered(7, 48, 3, 2, precision="fp64", seed=225)),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


@pytest.mark.parametrize("name,cad", CASES, ids=[c[0] for c in CASES])
def test_fp64_cadence_matches_oracle(name, cad):
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    p = make_peeler(cad, "fp64")
    resid, jones, st = p.cadence(to_dev(V, "fp64"), cad.sources())
    torch.cuda.synchronize()
    assert np.abs(resid.cpu().numpy() - R_ref).max() / rms_of(V) <= TOL["fp64"]
    assert jones_rel(jones.cpu().numpy(), J_ref) <= TOL["fp64"]
    check_status(name, st, st_ref, p.rel(cad.n_src), rel_ref, "fp64")
    p.close()


WALK_CASES = [
    ("one-time", Cadence(6, 600, 1, 2, precision="fp64", seed=226)),               # four groups share a time's tiles
    ("three-times", Cadence(6, 100, 3, 2, precision="fp64", seed=227)),            # two groups a time, two idle
    ("130-times", Cadence(4, 200, 130, 2, precision="fp64", seed=228)),            # tables of 78 times, then 52
]


@pytest.mark.parametrize("name,cad", WALK_CASES, ids=[c[0] for c in WALK_CASES])
def test_fp64_walk_of_tiles_matches_oracle(name, cad):
    test_fp64_cadence_matches_oracle(name, cad)
