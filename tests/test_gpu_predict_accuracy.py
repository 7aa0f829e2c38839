"""Rounding of the FP32 prediction where its sources add up coherently: antennas within
a metre, so every phase is small and a sample is the sum of the fluxes' models.  The
compensated sum of 128 terms is rounded once (2^-25 of its binade, 2.4e-8 of the value
in the mean) and a term is good to about 1e-7, random from term to term (1e-8 of the
sum); eight terms at a time in plain FP32 add 0.6e-8.  Plain sums of 32 sources would
be off by 7e-8."""
import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import make_peeler  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_chan", [40, 200])
def test_prediction_sums_are_compensated(n_chan):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()
    cad = Cadence(12, n_chan, 3, 128, radius_m=1.0, smax=1.5, seed=291)
    J = cad.jones().astype(np.complex64)
    ref = oracle.predict(cad.uvw(), cad.freqs(), cad.sources(), J.astype(np.complex128))
    p = make_peeler(cad, "mixed")
    got = p.predict(cad.sources(), torch.from_numpy(J).cuda()).cpu().numpy()
    p.close()
    d = (got - ref)[..., [0, 3]]               # XX and YY, where the fluxes add up
    err = np.sqrt(np.mean(np.abs(d) ** 2)) / np.sqrt(np.mean(np.abs(ref[..., [0, 3]]) ** 2))
    print(f"{n_chan} channels: {err:.2e} of the sample")
    assert err <= 5e-8
