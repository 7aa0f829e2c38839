"""Antenna coordinates about a far origin: only differences uvw_i - uvw_j mean
anything, so the results are those of the oracle, which takes the differences,
whatever the origin.  FP64 about a geocentric one (6.4e6 m: a phase of the
coordinates themselves is off by 8.6e-10 radian, tolerance 1e-10); FP32 about a
barycentric one (1.5e11 m: off by 2e-5 radian, tolerance 1e-5 x rms, gradients
1e-4).  The coordinates' own rounding is in both sides' input."""
import dataclasses

import numpy as np
import pytest

import oracle
from synth import Cadence

torch = pytest.importorskip("torch")
from _parity import TOL, jones_rel, make_peeler, oracle_case, rms_of, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@dataclasses.dataclass(frozen=True)
class Far(Cadence):
    origin_m: float = 0.0

    def uvw(self):
        return super().uvw() + self.origin_m * np.array([0.6, -0.5, 0.62])


FP64 = Far(13, 70, 3, 4, precision="fp64", seed=261, origin_m=6.4e6)
FP32 = Far(13, 70, 3, 4, pos_sigma_rad=2.909e-4, seed=262, origin_m=1.5e11)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import build
    build.build()


@pytest.mark.parametrize("cad", [FP64, FP32.with_(pos_sigma_rad=0.0)], ids=["fp64", "mixed"])
def test_cadence_about_a_far_origin(cad):
    V, R_ref, J_ref, _, _ = oracle_case(cad)
    p = make_peeler(cad, cad.precision)
    resid, jones, _ = p.cadence(to_dev(V, cad.precision), cad.sources())
    torch.cuda.synchronize()
    assert np.abs(resid.cpu().numpy() - R_ref).max() / rms_of(V) <= TOL[cad.precision]
    assert jones_rel(jones.cpu().numpy(), J_ref) <= TOL[cad.precision]
    p.close()


def test_prediction_about_a_far_origin():
    J = FP32.jones().astype(np.complex64)
    ref = oracle.predict(FP32.uvw(), FP32.freqs(), FP32.sources(), J.astype(np.complex128))
    p = make_peeler(FP32, "mixed")
    got = p.predict(FP32.sources(), torch.from_numpy(J).cuda()).cpu().numpy()
    assert np.abs(got - ref).max() <= TOL["mixed"] * rms_of(ref)
    p.close()


def test_adjoint_about_a_far_origin():
    V = oracle.simulate(FP32.with_(pos_sigma_rad=0.0)).astype(np.complex64).astype(np.complex128)
    src, J = FP32.perturbed_sources(), FP32.jones().astype(np.complex64)
    L_ref, gJ_ref, gl_ref, gm_ref, _ = oracle.loss_grad(FP32.uvw(), FP32.freqs(), V, src, J.astype(np.complex128))
    p = make_peeler(FP32, "mixed")
    loss, gJ, gs = p.grad(to_dev(V, "mixed"), torch.from_numpy(J).cuda(), torch.from_numpy(src).cuda())
    assert abs(loss.item() - L_ref) <= 1e-5 * L_ref
    assert np.abs(gJ.cpu().numpy() - gJ_ref).max() <= 1e-4 * np.abs(gJ_ref).max()
    for col, ref in ((0, gl_ref), (1, gm_ref)):
        assert np.abs(gs[:, col].cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max(), col
    p.close()
