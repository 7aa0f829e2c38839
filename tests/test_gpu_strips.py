"""The FP32 kernels that work on strips (strip_kernels.cuh) at the edges of their
tiles: the blocked pass, the prediction and the adjoint, against the oracle.
Strips hold 64, 128 or 256 channels in tiles of 16, sources go 32 or 64 at a
time, a CTA's warps take 8 (pass, prediction) or 12 (adjoint) strips.

Tolerances as test_gpu_parity.py.  The pass's cases are well conditioned: the
FP64 oracle moves by at most 1.5e-7 (Jones) and 7e-8 x rms (residual) under an
input perturbation of 1e-7 x rms."""
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


PASS_CASES = [
    ("17-channels", Cadence(40, 17, 8, 2, freq0_hz=167e6, seed=216), 64),
    ("64-channels-one-time", Cadence(20, 64, 1, 3, freq0_hz=167e6, seed=211), 64),      # eight baselines a CTA
    ("65-channels-9-times", Cadence(20, 65, 9, 33, freq0_hz=167e6, seed=212), 64),      # a warp's second time; 33 sources
    ("65-channels-blocks-of-16", Cadence(20, 65, 9, 33, freq0_hz=167e6, seed=212), 16),
    ("128-channels", Cadence(24, 128, 3, 6, freq0_hz=167e6, seed=213), 64),             # two baselines a CTA, odd count
    ("129-channels", Cadence(24, 129, 5, 8, freq0_hz=167e6, seed=214), 8),
    ("256-channels-17-times", Cadence(30, 256, 17, 35, freq0_hz=167e6, seed=215), 64),
]


@pytest.mark.parametrize("name,cad,per_pass", PASS_CASES, ids=[c[0] for c in PASS_CASES])
def test_strip_pass_matches_oracle(name, cad, per_pass):
    V, R_ref, J_ref, st_ref, rel_ref = oracle_case(cad)
    p = make_peeler(cad, "mixed", per_pass=per_pass, block_kernel=1)
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


PREDICT_CASES = [
    ("one-channel-one-source", Cadence(6, 1, 1, 1, seed=231)),
    ("64-channels-32", Cadence(7, 64, 9, 32, seed=232)),                     # QH = 2, a warp's second strip
    ("65-channels-33", Cadence(7, 65, 3, 33, seed=233)),
    ("128-channels-64", Cadence(6, 128, 8, 64, seed=234)),                   # one full launch
    ("129-channels-65", Cadence(6, 129, 2, 65, seed=235)),                   # two launches, a second tile of one channel
    ("300-channels", Cadence(5, 300, 5, 100, seed=236)),
]


@pytest.mark.parametrize("name,cad", PREDICT_CASES, ids=[c[0] for c in PREDICT_CASES])
def test_strip_prediction_matches_oracle(name, cad):
    J = cad.jones().astype(np.complex64)
    ref = oracle.predict(cad.uvw(), cad.freqs(), cad.sources(), J.astype(np.complex128))
    p = make_peeler(cad, "mixed")
    got = p.predict(cad.sources(), torch.from_numpy(J).cuda())
    base = torch.ones(p.cube_shape, dtype=torch.complex64, device="cuda")
    added = p.predict(cad.sources(), torch.from_numpy(J).cuda(), out=base, accumulate=True)
    assert np.abs(got.cpu().numpy() - ref).max() <= TOL["mixed"] * rms_of(ref)
    assert np.abs(added.cpu().numpy() - (ref + 1.0)).max() <= TOL["mixed"] * rms_of(ref) + 1e-6
    p.close()


def test_strip_prediction_takes_gains_on_an_element_boundary():
    cad = Cadence(7, 33, 2, 3, seed=237)
    J = torch.from_numpy(cad.jones().astype(np.complex64)).cuda()
    odd = torch.empty(J.numel() + 1, dtype=J.dtype, device="cuda")[1:].view(J.shape).copy_(J)
    assert odd.data_ptr() % 16 == 8
    p = make_peeler(cad, "mixed")
    assert torch.equal(p.predict(cad.sources(), odd), p.predict(cad.sources(), J))
    p.close()


GRAD_CASES = [
    ("one-channel", Cadence(6, 1, 1, 2, pos_sigma_rad=2.909e-4, seed=241)),
    ("255-channels-63", Cadence(5, 255, 1, 63, pos_sigma_rad=2.909e-4, seed=242)),       # one strip a baseline
    ("256-channels-64", Cadence(5, 256, 2, 64, pos_sigma_rad=2.909e-4, seed=243)),
    ("257-channels-65", Cadence(5, 257, 3, 65, pos_sigma_rad=2.909e-4, seed=244)),       # a strip of one channel
    ("520-channels-13-times", Cadence(4, 520, 13, 33, pos_sigma_rad=2.909e-4, seed=245)),   # 39 strips: five rounds
    ("12-strips", Cadence(5, 300, 6, 20, pos_sigma_rad=2.909e-4, seed=246)),               # one CTA an SM, 12 sources left
    ("161-sources", Cadence(4, 300, 4, 161, pos_sigma_rad=2.909e-4, seed=247)),           # totals outside shared memory
]


@pytest.mark.parametrize("name,cad", GRAD_CASES, ids=[c[0] for c in GRAD_CASES])
def test_strip_adjoint_matches_oracle(name, cad):
    V = oracle.simulate(cad.with_(pos_sigma_rad=0.0)).astype(np.complex64).astype(np.complex128)
    src = cad.perturbed_sources()
    src[-1, 2] = 0.0                                        # a source without flux still has dL/dS
    J = cad.jones().astype(np.complex64)
    L_ref, gJ_ref, gl_ref, gm_ref, gS_ref = oracle.loss_grad(cad.uvw(), cad.freqs(), V, src, J.astype(np.complex128))
    p = make_peeler(cad, "mixed")
    args = (to_dev(V, "mixed"), torch.from_numpy(J).cuda(), torch.from_numpy(src).cuda())
    loss, gJ, gs = p.grad(*args)
    again = p.grad(*args)
    torch.cuda.synchronize()
    assert abs(loss.item() - L_ref) <= 1e-5 * L_ref
    assert np.abs(gJ.cpu().numpy() - gJ_ref).max() <= 1e-4 * np.abs(gJ_ref).max()
    g = gs.cpu().numpy()
    for col, ref in ((0, gl_ref), (1, gm_ref), (2, gS_ref)):
        assert np.abs(g[:, col] - ref).max() <= 1e-4 * np.abs(ref).max(), col
    assert torch.equal(again[1], gJ) and torch.equal(again[2], gs)           # deterministic
    odd = torch.empty(J.size + 1, dtype=torch.complex64, device="cuda")[1:].view(J.shape).copy_(args[1])
    assert torch.equal(p.grad(args[0], odd, args[2])[1], gJ)                # gains on an element's boundary only
    p.close()
