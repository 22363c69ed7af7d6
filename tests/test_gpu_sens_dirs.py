"""The sensitivity pass's direction choices (the law's coefficients, or the
free parameters where they are fewer) and its two layouts: against the
oracle's FP64 normal equations, and bit for bit between the layouts."""
import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W
from common import NM

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_E, _H = (0, 1e8, 1e10, True), (1, 1e-20, 1e-19, True)
_R, _A0, _ETA = (2, 5e-9, 30e-9, False), (3, 0.2e-9, 0.5e-9, False), (4, 0.0, 500.0, False)
_FIX = [1e9, 5e-20, 10e-9, 0.3e-9, 200.0]
_K, _HD, _Z = (0, 0.5, 8.0, True), (1, -2e-9, 4e-9, False), (2, 0.0, 2e-7, False)


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    assert torch.cuda.is_available()
    return afminv


@pytest.mark.parametrize("force,free,fixed,modes,n", [
    ("dmt", [_R], _FIX, 3, 200), ("dmt", [_E, _A0], _FIX, 3, 161), ("dmt", [_A0, _R, _E], _FIX, 3, 193),
    ("dmt", [_H, _E, _A0, _R], _FIX, 2, 160), ("dmt", [_E, _H, _R, _A0], _FIX, 1, 1),
    ("dmt_kv", [_ETA], _FIX, 3, 96), ("dmt_kv", [_E, _ETA, _R], _FIX, 3, 97),
    ("dmt_kv", [_E, _H, _ETA, _A0], _FIX, 3, 95), ("dmt_kv", [_E, _H, _R, _A0, _ETA], _FIX, 1, 130),
    ("hooke", [_HD], [3.0, 0, 0, 0, 0], 3, 130), ("hooke", [_HD, _K], [0.0] * 5, 3, 130),
    ("linear_spring", [(1, 10e-9, 20e-9, False), (0, 2.0, 20.0, False)], [0.0] * 5, 3, 130),
    ("spring_damper", [_Z, _K], [0, 1e-9, 0, 0, 0], 3, 130),
    ("spring_damper", [_K, _HD, _Z], [0.0] * 5, 3, 130)])
def test_directions_and_layouts(orc, afm, force, free, fixed, modes, n):
    spec = W.get("c2", force=force, free=free, fixed=fixed, n_modes=modes)
    D = len(free)
    P = 4870                                   # past the lane layout for 2 and 4 lanes at 9728
    P = P if D > 2 else 9730
    x = W.sample_x(D, P, seed=8, lo=0.05, hi=0.95)
    prob = afm.make_problem(spec, n_steps=n)
    U_m = 10e-9 * np.cos(0.02 * np.arange(n))
    U = torch.from_numpy((U_m / NM).astype(np.float32)).cuda()
    S, H, b = afm.normal_equations(prob, torch.from_numpy(x).cuda(), U)
    few = 21
    xs = torch.from_numpy(np.ascontiguousarray(x[:, :few])).cuda()
    S1, H1, b1 = afm.normal_equations(prob, xs, U)
    assert torch.equal(S1, S[:few]) and torch.equal(H1, H[:few]) and torch.equal(b1, b[:few])
    _, S_fwd = afm.forward_batch(prob, xs, U, want_defl=False)
    assert torch.equal(S1, S_fwd)
    assert torch.equal(H, H.transpose(1, 2))
    c, pm = orc.make_case(spec), orc.make_pmap(spec)
    U32 = U.double().cpu().numpy() * NM
    for p in range(0, few, 5):
        _, Ho, bo = orc.normal_eq(c, pm, x[:, p].astype(np.float64), U32)
        Ho, bo = Ho / NM ** 2, bo / NM ** 2
        # FP32 tangents over n <= 200 steps: 1e-4 of the largest entry (as over
        # the 20-cycle records of test_gpu_lm.py, 1e-3)
        assert np.max(np.abs(H1[p].cpu().numpy() - Ho)) <= 1e-4 * np.max(np.abs(Ho))
        assert np.max(np.abs(b1[p].cpu().numpy() - bo)) <= 1e-4 * np.max(np.abs(bo)) + 1e-12
