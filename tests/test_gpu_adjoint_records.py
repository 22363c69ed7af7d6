"""Both forms of the adjoint on records long enough for the segments at once
(kern_adjoint.cu: more than 110 to 170 steps), chosen by the workspace: S and G of
each against the oracle's complex step.  Step counts around the 32-step
segments, particle counts up to the form's bound for them."""
import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W
from common import NM

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_E, _H = (0, 1e8, 1e10, True), (1, 1e-20, 1e-19, True)
_A0, _ETA = (3, 0.2e-9, 0.5e-9, False), (4, 0.0, 500.0, False)
_FIX = [1e9, 5e-20, 10e-9, 0.3e-9, 200.0]
_K, _HD, _Z = (0, 0.5, 8.0, True), (1, -2e-9, 4e-9, False), (2, 0.0, 2e-7, False)


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    assert torch.cuda.is_available()
    return afminv


@pytest.mark.parametrize("force,free,fixed,modes,n,few", [
    ("dmt", [_E, _H, _A0], _FIX, 3, 181, 12), ("dmt", [_E, _H, _A0], _FIX, 3, 193, 33),
    ("dmt", [_A0, _E], _FIX, 1, 191, 5), ("dmt", [_E, _H], _FIX, 2, 192, 64),
    ("dmt_kv", [_E, _ETA], _FIX, 3, 200, 40), ("dmt_kv", [_ETA, _H], _FIX, 5, 192, 31),
    ("hooke", [_HD, _K], [0.0] * 5, 8, 193, 7), ("hooke", [_HD], [3.0, 0, 0, 0, 0], 1, 183, 2),
    ("linear_spring", [(1, 10e-9, 20e-9, False), (0, 2.0, 20.0, False)], [0.0] * 5, 3, 200, 32),
    ("spring_damper", [_K, _HD, _Z], [0.0] * 5, 3, 191, 9),
    ("spring_damper", [_Z, _K], [0, 1e-9, 0, 0, 0], 1, 200, 240)])
def test_both_forms(orc, afm, force, free, fixed, modes, n, few):
    spec = W.get("f2_hooke" if modes == 8 else "c2", force=force, free=free, fixed=fixed, n_modes=modes)
    D = len(free)
    prob = afm.make_problem(spec, n_steps=n)
    x = W.sample_x(D, few, seed=3, lo=0.05, hi=0.95).astype(np.float32)
    U_m = 10e-9 * np.cos(0.02 * np.arange(n))
    U = torch.from_numpy((U_m / NM).astype(np.float32)).cuda()
    xs = torch.from_numpy(x).cuda()
    least = -(-(16 * -(-n // 32) * (modes if modes in (1, 3) else 8) * few) // 256) * 256
    assert afm.adjoint_workspace_size(prob, few) > least
    forms = [afm.adjoint(prob, xs, U),
             afm.adjoint(prob, xs, U, workspace=torch.empty(least, dtype=torch.uint8, device="cuda"))]
    c, pm = orc.make_case(spec), orc.make_pmap(spec)
    U32 = U.double().cpu().numpy() * NM
    for p in range(0, few, 1 + few // 6):
        S_o, g_o = orc.grad_cs(c, pm, x[:, p].astype(np.float64), U32)
        _, H_o, _ = orc.normal_eq(c, pm, x[:, p].astype(np.float64), U32)
        # FP32 over n <= 200 steps: 1e-4, as the tangents over 200 steps, of
        # the largest value that sum 2 r_n du_n/dx can take (Cauchy-Schwarz)
        bound = 1e-4 * 2 * np.sqrt(S_o * np.max(np.diag(H_o))) / NM ** 2
        for S, G in forms:
            assert abs(float(S[p]) - S_o / NM ** 2) <= 2e-5 * S_o / NM ** 2
            got = G[:, p].double().cpu().numpy()
            assert np.max(np.abs(got - np.asarray(g_o) / NM ** 2)) <= bound
