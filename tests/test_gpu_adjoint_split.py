"""The adjoint of few particles on one record (segments at once, joined by
their maps of the adjoint state): S and G of it, and of the one-kernel form
which takes over for larger batches, against the oracle's complex step.  Step
counts around the 32-step segments."""
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
    ("dmt", [_E, _H, _A0], _FIX, 3, 1, 1), ("dmt", [_E, _H, _A0], _FIX, 3, 16, 33),
    ("dmt", [_A0, _E], _FIX, 1, 31, 5), ("dmt", [_E, _H], _FIX, 2, 97, 64),
    ("dmt_kv", [_E, _ETA], _FIX, 3, 32, 40), ("dmt_kv", [_ETA, _H], _FIX, 5, 130, 31),
    ("hooke", [_HD, _K], [0.0] * 5, 8, 33, 7), ("hooke", [_HD], [3.0, 0, 0, 0, 0], 1, 17, 2),
    ("linear_spring", [(1, 10e-9, 20e-9, False), (0, 2.0, 20.0, False)], [0.0] * 5, 3, 47, 32),
    ("spring_damper", [_K, _HD, _Z], [0.0] * 5, 3, 95, 9),
    ("spring_damper", [_Z, _K], [0, 1e-9, 0, 0, 0], 1, 49, 130)])
def test_split_form(orc, afm, force, free, fixed, modes, n, few):
    spec = W.get("f2_hooke" if modes == 8 else "c2", force=force, free=free, fixed=fixed, n_modes=modes)
    D = len(free)
    prob = afm.make_problem(spec, n_steps=n)
    x = W.sample_x(D, few, seed=3, lo=0.05, hi=0.95).astype(np.float32)
    U_m = 10e-9 * np.cos(0.02 * np.arange(n))
    U = torch.from_numpy((U_m / NM).astype(np.float32)).cuda()
    xs = torch.from_numpy(x).cuda()
    S, G = afm.adjoint(prob, xs, U)
    if n >= 16:    # the same points in a batch past the split form's bounds
        reps = (2 ** 26 // (5 * n)) // few + 2
        Sg, Gg = afm.adjoint(prob, xs.repeat(1, reps), U)
        torch.testing.assert_close(Sg[:few], S, rtol=2e-5, atol=0)
        assert torch.equal(Sg[-few:], Sg[:few])
        Gg = Gg[:, :few].double().cpu().numpy()
    G = G.double().cpu().numpy()
    c, pm = orc.make_case(spec), orc.make_pmap(spec)
    U32 = U.double().cpu().numpy() * NM
    for p in range(0, few, 1 + few // 6):
        S_o, g_o = orc.grad_cs(c, pm, x[:, p].astype(np.float64), U32)
        _, H_o, _ = orc.normal_eq(c, pm, x[:, p].astype(np.float64), U32)
        assert abs(float(S[p]) - S_o / NM ** 2) <= 2e-5 * S_o / NM ** 2
        # FP32 over n <= 130 steps: 1e-4, as the tangents over 200 steps, of
        # the largest value that sum 2 r_n du_n/dx can take (Cauchy-Schwarz)
        bound = 1e-4 * 2 * np.sqrt(S_o * np.max(np.diag(H_o))) / NM ** 2
        assert np.max(np.abs(G[:, p] - np.asarray(g_o) / NM ** 2)) <= bound
        if n >= 16:
            assert np.max(np.abs(Gg[:, p] - np.asarray(g_o) / NM ** 2)) <= bound
