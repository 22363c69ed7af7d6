"""The one-warp time loop of small batches (edges of its record blocks, of its
warps and of the batch size it serves) against the one-thread and paired
kernels of larger batches, bit for bit."""
import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    assert torch.cuda.is_available()
    return afminv


_LAWS = {"linear_spring": [(0, 2.0, 20.0, False), (1, 10e-9, 20e-9, False)]}


@pytest.mark.parametrize("name,modes,n", [
    ("c1", 1, 1), ("c1", 1, 433), ("c2", 1, 64), ("c2", 2, 97), ("c2", 3, 31), ("c2", 3, 32),
    ("c2", 3, 600), ("c2", 4, 70), ("c2", 5, 70), ("c4", 1, 65), ("c4", 3, 300),
    ("linear_spring", 3, 65), ("f2_hooke", 3, 65), ("f2_hooke", 8, 530),
    ("f2_spring_damper", 3, 65), ("f2_spring_damper", 8, 530)])
def test_small_batches_equal_large_ones(afm, name, modes, n):
    if name in _LAWS:
        spec = W.get("c2", force=name, free=_LAWS[name], fixed=[0.0] * 5)
    else:
        spec = W.get(name)
    if spec["model"] != "point_mass":
        spec["n_modes"] = modes
    D = len(spec["free"])
    big = 65537                              # paired kernel where the law has one
    x = W.sample_x(D, big, seed=5)
    prob = afm.make_problem(spec, n_steps=n)
    U = torch.from_numpy((10.0 * np.cos(0.02 * np.arange(n))).astype(np.float32)).cuda()
    _, S_big = afm.forward_batch(prob, torch.from_numpy(x).cuda(), U, want_defl=False)
    mid = 19457                              # one thread per particle
    xm = torch.from_numpy(np.ascontiguousarray(x[:, :mid])).cuda()
    defl_mid, S_mid = afm.forward_batch(prob, xm, U)
    assert torch.equal(S_mid, S_big[:mid])
    for P in (1, 33, 4864, 4865, 9700, 19456):
        xs = torch.from_numpy(np.ascontiguousarray(x[:, :P])).cuda()
        defl, S = afm.forward_batch(prob, xs, U)
        assert torch.equal(S, S_mid[:P]), P
        assert torch.equal(defl, defl_mid[:, :P]), P
        _, S_only = afm.forward_batch(prob, xs, U, want_defl=False)
        assert torch.equal(S_only, S), P
        d_only, _ = afm.forward_batch(prob, xs, None)
        assert torch.equal(d_only, defl), P
