"""A finite-element particle's result must not depend on how many particles
share its launch: the two lane layouts (4 or 8 lanes per particle, chosen by
the particle count) give the same bits, and a swarm split into slices is the
whole swarm bit for bit where the slices take another layout than the whole."""
import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W
from common import oracle_record
from test_gpu_split import _split_run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    assert torch.cuda.is_available()
    return afminv


@pytest.mark.parametrize("force,n_elem,n", [("dmt", 32, 300), ("dmt", 5, 513), ("hooke", 32, 200),
                                            ("linear_spring", 3, 200)])
def test_layouts_give_the_same_bits(afm, force, n_elem, n):
    over = dict(n_elem=n_elem)
    if force != "dmt":
        over.update(force=force, fixed=[0.0] * 5,
                    free=[(0, 0.5, 8.0, True), (1, -2e-9, 14e-9, False)])
    spec = W.get("c5", **over)
    x = torch.from_numpy(W.sample_x(len(spec["free"]), 7300, seed=6, lo=0.05, hi=0.95)).cuda()
    prob = afm.make_problem(spec, n_steps=n)
    U = torch.from_numpy((15.0 * np.cos(0.0123 * np.arange(n))).astype(np.float32)).cuda()
    base = None
    for P in (2432, 2433, 4865, 7297):           # 8, 4, 8, 4 lanes per particle
        defl, S = afm.forward_batch(prob, x[:, :P].contiguous(), U)
        if base is None:
            base = (defl, S)
        assert torch.equal(defl[:, :2432], base[0]), P
        assert torch.equal(S[:2432], base[1]), P


def test_split_swarm_equals_one_swarm(orc, afm):
    spec = W.get("c5", cycles=2, P=2433, iters=4)      # whole: 4 lanes; slices: 8
    U32, _, _ = oracle_record(orc, spec)
    U = torch.from_numpy(U32).cuda()
    prob = afm.make_problem(spec)
    cfg = afm.make_pso(spec)
    keys, pos = _split_run(afm, prob, U, cfg, 2)
    res, hist = afm.invert(prob, U, cfg)
    torch.cuda.synchronize()
    r = afm.decode_result(res)
    assert r["winner"] == keys[-1] & 0xFFFFFFFF
    np.testing.assert_array_equal(r["x"][:len(spec["free"])], pos.double().cpu().numpy())
    S_hist = [np.uint32(k >> 32).view(np.float32) for k in keys]
    np.testing.assert_array_equal(hist.cpu().numpy(), np.array(S_hist, dtype=np.float32))
