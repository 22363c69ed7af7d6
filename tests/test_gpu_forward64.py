"""The FP64 forward solve's two layouts (several lanes per candidate for few
candidates, one thread each for many) against each other and the oracle."""
import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W
from common import NM

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    assert torch.cuda.is_available()
    return afminv


@pytest.mark.parametrize("name,modes,n", [
    ("c1", 1, 401), ("c2", 1, 300), ("c2", 2, 257), ("c2", 3, 1), ("c2", 3, 515), ("c2", 5, 300),
    ("c4", 1, 260), ("c4", 3, 300), ("f2_hooke", 8, 520), ("f2_spring_damper", 8, 520),
    ("f2_spring_damper", 3, 600)])
def test_lane_layouts_agree_with_each_other_and_the_oracle(orc, afm, name, modes, n):
    spec = W.get(name)
    if spec["model"] != "point_mass":
        spec["n_modes"] = modes
    D = len(spec["free"])
    lanes = 2 if modes == 1 else 4 if modes == 3 else 8
    P = 152 * 4 * (32 // lanes) + 1          # one warp too many for the lane layout
    x = W.sample_x(D, P, seed=3).astype(np.float64)
    prob = afm.make_problem(spec, n_steps=n)
    U = torch.from_numpy(10.0 * np.cos(0.02 * np.arange(n))).cuda()
    many, S_many = afm.forward_batch_f64(prob, torch.from_numpy(x).cuda(), U)
    few = 13                                  # an odd last warp
    xs = torch.from_numpy(np.ascontiguousarray(x[:, :few])).cuda()
    got, S = afm.forward_batch_f64(prob, xs, U)
    # rounding of n <= 600 compensated steps, amplified at contact: < 1e-11
    scale = float(many.abs().max())
    assert float((got - many[:, :few]).abs().max()) <= 1e-11 * scale
    assert float(((S - S_many[:few]) / S).abs().max()) <= 1e-10
    c, pm = orc.make_case(spec), orc.make_pmap(spec)
    for p in (0, 7, 12):
        ref = orc.forward(c, orc.map_x(pm, x[:, p]), n) / NM
        assert np.max(np.abs(got[:, p].cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
