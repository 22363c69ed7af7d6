"""The finite-element kernel's lane layouts (chosen by the particle count):
against the oracle at odd sizes on either side of each change of layout, and
against each other."""
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


@pytest.mark.parametrize("force,n_elem,n", [("dmt", 32, 300), ("dmt", 5, 513), ("hooke", 32, 200),
                                            ("linear_spring", 3, 200)])
def test_layouts_agree(orc, afm, force, n_elem, n):
    over = dict(n_elem=n_elem)
    if force != "dmt":
        over.update(force=force, fixed=[0.0] * 5,
                    free=[(0, 0.5, 8.0, True), (1, -2e-9, 14e-9, False)])
    spec = W.get("c5", **over)
    D = len(spec["free"])
    x = W.sample_x(D, 7300, seed=6, lo=0.05, hi=0.95)
    prob = afm.make_problem(spec, n_steps=n)
    U = torch.from_numpy((15.0 * np.cos(0.0123 * np.arange(n))).astype(np.float32)).cuda()
    base = None
    for P in (1, 2431, 2433, 4865, 7297):           # 8, 8, 4, 8, 4 lanes per particle
        defl, S = afm.forward_batch(prob, torch.from_numpy(np.ascontiguousarray(x[:, :P])).cuda(), U)
        d, s = defl[:, :1].double(), S[:1].double()
        if base is None:
            base = (d, s)
        # FP32 trajectories that differ in summation order only: as the
        # parity bounds, 1e-5 of the deflection and 1e-4 of the misfit
        assert float((d - base[0]).abs().max()) <= 1e-5 * float(base[0].abs().max()), P
        assert float(((s - base[1]) / base[1]).abs().max()) <= 1e-4, P
        last = P - 1
        c, pm = orc.make_case(spec), orc.make_pmap(spec)
        ref = orc.fe_forward(c, orc.map_x(pm, x[:, last].astype(np.float64)), n) / NM
        got = defl[:, last].double().cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), P
