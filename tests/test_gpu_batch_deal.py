"""Batches in which every pixel has a block of its own (dealt to the SMs)
against batches whose blocks pull pixels from a queue: the same results for
every pixel, at pixel counts around whole layers of SMs."""
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


@pytest.mark.parametrize("kp,P,force", [(1, 64, "dmt"), (2, 64, "dmt"), (4, 90, "dmt"), (1, 33, "dmt_kv")])
def test_dealt_and_queued(afm, kp, P, force):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = 32 * sms + 5                       # more than the blocks an SM holds
    rng = np.random.default_rng(kp)
    n_i = rng.integers(1, 90, many)
    off = np.concatenate([[0], np.cumsum(n_i)]).astype(np.int64)
    spec = W.get("c3" if force == "dmt" else "c4", P=P, iters=2)
    prob = afm.make_problem(spec, n_steps=90)
    U = torch.from_numpy((10 * np.cos(0.06 * np.arange(off[-1]))).astype(np.float32)).cuda()
    o = torch.from_numpy(off).cuda()
    cfg = afm.make_pso(spec)
    ref, _ = afm.invert_batch(prob, U, o, cfg, particles_per_thread=kp)
    for n in (1, 2, sms - 1, sms, sms + 1, 2 * sms, 2 * sms + 1, 3 * sms - 1, 4 * sms + 7):
        res, _ = afm.invert_batch(prob, U, o[:n + 1].contiguous(), cfg, particles_per_thread=kp)
        assert torch.equal(res, ref[:n]), n
