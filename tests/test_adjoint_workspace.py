"""The workspace of afm_adjoint: its size does not fall as the batch or the
record grows, and a buffer that is larger or only holds the checkpoints is
taken."""
import ctypes as C

import numpy as np
import pytest

from paper_1109_0334_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def afm():
    from paper_1109_0334_gb300 import build
    build.build()
    from paper_1109_0334_gb300 import afminv
    return afminv


def _checkpoints(n, modes, P):
    return -(-(16 * -(-n // 32) * modes * P) // 256) * 256


@pytest.mark.parametrize("load,modes", [("c1", 1), ("c2", 1), ("c2", 2), ("c2", 3), ("c4", 3),
                                        ("f2_spring_damper", 8)])
def test_size_is_monotone(afm, load, modes):
    M = modes if modes in (1, 3) else 8
    last = {}
    for n in (1, 31, 32, 200, 255, 256, 257, 512, 1280, 2560, 5120, 25600, 400000):
        probs = afm.make_problem(W.get(load, n_modes=modes), n_steps=n)
        prev = 0
        for P in (1, 2, 300, 1000, 2222, 2223, 4500, 5000, 5001, 9999, 10001, 30000):
            size = afm.adjoint_workspace_size(probs, P)
            assert size >= max(prev, last.get(P, 0), _checkpoints(n, M, P)), (n, P)
            assert size <= _checkpoints(n, M, P) + 2 ** 28 + 256, (n, P)
            prev = last[P] = size


@pytest.mark.parametrize("load,modes", [("c1", 1), ("c2", 3), ("f2_hooke", 8)])
def test_short_records_take_the_checkpoints_alone(afm, load, modes):
    """The segments at once are slower than the one kernel below ~110 steps
    (0.2 to 0.9 of its speed at 64), whatever the batch."""
    for n in (1, 32, 64, 110):
        prob = afm.make_problem(W.get(load, n_modes=modes), n_steps=n)
        for P in (1, 700, 10000):
            assert afm.adjoint_workspace_size(prob, P) == _checkpoints(n, modes, P), (n, P)


@pytest.mark.gpu
@pytest.mark.parametrize("load,modes,n", [("c2", 3, 640), ("c1", 1, 640), ("c4", 2, 300)])
def test_buffers_of_other_sizes_are_taken(afm, load, modes, n):
    spec = W.get(load, n_modes=modes)
    D, P = len(spec["free"]), 700
    prob = afm.make_problem(spec, n_steps=n)
    x = torch.from_numpy(W.sample_x(D, P, seed=2, lo=0.1, hi=0.9)).cuda()
    U = torch.from_numpy((15.0 * np.cos(0.0245 * np.arange(n))).astype(np.float32)).cuda()

    def call(nbytes, x):
        P = x.shape[1]
        ws = torch.full((nbytes + 256,), 0x5a, dtype=torch.uint8, device="cuda")
        S = torch.empty(P, dtype=torch.float32, device="cuda")
        G = torch.empty((D, P), dtype=torch.float32, device="cuda")
        afm._check(afm.lib().afm_adjoint(afm.context(), C.byref(prob), x.data_ptr(), P,
                                         U.data_ptr(), S.data_ptr(), G.data_ptr(), ws.data_ptr(),
                                         C.c_size_t(nbytes), afm._stream()))
        torch.cuda.synchronize()
        assert bool((ws[nbytes:] == 0x5a).all())          # nothing past the size given
        return S, G

    S, G = call(afm.adjoint_workspace_size(prob, P), x)
    for larger in (5001, 10001, 30000):                   # a larger batch's buffer: the same form
        S2, G2 = call(afm.adjoint_workspace_size(prob, larger), x)
        assert torch.equal(S2, S) and torch.equal(G2, G), larger
    least = _checkpoints(n, modes if modes in (1, 3) else 8, P)
    S1, G1 = call(least, x)                               # the checkpoints alone: one kernel,
    reps = 30000 // P + 1                                 # as in a batch past the other form
    Sb, Gb = call(afm.adjoint_workspace_size(prob, reps * P), x.repeat(1, reps))
    assert torch.equal(S1, Sb[:P]) and torch.equal(G1, Gb[:, :P])
    with pytest.raises(afm.AfmError) as ei:
        call(least - 256, x)
    assert ei.value.status == afm.ERR_INVALID_ARG
