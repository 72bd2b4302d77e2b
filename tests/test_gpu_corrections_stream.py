"""Gains and delays made by work queued on the handle's stream, or on the legacy
default stream, are the ones applied, however late that work runs."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu

N, K, S = 5, 512, 40
LATE = 1 << 27                       # clocks of a kernel in front of the values (~70 ms)


@pytest.fixture(scope="module")
def data():
    torch = pytest.importorskip("torch")
    packed, _ = synth.make_samples(N, S * K, K, seed=11020148 + 9)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    sets = []
    for seed in (3, 4):
        g, t = synth.gains_delays(N, seed)
        g, t = g.astype(np.complex64), t.astype(np.float32)
        R, _ = oracle.correlate(packed, N, K, gains=g.astype(np.complex128), delays=t.astype(np.float64))
        sets.append((torch.from_numpy(g).cuda(), torch.from_numpy(t).cuda(), R))
    torch.cuda.synchronize()
    return torch, x, sets


def _err(V, R):
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    return float(np.max(np.abs(V - R) / np.sqrt(A[ii] * A[jj])))


def test_binding_on_a_side_stream(lib, data):
    torch, x, sets = data
    from paper_1102_0148_gb300 import autograd
    s = torch.cuda.Stream()
    g = torch.ones(N, dtype=torch.complex64, device="cuda")
    t = torch.zeros(N, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    with lib.Correlator(N, K, "fp32") as c, torch.cuda.stream(s):
        for g0, t0, R in sets:               # the second call finds its stream set
            torch.cuda._sleep(LATE)
            g.copy_(g0)
            t.copy_(t0)
            V = autograd.visibilities(g, t, x, c)
            assert _err(V.cpu().numpy(), R) <= 1e-5
        torch.cuda._sleep(LATE)              # a cast made on the stream
        V = autograd.visibilities(sets[0][0].to(torch.complex128), sets[0][1].double(), x, c)
        assert _err(V.cpu().numpy(), sets[0][2]) <= 1e-5


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("legacy", [False, True])
def test_set_corrections_follows_its_producers(lib, data, legacy, pinned):
    torch, x, sets = data
    own = torch.cuda.Stream()
    with lib.Correlator(N, K, "fp32", stream=own.cuda_stream) as c:
        for g0, t0, R in sets:
            if pinned:
                g = torch.ones(N, dtype=torch.complex64).pin_memory()
                t = torch.zeros(N).pin_memory()
            else:
                g, t = torch.ones_like(g0), torch.zeros_like(t0)
            torch.cuda.synchronize()
            with torch.cuda.stream(torch.cuda.default_stream() if legacy else own):
                torch.cuda._sleep(LATE)
                g.copy_(g0, non_blocking=True)
                t.copy_(t0, non_blocking=True)
            lib.corr_set_corrections(c.h, g, t)
            g.zero_()                        # the values were copied before the return
            torch.cuda.synchronize()
            c.push(x, S * K)
            V, _ = c.dump(fp64=True)
            assert _err(V, R) <= 1e-5
