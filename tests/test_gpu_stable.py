"""corr_set_stable: the kernels and cuts it selects against the default ones
and the oracle, and its use by the autograd binding's forward pass."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


# a generic and a radix-16 FFT in place of the tensor-core first stage; one
# block of antennas and two, whose passes the two deals cut differently
@pytest.mark.parametrize("K,N,S", [(64, 5, 200), (128, 66, 1030), (256, 9, 96), (2048, 3, 65), (512, 66, 700)])
@pytest.mark.parametrize("dtype", ["fp32", "fp32_simt"])
def test_stable_and_default_routes(lib, K, N, S, dtype):
    torch = pytest.importorskip("torch")
    from paper_1102_0148_gb300 import autograd
    packed, _ = synth.make_samples(N, S * K, K, seed=7 + K)
    g, t = synth.gains_delays(N, 3)
    g, t = g.astype(np.complex64), t.astype(np.float32)
    R, _ = oracle.correlate(packed, N, K, gains=g, delays=t)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    torch.cuda.synchronize()
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    got = {}
    with lib.Correlator(N, K, dtype) as c:
        c.set_corrections(g, t)
        for on in (True, False):
            lib.corr_set_stable(c.h, on)
            c.push(x, S * K)
            got[on], n = c.dump(fp64=True)
            assert n == S
            assert np.max(np.abs(got[on] - R) / nrm) <= 1e-5
        if dtype == "fp32":
            V = autograd.visibilities(torch.from_numpy(g).cuda(), torch.from_numpy(t).cuda(), x, c)
            assert np.array_equal(V.cpu().numpy(), got[True])
            c.push(x, S * K)                     # the binding left the default on
            again, _ = c.dump(fp64=True)
            assert np.array_equal(again, got[False])
