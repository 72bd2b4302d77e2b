"""A bounded wait that runs out in a pair of CTAs (N > 64): the launch ends with
everything under way waited for in both CTAs, the host reports CORR_ETIMEOUT,
and the same handle then correlates correctly."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


# FP32: the framework's bound; FP16 and FP8 round every value once, by at most
# 2^-11 and 2^-4 of it (twice that per product, and second order)
@pytest.mark.parametrize("dtype,bound", [("fp32", 1e-5), ("fp16", 2.25 * 2.0 ** -11), ("fp8", 2.25 * 2.0 ** -4)])
# one stage of a lone group; several stages; groups on and off the diagonal
@pytest.mark.parametrize("K,N,S", [(16, 66, 32), (64, 66, 700), (16, 200, 300)])
def test_pair_wait_is_reported_and_recovered(lib, dtype, bound, K, N, S):
    torch = pytest.importorskip("torch")
    packed, _ = synth.make_samples(N, S * K, K, seed=11020148 + N + S)
    R, _ = oracle.correlate(packed, N, K)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    torch.cuda.synchronize()
    with lib.Correlator(N, K, dtype) as c:
        for _ in range(2):
            lib.corr_test_fault(c.h, 1, 0.02)
            c.push(x, S * K)
            with pytest.raises(lib.CorrError) as ei:
                c.dump(fp64=True)
            assert ei.value.code == lib.CORR_ETIMEOUT
        c.push(x, S * K)
        V, n = c.dump(fp64=True)
    assert n == S
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    d = np.abs(V - R)
    assert np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)) <= bound
