"""Coarse delays: the direct kernel (aligned input, whole 16-byte chunks)
against the general one, which takes the same samples one byte past an aligned
address, and the oracle."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


# frames around the CTAs' 1024 chunks (K / 32 per frame); K = 16 has no whole
# chunks and takes the general kernel either way
@pytest.mark.parametrize("K,S", [(16, 70), (32, 1023), (32, 1025), (128, 257), (512, 1), (512, 65), (4096, 9)])
def test_routes_agree(lib, K, S):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(K + S)
    N = 9
    D = np.concatenate([[0, K, 1, 2, K - 1], rng.integers(0, K + 1, N - 5)]).astype(np.int32)
    packed, _ = synth.make_samples(N, 2 * S * K, K, seed=61 + K)
    R, _ = oracle.correlate(packed, N, K, sample_delays=D)
    flat = torch.from_numpy(packed.reshape(-1))
    half = flat.numel() // 2
    out = []
    for shift in (0, 1):
        buf = torch.zeros(flat.numel() + 64, dtype=torch.uint8, device="cuda")
        buf[shift:shift + flat.numel()].copy_(flat)
        torch.cuda.synchronize()
        with lib.Correlator(N, K, "fp32_simt") as c:
            lib.corr_set_sample_delays(c.h, D)
            for p in (0, 1):                    # the second push starts from the first one's history
                c.push(buf[shift + p * half:shift + (p + 1) * half], S * K)
            V, n = c.dump(fp64=True)
        assert n == 2 * S
        out.append(V)
    # the delayed samples are the same bytes, in the same buffer: the same V
    assert np.array_equal(out[0], out[1])
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    d = np.abs(out[0] - R)
    assert np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)) <= 1e-5
