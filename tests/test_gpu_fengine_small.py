"""The general F-engine for K <= 256 (8 to 32 lanes per frame): edges of its
32-frame blocks, every output type it serves, against the oracle."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


def _norm(V, R, N):
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    d = np.abs(V - R)
    return float(np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)))


# FP32: the framework's bound.  FP16 and FP8 round every value once, by at most
# 2^-11 and 2^-4 of it: twice that per product, second order, and values below
# the normal range (FP16 at an address the wide loads cannot take)
@pytest.mark.parametrize("dtype,shift,bound", [("fp32", 0, 1e-5), ("fp32_simt", 0, 1e-5), ("fp32", 1, 1e-5),
                                               ("fp16", 1, 2.25 * 2.0 ** -11), ("fp8", 0, 2.25 * 2.0 ** -4)])
@pytest.mark.parametrize("K,N,S", [(16, 3, 1), (16, 2, 33), (32, 1, 31), (32, 5, 160), (64, 2, 32), (64, 3, 97),
                                   (128, 1, 129), (128, 4, 65), (256, 2, 1), (256, 3, 127)])
def test_against_oracle(lib, K, N, S, dtype, shift, bound):
    torch = pytest.importorskip("torch")
    packed, _ = synth.make_samples(N, S * K, K, seed=31 + K + S)
    g, t = synth.gains_delays(N, 3)
    g, t = g.astype(np.complex64), t.astype(np.float32)
    R, _ = oracle.correlate(packed, N, K, gains=g, delays=t)
    flat = torch.from_numpy(packed.reshape(-1))
    buf = torch.zeros(flat.numel() + 64, dtype=torch.uint8, device="cuda")
    x = buf[shift:shift + flat.numel()]
    x.copy_(flat)
    torch.cuda.synchronize()
    with lib.Correlator(N, K, dtype) as c:
        c.set_corrections(g, t)
        if dtype in ("fp16", "fp8"):
            lib.corr_set_scales(c.h, np.full((N, K // 2), (64.0 if dtype == "fp16" else 16.0) / np.sqrt(2.0 * K), np.float32))
        lib.corr_set_stable(c.h, True)
        c.push(x, S * K)
        V, n = c.dump(fp64=True)
        spec = torch.empty((N, S, K // 2), dtype=torch.complex64, device="cuda")
        lib.corr_debug_spectra(c.h, x.data_ptr(), S * K, spec.data_ptr())
    assert n == S and _norm(V, R, N) <= bound
    Y = np.sum(np.abs(spec.cpu().numpy().astype(np.complex128)) ** 2, axis=1)
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    assert np.all(np.abs(Y - R[autos].real) <= 1e-5 * np.maximum(R[autos].real, 1e-3 * Y.mean()))
