"""The next integration's pre-cast scales, made by the dump: the power of two
nearest to target / sqrt(P / 2) of the dumped autocorrelations, also where the
power is a power of two (the nearest exponent is a tie or exact) or zero."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,target", [("fp16", 64.0), ("fp8", 16.0)])
@pytest.mark.parametrize("N,K,S", [(1, 16, 33), (44, 512, 64), (65, 64, 130), (130, 256, 40)])
def test_scales_from_dumped_autos(lib, dtype, target, N, K, S):
    torch = pytest.importorskip("torch")
    packed, _ = synth.make_samples(N, S * K, K, seed=21 + N + K)
    packed = packed.copy()
    packed[:, 0, :] = 0x44              # constant 4: power (4 K)^2 in DC, none elsewhere
    if N > 2:
        packed[:, 2, :] = 0
    with lib.Correlator(N, K, dtype) as c:
        c.push(torch.from_numpy(packed.reshape(-1)).cuda(), S * K)
        V, n = c.dump(fp64=True)
        got = lib.corr_get_scales(c.h)
    assert n == S
    P = np.stack([V[oracle.baseline_index(i, i, N)].real for i in range(N)]) / S
    with np.errstate(divide="ignore"):
        e = np.log2(target) - 0.5 * np.log2(P * 0.5)
    assert np.all(got[P == 0] == 1.0)
    m = P > 0
    x = np.log2(got[m].astype(np.float64))
    assert np.all(x == np.rint(x))
    # nearest: at most half an exponent away (ties, and the 2^-60 rounding of
    # the logarithms next to them, may go either way)
    assert np.max(np.abs(x - np.clip(e[m], -60, 60))) <= 0.5 + 1e-9
