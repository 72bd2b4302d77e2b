"""FP16 and FP8 spectra of the tensor-core first stage, for every K that it
serves: strongly correlated antennas, so that every cross-correlation counts,
gains and delays, against the oracle's spectra rounded to the type, so that what
is left is FP32 arithmetic and the values that it rounds the other way."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


def _samples(N, K, S, seed):
    """4-bit samples, 90% of the power common, delayed by up to 3 samples."""
    rng = np.random.default_rng(seed)
    c = 2.0 * rng.standard_normal(S * K + 4)
    x = np.empty((N, S * K))
    for i in range(N):
        d = int(rng.integers(0, 4))
        x[i] = c[4 - d:4 - d + S * K] + 0.7 * rng.standard_normal(S * K)
    q = np.clip(np.rint(x), -8, 7).astype(np.int8).reshape(N, S, K)
    b = (q[..., 0::2] & 15) | ((q[..., 1::2] & 15) << 4)
    return np.ascontiguousarray(b.astype(np.uint8).transpose(1, 0, 2))


def _rounded(torch, packed, N, K, gains, delays, scale, dt):
    """Visibilities of the oracle's spectra, corrected, scaled and rounded to dt."""
    Y = oracle.spectra(oracle.unpack(packed, N, K), K)
    if gains is not None:
        Y = Y * oracle.correction_factors(K, gains.astype(np.complex128), delays.astype(np.float64))[:, None, :]
    parts = [torch.from_numpy(p.astype(np.float32) * scale).to(dt).to(torch.float64).numpy() for p in (Y.real, Y.imag)]
    return oracle.visibilities(parts[0] + 1j * parts[1]) / np.float64(scale) ** 2


# S well past the first frames of an FP8 integration, which take other kernels
# (N = 3: 896, N = 9: 1408)
@pytest.mark.parametrize("K,N,S", [(16, 3, 3000), (16, 9, 4001), (32, 3, 3000), (32, 9, 4001), (64, 3, 2400),
                                   (128, 3, 2400), (256, 3, 2400), (512, 3, 2400), (512, 9, 3200), (1024, 3, 2400),
                                   (2048, 3, 1800)])
@pytest.mark.parametrize("dtype,bits", [("fp16", 11), ("fp8", 4)])
@pytest.mark.parametrize("corrected", [False, True])
def test_rounded_spectra(lib, K, N, S, dtype, bits, corrected):
    torch = pytest.importorskip("torch")
    packed = _samples(N, K, S, 5 + K + N)
    g = t = None
    if corrected:
        g, t = synth.gains_delays(N, 5)
        g, t = g.astype(np.complex64), t.astype(np.float32)
    scale = np.float32((64.0 if dtype == "fp16" else 16.0) / np.sqrt(2.0 * K))
    V0 = _rounded(torch, packed, N, K, g, t, scale, torch.float16 if dtype == "fp16" else torch.float8_e4m3fn)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    torch.cuda.synchronize()
    with lib.Correlator(N, K, dtype) as c:
        if corrected:
            c.set_corrections(g, t)
        lib.corr_set_scales(c.h, np.full((N, K // 2), scale))
        c.push(x, S * K)
        V, n = c.dump(fp64=True)
    assert n == S
    A = np.abs(V0[[oracle.baseline_index(i, i, N) for i in range(N)]])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    cross = np.abs(V0 / nrm)[ii != jj]
    assert np.median(cross) > 0.5                    # a lost phase would show
    d = np.abs(V - V0) / nrm
    # FP32 sums: 1e-5.  Spectra within 5e-6 of their rms (the bound of the
    # spectra's own test) fall the other way at one value in u / 1e-5, u = 2^-bits
    # being the least spacing of a value's neighbours; each moves a value by 2 u of
    # it at most, the sums of an antenna and channel by 4 u sqrt(p / S) rms, and two
    # of them that meet in one sum, at values of 8 times the mean power, by 32 u / S
    u = 2.0 ** -bits
    assert np.sqrt(np.mean(d ** 2)) <= 1e-5 + 4.0 * u * np.sqrt(1e-5 / u / S)
    assert d.max() <= 1e-5 + 32.0 * u / S
