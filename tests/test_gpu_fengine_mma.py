"""F-engine kernels with the tensor-core first stage (K = 16 .. 2048): tile and
group edges, every output type, and the same samples through the general
kernel, which takes them at an address the wide loads cannot use."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu

# antennas around the groups a CTA takes (16 K-samples' worth: 2 at K = 256 ..
# 16 at K = 32) and frames around its 32-frame blocks and the 128-frame padding
SHAPES = [(16, 1, 1), (16, 17, 33), (16, 65, 160), (32, 16, 31), (32, 33, 129), (64, 1, 128),
          (64, 9, 127), (128, 5, 97), (128, 65, 40), (256, 2, 32), (256, 3, 65), (512, 1, 33),
          (512, 66, 130), (1024, 3, 31), (1024, 65, 33), (2048, 1, 1), (2048, 5, 161)]


def _dump(lib, torch, packed, N, K, dtype, shift=0, gains=None, delays=None, scales=None):
    """V [P][C] and n of one push of `packed` placed `shift` bytes past an
    aligned address."""
    flat = torch.from_numpy(packed.reshape(-1))
    buf = torch.zeros(flat.numel() + 64, dtype=torch.uint8, device="cuda")
    x = buf[shift:shift + flat.numel()]
    x.copy_(flat)
    torch.cuda.synchronize()
    with lib.Correlator(N, K, dtype) as c:
        if gains is not None or delays is not None:
            c.set_corrections(gains, delays)
        if scales is not None:
            lib.corr_set_scales(c.h, scales)
        c.push(x, flat.numel() * 2 // N)
        V, n = c.dump(fp64=True)
        used = lib.corr_get_scales(c.h) if dtype in (lib.CORR_FP16, lib.CORR_FP8E4M3) else None
    return V, n, used


def _norm(V, R, N):
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    d = np.abs(V - R)
    nrm = np.sqrt(A[ii] * A[jj])
    # (a channel without power, DC of a single short frame: V must be R)
    return float(np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)))


@pytest.fixture(scope="module")
def lib():
    return pytest.importorskip("paper_1102_0148_gb300.corr")


@pytest.fixture(scope="module")
def torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("K,N,S", SHAPES)
@pytest.mark.parametrize("corrected", [False, True])
def test_fp32_outputs_against_oracle(lib, torch, K, N, S, corrected):
    packed, _ = synth.make_samples(N, S * K, K, seed=11020148 + K + N)
    g = t = None
    if corrected:
        g, t = synth.gains_delays(N, 3)
        g, t = g.astype(np.complex64), t.astype(np.float32)
    R, _ = oracle.correlate(packed, N, K, gains=g, delays=t)
    for dtype in (lib.CORR_FP32, lib.CORR_FP32_SIMT):
        V, n, _ = _dump(lib, torch, packed, N, K, dtype, gains=g, delays=t)
        assert n == S
        assert _norm(V, R, N) <= 1e-5


# Each route rounds every scaled value once: a relative error of at most 2^-11
# (FP16) or 2^-4 (E4M3) of the value, so by Cauchy-Schwarz each visibility is
# within twice that (plus second order) of the unrounded one and the two routes
# within four times it, normalised.  Values below the formats' normal range (a
# thousandth of the rms and less) add less than the slack.
@pytest.mark.parametrize("K,N,S", SHAPES)
@pytest.mark.parametrize("dtype,bound", [("fp16", 4.5 * 2.0 ** -11), ("fp8", 4.5 * 2.0 ** -4)])
def test_narrow_outputs_against_general_kernel(lib, torch, K, N, S, dtype, bound):
    packed, _ = synth.make_samples(N, S * K, K, seed=11020148 + 2 * K + N)
    g, t = synth.gains_delays(N, 5)
    g, t = g.astype(np.complex64), t.astype(np.float32)
    d = lib.DTYPES[dtype]
    scales = np.full((N, K // 2), 64.0 / np.sqrt(2.0 * K) if dtype == "fp16" else 16.0 / np.sqrt(2.0 * K),
                     np.float32)
    V, n, _ = _dump(lib, torch, packed, N, K, d, gains=g, delays=t, scales=scales)
    G, m, _ = _dump(lib, torch, packed, N, K, d, shift=1, gains=g, delays=t, scales=scales)
    assert n == m == S
    assert _norm(V, G, N) <= bound


@pytest.mark.parametrize("K", [16, 64, 256, 512, 1024, 2048])
def test_silent_antenna_is_exactly_zero(lib, torch, K):
    """All-zero samples give exactly zero spectra (their offset of 8 cancels in
    exact arithmetic), so a silent antenna keeps scale 1."""
    N, S = 3, 40
    packed, _ = synth.make_samples(N, S * K, K, seed=7)
    packed = packed.copy()
    packed[:, 1, :] = 0
    for dtype in (lib.CORR_FP32, lib.CORR_FP32_SIMT, lib.CORR_FP16, lib.CORR_FP8E4M3):
        V, _, used = _dump(lib, torch, packed, N, K, dtype)
        for i, j in ((0, 1), (1, 1), (1, 2)):
            assert np.all(V[oracle.baseline_index(i, j, N)] == 0)
        if used is not None:
            assert np.all(used[1] == 1.0)
