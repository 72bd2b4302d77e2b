"""FP8 F-engine on both sides of the line between short integrations (FP32 FFT
kernels) and longer ones (tensor-core first stage): the same samples through
the general kernel, at an address the wide loads cannot use."""

import pytest
import numpy as np

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


# first S on the tensor-core side at N = 1, 2, 3, 5 (2 S^2 / N + S >= 420000):
# 458, 648, 793, 1024; each with the pass before it and a ragged longer one
@pytest.mark.parametrize("K", [16, 32, 64, 128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("N,S", [(1, 457), (1, 459), (2, 647), (2, 649), (3, 801), (5, 1023), (5, 1185)])
def test_fp8_both_sides_of_the_line(lib, K, N, S):
    torch = pytest.importorskip("torch")
    packed, _ = synth.make_samples(N, S * K, K, seed=8 + K + S)
    flat = torch.from_numpy(packed.reshape(-1))
    V = []
    for shift in (0, 1):
        buf = torch.zeros(flat.numel() + 64, dtype=torch.uint8, device="cuda")
        buf[shift:shift + flat.numel()].copy_(flat)
        torch.cuda.synchronize()
        with lib.Correlator(N, K, "fp8") as c:
            if V:
                lib.corr_set_scales(c.h, used)
            c.push(buf[shift:shift + flat.numel()], S * K)
            v, n = c.dump(fp64=True)
            used = lib.corr_get_scales(c.h) if not V else used
        assert n == S
        V.append(v)
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(V[1][autos])
    ii, jj = np.triu_indices(N)
    # each route rounds every value once, by at most 2^-4 of it: each is within
    # twice that of the unrounded one, and the two within four times it
    # (normalised by autocorrelations that are themselves so far off)
    assert np.all(np.abs(V[0] - V[1]) <= 4.5 * 2.0 ** -4 / (1 - 2.25 * 2.0 ** -4) * np.sqrt(A[ii] * A[jj]))
