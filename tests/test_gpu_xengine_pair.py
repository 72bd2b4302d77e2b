"""Tensor-core X-engine at N > 64 (pairs of CTAs sharing their MMAs): antenna
counts around the edges of blocks, block pairs and 64-column steps, passes of
one k-tile and of several windows, items whole and cut between pairs."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(16, 65, 33), (16, 96, 300), (32, 97, 64), (16, 127, 128), (16, 128, 1), (16, 129, 257),
          (16, 160, 130), (16, 161, 640), (16, 191, 31), (16, 192, 200), (16, 193, 96),
          (64, 256, 150), (16, 257, 2100), (16, 300, 128)]

# FP32 mode: the framework's bound.  FP16 and FP8 round every value once, by at
# most 2^-11 and 2^-4 of it: by Cauchy-Schwarz twice that, normalised, plus
# second order and values below the normal range.
BOUNDS = {"fp32": 1e-5, "fp16": 2.25 * 2.0 ** -11, "fp8": 2.25 * 2.0 ** -4}


@pytest.fixture(scope="module")
def data():
    memo = {}

    def get(K, N, S):
        if (K, N, S) not in memo:
            packed, _ = synth.make_samples(N, S * K, K, seed=11020148 + K + N)
            memo[K, N, S] = packed, oracle.correlate(packed, N, K)[0]
        return memo[K, N, S]
    return get


@pytest.mark.parametrize("K,N,S", SHAPES)
@pytest.mark.parametrize("dtype", ["fp32", "fp16", "fp8"])
@pytest.mark.parametrize("split", [0, 3])
def test_antenna_counts_against_oracle(data, K, N, S, dtype, split):
    lib = pytest.importorskip("paper_1102_0148_gb300.corr")
    torch = pytest.importorskip("torch")
    packed, R = data(K, N, S)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    torch.cuda.synchronize()
    with lib.Correlator(N, K, lib.DTYPES[dtype]) as c:
        if split:
            lib.corr_set_tiles(c.h, 0, 0, split, 0)
        for passes in (1, 2):                   # a first pass stores, a second one adds
            for _ in range(passes):
                c.push(x, S * K)
            V, n = c.dump(fp64=True)
            assert n == passes * S
            d = np.abs(V - passes * R)
            autos = [oracle.baseline_index(i, i, N) for i in range(N)]
            A = np.abs(passes * R[autos])
            ii, jj = np.triu_indices(N)
            nrm = np.sqrt(A[ii] * A[jj])
            # (a channel without power: V must be R)
            assert np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)) <= BOUNDS[dtype]
