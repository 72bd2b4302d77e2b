"""Passes of arrays above 64 antennas are cut into ranges that are summed in FP32
and combined in FP64: the number of ranges, which bounds the FP32 sums, and the
combination of 2 to 8 of them, in a first pass and a later one."""

import numpy as np
import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


# ranges: the count that minimises the busiest of 152 single CTAs, dealt one
# A block against two B blocks in turn, worked out apart from the library
@pytest.mark.parametrize("dtype,N,K,S,ranges", [
    ("fp32", 66, 64, 384, 2), ("fp32", 65, 32, 2048, 4), ("fp32", 100, 64, 4096, 2), ("fp32", 130, 32, 1000, 2),
    ("fp32", 200, 16, 3000, 6), ("fp32", 128, 128, 8192, 8), ("fp16", 300, 16, 2048, 4), ("fp8", 200, 16, 3000, 3)])
def test_ranges_of_a_pass(lib, dtype, N, K, S, ranges):
    torch = pytest.importorskip("torch")
    x, y = (synth.make_samples_torch(N, S * K, K, seed=s, device="cuda")[0].reshape(-1) for s in (1, 2))
    torch.cuda.synchronize()
    got = {}
    with lib.Correlator(N, K, dtype) as c:
        if dtype != "fp32":
            lib.corr_set_scales(c.h, np.ones((N, K // 2), np.float32))
        for split in (0, ranges, 1):
            lib.corr_set_tiles(c.h, 0, 0, split, 0)
            V = []
            for pushes in ((x,), (x, y)):            # the second pass is added to the first
                for p in pushes:
                    c.push(p, S * K)
                    lib.corr_sync(c.h)
                V.append(c.dump(fp64=True)[0])
            got[split] = V
    for a, b in zip(got[0], got[ranges]):
        assert np.array_equal(a, b)
    # a lone range rounds elsewhere: the counts above are not the same by chance
    assert not np.array_equal(got[0][0], got[1][0])


def test_infinities_pass_through_the_combination(lib):
    """An antenna whose scaled spectra overflow FP16: the combined ranges hold
    infinities and NaN where one range does."""
    torch = pytest.importorskip("torch")
    N, K, S = 66, 64, 384
    x = synth.make_samples_torch(N, S * K, K, seed=3, device="cuda")[0].reshape(-1)
    torch.cuda.synchronize()
    scales = np.ones((N, K // 2), np.float32)
    scales[[3, 65]] = 2.0 ** 20
    V = {}
    with lib.Correlator(N, K, "fp16") as c:
        lib.corr_set_scales(c.h, scales)
        for split in (1, 2):
            lib.corr_set_tiles(c.h, 0, 0, split, 0)
            c.push(x, S * K)
            V[split] = c.dump(fp64=True)[0]
    for part in (np.real, np.imag):
        a, b = part(V[1]), part(V[2])
        assert np.isinf(a).any() or np.isnan(a).any()
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isposinf(a), np.isposinf(b))
        assert np.array_equal(np.isneginf(a), np.isneginf(b))
