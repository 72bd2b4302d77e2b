"""corr_set_stream waits for the handle's queued work, also when it names the
stream that the handle has."""

import numpy as np
import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("same", [False, True])
def test_set_stream_waits_for_queued_work(lib, same):
    torch = pytest.importorskip("torch")
    N, K, S = 4, 64, 96
    packed, _ = synth.make_samples(N, S * K, K, seed=5)
    x = torch.from_numpy(packed.reshape(-1)).cuda()
    torch.cuda.synchronize()
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    out = torch.zeros((N * (N + 1) // 2, K // 2), dtype=torch.complex64).pin_memory()
    with lib.Correlator(N, K, "fp32", stream=s.cuda_stream) as c:
        assert lib.corr_get_stream(c.h) == s.cuda_stream
        c.push(x, S * K)
        want, _ = c.dump()
        with torch.cuda.stream(s):
            torch.cuda._sleep(1 << 27)               # ~70 ms in front of the work
        c.push(x, S * K)
        lib.corr_dump_async(c.h, out)
        lib.corr_set_stream(c.h, (s if same else other).cuda_stream)
        assert np.array_equal(out.numpy(), want)     # complete without another wait
        assert lib.corr_get_stream(c.h) == (s if same else other).cuda_stream
