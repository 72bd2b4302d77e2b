"""The profile of a batch counts the X-engine launches that a push takes: one
for the modes of one antenna block, one for those of several."""

import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("modes,launches", [([(44, 512), (5, 64)], 1), ([(66, 64)], 1), ([(130, 64), (70, 64)], 1),
                                            ([(66, 64), (5, 128)], 2), ([(5, 128), (66, 64), (8, 64)], 2)])
def test_xengine_launches_of_a_push(lib, modes, launches):
    torch = pytest.importorskip("torch")
    x = [synth.make_samples_torch(N, 128 * K, K, seed=1, device="cuda")[0].reshape(-1) for N, K in modes]
    torch.cuda.synchronize()
    with lib.CorrelatorBatch(modes, "fp16") as b:
        b.push(x)
        b.dump()
        for h in b.handles:
            lib.corr_profile_enable(h, True)
        for _ in range(3):
            b.push(x)
        b.sync()
        assert sum(lib.corr_profile_read(h)["xengine"][0] for h in b.handles) == 3 * launches
        b.dump()
