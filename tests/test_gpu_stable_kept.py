"""The autograd binding leaves the handle's corr_set_stable as it was, and a
batch's modes keep theirs."""

import numpy as np
import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("on", [False, True])
def test_binding_keeps_the_setting(lib, on):
    torch = pytest.importorskip("torch")
    from paper_1102_0148_gb300 import autograd
    N, K, S = 3, 64, 40
    x = torch.from_numpy(synth.make_samples(N, S * K, K, seed=6)[0].reshape(-1)).cuda()
    g = torch.ones(N, dtype=torch.complex64, device="cuda")
    t = torch.zeros(N, device="cuda")
    torch.cuda.synchronize()
    with lib.Correlator(N, K, "fp32") as c:
        assert lib.corr_get_stable(c.h) is False
        lib.corr_set_stable(c.h, on)
        autograd.visibilities(g, t, x, c)
        assert lib.corr_get_stable(c.h) is on
        with pytest.raises(lib.CorrError):                   # samples of no whole frame
            autograd.visibilities(g, t, x[: N * (K // 2) + 16 * N], c)
        assert lib.corr_get_stable(c.h) is on


def test_batch_mode_is_stable_throughout(lib):
    torch = pytest.importorskip("torch")
    modes, S = [(66, 64), (5, 256)], 384
    x = [torch.from_numpy(synth.make_samples(N, S * K, K, seed=7)[0].reshape(-1)).cuda() for N, K in modes]
    torch.cuda.synchronize()
    for m, (N, K) in enumerate(modes):
        with lib.Correlator(N, K, "fp32") as c, lib.CorrelatorBatch([(N, K)], "fp32") as b:
            for h in (c.h, b.handles[0]):
                lib.corr_set_stable(h, True)
            c.push(x[m], S * K)
            b.push([x[m]])
            V, _ = c.dump(fp64=True)
            W, _ = b.dump(fp64=True)
        assert np.array_equal(V, W[0])
