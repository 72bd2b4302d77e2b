"""The accumulator after a dump counts as zeros without being cleared: empty
dumps, checkpoints, fused and captured steps that follow one see zeros."""

import numpy as np
import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu


def _dev(torch, N, K, S, seed):
    p, _ = synth.make_samples(N, S * K, K, seed=seed)
    return torch.from_numpy(p.reshape(-1)).cuda()


@pytest.mark.parametrize("dtype,N,K", [("fp32", 5, 64), ("fp16", 66, 64), ("fp32_simt", 7, 128),
                                       ("fp8", 3, 512)])
def test_after_a_dump(lib, dtype, N, K):
    torch = pytest.importorskip("torch")
    S = 130
    A, B = (_dev(torch, N, K, S, s) for s in (1, 2))
    P, C = N * (N + 1) // 2, K // 2
    scales = np.ones((N, C), np.float32) if dtype in ("fp16", "fp8") else None

    def handle():
        c = lib.Correlator(N, K, dtype)
        if scales is not None:
            lib.corr_set_scales(c.h, scales)
        return c

    with handle() as c:
        c.push(B)
        want, _ = c.dump(fp64=True)
    with handle() as c, handle() as r:
        c.push(A)
        c.dump()
        V, n = c.dump(fp64=True)                    # an empty integration
        assert n == 0 and np.all(V == 0)
        c.push(B)
        V, n = c.dump(fp64=True)
        assert n == S and np.array_equal(V, want)
        lib.corr_load_state(r.h, lib.corr_save_state(c.h))   # a checkpoint of nothing yet
        r.push(B)
        V, n = r.dump(fp64=True)
        assert n == S and np.array_equal(V, want)
        V, n = c.dump(fp64=True)
        assert n == 0 and np.all(V == 0)


def test_fused_after_a_dump(lib):
    torch = pytest.importorskip("torch")
    N, K, S = 4, 512, 96
    A, B = (_dev(torch, N, K, S, s) for s in (3, 4))
    with lib.Correlator(N, K, "fp32") as c:
        lib.corr_set_fused(c.h, True)
        c.push(B)
        want, _ = c.dump(fp64=True)
        lib.corr_set_fused(c.h, False)
        c.push(A)
        c.dump()                                     # leaves A's sums in memory
        lib.corr_set_fused(c.h, True)
        c.push(B)
        V, _ = c.dump(fp64=True)
    assert np.array_equal(V, want)


def test_captured_step_with_an_empty_mode(lib):
    torch = pytest.importorskip("torch")
    modes = [(4, 64), (3, 128)]
    A, B = (_dev(torch, N, K, 64, 5) for N, K in modes)
    vis = [torch.empty((N * (N + 1) // 2, K // 2), dtype=torch.complex64, device="cuda") for N, K in modes]
    with lib.CorrelatorBatch(modes, "fp32") as b:
        b.capture([A, B], vis, n=[64 * 64, 0])
        b.push([A, B])                               # the empty mode used in between
        b.dump()
        for v in vis:
            v.fill_(7)
        torch.cuda.synchronize()
        n = b.replay()
        b.sync()
        assert n == [64, 0]
        assert torch.all(vis[1] == 0) and torch.any(vis[0] != 0)
        V, n = b.dump()
        assert n == [0, 0] and all(np.all(v == 0) for v in V)
