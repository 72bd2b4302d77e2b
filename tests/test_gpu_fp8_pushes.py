"""FP8: the same samples give the same spectra in any pushes of whole 128-frame
blocks, on both sides of the frame at which an integration changes F-engine
kernels."""

import numpy as np
import pytest

import oracle
from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu

# the change comes at the first whole 128 frames T with 2 T^2 / N + T >= 420000
LINE = {1: 512, 2: 768, 5: 1024}


def _norm(V, R, N):
    autos = [oracle.baseline_index(i, i, N) for i in range(N)]
    A = np.abs(R[autos])
    ii, jj = np.triu_indices(N)
    nrm = np.sqrt(A[ii] * A[jj])
    d = np.abs(V - R)
    return float(np.max(np.divide(d, nrm, out=np.where(d > 0, np.inf, 0.0), where=nrm > 0)))


@pytest.mark.parametrize("K", [16, 64, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("N", [1, 2, 5])
def test_pushes_do_not_change_the_spectra(lib, N, K):
    torch = pytest.importorskip("torch")
    S = LINE[N] + 300
    packed, _ = synth.make_samples(N, S * K, K, seed=21 + K + N)
    x = torch.from_numpy(packed).cuda()
    host = torch.from_numpy(packed).pin_memory()
    torch.cuda.synchronize()
    scales = np.full((N, K // 2), 16.0 / np.sqrt(2.0 * K), np.float32)

    def run(cuts, data=x):
        with lib.Correlator(N, K, "fp8") as c:
            lib.corr_set_scales(c.h, scales)
            for a, b in zip([0] + cuts, cuts + [S]):
                c.push(data[a:b], (b - a) * K)
            V, n = c.dump(fp64=True)
        assert n == S
        return V

    one = run([])
    # whole 128-frame blocks: one pass of the same values, so the same bits
    for cuts in ([128], list(range(128, S, 128)), [LINE[N] - 128], [LINE[N]], [LINE[N] + 128]):
        assert np.array_equal(run(cuts), one)
    assert np.array_equal(run([], host), one)


def test_batch_pushes(lib):
    torch = pytest.importorskip("torch")
    modes = [(2, 512), (5, 64)]
    S = [LINE[N] + 300 for N, _ in modes]
    x = [torch.from_numpy(synth.make_samples(N, s * K, K, seed=5)[0]).cuda() for (N, K), s in zip(modes, S)]
    torch.cuda.synchronize()

    def run(cuts):
        with lib.CorrelatorBatch(modes, "fp8") as b:
            for h, (N, K) in zip(b.handles, modes):
                lib.corr_set_scales(h, np.full((N, K // 2), 16.0 / np.sqrt(2.0 * K), np.float32))
            for c0, c1 in zip([[0, 0]] + cuts, cuts + [S]):
                b.push([d[p:q].reshape(-1) for d, p, q in zip(x, c0, c1)])
            V, n = b.dump(fp64=True)
        assert n == S
        return V

    one = run([])
    for cuts in ([[128, 256]], [[500, 100], [700, 1100]], [[768, 1024]]):
        for (N, _), a, b in zip(modes, run(cuts), one):
            assert _norm(a, b, N) <= 1e-5
    # a captured step takes the kernels that a push of it takes
    vis = [torch.empty((N * (N + 1) // 2, K // 2), dtype=torch.complex128, device="cuda") for N, K in modes]
    with lib.CorrelatorBatch(modes, "fp8") as b:
        for h, (N, K) in zip(b.handles, modes):
            lib.corr_set_scales(h, np.full((N, K // 2), 16.0 / np.sqrt(2.0 * K), np.float32))
        b.capture([d.reshape(-1) for d in x], vis, fp64=True)
        b.replay()
        b.sync()
    assert all(np.array_equal(v.cpu().numpy(), w) for v, w in zip(vis, one))
