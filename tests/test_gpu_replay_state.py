"""A captured step leaves its sums in the accumulator, which then counts as
zeros: empty dumps, checkpoints and pushes that follow a replay see zeros,
whatever ran between the capture and the replay."""

import numpy as np
import pytest

from paper_1102_0148_gb300 import synth

pytestmark = pytest.mark.gpu

MODES = [(4, 64), (66, 64)]          # one antenna block; two (pass result in the FP32 slot)
S = 64


@pytest.fixture()
def step(lib):
    """A batch with a captured step over A, its outputs, another input B and
    B's visibilities as a batch that never replayed gives them."""
    torch = pytest.importorskip("torch")
    A, B = ([torch.from_numpy(synth.make_samples(N, S * K, K, seed=s + K)[0].reshape(-1)).cuda()
             for N, K in MODES] for s in (1, 2))
    vis = [torch.empty((N * (N + 1) // 2, K // 2), dtype=torch.complex128, device="cuda") for N, K in MODES]
    torch.cuda.synchronize()
    with lib.CorrelatorBatch(MODES, "fp32") as b:
        b.push(B)
        want, _ = b.dump(fp64=True)
    with lib.CorrelatorBatch(MODES, "fp32") as b:
        b.capture(A, vis, fp64=True)
        yield b, vis, B, want


def _replay(b):
    assert b.replay() == [S, S]
    b.sync()


def _push_equals(b, B, want):
    b.push(B)
    V, n = b.dump(fp64=True)
    assert n == [S, S]
    assert all(np.array_equal(v, w) for v, w in zip(V, want))


def _empty(b):
    V, n = b.dump(fp64=True)
    assert n == [0, 0] and all(np.all(v == 0) for v in V)


def test_push_after_loading_an_empty_state_and_a_replay(lib, step):
    b, _, B, want = step
    for h, (N, K) in zip(b.handles, MODES):
        with lib.Correlator(N, K, "fp32") as c:
            lib.corr_load_state(h, lib.corr_save_state(c.h))
    _replay(b)
    _push_equals(b, B, want)


def test_checkpoints_between_replays(lib, step):
    b, _, B, want = step
    for _ in range(2):
        _replay(b)
        states = [lib.corr_save_state(h) for h in b.handles]
    with lib.CorrelatorBatch(MODES, "fp32") as r:
        for h, st in zip(r.handles, states):
            lib.corr_load_state(h, st)
        _push_equals(r, B, want)
    _push_equals(b, B, want)


def test_empty_dumps_around_replays(lib, step):
    b, vis, B, want = step
    first = [v.clone() for v in vis]
    for _ in range(2):
        _empty(b)
        _replay(b)
        assert all(bool((v == f).all()) for v, f in zip(vis, first))
        _empty(b)
    _push_equals(b, B, want)


@pytest.mark.parametrize("mode", [0, 1])
def test_failed_capture_leaves_no_sums(lib, step, mode):
    """Recording fails at one mode's dump, with the passes recorded and never
    run: every mode is as the eager step's dump left it."""
    b, vis, B, want = step
    lib.corr_test_fault(b.handles[mode], 3, 0.05)
    with pytest.raises(lib.CorrError) as ei:
        b.capture(B, vis, fp64=True)
    assert ei.value.code == lib.CORR_ECUDA
    with pytest.raises(lib.CorrError) as ei:
        b.replay()
    assert ei.value.code == lib.CORR_ESTATE
    _push_equals(b, B, want)
    _empty(b)
    b.capture(B, vis, fp64=True)
    for v in vis:
        v.zero_()
    _replay(b)
    assert all(np.array_equal(v.cpu().numpy(), w) for v, w in zip(vis, want))
