"""Sets shared by contexts: the exact l2 scan never reads row norms whose pass another
context has only enqueued, and a set is prepared only once every pass of it has finished.
A delay kernel in front of the other context's work keeps that pass pending meanwhile."""
import numpy as np
import pytest

import oracle
from paper_2307_03043_gb300 import binding as ch
from paper_2307_03043_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NA, NB, D, T = 900, 4000, 64, 1100  # takes the certified form


@pytest.fixture()
def two():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03043_gb300 import build
    build.build()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctxs = [ch.ch_ctx_create(0, s) for s in streams]
    yield ctxs, streams
    torch.cuda.synchronize()
    for c in ctxs:
        ch.ch_ctx_destroy(c)


class _Pair:
    def __init__(self, ctx, seed):
        self.A, self.B = workloads.gaussian_mixture(NA, NB, D, seed, clusters=5)
        self.dA, self.dB = torch.from_numpy(self.A).cuda(), torch.from_numpy(self.B).cuda()
        self.idx = np.random.default_rng(seed).integers(0, NA, T).astype(np.int64)
        self.didx = torch.from_numpy(self.idx).cuda()
        self.m = torch.full((T,), -1.0, device="cuda")
        self.am = torch.full((T,), -7, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        self.sA = ch.ch_set_create(ctx, self.dA, 2, NA, D)
        self.sB = ch.ch_set_create(ctx, self.dB, 2, NB, D)
        ch.ch_ctx_sync(ctx)

    def scan(self, ctx, screen=ch.CH_SCREEN_EXACT):
        ch.ch_sampled_nn(ctx, self.sA, self.didx, T, self.sB, ch.CH_L2, screen, 8, self.m, self.am)

    def check(self):
        torch.cuda.synchronize()
        mo, amo = oracle.scan(self.A, self.idx, self.B, ch.CH_L2)
        assert np.array_equal(self.m.cpu().numpy().view(np.uint32), mo.view(np.uint32))
        assert np.array_equal(self.am.cpu().numpy(), amo)

    def close(self):
        torch.cuda.synchronize()
        ch.ch_set_destroy(self.sA)
        ch.ch_set_destroy(self.sB)


def _delay(stream, ms=60):
    with torch.cuda.stream(stream):
        torch.cuda._sleep(int(ms * 2e6))


def _pending_screen(ctx, stream, pair):
    """A screened scan (which makes B's norms) waiting behind a delay on ctx's stream."""
    out = torch.empty(T, device="cuda")
    warm = _Pair(ctx, 90)
    warm.scan(ctx, ch.CH_SCREEN_AUTO)  # the context's workspace stays as it is from here on
    warm.close()
    _delay(stream)
    ch.ch_sampled_nn(ctx, pair.sA, pair.didx, T, pair.sB, ch.CH_L2, ch.CH_SCREEN_AUTO, 8, out)
    return out


def test_owners_exact_scan_beside_another_contexts_pending_norms(two):
    (c1, c2), (s1, s2) = two
    warm = _Pair(c1, 91)
    warm.scan(c1)
    warm.close()
    p = _Pair(c1, 1)
    keep = _pending_screen(c2, s2, p)
    p.scan(c1)
    p.check()
    del keep
    p.close()


def test_prepare_waits_for_another_contexts_pending_norms(two):
    (c1, c2), (s1, s2) = two
    warm = _Pair(c2, 92)
    warm.scan(c2)
    ch.ch_set_prepare(c2, warm.sA)
    warm.close()
    p = _Pair(c1, 2)
    keep = _pending_screen(c1, s1, p)
    ch.ch_set_prepare(c2, p.sB)
    assert s1.query()  # the owner's pass is over
    p.scan(c2)
    p.check()
    del keep
    p.close()


def test_captured_exact_scan_leaves_no_norms_behind(two):
    """Captured work has not run: a later call makes the norms it needs, and so does the
    graph when it is launched."""
    (c1, _), (s1, _) = two
    warm = _Pair(c1, 93)
    warm.scan(c1)
    warm.close()
    p = _Pair(c1, 3)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s1):
        p.scan(c1)
    p.scan(c1)
    p.check()
    p.m.fill_(-1.0)
    p.am.fill_(-7)
    torch.cuda.synchronize()
    g.replay()
    p.check()
    p.close()
