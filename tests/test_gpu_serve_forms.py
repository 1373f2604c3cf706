"""Serving exact scans under a tight budget: the faster forms' extra scratch never costs
a request its admission, its place beside others, or a bit of its result."""
import os
import time

import pytest

from paper_2307_03043_gb300 import binding as ch
from paper_2307_03043_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, D, SLOTS = 20000, 64, 4
KINDS = {"chained": dict(metric=ch.CH_L1), "certified": dict(metric=ch.CH_L2, screen=ch.CH_SCREEN_EXACT)}


def _params(kind, k=0):
    return ch.est_params(levels=10, proj_dim=16, hash_seed=k, eps=0.1, sample_seed=100 + k, **KINDS[kind])


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03043_gb300 import build
    build.build()
    c = ch.ch_ctx_create(0, None)
    yield c
    ch.ch_ctx_destroy(c)


@pytest.fixture(scope="module")
def data():
    return workloads.gaussian_mixture(N, N, D, 8, clusters=10)


class _Server:
    def __init__(self, ctx, data, budget, slots=SLOTS, fault=None):
        if fault:
            os.environ["CH_SERVE_FAULT"] = fault
        try:
            self.h = ch.ch_serve_create(ctx, budget, slots, 64)
        finally:
            os.environ.pop("CH_SERVE_FAULT", None)
        self.ids = [ch.ch_serve_register(self.h, X, 0, N, D) for X in data]

    def __enter__(self):
        return self

    def __exit__(self, *_):
        ch.ch_serve_destroy(self.h)

    def submit(self, p):
        return ch.ch_serve_submit(self.h, *self.ids, p)

    def wait(self, ticket):
        st, eta, rs = ch.ch_serve_wait(self.h, ticket, 60000)
        assert st == ch.CH_OK and rs == ch.CH_OK
        return eta

    def peak(self):
        return int(ch.ch_serve_stats_get(self.h).peak_bytes)


def _footprints(ctx, data, kind):
    """(faster form's, plain form's) admitted bytes of one request, and its result in each."""
    with _Server(ctx, data, 8 << 30) as s:
        eta = s.wait(s.submit(_params(kind))[1])
        fast = s.peak()
    with _Server(ctx, data, fast - 1, slots=1) as s:  # between the two footprints
        st, t = s.submit(_params(kind))
        assert st == ch.CH_OK
        assert s.wait(t) == eta
        plain = s.peak()
    with _Server(ctx, data, plain - 1) as s:
        assert s.submit(_params(kind))[0] == ch.CH_EBUSY
    assert plain < fast
    return fast, plain


@pytest.mark.parametrize("kind", list(KINDS))
def test_a_full_set_of_plain_footprints_runs_side_by_side(ctx, data, kind):
    """A budget of SLOTS plain footprints runs SLOTS requests at once: each sleeps 50 ms on
    the host here, so one after another they would take SLOTS x 50 ms."""
    fast, plain = _footprints(ctx, data, kind)
    alone = {}
    with _Server(ctx, data, 8 << 30) as s:
        for k in range(SLOTS):
            alone[k] = s.wait(s.submit(_params(kind, k))[1])
    with _Server(ctx, data, SLOTS * plain, fault="slow") as s:
        s.wait(s.submit(_params(kind))[1])  # the pool and the contexts are warm
        wall = []
        for _ in range(4):
            t0 = time.perf_counter()
            ts = [s.submit(_params(kind, k))[1] for k in range(SLOTS)]
            got = [s.wait(t) for t in ts]
            wall.append(time.perf_counter() - t0)
            assert got == [alone[k] for k in range(SLOTS)]
        assert s.peak() <= SLOTS * plain
    assert min(wall) < 0.095, wall  # two in a row: 100 ms at least


def test_a_wide_budget_admits_the_faster_form(ctx, data):
    for kind in KINDS:
        fast, plain = _footprints(ctx, data, kind)
        with _Server(ctx, data, SLOTS * fast) as s:
            s.wait(s.submit(_params(kind))[1])
            assert s.peak() == fast
