"""The exact scan of d <= 4 on clouds away from the origin and on lattices (many equal
distances): bit for bit the oracle's, lone and batched, at both sample counts per thread
and on both sides of the second walk's rule; and at the origin's speed wherever the cloud
lies."""
import numpy as np
import pytest

import oracle
from paper_2307_03043_gb300 import binding as ch
from paper_2307_03043_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03043_gb300 import build
    build.build()
    c = ch.ch_ctx_create(0, torch.cuda.current_stream())
    yield c
    ch.ch_ctx_destroy(c)


def _sets(ctx, *hosts):
    dev = [torch.from_numpy(h).cuda() for h in hosts]
    return dev, [ch.ch_set_create(ctx, x, 2, x.shape[0], x.shape[1]) for x in dev]


def _check(ctx, A, B, idx, metric=ch.CH_L2):
    dev, (sA, sB) = _sets(ctx, A, B)
    T = idx.size
    m = torch.full((T,), -1.0, device="cuda")
    am = torch.full((T,), -7, dtype=torch.int64, device="cuda")
    ch.ch_sampled_nn(ctx, sA, torch.from_numpy(idx).cuda(), T, sB, metric, ch.CH_SCREEN_EXACT, 8, m, am)
    mo, amo = oracle.scan(A, idx, B, metric)
    assert np.array_equal(m.cpu().numpy().view(np.uint32), mo.view(np.uint32))
    some = np.isfinite(mo)  # a sample all of whose distances overflow has no nearest point
    assert np.array_equal(am.cpu().numpy()[some], amo[some])
    for s in (sA, sB):
        ch.ch_set_destroy(s)


def _lattice(n, d, cells, seed, shift=0.0, scale=1.0):
    g = np.random.default_rng(seed)
    return (g.integers(0, cells, (n, d)) * np.float32(scale) + np.float32(shift)).astype(np.float32)


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("cells,shift,off", [(2, 0.0, 0.0), (5, 0.0, 0.25), (16, 100.0, 0.0), (40, -7.0, 0.3)])
def test_lattice_ties(ctx, d, cells, shift, off):
    A, B = _lattice(700, d, cells, 1, shift + off), _lattice(6001, d, cells, 2, shift)
    idx = np.random.default_rng(3).integers(0, 700, 1300).astype(np.int64)
    _check(ctx, A, B, idx)


def test_lattice_ties_two_samples_per_thread(ctx):
    A, B = _lattice(2000, 3, 12, 4, 0.5), _lattice(90001, 3, 12, 5)
    idx = np.random.default_rng(6).integers(0, 2000, 3100).astype(np.int64)
    _check(ctx, A, B, idx)


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", ["far", "far_and_wide", "a_few_ties", "all_equal", "one_sample_far_off", "sparse_out_of_range"])
def test_offsets_and_few_wide_samples(ctx, d, kind):
    A, B = workloads.gaussian_mixture(900, 7001, d, 31 + d, clusters=4)
    if kind == "far":
        A += 30000
        B += 30000
    elif kind == "far_and_wide":
        A[::3] -= 90000
        B[::2] += 30000
    elif kind == "a_few_ties":  # below the second walk's rule: warps look single samples over
        B[100::50] = A[5] + 1
    elif kind == "all_equal":
        B[:] = B[11]
    elif kind == "one_sample_far_off":  # the block's pivot
        A[0] *= np.float32(1e17)
    elif kind == "sparse_out_of_range":
        A[7::100] *= np.float32(3e20)
    idx = np.random.default_rng(8).integers(0, 900, 1100).astype(np.int64)
    idx[0] = 0
    _check(ctx, A, B, idx)


@pytest.mark.parametrize("metric", [ch.CH_L1, ch.CH_L2], ids=["l1", "l2"])
def test_batched_lattices_equal_lone(ctx, metric):
    hosts = []
    for i, (cells, shift, off) in enumerate([(6, 0.0, 0.0), (6, 50.0, 0.25), (30, 0.0, 0.1), (300, 1e4, 0.0)]):
        hosts += [_lattice(3000 + 501 * i, 3, cells, 2 * i, shift + off), _lattice(20000 + 77 * i, 3, cells, 2 * i + 1, shift)]
    dev, sets = _sets(ctx, *hosts)
    A, B = sets[0::2] * 3, sets[1::2] * 3
    ps = [ch.est_params(metric, 10, 16, None, i, eps=0.1, sample_seed=i) for i in range(len(A))]
    etas, status = ch.ch_estimate_batch(ctx, A, B, ps)
    assert status == [ch.CH_OK] * len(A)
    assert etas == [ch.ch_estimate(ctx, a, b, p) for a, b, p in zip(A, B, ps)]
    for s in sets:
        ch.ch_set_destroy(s)


def test_a_cloud_away_from_the_origin_costs_no_more(ctx):
    """The same surface at the origin and 1000 extents off: the same work, so the same time.
    (Before the pivot it took 4 to 14 times as long; 1.5 leaves room for noise.)"""
    A, B = workloads.shape_surface(20000, 200000, 3)
    idx = torch.from_numpy(np.random.default_rng(1).integers(0, 20000, 4606).astype(np.int64)).cuda()
    m = torch.empty(4606, device="cuda")
    best = {}
    for off in (0.0, 1000.0):
        dev, (sA, sB) = _sets(ctx, A + np.float32(off), B + np.float32(off))
        times = []
        for _ in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            ch.ch_sampled_nn(ctx, sA, idx, 4606, sB, ch.CH_L2, ch.CH_SCREEN_EXACT, 8, m)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        best[off] = min(times[2:])
        for s in (sA, sB):
            ch.ch_set_destroy(s)
    assert best[1000.0] < 1.5 * best[0.0], best
