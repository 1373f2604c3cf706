"""The certified exact l2 scan (tensor-core screen with a proven error bound,
canonical distances for every column the bound does not exclude) against the
oracle, bit for bit: minima and argmins at the edges of its tiles, slices and
row widths, where ties, offsets or extreme magnitudes send samples to the
CUDA-core form, and with a wait budget that stops the screen."""
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


def _scan(ctx, A, B, idx, dtype=ch.CH_F32, metric=ch.CH_L2):
    """(min_d, argmin) of the exact scan on the GPU, and the values the library saw."""
    T = idx.size
    if dtype == ch.CH_BF16:
        hA, hB = workloads.to_bf16_bits(A), workloads.to_bf16_bits(B)
        A, B = workloads.bf16_bits_to_f32(hA), workloads.bf16_bits_to_f32(hB)
        dA, dB = (torch.from_numpy(h.view(np.int16)).cuda() for h in (hA, hB))
    else:
        dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    sA = ch.ch_set_create(ctx, dA, 2, A.shape[0], A.shape[1], dtype)
    sB = ch.ch_set_create(ctx, dB, 2, B.shape[0], B.shape[1], dtype)
    m = torch.full((T,), -1.0, device="cuda")
    am = torch.full((T,), -7, dtype=torch.int64, device="cuda")
    ch.ch_sampled_nn(ctx, sA, torch.from_numpy(idx).cuda(), T, sB, metric, ch.CH_SCREEN_EXACT, 8, m, am)
    out = m.cpu().numpy(), am.cpu().numpy()
    ch.ch_set_destroy(sA)
    ch.ch_set_destroy(sB)
    return out, A, B


def _check(ctx, A, B, idx, dtype=ch.CH_F32, metric=ch.CH_L2):
    (m, am), A, B = _scan(ctx, A, B, idx, dtype, metric)
    ok = idx >= 0
    mo, amo = oracle.scan(A, idx[ok], B, metric)
    assert np.array_equal(m[ok].view(np.uint32), mo.view(np.uint32))
    assert np.array_equal(am[ok], amo)
    assert np.all(m[~ok] == 0) and np.all(am[~ok] == -1)


@pytest.mark.parametrize("dtype", [ch.CH_F32, ch.CH_BF16], ids=["f32", "bf16"])
@pytest.mark.parametrize("nB,d,T", [(257, 8, 4200), (1000, 16, 1100), (5003, 24, 600), (2560, 32, 520),
                                    (4099, 40, 530), (2049, 128, 640), (3001, 200, 560), (1537, 384, 700),
                                    (1111, 768, 1000), (700, 1000, 1500), (40000, 16, 256)])
def test_certified_scan_shapes(ctx, dtype, nB, d, T):
    A, B = workloads.gaussian_mixture(900, nB, d, nB + d, clusters=5)
    idx = np.random.default_rng(d).integers(0, 900, T).astype(np.int64)
    idx[3::29] = -1
    _check(ctx, A, B, idx, dtype)


@pytest.mark.parametrize("case", ["duplicates", "all_equal", "offset", "offset_mixed", "tiny", "huge", "one_far",
                                  "queries_in_B"])
def test_certified_scan_data(ctx, case):
    A, B = workloads.gaussian_mixture(600, 3000, 32, 11, clusters=4)
    if case == "duplicates":
        B[1500:] = B[:1500]
    elif case == "all_equal":
        B[:] = B[7]
    elif case == "offset":  # the bound excludes almost nothing: every sample is listed
        A += 3000
        B += 3000
    elif case == "offset_mixed":
        A[::2] += 3000
        B[::3] += 3000
    elif case == "tiny":  # squares underflow
        A *= np.float32(1e-22)
        B *= np.float32(1e-22)
    elif case == "huge":  # squared norms overflow, distances do not
        A = (A * 1e-3 + 2e19).astype(np.float32)
        B = (B * 1e-3 + 2e19).astype(np.float32)
    elif case == "one_far":
        B[17] *= np.float32(1e15)
        A[5] *= np.float32(1e15)
    elif case == "queries_in_B":
        B[100:700] = A
    idx = np.random.default_rng(1).integers(0, 600, 1300).astype(np.int64)
    _check(ctx, A, B, idx)


@pytest.mark.parametrize("metric", [ch.CH_L1, ch.CH_L2], ids=["l1", "l2"])
@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("case", ["plain", "duplicates", "offset", "offset_mixed", "tiny", "huge", "few_rows"])
def test_small_d_scan_data(ctx, metric, d, case):
    """d <= 4: sub-tile minima under the error bound, with the second-best sub-tile
    and whole-chunk evaluations that ties, offsets and extreme magnitudes call for."""
    A, B = workloads.gaussian_mixture(700, 5000, d, 21 + d, clusters=4)
    if case == "duplicates":
        B[2500:] = B[:2500]
    elif case == "offset":
        A += 3000
        B += 3000
    elif case == "offset_mixed":
        A[::2] += 3000
        B[::3] += 3000
    elif case == "tiny":
        A *= np.float32(1e-22)
        B *= np.float32(1e-22)
    elif case == "huge":
        A = (A * 1e-3 + 2e19).astype(np.float32)
        B = (B * 1e-3 + 2e19).astype(np.float32)
    elif case == "few_rows":
        B = B[:33]
    idx = np.random.default_rng(4).integers(0, 700, 1500).astype(np.int64)
    idx[2::37] = -1
    _check(ctx, A, B, idx, metric=metric)


@pytest.mark.parametrize("dtype", [ch.CH_F32, ch.CH_BF16], ids=["f32", "bf16"])
@pytest.mark.parametrize("metric", [ch.CH_L1, ch.CH_L2], ids=["l1", "l2"])
@pytest.mark.parametrize("nB,d,T", [(9000, 33, 1900), (1801, 300, 1000), (10007, 97, 560), (5003, 127, 900),
                                    (2500, 50, 4400), (30000, 5, 3700)])
def test_chained_scan_shapes(ctx, metric, dtype, nB, d, T):
    """Rows the screen cannot read, and l1: the chained form's tiles, slabs and sample
    block widths (both metrics at sizes past its rule)."""
    A, B = workloads.gaussian_mixture(400, nB, d, nB + d, clusters=5)
    idx = np.random.default_rng(d).integers(0, 400, T).astype(np.int64)
    idx[3::29] = -1
    _check(ctx, A, B, idx, dtype, metric)


@pytest.mark.parametrize("case", ["duplicates", "all_equal", "offset", "tiny", "huge", "one_far", "queries_in_B"])
def test_chained_scan_data(ctx, case):
    A, B = workloads.gaussian_mixture(600, 3000, 32, 11, clusters=4)
    if case == "duplicates":
        B[1500:] = B[:1500]
    elif case == "all_equal":
        B[:] = B[7]
    elif case == "offset":
        A += 3000
        B += 3000
    elif case == "tiny":
        A *= np.float32(1e-33)
        B *= np.float32(1e-33)
    elif case == "huge":  # l1 sums overflow for the far rows
        with np.errstate(over="ignore"):
            B[::2] *= np.float32(3e36)
    elif case == "one_far":
        B[17] *= np.float32(1e15)
        A[5] *= np.float32(1e15)
    elif case == "queries_in_B":
        B[100:700] = A
    idx = np.random.default_rng(1).integers(0, 600, 5700).astype(np.int64)
    _check(ctx, A, B, idx, metric=ch.CH_L1)


@pytest.mark.parametrize("metric,d", [(ch.CH_L1, 24), (ch.CH_L2, 27)])
def test_chained_brute_force_over_slices(ctx, metric, d):
    A, B = workloads.uniform(17000, 1400, d, 6)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    sA, sB = ch.ch_set_create(ctx, dA, 2, 17000, d), ch.ch_set_create(ctx, dB, 2, 1400, d)
    mins = torch.zeros(17000, device="cuda")
    v = ch.ch_exact(ctx, sA, sB, metric, 0, mins)
    vo, mo = oracle.exact_canonical(A, B, metric)
    assert np.array_equal(mins.cpu().numpy(), mo) and abs(v / vo - 1) < 1e-12
    ch.ch_set_destroy(sA)
    ch.ch_set_destroy(sB)


def test_certified_brute_force_over_slices(ctx):
    """More samples than one slice of the scan, in A's order (ch_exact)."""
    A, B = workloads.uniform(17000, 333, 12, 5)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    sA, sB = ch.ch_set_create(ctx, dA, 2, 17000, 12), ch.ch_set_create(ctx, dB, 2, 333, 12)
    mins = torch.zeros(17000, device="cuda")
    v = ch.ch_exact(ctx, sA, sB, ch.CH_L2, 0, mins)
    vo, mo = oracle.exact_canonical(A, B, ch.CH_L2)
    assert np.array_equal(mins.cpu().numpy(), mo) and abs(v / vo - 1) < 1e-12
    ch.ch_set_destroy(sA)
    ch.ch_set_destroy(sB)


def test_certified_scan_survives_a_stopped_screen(ctx):
    """A wait budget that runs out inside the screen leaves the samples to the
    CUDA-core form: the exact scan never times out."""
    A, B = workloads.gaussian_mixture(500, 20000, 64, 3, clusters=6)
    idx = np.random.default_rng(2).integers(0, 500, 520).astype(np.int64)
    ch.ch_ctx_set_wait_cycles(ctx, 8)
    try:
        _check(ctx, A, B, idx)
    finally:
        ch.ch_ctx_set_wait_cycles(ctx, 0)
