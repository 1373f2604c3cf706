"""The workloads this library's performance is measured on.

Each listed case is one call (or the stage-by-stage sequence of calls) that a program linked
against libchamfer makes through the binding; `draw` gives more of the same kinds over the
same ranges.  Inputs are drawn on the GPU from the seed with the distributions of
`paper_2307_03043_gb300/workloads.py` (uniform cubes, Gaussian mixtures, unit-norm mixtures,
d = 3 surface samples); sizes are the ones of the benchmark, the tests and the serving mix.
"""
import math

import numpy as np
import torch

from paper_2307_03043_gb300 import binding as ch

EPS = 0.1
LEVELS = 10
PROJ = 16
DTYPES = {"f32": (ch.CH_F32, 4), "bf16": (ch.CH_BF16, 2), "fp8": (ch.CH_FP8E4M3, 1)}
METRICS = {"l1": ch.CH_L1, "l2": ch.CH_L2}


def listed():
    return [
        # The smallest plain call: a lone estimate of two 2000-point sets, all launches and latency.
        {"name": "estimate_2k_d16_l2", "call": "estimate", "data": "uniform", "nA": 2000, "nB": 2000, "d": 16,
         "dtype": "f32", "metric": "l2"},
        # The ordinary call: the benchmark's 100k x 100k, d = 128 mixture (TF32 screen).
        {"name": "estimate_100k_d128_l2", "call": "estimate", "data": "mixture", "nA": 100000, "nB": 100000, "d": 128,
         "dtype": "f32", "metric": "l2"},
        # The large call: the benchmark's default 1M x 1M, d = 384 unit vectors stored as bf16.
        {"name": "estimate_1m_d384_bf16", "call": "estimate", "data": "unit", "nA": 1000000, "nB": 1000000, "d": 384,
         "dtype": "bf16", "metric": "l2"},
        # The same vectors as fp8 with row scales, stage by stage (a program that keeps b(a), the
        # draws and the nearest points), ragged sizes.
        {"name": "stages_700k_d384_fp8", "call": "stages", "data": "unit", "nA": 700001, "nB": 899999, "d": 384,
         "dtype": "fp8", "metric": "l2"},
        # The default metric (l1) with every stage's outputs kept, ragged sizes, d of the batched mixtures.
        {"name": "stages_70k_d64_l1", "call": "stages", "data": "mixture", "nA": 70001, "nB": 99991, "d": 64,
         "dtype": "f32", "metric": "l1"},
        # Many small pairs in one call: ShapeNet-like d = 3 surfaces, sizes log-uniform in [256, 50000].
        {"name": "batch_512_d3_l2", "call": "batch", "data": "surface", "pairs": 512, "lo": 256, "hi": 50000, "d": 3,
         "dtype": "f32", "metric": "l2", "size_seed": 1},
        # The same call on d = 64 mixtures (a tensor-core screen per pair).
        {"name": "batch_128_d64_l2", "call": "batch", "data": "mixture", "pairs": 128, "lo": 256, "hi": 50000, "d": 64,
         "dtype": "f32", "metric": "l2", "size_seed": 2},
        # A request against an index: resident bf16 d = 768 embeddings, the l2 embedding kept with the sets.
        {"name": "indexed_200k_d768_bf16", "call": "indexed", "data": "uniform", "nA": 120000, "nB": 200000, "d": 768,
         "dtype": "bf16", "metric": "l2"},
        # The brute force that estimates are checked against, every per-point minimum kept.
        {"name": "exact_20k_d128_l2", "call": "exact", "data": "mixture", "nA": 20011, "nB": 30011, "d": 128,
         "dtype": "f32", "metric": "l2"},
        # The large-scale CrudeNN variant of Section 3: 4 structures x a window of 16 points.
        {"name": "crude_4x16_50k_d128", "call": "crude", "data": "mixture", "nA": 50000, "nB": 50000, "d": 128,
         "dtype": "f32", "metric": "l2", "repeats": 4, "window": 16},
        # Both directions of a pair of unequal sets whose rows are too short for the tensor-core screen.
        {"name": "symmetric_60k_d16_l2", "call": "symmetric", "data": "mixture", "nA": 60000, "nB": 100000, "d": 16,
         "dtype": "f32", "metric": "l2"},
        # Word-embedding clouds (d = 300, bf16) under l1: the sampled scan alone, with its argmins.
        {"name": "scan_3k_x_20k_d300_l1", "call": "scan", "data": "mixture", "nA": 5003, "nB": 20011, "d": 300,
         "dtype": "bf16", "metric": "l1", "T": 3001},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["estimate", "estimate", "stages", "batch", "indexed", "exact", "crude", "symmetric", "scan"])
    metric = rng.choice(["l1", "l2", "l2"])
    if call == "estimate":
        if rng.random() < 0.5:  # unit vectors under l2, any storage type
            d, dtype = rng.choice([96, 128, 200, 256, 384]), rng.choice(["bf16", "fp8", "f32"])
            d = 16 * (d // 16)
            n = 1000000 if dtype != "f32" else 300000
            return {"call": call, "data": "unit", "nA": _log(rng, 20000, n), "nB": _log(rng, 20000, n), "d": d,
                    "dtype": dtype, "metric": "l2"}
        d = rng.choice([2, 3, 5, 16, 24, 33, 50, 64, 100, 128])
        hi = 100000 if metric == "l2" else 40000
        return {"call": call, "data": rng.choice(["mixture", "uniform"]), "nA": _log(rng, 1000, hi),
                "nB": _log(rng, 1000, hi), "d": d, "dtype": "f32", "metric": metric}
    if call == "stages":
        if metric == "l1":
            return {"call": call, "data": "mixture", "nA": _log(rng, 2000, 60000), "nB": _log(rng, 2000, 60000),
                    "d": rng.choice([16, 37, 64, 100, 128]), "dtype": rng.choice(["f32", "bf16"]), "metric": metric}
        return {"call": call, "data": "unit", "nA": _log(rng, 10000, 600000), "nB": _log(rng, 10000, 600000),
                "d": rng.choice([128, 256, 384]), "dtype": rng.choice(["fp8", "bf16"]), "metric": metric}
    if call == "batch":
        d = rng.choice([3, 3, 64])
        pairs = rng.randint(64, 400) if d == 3 else rng.randint(16, 100) if metric == "l2" else rng.randint(4, 24)
        return {"call": call, "data": "surface" if d == 3 else "mixture", "pairs": pairs, "lo": 256,
                "hi": 50000, "d": d, "dtype": "f32", "metric": metric, "size_seed": rng.randint(3, 1 << 20)}
    if call == "indexed":
        dtype = rng.choice(["f32", "bf16"])
        return {"call": call, "data": "uniform", "nA": _log(rng, 1000, 200000), "nB": _log(rng, 1000, 200000),
                "d": rng.choice([3, 128, 768]), "dtype": dtype, "metric": "l2"}
    if call == "exact":
        n = 20000 if metric == "l2" else 8000
        return {"call": call, "data": rng.choice(["mixture", "uniform"]), "nA": _log(rng, 500, n),
                "nB": _log(rng, 500, n), "d": rng.choice([3, 16, 40, 64, 128]), "dtype": rng.choice(["f32", "bf16"]),
                "metric": metric}
    if call == "crude":
        return {"call": call, "data": "mixture", "nA": _log(rng, 2000, 50000), "nB": _log(rng, 2000, 50000),
                "d": rng.choice([12, 64, 128]), "dtype": "f32", "metric": "l2", "repeats": rng.choice([1, 2, 4]),
                "window": rng.choice([4, 8, 16])}
    if call == "symmetric":
        return {"call": call, "data": "mixture", "nA": _log(rng, 2000, 60000), "nB": _log(rng, 2000, 60000),
                "d": rng.choice([10, 16, 24, 128]), "dtype": "f32", "metric": metric}
    return {"call": call, "data": "mixture", "nA": _log(rng, 500, 6000), "nB": _log(rng, 2000, 25000),
            "d": rng.choice([100, 128, 300]), "dtype": rng.choice(["f32", "bf16"]), "metric": metric,
            "T": _log(rng, 64, 3000)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mixture(nA, nB, d, g, clusters=100):
    c = torch.rand(clusters, d, device="cuda", generator=g) * 20 - 10
    cb = c + 0.5 * torch.randn(clusters, d, device="cuda", generator=g)
    out = []
    for n, centre in ((nA, c), (nB, cb)):
        lab = torch.randint(0, clusters, (n,), device="cuda", generator=g)
        out.append(centre[lab] + torch.randn(n, d, device="cuda", generator=g))
    return out


def _unit(nA, nB, d, g, clusters=1000, sigma=0.3):
    c = torch.nn.functional.normalize(torch.randn(clusters, d, device="cuda", generator=g), dim=1)
    out = []
    for n in (nA, nB):
        x = torch.randn(n, d, device="cuda", generator=g).mul_(sigma / math.sqrt(d))
        x += c[torch.randint(0, clusters, (n,), device="cuda", generator=g)]
        out.append(torch.nn.functional.normalize(x, dim=1))
    return out


def _uniform(nA, nB, d, g):
    return [torch.rand(n, d, device="cuda", generator=g) for n in (nA, nB)]


def _stored(x, dtype):
    """x as stored on the device: (tensor, row scales or None)."""
    if dtype == "f32":
        return x.contiguous(), None
    if dtype == "bf16":
        return x.to(torch.bfloat16), None
    s = x.abs().amax(dim=1) / 448.0
    s = torch.where(s > 0, s, torch.ones_like(s))
    return (x / s[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), s


def _widened(x, scales):
    """The values the library sees, in 64 bits."""
    if scales is not None:
        return x.view(torch.float8_e4m3fn).to(torch.float32).mul(scales[:, None]).double()
    return x.double()


def _pair(case, seed):
    make = {"mixture": _mixture, "unit": _unit, "uniform": _uniform}[case["data"]]
    return [_stored(x, case["dtype"]) for x in make(case["nA"], case["nB"], case["d"], _gen(seed))]


def _sizes(case):
    r = np.random.Generator(np.random.PCG64(case["size_seed"]))
    n = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), size=(case["pairs"], 2)))
    return n.astype(np.int64)


def _batch_sets(case, seed):
    """All pairs' sets as views of one tensor, each starting on a 16-byte boundary."""
    g, d, sizes = _gen(seed), case["d"], _sizes(case)
    P = case["pairs"]
    flat = torch.as_tensor(sizes.reshape(-1), device="cuda")
    room = (flat + 3) // 4 * 4
    start = (torch.cumsum(room, 0) - room).tolist()
    total = int(room.sum())
    pair = torch.repeat_interleave(torch.arange(P, device="cuda").repeat_interleave(2), room, output_size=total)
    if case["data"] == "surface":
        axes = 0.2 + 0.8 * torch.rand(P, 3, device="cuda", generator=g)
        w, i, j, k = torch.nn.functional.normalize(torch.randn(P, 4, device="cuda", generator=g), dim=1).unbind(1)
        q = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - k * w), 2 * (i * k + j * w),
                         2 * (i * j + k * w), 1 - 2 * (i * i + k * k), 2 * (j * k - i * w),
                         2 * (i * k - j * w), 2 * (j * k + i * w), 1 - 2 * (i * i + j * j)], 1).reshape(P, 3, 3)
        box = torch.rand(P, device="cuda", generator=g) < 0.5
        ball = torch.nn.functional.normalize(torch.randn(total, 3, device="cuda", generator=g), dim=1)
        cube = torch.rand(total, 3, device="cuda", generator=g) * 2 - 1
        face = torch.randint(0, 6, (total, 1), device="cuda", generator=g)
        cube.scatter_(1, face // 2, (face % 2).float() * 2 - 1)
        x = torch.where(box[pair, None], cube, ball) * axes[pair]
        x = torch.bmm(x[:, None, :], q[pair].transpose(1, 2))[:, 0]
        x += 0.01 * axes.amax(dim=1)[pair, None] * torch.randn(total, 3, device="cuda", generator=g)
    else:
        c = torch.rand(P, 10, d, device="cuda", generator=g) * 20 - 10
        cb = c + 0.5 * torch.randn(P, 10, d, device="cuda", generator=g)
        both = torch.stack([c, cb], 1).reshape(P * 2, 10, d)
        which = torch.repeat_interleave(torch.arange(2 * P, device="cuda"), room, output_size=total)
        x = both[which, torch.randint(0, 10, (total,), device="cuda", generator=g)]
        x += torch.randn(total, d, device="cuda", generator=g)
    x = x.contiguous()
    return [x[s:s + int(n)] for s, n in zip(start, sizes.reshape(-1))]


# ------------------------------------------------------------------ a program's state
_CTX = []


def _context():
    """The one context a program keeps, on torch's stream."""
    if not _CTX:
        _CTX.append(ch.ch_ctx_create(torch.cuda.current_device(), torch.cuda.current_stream()))
    return _CTX[0]


class _State:
    def __init__(self, case):
        self.case, self.sets, self.keep = case, [], []

    def add(self, x, scales, dtype):
        """Registers device data (adopted; fp8 rows are copied beside their scales)."""
        self.keep.append((x, scales))
        s = ch.ch_set_create(_context(), x, 2 if scales is None else 1, x.shape[0], x.shape[1], DTYPES[dtype][0], scales)
        self.sets.append(s)
        return s

    def __del__(self):
        for s in self.sets:
            ch.ch_set_destroy(s)


def prepare(case, seed):
    st = _State(case)
    call, metric = case["call"], METRICS[case["metric"]]
    st.seed = seed
    if call == "batch":
        views = _batch_sets(case, seed)
        sets = [st.add(v, None, case["dtype"]) for v in views]
        st.A, st.B = sets[0::2], sets[1::2]
        st.params = [ch.est_params(metric, LEVELS, PROJ, None, seed * 7919 + i, eps=EPS, sample_seed=seed + i)
                     for i in range(case["pairs"])]
        return st
    st.data = _pair(case, seed)
    st.hash = ch.hash_params(metric, LEVELS, PROJ, None, seed, window=case.get("window", 1),
                             repeats=case.get("repeats", 1))
    st.params = ch.est_params(metric, LEVELS, PROJ, None, seed, eps=EPS, sample_seed=seed + 1)
    nA, dev = case["nA"], "cuda"
    if call in ("stages", "crude"):
        st.b = torch.empty(nA, dtype=torch.int64, device=dev)
        st.D = torch.empty(nA, dtype=torch.float32, device=dev)
        st.level = torch.empty(nA, dtype=torch.uint8, device=dev)
    if call in ("stages", "scan"):
        st.T = _samples(case)
        st.idx = torch.randint(0, nA, (st.T,), device=dev, generator=_gen(seed + 2))
        st.w = torch.empty(nA, dtype=torch.int64, device=dev)
        st.min_d = torch.empty(st.T, dtype=torch.float32, device=dev)
        st.argmin = torch.empty(st.T, dtype=torch.int64, device=dev)
    if call == "exact":
        st.mins = torch.empty(nA, dtype=torch.float32, device=dev)
    if call == "indexed":  # the sets and their embeddings are resident, as a server keeps them
        for x, s in st.data:
            ch.ch_set_embed(_context(), st.add(x, s, case["dtype"]), st.hash)
    return st


def run(st):
    ctx, case = _context(), st.case
    call, metric = case["call"], METRICS[case["metric"]]
    if call == "batch":
        etas, status = ch.ch_estimate_batch(ctx, st.A, st.B, st.params)
        return {"eta": np.array(etas), "status": np.array(status)}
    if call == "indexed":
        return ch.ch_estimate(ctx, st.sets[0], st.sets[1], st.params)
    # the sets are registered for this call and released after it: their own passes belong to it
    one = _State(case)
    A, B = (one.add(x, s, case["dtype"]) for x, s in st.data)
    if call == "estimate":
        return ch.ch_estimate(ctx, A, B, st.params)
    if call == "symmetric":
        return list(ch.ch_estimate_sym(ctx, A, B, st.params))
    if call == "exact":
        return {"sum": ch.ch_exact(ctx, A, B, metric, 0, st.mins), "min": st.mins}
    out = {}
    if call in ("stages", "crude"):
        ch.ch_crude_nn(ctx, A, B, st.hash, st.b, st.D, st.level)
        out.update(b=st.b, D=st.D, level=st.level)
    if call == "stages":
        ch.ch_sample(ctx, st.D, case["nA"], st.T, st.seed + 1, st.idx, st.w)
        out.update(idx=st.idx, w=st.w)
    if call in ("stages", "scan"):
        ch.ch_sampled_nn(ctx, A, st.idx, st.T, B, metric, ch.CH_SCREEN_AUTO, 8, st.min_d, st.argmin)
        out.update(min=st.min_d, argmin=st.argmin)
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def _samples(case):
    return case.get("T") or math.ceil(4 * math.log(max(case["nA"], case["nB"], 2)) / EPS ** 2)


def work(case):
    d, elem = case["d"], DTYPES[case["dtype"]][1]
    l2, call = case["metric"] == "l2", case["call"]
    if call == "batch":
        n_bytes = n_flops = 0
        for a, b in _sizes(case).tolist():
            T = math.ceil(4 * math.log(max(a, b, 2)) / EPS ** 2)
            n_bytes += (a + b) * d * elem
            n_flops += 2 * T * b * d + (2 * (a + b) * d * PROJ if l2 else 0)
        return {"bytes": n_bytes + 8 * case["pairs"], "flops": n_flops}
    nA, nB = case["nA"], case["nB"]
    row = d * elem + (4 if case["dtype"] == "fp8" else 0)
    both = (nA + nB) * row
    embed = 2 * (nA + nB) * d * PROJ if l2 else 0
    if call == "exact":
        return {"bytes": both + 4 * nA, "flops": 2 * nA * nB * d}
    if call == "crude":
        k, w = case.get("repeats", 1), case.get("window", 1)
        return {"bytes": both + 13 * nA, "flops": k * embed + 2 * nA * k * w * d}
    T = _samples(case)
    if call == "scan":
        return {"bytes": (min(T, nA) + nB) * row + 20 * T, "flops": 2 * T * nB * d}
    if call == "indexed":  # the scan's rows and the resident embeddings
        return {"bytes": both + (nA + nB) * PROJ * 4, "flops": 2 * T * nB * d}
    if call == "symmetric":
        return {"bytes": both, "flops": embed + 2 * T * (nA + nB) * d}
    out = 21 * nA + 20 * T if call == "stages" else 0
    return {"bytes": both + out, "flops": embed + 2 * T * nB * d}


def exact(case, seed):
    """The minima of the brute force and of the bare scan in 64 bits; the other calls' outputs
    follow from draws that only the library makes."""
    if case["call"] not in ("exact", "scan"):
        return None
    (A, sA), (B, sB) = _pair(case, seed)
    p = 1.0 if case["metric"] == "l1" else 2.0
    A, B = _widened(A, sA), _widened(B, sB)
    if case["call"] == "scan":
        A = A[torch.randint(0, case["nA"], (case["T"],), device="cuda", generator=_gen(seed + 2))]
    step = max(1, (1 << 24) // B.shape[0])
    mins = torch.cat([torch.cdist(A[i:i + step], B, p=p, compute_mode="donot_use_mm_for_euclid_dist").amin(dim=1)
                      for i in range(0, A.shape[0], step)])
    if case["call"] == "scan":
        return {"min": mins, "argmin": None}
    return {"sum": float(mins.sum()), "min": mins}
