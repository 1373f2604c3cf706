"""The error bound of the certified exact l2 scan against the scores the tensor cores give,
in 64 bits.  The bound's operand rounding and norm terms follow from the formats; its
accumulation term (each of the d products added with an error of at most 4 x 2^-23 of
|q||b|) is a model of hardware whose internals are not documented, so it is measured here:
on operands that TF32 and BF16 hold exactly the whole error must stay within a quarter of
that term -- the model without its factor of four -- and on arbitrary ones within the whole
bound."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2307_03043_gb300 import binding as ch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
T, NB = 256, 512
U23 = 2.0 ** -23


@pytest.fixture(scope="module")
def scores(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03043_gb300 import build
    lib = build.build()
    so = str(tmp_path_factory.mktemp("scores") / "screen_scores.so")
    cmd = [build._nvcc(), "-shared", os.path.join(ROOT, "tests", "native", "screen_scores.cu"), "-o", so, lib,
           "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib)]
    r = subprocess.run(cmd + build.NVCC_FLAGS, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    h = ctypes.CDLL(so)
    p, i, q = ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong
    h.scores_workspace.restype, h.scores_workspace.argtypes = q, [q, q, i, i, i]
    h.scores_run.argtypes = [p, p, i, q, q, i, p, q, p, p, p, p, i]
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def run(Q, B, dtype):
        """(class minima [parts, T, 32], first columns) of the screen of samples Q against B."""
        d, es = Q.shape[1], 4 if dtype == ch.CH_F32 else 2
        tq, tb = (torch.from_numpy(x).cuda().to(torch.float32 if dtype == ch.CH_F32 else torch.bfloat16).contiguous()
                  for x in (Q, B))
        idx = torch.arange(T, device="cuda")
        idx[(2 * torch.arange(16, device="cuda") + 1) * T // 32] = -1  # the pilots: no votes, so the screen runs
        size = h.scores_workspace(T, NB, d, dtype, sms)
        work = torch.zeros(size, dtype=torch.uint8, device="cuda")
        norms = torch.empty(NB, device="cuda")
        m, am = torch.empty(T, device="cuda"), torch.empty(T, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert h.scores_run(tq.data_ptr(), tb.data_ptr(), dtype, T, NB, d, idx.data_ptr(), T, norms.data_ptr(),
                            work.data_ptr(), m.data_ptr(), am.data_ptr(), sms) == 0
        al = lambda n: (n + 255) & ~255
        at = 256 + al(T * 4) + al(T * 8) + al(T * d * es)
        parts = (size - at - 768) // (3 * T * 32 * 4)
        n = parts * T * 32
        part_s = work[at:at + 4 * n].view(torch.float32).reshape(parts, T, 32).cpu().numpy()
        part_i = work[at + al(4 * n):at + al(4 * n) + 4 * n].view(torch.int32).reshape(parts, T, 32).cpu().numpy()
        live = (idx >= 0).cpu().numpy()
        return part_s[:, live], part_i[:, live], live

    return run


def _terms(d, dtype):
    c_in = 2.0 ** -9 * (1 + 2.0 ** -10) if dtype == ch.CH_F32 else 0.0
    a = 2 * (c_in + 4 * d * U23) + 2.0 ** -22
    b1 = (d + 2) * U23
    shrink = np.float32((1 - a / 2 - b1) * (1 - U23))
    return c_in, a, b1, float(shrink)


def _data(kind, d, exact_bits, seed):
    g = np.random.default_rng(seed)
    q, b = g.standard_normal((T, d)), g.standard_normal((NB, d))
    if kind == "positive":  # every product adds up
        q, b = np.abs(q), np.abs(b)
    elif kind == "cancelling":  # large products that cancel in pairs, small ones left
        q[:, 1::2], b[:, 1::2] = q[:, ::2], -b[:, ::2]
        q[:, ::16] *= 1024
        b[:, 3::16] *= 2.0 ** -9
    elif kind == "spread":  # forty powers of two
        q *= 2.0 ** g.integers(-20, 20, q.shape)
        b *= 2.0 ** g.integers(-20, 20, b.shape)
    elif kind == "mixed_rows":  # norms from 2^-15 to 2^15 side by side
        q *= 2.0 ** g.integers(-15, 15, (T, 1))
        b *= 2.0 ** g.integers(-15, 15, (NB, 1))
    elif kind == "ones":  # mantissas of ones: rounding and truncation at their worst
        q, b = (np.float64(2 - 2.0 ** -23) * 2.0 ** g.integers(-1, 2, x.shape) for x in (q, b))
    elif kind == "far":
        q, b = q + 1000, b + 1000
    q, b = q.astype(np.float32), b.astype(np.float32)
    if exact_bits:  # keep 7 explicit mantissa bits: exact in TF32 and BF16
        q, b = ((x.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32) for x in (q, b))
    return np.ascontiguousarray(q), np.ascontiguousarray(b)


KINDS = ["normal", "positive", "cancelling", "spread", "mixed_rows", "ones", "far"]


@pytest.mark.parametrize("dtype", [ch.CH_F32, ch.CH_BF16], ids=["tf32", "bf16"])
@pytest.mark.parametrize("d", [8, 32, 128, 384, 1024, 1408])
def test_scores_stay_within_the_bound(scores, dtype, d):
    c_in, a, b1, shrink = _terms(d, dtype)
    worst = {}
    for kind in KINDS:
        for exact_bits in (True, False):
            if dtype == ch.CH_BF16 and not exact_bits:
                continue  # BF16 operands are what the set holds: always exact
            Q, B = _data(kind, d, exact_bits, d)
            S, first, live = scores(Q, B, dtype)
            Q64, B64 = Q[live].astype(np.float64), B.astype(np.float64)
            nb = (B64 * B64).sum(1)
            X = shrink * nb[None] - 2 * (Q64 @ B64.T)  # the scores without error
            qn, bn = np.linalg.norm(Q64, axis=1), np.sqrt(nb)
            acc = 2 * 4 * d * U23 * qn[:, None] * bn[None]           # the accumulation term
            rest = 2.0 ** -22 * qn[:, None] * bn[None] + b1 * nb[None]  # last fma, norms
            bound = acc / 4 + rest if exact_bits else a * qn[:, None] * bn[None] + b1 * nb[None]
            ratio = 0.0
            for p in range(S.shape[0]):
                for cls in range(32):
                    col = first[p, :, cls]
                    rows = np.nonzero(col >= 0)[0]
                    c4 = col[rows, None] + 32 * np.arange(4)[None]  # the entry's columns
                    ok = c4 < NB
                    c4 = np.where(ok, c4, 0)
                    x = np.where(ok, X[rows[:, None], c4], np.inf)
                    lim = np.where(ok, bound[rows[:, None], c4], 0.0).max(1)
                    err = np.abs(S[p, rows, cls].astype(np.float64) - x.min(1))
                    ratio = max(ratio, float((err / lim).max()))
            worst[kind, exact_bits] = ratio
    print(d, {k: round(v, 4) for k, v in worst.items()})
    assert max(worst.values()) <= 1.0, worst
