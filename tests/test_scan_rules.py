"""The exact scan's dispatch rules (host code of the built library, no GPU): which
calls the certified and the chained forms take, at the edges of what their 32-bit
column and sample numbers, row reads and loads can hold."""
import os
import subprocess

import pytest

from paper_2307_03043_gb300 import binding as ch
from paper_2307_03043_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("rules") / "scan_rules")
    src = os.path.join(ROOT, "tests", "native", "scan_rules.cu")
    cmd = [build._nvcc(), src, "-o", exe, lib, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib)]
    r = subprocess.run(cmd + build.NVCC_FLAGS, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def ask(*cases):
        text = "\n".join(" ".join(map(str, c)) for c in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
        return [(int(out[2 * i]), int(out[2 * i + 1])) for i in range(len(cases))]

    return ask


def _case(T=4096, nB=100000, d=64, dtype=ch.CH_F32, nA=None, alignA=0, alignB=0):
    return dtype, T if nA is None else nA, nB, d, T, alignA, alignB


def test_samples_past_32_bits_take_neither_form(rules):
    """A sample's number goes through a 32-bit list: 2^31 samples and more (brute
    force over that many points, or that many draws) stay with the plain scan."""
    most = 2 ** 31
    for dtype, d in ((ch.CH_BF16, 8), (ch.CH_F32, 8)):
        ok, past, far = rules(_case(most - 1, 1000, d, dtype), _case(most, 1000, d, dtype),
                              _case(most + 12345, 1000, d, dtype))
        assert ok == (1, 1) and past == (0, 0) and far == (0, 0)
    drawn = rules(_case(most, 1000, 8, ch.CH_BF16, nA=5000))
    assert drawn == [(0, 0)]


def test_rules_at_their_other_edges(rules):
    cases = {
        (1, 1): [_case(), _case(d=384, dtype=ch.CH_BF16)],
        (0, 1): [_case(d=33), _case(d=64, alignB=4), _case(d=64, alignA=8), _case(d=64, dtype=ch.CH_FP8E4M3)],
        (1, 0): [_case(T=256, nB=40000, d=16), _case(T=1024, nB=1024, d=32), _case(T=3000, nB=2000, d=16),
                 _case(T=3000, nB=4000, d=8), _case(T=3000, nB=2000, d=40)],
        (0, 0): [_case(d=4), _case(nB=2 ** 31), _case(T=100), _case(T=512, nB=200, d=16),
                 _case(T=1024, nB=1024, d=16), _case(T=3000, nB=3000, d=8), _case(T=1000, nB=2000, d=64)],
    }
    for want, cs in cases.items():
        assert rules(*cs) == [want] * len(cs), want
