"""Partner chunks of launches with few items (pick_split_small, csrc/tc_setup.cpp), on the CPU: the count
of pick_split unless 9 .. 32 chunks, within two waves of CTAs, cut waves x pairs per CTA by a tenth."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_07420_gb300", "csrc")


def _rounds(items, partners, sms, s):
    return -(-items * s // sms) * -(-partners // s)


def test_pick_split_small(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "small_probe")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe,
                        os.path.join(ROOT, "tests", "host", "small_probe.cpp"), os.path.join(CSRC, "tc_setup.cpp")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    cases = [(i, m, sms) for i in (1, 3, 7, 12, 14, 32, 64, 512) for m in (1, 7, 8, 9, 12, 16, 40, 256)
             for sms in (1, 76, 152)]
    out = subprocess.run([exe], input="\n".join("%d %d %d" % c for c in cases), capture_output=True, text=True)
    got = [tuple(int(x) for x in line.split()) for line in out.stdout.splitlines()]
    assert len(got) == len(cases)
    for (items, partners, sms), (s0, s) in zip(cases, got):
        assert 1 <= s <= max(1, min(32, partners))
        better = [x for x in range(9, min(32, partners) + 1) if items * x <= 2 * sms
                  and 10 * _rounds(items, partners, sms, x) <= 9 * _rounds(items, partners, sms, s0)]
        if not better:
            assert s == s0
        else:
            assert s in better and _rounds(items, partners, sms, s) == min(_rounds(items, partners, sms, x)
                                                                           for x in better)
    assert got[cases.index((12, 12, 152))][1] == 12      # one pair per CTA instead of one or two
