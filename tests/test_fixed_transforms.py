"""Rounding of the 64-bit fixed-point transforms (csrc/tc_fixed.cuh, codelets of csrc/tc_fft.cuh) on the CPU,
against long double: every box that runs them, both directions, spectra flat and falling off.

Bounds.  A rounding to nearest is off by at most half a unit, a product by the cut digits a quarter more; an
output of a codelet has passed at most six such roundings per component, so its error is of variance
v <= 6 (0.75)^2 / 3 = 1.1 per component.  Independent errors of the first pass are summed over N^2 pencil
values, those of the second over N: sqrt(2 v (1 + 1/N + 1/N^2)) N < 1.6 N units in the root mean square of a
complex output, and five times that at the worst of at most 24^3 outputs.  (Errors of products that are cut off have
one sign and add up to as much as 2500 units at one point.)
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_07420_gb300", "csrc")


def _probe(path, *flags):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = str(path / "fixed_probe")
    r = subprocess.run([gxx, "-std=c++17", "-w", *flags, "-I", os.path.join(ROOT, "tests", "host", "cuda"), "-I", CSRC,
                        "-o", exe, os.path.join(ROOT, "tests", "host", "fixed_probe.cpp")],
                       capture_output=True, text=True)
    if "-fsanitize=undefined" in flags and "ubsan" in r.stderr:
        pytest.skip("no sanitizer library")
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0
    return out


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    return [line.split() for line in _probe(tmp_path_factory.mktemp("fixed"), "-O2").stdout.splitlines()]


def test_no_undefined_arithmetic(tmp_path):
    """No signed overflow and no left shift of a negative value in the transforms and their scales."""
    assert _probe(tmp_path, "-O1", "-fsanitize=undefined").stderr == ""


@pytest.mark.parametrize("direction", ["inv", "fwd"])
@pytest.mark.parametrize("box", [(24, 17), (20, 17), (18, 17), (16, 13), (16, 16), (15, 15), (12, 12), (9, 9)])
def test_fixed_point_rounding(lines, direction, box):
    got = [x for x in lines if x[0] == direction and (int(x[1]), int(x[2])) == box]
    assert [x[3] for x in got] == ["flat", "gauss", "exponential"]
    n = box[0]
    for x in got:
        rms, top, unit = (float(v) for v in x[4:7])
        assert rms < 1.6 * n * unit, x
        assert top < 8.0 * n * unit, x
