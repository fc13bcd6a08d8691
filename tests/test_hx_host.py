"""The block-scaled arithmetic (csrc/pp_hx.cuh) on the host: the library's own header, compiled by g++ with the
compiler's check of signed overflow, around the recipes of the line kernels (tests/c/hx_lines.cpp), against direct
sums in long double.  No sum may leave 32 bits, and a line may differ by a quarter of the solver's 1e-12 (a solve
takes four transforms)."""
import concurrent.futures as cf
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1909_05423_gb300", "csrc")
TOL = 2.5e-13


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("hx") / "hx_lines")
    cmd = ["g++", "-O2", "-std=c++17", "-Wall", "-ffp-contract=off", "-fcx-limited-range",
           "-fsanitize=signed-integer-overflow", "-I", os.path.join(HERE, "c", "host_cuda"), "-I", CSRC,
           os.path.join(HERE, "c", "hx_lines.cpp"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


# random: dense lines.  fours, few: lines of a few cells, whose scale the sum of magnitudes sets.  aligned: lines whose
# cells add up in one of the values that the butterflies take re + im or re - im of.  modes: one or two coefficients.
# huge: magnitudes whose sum is beyond FP32's range while every result is within it.
@pytest.mark.parametrize("family", ["random", "fours", "few", "aligned", "modes", "huge"])
def test_lines(exe, family):
    with cf.ThreadPoolExecutor(5) as ex:
        runs = list(ex.map(lambda M: subprocess.run([exe, family, str(M)], capture_output=True, text=True, timeout=300),
                           [64, 128, 256, 512, 1024]))
    for r in runs:
        assert r.returncode == 0 and r.stderr == "", r.stderr[:500]
        rows = [line.split() for line in r.stdout.splitlines()]
        assert len(rows) == 10
        for kind, m, lines, err in rows:
            assert float(err) <= TOL, (family, kind, m, err)
