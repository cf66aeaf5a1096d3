"""The fixed-point collision (csrc/fixed64.cuh) on the host, against the same
equations in long double and beside FP64 arithmetic, over relaxation rates,
velocities, forces and cells with and without a particle.

Bounds, in result units u = 2^(E - 57) and apart from the final rounding to
FP64.  A product by a coefficient errs by at most 1.75 u, a square or a general
product by 2 u, a converted input by u/4, a table constant by u/2.  The
longest chain is the rest direction's: density product 1.75, three squares 6,
twice the relaxation product 3.5, constants and compensation 1.5, inputs (19
at u/4, through coefficients below 1, twice for x_0): 5.5; so 18.25 u.  A
covered cell adds 2 (S - F) B/4: at most the errors of S and F and 1.75, S's
rest direction with twice three products 12/2 (its unit is u/2), below 24 u.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2303_11811_gb300", "csrc")


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fixed64") / "check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "fixed64_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    r = []
    for line in out.splitlines():
        p = line.split()
        r.append(dict(kind=p[0], wild=int(p[1]), tau=float(p[2]), trt=int(p[3]), u=float(p[4]),
                      f=float(p[5]), worst=float(p[6]), force=float(p[7]), rms=float(p[8]),
                      rms64=float(p[9]), out=int(p[10]), cells=int(p[11])))
    return r


@pytest.mark.parametrize("kind", ["fluid", "mixed", "full", "none"])
def test_error_bound(rows, kind):
    """Every result within the unit bound, adversarial values included: a sum
    or product that overflowed would be off by orders of magnitude."""
    for r in rows:
        if r["kind"] == kind:
            assert r["worst"] <= 24.0 and r["force"] <= 24.0, r


def test_range(rows):
    """Ordinary flows are inside the fixed-point range, values of 1/8 and more
    outside it."""
    for r in rows:
        if r["u"] <= 1e-3:
            assert r["out"] == 0, r
        if r["wild"] and r["u"] == 0.3:
            assert r["out"] > 0.3 * r["cells"], r


def test_no_less_accurate_than_fp64(rows):
    """Near equilibrium, rms error over all settings of a kind, relative to the
    cell's largest value: at most that of FP64 arithmetic."""
    for kind in ("fluid", "mixed", "full", "none"):
        sel = [r for r in rows if r["kind"] == kind and not r["wild"]
               and r["u"] in (1e-5, 1e-3, 2e-2) and r["f"] <= r["u"]]
        fixed = sum(r["rms"] ** 2 for r in sel) ** 0.5
        fp64 = sum(r["rms64"] ** 2 for r in sel) ** 0.5
        assert fixed <= fp64, (kind, fixed, fp64)
