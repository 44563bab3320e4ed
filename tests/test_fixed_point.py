"""The fixed-point arithmetic of the FP64 link update (csrc/su2_fixed.cuh),
compiled for the host, against long double: each function within the error
its place in the update allows, and the new link closer to the exact one than
the same update in doubles, over couplings from 0.1 to 1e5 and links from
ordered to random (all components together; the vector part alone up to the
coupling FIX_BETA_MAX, above which the kernels take the FP64 sequence)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1104_5432_gb300", "csrc")


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_point")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "fixed_point_main.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return [ln.split() for ln in out.splitlines()]


def test_functions(lines):
    got = {ln[0]: [float(x) for x in ln[1:]] for ln in lines if ln[0] not in ("link", "vector")}
    u = 2.0 ** -57
    # -ln u at 2^-61 (u > 1/2) and 2^-57, a truncation or two each
    assert got["ln"][0] <= 2.0 ** -59 and got["ln"][1] <= 2 * u
    assert max(got["arc"]) <= u
    assert got["root"][0] <= 2.0 ** -59 and got["root"][1] <= u
    # a link component to one unit of 2^-61, a double to half a unit in its
    # last place (the lines carry four digits)
    assert got["convert"][0] <= 1.001 * 2.0 ** -61 and got["convert"][1] <= 1.001 * 2.0 ** -53
    worst, worst_d, rms, rms_d = got["haar"]
    assert worst <= worst_d and rms <= 0.5 * rms_d


def test_new_links_are_no_further_off_than_in_doubles(lines):
    rows = [[float(x) for x in ln[1:]] for ln in lines if ln[0] == "link"]
    assert len(rows) == 18
    for beta, spread, n, flips, worst, worst_d, rms, rms_d in rows:
        assert n > 10000 and flips == 0, (beta, spread)
        assert rms <= 0.5 * rms_d, (beta, spread, rms, rms_d)
        assert worst <= worst_d, (beta, spread, worst, worst_d)


def test_vector_parts_up_to_the_largest_coupling(lines):
    """At coupling beta the vector part of a link is of the size of beta^-1/2 and
    a double's error shrinks with it, an absolute error at 2^-61 .. 2^-57 does
    not: up to FIX_BETA_MAX the fixed point is still the closer, and at 1e5,
    where the kernels do not use it, it is not (so the limit is needed)."""
    limit = [float(ln[1]) for ln in lines if ln[0] == "limit"][0]
    rows = [[float(x) for x in ln[1:]] for ln in lines if ln[0] == "vector"]
    assert [r[0] for r in rows] == [2.3, 2.3, limit, limit, 1e5, 1e5]
    for beta, spread, n, flips, worst, worst_d, rms, rms_d in rows:
        assert n > 50000 and flips == 0, (beta, spread)
        if beta <= limit:
            assert rms <= 0.6 * rms_d and worst <= worst_d, (beta, spread, rms, rms_d, worst, worst_d)
        else:
            assert rms > rms_d, (beta, spread, rms, rms_d)
