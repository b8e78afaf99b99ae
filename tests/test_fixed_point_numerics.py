"""The arithmetic of csrc/fx.cuh on the host (tests/fixed_point_host.cpp compiles it with a C++ compiler),
against long double and beside the FP64 path, over propagators whose rows and columns differ in size and
tolerances that let every pivot pass."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="no host C++ compiler")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fx") / "fixed_point_host")
    subprocess.run(["g++", "-O2", "-w", "-std=c++17", "-I", os.path.join(HERE, "host_stub"), "-o", exe,
                    os.path.join(HERE, "fixed_point_host.cpp")], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [float(x) for x in out.split()]

    return run


@pytest.mark.parametrize("pivots", [13, 4096])  # the default pivot guard, and none
@pytest.mark.parametrize("pattern, spread", [("rows", 0), ("rows", 4), ("rows", 10), ("rows", 30), ("cols", 4),
                                             ("cols", 20), ("both", 4), ("onerow", 8), ("onecol", 8), ("onecol", 30)])
@pytest.mark.parametrize("n", [2, 3, 6, 12, 18])
def test_solves(host, n, pattern, spread, pivots):
    """An accepted solve has a unit in 2^55 times a spread of 2^3 at every place where FP64 has one in
    2^53: four times the error, and sixteen in the extremes, where a small w meets a large pivot (2^-47)."""
    blocks, refused, sinks, left, med, worst, med64, worst64 = host(n, pattern, spread, pivots, 10)[:8]
    assert med <= 4 * med64 + 2.0 ** -53 and worst <= 16 * worst64 + 2.0 ** -47
    if spread == 0:
        assert refused <= 0.01 * blocks and left <= 0.05 * sinks


@pytest.mark.parametrize("guard", [10, 30, 4096])  # the default lemma guard, a lower one, and none
@pytest.mark.parametrize("pattern, spread", [("rows", 0), ("rows", 4), ("cols", 4), ("cols", 20), ("onecol", 8), ("onerow", 8),
                                             ("unused", 5), ("unused", 10), ("unused", 25), ("unused", 45)])
@pytest.mark.parametrize("n", [3, 6, 12, 18])
def test_determinants(host, n, pattern, spread, guard):
    """An accepted determinant: a value of 2^-7 of the scale is off by a few units of 2^-56 of it, 2^-46 at
    the most; beyond that as the solves, four times FP64's error and sixteen in the extremes."""
    out = host(n, pattern, spread, 13 if guard == 10 else 4096, guard)
    accepted, left, med, worst, med64, worst64 = out[8:14]
    assert med <= 4 * med64 + 2.0 ** -49 and worst <= 16 * worst64 + 2.0 ** -46
    if spread == 0:
        assert left <= 0.005 * accepted


@pytest.mark.parametrize("pattern, spread, flat", [
    ("rows", 0, 1), ("rows", 1, None), ("rows", 2, None), ("rows", 3, 0), ("rows", 30, 0), ("cols", 2, None), ("cols", 3, 0),
    ("cols", 20, 0), ("both", 2, None), ("both", 3, 0), ("decay", 1, None), ("decay", 3, 0), ("decay", 8, 0), ("onerow", 4, 0),
    ("onecol", 4, 0), ("flip", 8, 0), ("unused", 3, 1), ("unused", 40, 1)])
@pytest.mark.parametrize("n", [4, 6, 12, 18])
def test_flat_propagators(host, n, pattern, spread, flat):
    """What the scan lets pass is as good in fixed point as in FP64: three times its error at most, eight in
    the extremes (the maxima of some 10 000 determinants); rows or columns over 2^3 do not pass."""
    out = host(n, pattern, spread, 13, 10)
    accepted, left, med, worst, med64, worst64, is_flat = out[8:]
    assert flat is None or is_flat == flat
    if is_flat:
        assert accepted > 0 and med <= 3 * med64 and worst <= 8 * worst64
