"""The line plans of the spectral solve (csrc/fft_plan.h), compiled with the
host C++ compiler and checked for every grid size without a GPU: which sizes
have one, the shared-memory layout of each (also above 48 KB and with four
lines per CTA), the transform that its steps make, and that asking for one
allocates nothing."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0812_2801_gb300", "csrc")


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fft_plan") / "driver")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC,
                    os.path.join(HERE, "host", "fft_plan_driver.cpp"), "-o", exe], check=True)
    return lambda *a: subprocess.run([exe, *map(str, a)], capture_output=True, text=True,
                                     check=True).stdout.strip()


def _smooth(n):
    for p in (2, 3, 5, 7, 11, 13):
        while n % p == 0:
            n //= p
    return n == 1


def test_every_13_smooth_size_has_a_plan(ask):
    rows = [[int(x) for x in line.split()] for line in ask("plans").split("\n")]
    assert [r[0] for r in rows] == [n for n in range(2, 1025) if _smooth(n)]
    # both sides of the two limits occur
    assert {r[1] for r in rows} == {4, 8}
    assert any(r[2] > 49152 for r in rows) and any(r[2] <= 49152 for r in rows)


def test_layouts_are_sound(ask):
    assert ask("layout") == "ok"


@pytest.mark.parametrize("n", [2, 3, 13, 16, 48, 64, 105, 189, 192, 343, 480, 729, 750, 768, 1000, 1024])
def test_steps_make_the_transform(ask, n):
    """Direct sums of up to 1024 unit-size terms: 1024 rounding errors of up to
    1e-16 each and of the roots' angles, over sqrt(n)."""
    assert float(ask("fft", n)) <= 1e-11


def test_plans_allocate_nothing(ask):
    """emd_poisson_static promises to allocate nothing; its plan is kept too."""
    assert ask("allocs") == "0"
