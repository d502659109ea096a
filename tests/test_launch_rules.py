"""The launch rules (csrc/launch_rules.h), compiled with the host C++ compiler
and checked over their whole range without a GPU."""
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
    exe = str(tmp_path_factory.mktemp("launch_rules") / "driver")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC,
                    os.path.join(HERE, "host", "launch_rules_driver.cpp"), "-o", exe], check=True)

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True,
                             check=True).stdout.split()
        assert len(out) == len(lines)
        return [int(x) for x in out]
    return run


def test_gram_chunks_never_lengthen_the_sums(ask):
    """An entry of X^H Y is one FP64 chain per row chunk: the chains are no
    longer than with n^3 / 4096 chunks (at most 64), whatever the number of
    states, and a chunk has at least 96 rows."""
    cases = [(n ** 3, m) for n in (8, 16, 24, 33, 48, 64, 96, 128, 160)
             for m in (1, 9, 16, 17, 64, 96, 97, 138, 200, 512, 800, 1100)]
    for (n3, m), c in zip(cases, ask([f"gram {a} {b}" for a, b in cases])):
        assert c >= max(1, min(64, n3 // 4096)), (n3, m)
        assert c == 1 or n3 // c >= 96, (n3, m)
        # small m: the GPU is filled as far as 96 rows per chunk allow
        tiles = (-(-m // 16)) ** 2
        assert c * tiles >= min(16 * 152, n3 // 96 * tiles)
