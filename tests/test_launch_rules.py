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


def _complex64_zchunk(n, M, cols):
    best, cost = n, None
    for nz in range(1, max(1, n // 4) + 1):
        zc = -(-n // nz)
        load = (cols * -(-n // zc) + 151) // 152
        c = max(load, 1.4) * (zc + 2 * M + 2)
        if cost is None or c < 0.98 * cost:
            best, cost = zc, c
    return best


def _double_float_zchunk(n, M, cols):
    best, cost = n, 1e300
    for nz in range(1, n // 4 + 1):
        zc = -(-n // nz)
        load = (cols * -(-n // zc) + 151) // 152
        t = max(load, 1.4) * (zc + 0.3 * 2 * M)
        if t < 0.98 * cost:
            best, cost = zc, t
    return best


def test_one_zchunk_rule_for_both_stages(ask):
    """The chunks that the two stages were measured with, each by the formula it
    had of its own."""
    cases = [(n, M, cols) for n in (8, 16, 31, 48, 64, 96, 120, 160, 1024) for M in (1, 2, 3, 4)
             for cols in (1, 7, 36, 72, 151, 152, 153, 640, 2304, 100000)]
    got = ask([f"zchunk {n} {M} {c} 1 2" for n, M, c in cases] +
              [f"zchunk {n} {M} {c} 0.3 0" for n, M, c in cases])
    assert got == [_complex64_zchunk(*c) for c in cases] + [_double_float_zchunk(*c) for c in cases]


def test_gather_splits_fit_their_scratch(ask):
    cases = [(p, c) for p in (1, 6, 227, 228, 229, 455, 456, 457, 911, 912, 1823, 1824, 50000)
             for c in (1, 4095, 4096, 8191, 8192, 16383, 16384, 10 ** 6)]
    for (pairs, cap), s in zip(cases, ask([f"split {p} {c}" for p, c in cases])):
        assert s in (1, 2, 4, 8)
        if s > 1:                                     # scratch: 3648 CTAs, 1824 counters
            assert pairs * s < 3648 and pairs < 1824
            assert cap // 2 >= 1024 * s               # a full round of 1024 entries each
