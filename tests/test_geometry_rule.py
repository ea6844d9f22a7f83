"""The library's choices by size (csrc/lorads_geometry.h), compiled for the host: the CTAs of a single
solve, the operators' forms for short rows."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_09133_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lorads_geometry.h"
int main(int argc, char** argv) {
  if (argc == 5 && argv[1][0] == 's') {
    std::printf("%d\n", (int)lorads::short_rows(atol(argv[2]), atol(argv[3]), atoi(argv[4])));
    return 0;
  }
  if (argc == 6 && argv[1][0] == 'u') {
    const int G = lorads::unit_lanes((lorads::UnitWork)atoi(argv[2]), atoi(argv[3]), atol(argv[4]),
                                     atoi(argv[5]));
    std::printf("%d\n%d\n", G, lorads::unit_count(atoi(argv[3]), G));
    return 0;
  }
  for (int i = 1; i + 5 < argc; i += 6) {
    lorads::SolveSize s{};
    s.n = atol(argv[i]);
    s.fp64 = atoi(argv[i + 1]) != 0;
    s.diag_only = atoi(argv[i + 2]) != 0;
    s.threads = atoi(argv[i + 3]);
    s.sms = atoi(argv[i + 4]);
    s.lanes = atoi(argv[i + 5]);
    std::printf("%d\n", lorads::default_ctas(s));
  }
}
"""


@pytest.fixture(scope="module")
def ctas(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("geometry")
    (d / "g.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "g.cpp"), "-o", str(d / "g")],
                   check=True)

    def run(cases):
        args = [str(int(x)) for c in cases for x in (*c, 4)[:6]]
        return call(*args)

    def call(*args):
        out = subprocess.run([str(d / "g"), *map(str, args)], capture_output=True, text=True,
                             check=True)
        return list(map(int, out.stdout.split()))
    run.call = call
    return run


def test_a_cta_size_of_the_one_cta_kernel_keeps_small_solves_there(ctas):
    """352 and 384 threads fit only the one-CTA kernel: below n = 512 they choose it, in both forms."""
    cases = [(n, fp64, diag, th, 152) for n in (1, 39, 40, 60, 255, 256, 300, 511)
             for fp64 in (0, 1) for diag in (0, 1) for th in (352, 384)]
    assert ctas(cases) == [1] * len(cases)


def test_thresholds(ctas):
    one = [(39, 1, 0, 0, 152), (255, 1, 1, 0, 152), (511, 0, 0, 0, 152), (511, 0, 1, 0, 152)]
    assert ctas(one) == [1] * len(one)
    more = [(40, 1, 0, 0, 152), (40, 1, 0, 320, 152), (256, 1, 1, 0, 152), (256, 1, 1, 320, 152)]
    assert min(ctas(more)) > 1
    whole = [(512, f, d, 0, 148) for f in (0, 1) for d in (0, 1)]
    assert ctas(whole) == [148] * len(whole)


def test_no_more_ctas_than_the_rows_fill(ctas):
    """From the thresholds to n = 511 an FP64 solve takes the CTAs that its rows fill: with fewer rows than
    that many SMs hold, callers side by side share the GPU."""
    diag = [(n, 1, 1, th, 152, lanes) for n in (256, 257, 300, 511) for th in (0, 128, 256, 320)
            for lanes in (1, 2, 4, 8, 32)]
    want = [max(2, min(152, -(-n * lanes // (th or 128)))) for n, _, _, th, _, lanes in diag]
    assert ctas(diag) == want
    general = [(n, 1, 0, threads, 152) for n in (40, 41, 60, 120, 400, 511) for threads in (0, 320)]
    want = [max(2, min(152, -(-n * 32 // (th or 128)))) for n, _, _, th, _ in general]
    assert ctas(general) == want
    assert ctas([(511, 1, 0, 0, 100)]) == [100]


def test_short_rows(ctas):
    """At most one entry per sub-team of a warp on average."""
    for lanes in (2, 4, 8, 32, 64):
        S = 32 // min(lanes, 32)
        for n in (1, 20000):
            assert ctas.call("s", n, n * S, lanes) == [1]
            assert ctas.call("s", n, n * S + 1, lanes) == [0]


def test_unit_lanes(ctas):
    """FP64 operators: at most 8 units per lane and a lane for every unit at most; two lanes with many
    rows, eight with few; no widening where it was measured to lose."""
    SDDMM_DIAG, SDDMM, HESSIAN, SPMM = range(4)

    def lanes(work, ld, rows):
        G, N = ctas.call("u", work, ld, rows, 152)
        assert G in (2, 4, 8, 16) and N <= 8 and (N - 1) * G < ld // 2 <= N * G
        return G

    for work in range(4):
        for ld in range(4, 257, 4):
            least = next(G for G in (2, 4, 8, 16) if G * 8 >= ld // 2)
            if work == SPMM and least < 8 and -(-(ld // 2) // least) == 8:
                least *= 2
            assert lanes(work, ld, 10 ** 7) == least
            few = lanes(work, ld, 100)
            assert few == max(least, min(8, 1 << (ld // 2).bit_length() - 1))
            sizes = [lanes(work, ld, rows) for rows in (100, 1000, 10 ** 4, 10 ** 5, 10 ** 6)]
            assert sizes == sorted(sizes, reverse=True)
    assert lanes(SDDMM_DIAG, 12, 30000) == 2 and lanes(SDDMM, 12, 30000) == 2
    assert lanes(HESSIAN, 12, 30000) == 2 and lanes(HESSIAN, 32, 20000) == 4
    assert lanes(HESSIAN, 48, 12000) == 8
    assert lanes(SDDMM_DIAG, 32, 10000) == 4 and lanes(SPMM, 48, 10000) == 8
    assert lanes(SPMM, 32, 10 ** 6) == 4 and lanes(SPMM, 48, 80000) == 8 and lanes(SPMM, 20, 80000) == 2
