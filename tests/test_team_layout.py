"""Shared memory of the team kernels over every mechanism size that the loader
accepts, from the layout header as the host compiles it (no GPU).
"""
import shutil
import subprocess

import pytest

from paper_1608_05794_gb300.build import ARCH, CSRC, INCLUDE, _nvcc

MAX_SMEM = 227 * 1024  # dynamic and static shared memory of a CTA

PROGRAM = r"""
#include <cstdio>
#include "ck_layout.cuh"
// lines "S R typed" -> sizes in bytes
int main() {
  int S, R, typed;
  while (std::scanf("%d %d %d", &S, &R, &typed) == 3) {
    const ck::TeamChunks c = ck::team_chunks(S, R, typed);
    auto scratch = [&](int chunk) {  // as the loader sizes a table: the typed reactions come last
      int most = 0;
      for (int b = 0; b < R; b += chunk) {
        const int end = b + chunk < R ? b + chunk : R, from = b > R - typed ? b : R - typed;
        if (end - from > most) most = end - from;
      }
      return ck::JAC_PER_RXN * chunk + most;
    };
    ck::DevMech d{};
    d.S = S;
    d.R = R;
    d.n = S + 1;
    d.first_typed = R - typed;
    d.rhs_chunk = c.rhs;
    d.wide.scratch = scratch(c.wide);
    d.narrow.scratch = scratch(c.narrow);
    std::printf("%d %d %d %zu %zu %d\n", c.rhs, c.wide, c.narrow, 8 * ck::Ros4Layout(d, true).doubles,
                8 * ck::Ros4Layout(d, false).doubles, 8 * ck::rhs_doubles(d));
  }
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    try:
        nvcc = _nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cu").write_text(PROGRAM)
    subprocess.run([nvcc, *ARCH, "-std=c++17", "-I", CSRC, "-I", INCLUDE, "--expt-relaxed-constexpr",
                    str(d / "layout.cu"), "-o", str(d / "layout")], check=True)

    def run(cases):
        text = "".join("%d %d %d\n" % c for c in cases)
        out = subprocess.run([str(d / "layout")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def test_every_accepted_size_fits_a_cta(layout):
    cases = [(S, R, typed) for S in (1, 10, 23, 24, 31, 32, 33, 53, 63, 64, 100, 111, 112, 127, 128)
             for R in (0, 1, 20, 325, 511, 512, 513, 784, 2000, 28001, 32767)
             for typed in sorted({0, R // 6, R})]
    for (S, R, typed), (rhs, wide, narrow, ros4, ros4_narrow, rates) in zip(cases, layout(cases)):
        assert max(ros4, ros4_narrow) <= MAX_SMEM - 256, (S, R, typed)
        # the kernels without a matrix: eight vectors, the species arrays and the rates
        assert rates + 8 * (8 * (S + 1) + 64 + 4 * (S + 1) + 2 * S) <= MAX_SMEM - 256, (S, R, typed)
        assert 1 <= rhs <= max(R, 1) and 1 <= wide <= max(R, 1) and 1 <= narrow <= max(R, 1)


def _ctas(size):
    return 228 * 1024 // (size + 1024 + 80)


def test_chunks_follow_the_shared_memory(layout):
    # no step in the number of passes just above the sizes of any one mechanism:
    # as many reactions at a time as the residency of the kernel leaves room for
    sizes = [(S, R, R // 7) for S in (10, 23, 24, 40, 53, 58, 64, 80, 106, 111, 112, 128)
             for R in (20, 200, 325, 340, 400, 650, 784, 785, 800, 852, 1568, 5000)]
    for (S, R, typed), (rhs, wide, narrow, ros4, ros4_narrow, _) in zip(sizes, layout(sizes)):
        n = S + 1
        species = 64 + 4 * (S + 1) + 2 * S
        before = (n * (n | 1) + 5 * n + (n + 1) // 2 + 1 + species) & ~1  # matrix, vectors, species arrays, row table
        want = 8 if n <= 24 else (6 if n <= 64 else 2)
        while want > 1 and _ctas(8 * (before + 4 * n)) < want:
            want -= 1
        assert _ctas(ros4) >= want and _ctas(ros4_narrow) >= want, (S, R)
        # the separate Jacobian kernel's values
        assert _ctas(8 * (9 * wide + 2 * n + species + 3 * S)) >= (8 if n <= 24 else (6 if n <= 64 else 2)), (S, R)
        # one pass fewer would not have fitted
        room = ((228 * 1024 // want - 1024 if want > 1 else 227 * 1024) - 80) // 8
        fewer = lambda chunk: -(-R // (-(-R // chunk) - 1))  # noqa: E731
        if rhs < R:
            assert before + fewer(rhs) > room, (S, R)
        if narrow < R:
            assert n * (n | 1) + 2 * n + species + 3 * S + (9 * R + typed if fewer(narrow) >= R else 10 * fewer(narrow)) > room
    assert [c[:2] for c in layout([(53, 325, 50), (53, 340, 52), (53, 380, 58)])] == [(325, 325), (340, 340), (380, 380)]
    assert [c[:2] for c in layout([(111, 784, 120), (111, 785, 120), (111, 852, 130)])] == [(392, 784), (393, 785),
                                                                                          (426, 852)]


def test_latency_form_holds_all_reactions(layout):
    # up to 32 species and 64 reactions the kernels take them in one pass
    cases = [(S, R, typed) for S in (1, 2, 10, 23, 24, 25, 31, 32) for R in (1, 20, 63, 64) for typed in sorted({0, R // 7, R})]
    for (S, R, typed), (rhs, wide, narrow, *_) in zip(cases, layout(cases)):
        assert rhs == wide == narrow == R, (S, R, typed)
