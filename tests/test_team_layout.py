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
