"""The split products' sums stay exact: the rows that a contraction sums in one
set of FP32 accumulators follow from the table's digits (csrc/split_tables.h,
compiled here for the host)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1111_4971_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "split_tables.h"
int main(int argc, char** argv) {
  const int rows = std::atoi(argv[1]), slots = std::atoi(argv[2]);
  const bool halves = std::atoi(argv[3]) != 0;
  std::vector<double> t(size_t(rows) * slots);
  if (std::fread(t.data(), sizeof(double), t.size(), stdin) != t.size()) return 1;
  std::vector<int> s(pp::split_padded(rows));
  const pp::RowScale p = pp::table_scales(t.data(), rows, slots, s.data());
  std::printf("%d %d %d\n", pp::contract_steps(t.data(), s.data(), rows, slots, halves), p.plain0, p.plain1);
  for (int r = 0; r < rows; ++r) {
    std::printf("%d", s[pp::scale_index(r)] >> 20);
    for (int k = 0; k < slots; ++k) {
      long d[6];
      pp::table_digits(t.data(), s.data(), slots, r, k, d);
      for (int j = 0; j < 6; ++j) std::printf(" %ld", d[j]);
    }
    std::printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("split")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def run(table, halves):
        rows, slots = table.shape
        out = subprocess.run([str(d / "main"), str(rows), str(slots), str(int(halves))], check=True,
                             input=np.ascontiguousarray(table, dtype=np.float64).tobytes(), capture_output=True).stdout
        lines = out.decode().split("\n")
        steps, plain0, plain1 = map(int, lines[0].split())
        body = np.array([list(map(int, x.split())) for x in lines[1:rows + 1]])
        return steps, (plain0, plain1), body[:, 0], body[:, 1:].reshape(rows, slots, 6)
    return run


def worst(digits, halves, steps):
    """The largest sum of a weight 0 .. 4 over 16 * steps rows, for data digits of the largest size."""
    out = 0
    for r0 in range(0, len(digits), 16 * steps):
        t = digits[r0:r0 + 16 * steps].sum(0)
        for w in range(5):
            out = max(out, (256 * t[:, :w].sum(1) + (512 if halves else 256) * t[:, w]).max())
    return out


@pytest.mark.parametrize("kind,ny", [("centred", n) for n in (16, 48, 128, 144, 1024, 2064)] +
                         [("wall", n) for n in (16, 80, 256, 2064)] + [("x", n) for n in (16, 80, 1024)])
def test_spanning_meshes_sum_64_rows(program, kind, ny):
    n = np.arange(1, 33)
    j = np.arange(ny if kind == "x" else ny // 2) + (0.0 if kind == "wall" else 0.5)
    table = np.sin(np.pi * n[None, :] * j[:, None] / ny)
    if kind == "wall":
        table[0] = np.sin(np.pi * n / 2) * (n % 2)
    steps, plain, scale, digits = program(table, kind != "x")
    assert steps == 4 and worst(digits, kind != "x", 4) <= 2 ** 24
    # each row's largest value comes into [1/2, 1]; the plain steps have no scale
    top = np.abs(table).max(1) * 2.0 ** scale
    assert ((top >= 0.5) & (top <= 1.0)).all()
    assert not scale[16 * plain[0]:16 * plain[1]].any()


@pytest.mark.parametrize("halves,value,steps", [
    (True, 255, 2), (False, 255, 2),            # every digit 255: 64 rows of 5 or 6 products pass 2^24
    (False, 200, 4), (True, 170, 4),
])
def test_tables_of_large_digits_sum_fewer_rows(program, halves, value, steps):
    x = sum(value << (9 * k) for k in range(6)) * 2.0 ** -53
    table = np.full((80, 4), x)
    table[::2, 1] *= -1
    got, plain, scale, digits = program(table, halves)
    assert (digits[..., :5] >= value - 1).all()
    assert got == steps and worst(digits, halves, got) <= 2 ** 24
    assert got == 4 or worst(digits, halves, 2 * got) > 2 ** 24


def test_rows_of_zeros(program):
    table = np.zeros((40, 2))
    table[5] = 2.0 ** -20
    steps, plain, scale, digits = program(table, False)
    assert scale[5] == 19 and (scale[np.arange(40) != 5] == 2047).all() and plain == (0, 0)
