"""The item count of the half-pair schedule where nbk (nbk + 1) passes 2^31, on
the host: the header compiled into a small program."""
import subprocess

import pytest

from paper_2106_11143_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "nb_symsched.cuh"
int main(int argc, char **argv) {
  for (int k = 1; k < argc; ++k) {
    const int nbk = std::atoi(argv[k]);
    const long long items = (long long)nb::sym_items(nbk);
    const nb::SymItem a = nb::sym_item((int)(items - 1), nbk);
    std::printf("%d %lld %u %d %d %d\n", nbk, items, (unsigned)nb::sym_items(nbk), a.P, a.Q, a.round);
  }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("sched")
    (d / "p.cu").write_text(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-o", str(d / "p"),
                           str(d / "p.cu"), "-ldl"])
    out = subprocess.check_output([str(d / "p"), "46340", "46341", "46875", "58594", "60000"], text=True)
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]


def test_item_count_past_the_32_bit_product(rows):
    """46341 is the first nbk whose product passes 2^31 - 1; 46875 and 58594 are
    the 256-ion blocks of 12e6 and 15e6 ions."""
    for nbk, items, grid, P, Q, last in rows:
        assert items == nbk * (nbk + 1) // 2 == grid
        assert items < 2 ** 31
        assert 0 <= P <= Q < nbk and last == nbk - 1


def test_plans_reach_these_counts():
    from paper_2106_11143_gb300 import api
    build.build()
    for n, nbk in ((12_000_000, 46875), (15_000_000, 58594)):
        for prec in ("fp64", "df64"):
            p = api.plan_info("force", prec, n)
            assert p["symmetric"] and p["n_it"] == nbk and p["n_jc"] == 1, (prec, n, p)
