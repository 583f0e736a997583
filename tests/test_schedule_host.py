"""Host-side parts of the half-pair kernels that the C ABI does not show, from small
programs compiled against the library: the item count of the schedule where nbk
(nbk + 1) passes 2^31, and the potential's own plan against the fixed scratch of
nb_energy_noalloc."""
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


PHI_PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "nb_symsched.cuh"
#include "nb_tri.cuh"
int main(int argc, char **argv) {
  for (int k = 1; k < argc; ++k) {
    const long long n = std::atoll(argv[k]);
    const nb::PhiPlan p = nb::make_phi_plan(n);
    std::printf("%lld %d %d %d %zu %lld\n", n, p.G, p.nbk, p.n_slots, p.out_doubles(n),
                p.G ? (long long)nb::sym_sync_ints(p.nbk) : 0LL);
  }
}
"""


def test_potential_plan_fits_the_fixed_scratch(tmp_path):
    """Its blocks cover the ions; its slots and counters, the 3 * 128 reduction
    doubles, the energies and the error word fit 2^20 doubles up to 1e6 ions; the
    in-place output takes over where the slots would pass 1e6 doubles."""
    import numpy as np
    build.build()
    (tmp_path / "p.cu").write_text(PHI_PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-o", str(tmp_path / "p"),
                           str(tmp_path / "p.cu"), build.LIB, "-Xlinker", "-rpath=" + build.HERE])
    ns = sorted(set(np.geomspace(1, 1_000_000, 500).astype(int).tolist()
                    + [1999, 2000, 9999, 10000, 15871, 15872, 22500, 22750, 999_999, 1_000_000, 12_000_000, 40_000_000]))
    out = subprocess.check_output([str(tmp_path / "p")] + [str(n) for n in ns], text=True)
    forms = set()
    for line in out.splitlines():
        n, G, nbk, slots, doubles, ints = (int(v) for v in line.split())
        assert (G > 0) == (2000 <= n <= 60000 * 512), n
        if G:
            assert G in (4, 8, 16) and nbk == -(-n // (32 * G)) and slots in (1, nbk)
            assert (slots == 1) == (nbk * n > 1_000_000)
            assert 8 * (doubles - slots * n) >= 4 * ints
            forms.add((G, slots == 1))
        if n <= 1_000_000:
            assert doubles + 3 * 128 + 5 <= 1 << 20, (n, G, nbk, slots)
    assert forms >= {(4, False), (8, False), (16, False), (8, True)}
