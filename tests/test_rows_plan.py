"""CPU-only checks of how the row kernels cut lattices into items
(csrc/lbm_rows_plan.h), through a small host program around that header.

An item of h rows pulls and computes six more, and a pair of warps marches
down its rows one after another, so a launch lasts at least as long as its
tallest item.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PAIRS = 152 * 8  # pairs of warps that a GB300 holds

MAIN = r"""
#include <cstdio>
#include "lbm_rows_plan.h"
using namespace pplbm;
int main() {
    long n, nx, ny;
    while (std::scanf("%ld", &n) == 1) {
        std::vector<LatDev> lats;
        for (long k = 0; k < n; ++k) {
            if (std::scanf("%ld %ld", &nx, &ny) != 2) return 1;
            LatDev L{};
            L.nx = (int)nx;
            L.ny = (int)ny;
            lats.push_back(L);
        }
        const int h = pair_item_height(lats, %PAIRS%);
        std::vector<int4> t;
        for (size_t l = 0; l < lats.size(); ++l) row_items(lats[l], (int)l, h, t, kPairCols);
        std::printf("%d %zu\n", h, t.size());
        for (const int4& i : t) std::printf("%d %d %d %d\n", i.x, i.y, i.z, i.w);
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2003_07968_gb300 import build

    d = tmp_path_factory.mktemp("plan")
    src, exe = str(d / "plan.cu"), str(d / "plan")
    open(src, "w").write(MAIN.replace("%PAIRS%", str(PAIRS)))
    subprocess.run([build.nvcc(), "-std=c++17", *build.ARCH, "--expt-relaxed-constexpr", "-I",
                    build.CSRC, src, "-o", exe], check=True)

    def run(lats):
        text = f"{len(lats)}\n" + "".join(f"{nx} {ny}\n" for nx, ny in lats)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        lines = [tuple(int(v) for v in ln.split()) for ln in out.splitlines()]
        assert len(lines) == 1 + lines[0][1]
        return lines[0][0], [(l, x, y, w & 0xFFFFFF, w >> 24) for l, x, y, w in lines[1:]]

    return run


MIXES = [[(16, 16)] * 2000 + [(512, 512)], [(512, 512)] + [(16, 16)] * 1200,
         [(32, 32)] * 5000 + [(2048, 2048)], [(56, 20000)] * 2 + [(16, 16)] * 1300,
         [(64, 64)] * 300 + [(4096, 100)], [(64 + 7 * k % 449, 64 + 13 * k % 449) for k in range(512)],
         [(2, 2)] * 3000 + [(61, 999)], [(700, 720)] * 2, [(5, 3)], [(8192, 8192)], [(300000, 40)]]


@pytest.mark.parametrize("k", range(len(MIXES)))
def test_pair_items_cover_and_share(plan, k):
    lats = MIXES[k]
    h, items = plan(lats)
    # every site once: an item's strip and band, and the sum of the areas
    seen = set()
    area = [0] * len(lats)
    for l, x, y, rows, width in items:
        nx, ny = lats[l]
        assert 0 < width <= 56 and x % 2 == 0 and x + width <= nx
        assert 0 < rows <= h and y + rows <= ny
        assert (l, x, y) not in seen
        seen.add((l, x, y))
        area[l] += rows * width
    assert area == [nx * ny for nx, ny in lats]
    # no item much taller than its pair's share of all rows (one wave of up to
    # 108 rows is even; a lattice alone is cut into four waves at most)
    if len(lats) > 1:
        units = sum(-(-nx // 56) * ny for nx, ny in lats)
        assert max(i[3] for i in items) <= max(108, 2 * -(-units // PAIRS))


PAY = r"""
#include <cstdio>
#include "lbm_rows_plan.h"
using namespace pplbm;
int main() {
    int f16, mrt, tensor;
    long n, nx, ny;
    while (std::scanf("%d %d %d %ld", &f16, &mrt, &tensor, &n) == 4) {
        std::vector<LatDev> lats;
        for (long k = 0; k < n; ++k) {
            if (std::scanf("%ld %ld", &nx, &ny) != 2) return 1;
            LatDev L{};
            L.nx = (int)nx;
            L.ny = (int)ny;
            lats.push_back(L);
        }
        const int64_t sms = 152;
        const int h = f16 ? row_item_height(lats, sms * 4 * kRowWarps)
                          : pair_item_height(lats, sms * 2 * kPairs);
        std::printf("%d\n", (int)rows_pay(lats, h, f16, mrt, n == 1, tensor, sms));
    }
}
"""
# shapes, storage (1 FP32, 2 FP16), whether the arena is one tensor, and which
# kernel was measured faster, by 10 % or more in BGK and MRT
TILES = [([(64, 64)] * 310, 1, 1), ([(64, 64)] * 310, 2, 1), ([(64, 64)] * 1000, 1, 1),
         ([(64, 64)] * 4000, 2, 1), ([(60, 60)] * 400, 1, 1), ([(32, 32)] * 1000, 1, 1),
         ([(32, 32)] * 1000, 2, 1), ([(64, 16)] * 400, 1, 1), ([(64, 18750)], 1, 1),
         ([(64, 62500)], 2, 1), ([(61, 19672)], 2, 1), ([(8, 8)] * 5000, 1, 0)]
ROWS = [([(56, 56)] * 400, 1, 1), ([(48, 48)] * 400, 1, 1), ([(100, 100)] * 200, 1, 1),
        ([(100, 100)] * 200, 2, 1), ([(256, 256)] * 30, 1, 1), ([(1024, 1024)], 1, 1),
        ([(4096, 4096)], 2, 1), ([(8192, 8192)], 1, 1), ([(8192, 8192)], 2, 1),
        ([(70, 70)] * 300, 1, 1), ([(500, 500)] * 30, 1, 1), ([(600000, 2)], 1, 1),
        ([(64 + 7 * k % 449, 64 + 13 * k % 449) for k in range(512)], 1, 1),
        ([(64 + 7 * k % 449, 64 + 13 * k % 449) for k in range(128)], 2, 1)]


def test_row_kernels_only_where_they_pay(tmp_path):
    from paper_2003_07968_gb300 import build

    src, exe = str(tmp_path / "pay.cu"), str(tmp_path / "pay")
    open(src, "w").write(PAY)
    subprocess.run([build.nvcc(), "-std=c++17", *build.ARCH, "--expt-relaxed-constexpr", "-I",
                    build.CSRC, src, "-o", exe], check=True)
    cases = [(c, mrt, want) for cs, want in ((TILES, 0), (ROWS, 1)) for c in cs for mrt in (0, 1)]
    text = "".join(f"{int(st == 2)} {mrt} {tensor} {len(lats)}\n" +
                   "".join(f"{nx} {ny}\n" for nx, ny in lats)
                   for (lats, st, tensor), mrt, _ in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(cases)
    for got, ((lats, st, _), mrt, want) in zip(out, cases):
        assert int(got) == want, (lats[0], len(lats), st, mrt)
