"""The rules of the launches, evaluated on the host from the headers that the kernels use.

A kernel ends with its longest unit.  Bodies of more than 8 particles per cell have fewer and fuller blocks, so a count
of parts made for 512 particles a block leaves long units and idle warps.  For blocks of 641 to 8000 particles (up to
125 per cell) the longest unit must be no longer than the one that the body is cut into, or than that of a count of
parts by the particle number alone (two units of 512 for each of 20 warps per SM, at most eight parts, in whole chunks).
Blocks of up to 640 keep the parts measured for them; no body is cut into more units than the limit.

The grid update loops over its blocks in whole waves of the CTAs that are resident together.  One CTA scans the tile
sums of a large key space, 1024 an iteration: in iterations of no less than 4 million keys."""
import shutil
import subprocess

import pytest

from paper_2412_10399_gb300 import build

SMS = 152
SRC = r"""
#include <cstdio>
#include "launch.h"
int main(int argc, char**) {
  long long which, n, kind, transfer, npb, cnt;
  while (argc == 3 && std::scanf("%lld", &n) == 1)
    std::printf("%d %u\n", (int)ck::scan_fused((unsigned)n), ck::scan_tiles((unsigned)n));
  while (argc == 2 && std::scanf("%lld %lld %lld", &kind, &n, &cnt) == 3)
    std::printf("%d\n", ck::update_ctas((int)kind, 152, (unsigned)cnt, (unsigned)n));
  while (std::scanf("%lld %lld %lld %lld %lld %lld", &which, &n, &kind, &transfer, &npb, &cnt) == 6) {
    const int warps = which == 0 ? ck::p2g_warps(kind, transfer, kind == 1 && transfer == 0 ? 2 : 1)
                                 : ck::g2p_warps(kind, transfer, 5);
    const ck::Units h = ck::step_units((int)which, n, 152, warps);
    const ck::Units w = ck::limit_units(h, (unsigned)npb, ck::p2g_ctas(152), (unsigned)cnt);
    std::printf("%u %u %u %u\n", h.splits, h.unit, w.splits, ck::part_size(w, (unsigned)cnt, which == 0 ? 96u : 32u));
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("units")
    (d / "rule.cu").write_text(SRC)
    exe = str(d / "rule")
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", f"-I{build.CSRC}", f"-I{build.INCLUDE}", str(d / "rule.cu"),
                    "-o", exe], check=True, capture_output=True)

    def ask(rows, *args):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([exe, *args], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return ask


def _rows(counts):
    for which in (0, 1):
        for kind in (0, 1):
            for transfer in (0, 1, 2):
                for n in (3000, 20000, 50000, 97280, 150000, 224000, 346112, 600000, 1000000, 1500000):
                    for cnt in counts:
                        yield which, n, kind, transfer, max(1, -(-n // cnt)), cnt


def test_dense_blocks_are_cut_into_units(rule):
    rows = list(_rows((641, 900, 1728, 4096, 8000)))
    for (which, n, kind, transfer, npb, cnt), (_, unit, splits, longest) in zip(rows, rule(rows)):
        chunk = 96 if which == 0 else 32
        parts = max(1, min(8, SMS * 20 * 2 * 512 // n))
        fixed = -(-(-(-cnt // parts)) // chunk) * chunk
        assert longest <= max(unit, fixed), (which, n, kind, transfer, cnt)
        assert (splits - 1) * npb < SMS * 32


def test_ordinary_blocks_keep_their_parts(rule):
    rows = list(_rows((64, 512, 640)))
    for r, (host, unit, splits, longest) in zip(rows, rule(rows)):
        assert splits == min(host, -(-SMS * 32 // r[4])) and longest >= unit


def test_grid_update_launches_whole_waves(rule):
    rows = [(kind, n, pool) for kind in (0, 1) for n in (1, 4096, 32768, 150000, 346112, 1000000, 16273664)
            for pool in (64, 4608, 100000, 2000000)]
    for (kind, n, pool), (ctas,) in zip(rows, rule(rows, "update")):
        wave = (8 if kind else 10) * SMS
        assert ctas % wave == 0 and wave <= ctas <= 64 * SMS
        est = (min(pool, n // 64 + 256) + 1) // 2
        assert ctas + wave > min(est, 64 * SMS) and (ctas == wave or ctas <= est)


def test_one_cta_scans_wide_tiles(rule):
    rows = [(n,) for n in (1, 1024, 8192, 8193, 1 << 22, (1 << 22) + 1, 175 ** 3, 256 ** 3, 512 ** 3, 2 ** 31 - 1)]
    for (n,), (fused, tiles) in zip(rows, rule(rows, "scan", "tiles")):
        assert tiles == -(-n // (1024 if fused else 4096)) and fused == (n <= 1 << 22)
