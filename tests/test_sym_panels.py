"""The split of the products that evaluate each pair of one point set once (csrc/sym.cuh), on the CPU:
a host program fills every slot as the kernels do and adds them as the reductions do."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Columns and rows all weigh 1, so that a point's sums over all panels count the columns: NU * BN.  Slots
# start at -1 in every panel: reading one that was not written, or writing one twice, shows.
PROGRAM = r"""
#include "sym.cuh"
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace krr;
#define CHECK(c) do { if (!(c)) { std::printf("%s at NU %d RU %d entries %lld runs %d panel %d..%d\n", #c, g.NU, g.RU, \
                                              entries, maxruns, g.I0, g.I1); return 1; } } while (0)
static int one(int NU, int BN, int RU, long long entries, int maxruns, int* panels) {
    SyGrid whole{};
    whole.n = NU * BN;
    whole.BN = BN;
    whole.NU = NU;
    whole.RU = RU;
    whole.nblk = (NU + RU - 1) / RU;
    whole.W = whole.first(whole.nblk);
    whole.G = (int)(whole.W < maxruns ? whole.W : maxruns);
    std::vector<long long> total(NU, 0);           // by column unit: all its points are alike
    *panels = 0;
    for (int from = 0; from < whole.nblk;) {
        const SyPanel g(whole, from, entries, maxruns);
        ++*panels;
        CHECK(g.I0 == from && g.I1 > g.I0 && g.I1 <= g.nblk);
        CHECK(g.first_panel() == (from == 0) && g.last_panel() == (g.I1 == g.nblk));
        CHECK(g.col_entries() <= entries || g.I1 == g.I0 + 1);
        if (g.first_panel() && g.last_panel())     // the whole grid: the plain type's addresses
            for (int T = 0; T < NU; ++T) {
                CHECK(g.col_base(T) == whole.col_base(T) && g.slots(T / RU) == whole.slots(T / RU));
                CHECK(g.G == whole.G && g.run_begin(g.G / 2) == whole.run_begin(g.G / 2));
                CHECK(g.run_of(T) == whole.run_of(T) && g.slot(T) == whole.slot(T));
            }
        CHECK(g.G >= 1 && g.G <= maxruns && g.G <= g.W);
        CHECK(g.run_begin(0) == g.first(g.I0) && g.run_begin(g.G) == g.first(g.I1));
        CHECK(g.col_base(NU) <= g.col_entries());
        std::vector<long long> col(g.col_entries() / BN, -1), row(g.G + g.I1 - g.I0, -1);
        for (int run = 0; run < g.G; ++run) {
            long long u = g.run_begin(run);
            const long long u1 = g.run_begin(run + 1);
            CHECK(u < u1);
            for (int I = g.block_of(u); u < u1; ++I) {
                const long long ue = u1 < g.first(I + 1) ? u1 : g.first(I + 1);
                CHECK(I >= g.I0 && I < g.I1);
                long long& r = row.at(run + g.slot(I));
                CHECK(r == -1);
                r = (ue - u) * BN;
                for (; u < ue; ++u) {
                    CHECK(g.run_of(u) == run);
                    const int T = I * RU + (int)(u - g.first(I));
                    CHECK(T < NU);
                    if (T / RU <= I) continue;
                    CHECK(g.col_base(T) % BN == 0 && g.slot(I) < g.slots(T / RU));
                    long long& c = col.at(g.col_base(T) / BN + g.slot(I));
                    CHECK(c == -1);
                    c = (long long)g.row_tiles(I) * SY_T;
                }
            }
        }
        for (int T = 0; T < NU; ++T) {
            const int b = T / RU;
            for (int I = 0; I < g.slots(b); ++I) {
                const long long c = col.at(g.col_base(T) / BN + I);
                CHECK(c > 0);
                total[T] += c;
            }
            if (!g.has(b)) continue;
            for (int s = g.run_of(g.first(b)); s <= g.run_of(g.first(b + 1) - 1); ++s) {
                CHECK(row.at(s + g.slot(b)) > 0);
                total[T] += row.at(s + g.slot(b));
            }
        }
        from = g.I1;
        if (from < g.nblk) continue;
        for (int T = 0; T < NU; ++T) CHECK(total[T] == (long long)NU * BN);
    }
    return 0;
}
int main() {
    int many = 0, p = 0;
    for (int BN : {128, 256})
        for (int RU : {1, 2, 3, 4})
            for (int NU = 1; NU <= 41; ++NU)
                for (long long entries : {1LL, 1LL * BN, 5LL * BN, 17LL * BN, 100LL * BN, 1LL << 40})
                    for (int runs : {1, 2, 7, 152}) {
                        if (one(NU, BN, RU, entries, runs, &p)) return 1;
                        if (entries == 1LL << 40 && p != 1) return 2;
                        many += p > 3;
                    }
    // the largest sets the products take, with the limit as it is: panels within it (no slots filled)
    for (int w : {1024, 512, 256}) {
        SyGrid g{};
        g.BN = 128;
        g.RU = w / 128;
        g.n = 1 << 21;
        g.NU = g.n / 128;
        g.nblk = (g.NU + g.RU - 1) / g.RU;
        for (int I = 0, k = 0; I < g.nblk; ++k) {
            const SyPanel p(g, I, kSymBytes / 8, 304);
            if (8 * p.col_entries() > kSymBytes || k > 1000 || p.run_begin(0) < 0) return 3;
            I = p.I1;
        }
        if (g.first(g.nblk) > 0x7fffffffLL) return 4;   // pair numbers are int in the kernels
    }
    std::printf("ok %d\n", many);
    return 0;
}
"""


def test_panels_cover_every_pair_once(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "panels.cu", tmp_path / "panels"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-arch=sm_103a", "-I", os.path.join(ROOT, "paper_1905_10587_gb300", "csrc"), "-o", str(exe),
                    str(src)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
    assert int(res.stdout.split()[1]) > 500        # cases with four panels or more
