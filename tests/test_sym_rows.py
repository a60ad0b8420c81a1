"""The symmetric decomposition of the pair work (SymRows, make_sym_decomp),
checked on the CPU against the library's own host code: a small host program
links libnbsym.so, with no GPU.

What must hold for every launch the planner can make:
* every unordered pair of i-blocks is the tile of exactly one row, every block
  has its own, and rows, tiles and units number each other consistently;
* the tiles whose j side is a given block have the deltas 0 .. jslots - 1, so
  those bodies' j slots are all written, and by one tile each;
* no body has more partial sums (j slots plus the blocks of its row) than the
  rows reserved for its cluster, clusters do not overlap, and the rows needed
  stay within the limit (a violation would write past the storage);
* the launch order of several clusters' blocks is a permutation of the grid.
"""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1003_3896_gb300")

SRC = r"""
#include <cstdio>
#include <cstdint>
#include <vector>
#include "engine.h"

using namespace nb;

static uint64_t s_rng = 0x243F6A8885A308D3ull;
static uint64_t rnd() { s_rng ^= s_rng << 13; s_rng ^= s_rng >> 7; s_rng ^= s_rng << 17; return s_rng; }
static int64_t rnd_in(int64_t lo, int64_t hi) { return lo + (int64_t)(rnd() % (uint64_t)(hi - lo + 1)); }

int main()
{
    long long bad = 0, rows_checked = 0, fits = 0, refused = 0, shrunk = 0;
    for (int64_t n = 1; n <= 20000; n += n < 600 ? 1 : 131)
        for (int I : {1, 2, 4, 8}) {
            const int ipb = TILE * I;
            const SymRows sr(n, ipb);
            const int nb = sr.nb;
            std::vector<int> pair((size_t)nb * nb, 0), jw((size_t)nb * (sr.half + 1), 0);
            int64_t q = 0;
            for (int b = 0; b < nb; ++b) {
                bad += sr.row_first(b) != q;
                for (int t = 0; t < sr.row_tiles(b); ++t, ++q) {
                    bad += sr.row_of(q) != b;
                    const int c = (b + t) % nb;
                    ++pair[(size_t)b * nb + c];
                    if (c != b) ++pair[(size_t)c * nb + b];
                    ++jw[(size_t)c * (sr.half + 1) + t];
                }
            }
            bad += sr.tiles() != q || q != (int64_t)nb * (nb + 1) / 2;
            for (int v : pair) bad += v != 1;
            for (int c = 0; c < nb; ++c)
                for (int t = 0; t <= sr.half; ++t)
                    bad += jw[(size_t)c * (sr.half + 1) + t] != (t < sr.jslots(c) ? 1 : 0);
            ++rows_checked;
        }
    for (int trial = 0; trial < 4000; ++trial) {
        const int K = trial % 3 == 0 ? 1 : (int)rnd_in(2, 600);
        const int I = 1 << rnd_in(0, 3), ipb = TILE * I, jt = 128 >> rnd_in(0, 2);
        std::vector<int64_t> nk(K), uoff(K + 1), poff(K);
        for (auto &v : nk) v = K == 1 ? rnd_in(1, 400000) : rnd_in(1, 9000);
        sym_units(nk.data(), K, ipb, jt, uoff.data());
        const int64_t G = rnd_in(1, 152 * 36);
        const int64_t limit = rnd() % 3 ? (int64_t)1 << 40 : rnd_in(1000, 40000000);
        const bool jsum = rnd() % 4 != 0;
        Decomp d;
        int64_t rows = -1;
        if (!make_sym_decomp(nk.data(), K, uoff.data(), ipb, jt, G, limit, jsum, d, poff.data(),
                             &rows)) {
            bad += rows <= limit;
            ++refused;
            continue;
        }
        ++fits;
        bad += rows > limit || d.G < 1 || d.G > d.W || d.W != uoff[K] || d.sym != 1;
        if (d.G < (G < d.W ? G : d.W)) ++shrunk;
        for (int64_t g = 0; g < d.G; ++g) bad += d.U(g + 1) <= d.U(g);
        const int64_t upt = ipb / jt;
        if (K > 1 && d.G <= PERM_CAP) {
            ClusterSet C;
            C.K = K;
            C.nk = nk;
            C.uoff = uoff;
            block_order(C, d, I, false);
            std::vector<char> seen((size_t)d.G, 0);
            bad += (int64_t)C.bperm.size() != d.G;
            for (uint16_t g : C.bperm) bad += g >= d.G || seen[g]++;
        }
        for (int k = 0; k < K; ++k) {
            const SymRows sr(nk[k], ipb);
            const int64_t end = k + 1 < K ? poff[k + 1] : rows;
            for (int b = 0; b < sr.nb; ++b) {
                const int64_t u0 = uoff[k] + sr.row_first(b) * upt;
                const int64_t T = (int64_t)sr.row_tiles(b) * upt;
                const int64_t cnt = d.owner(u0 + T - 1) - d.owner(u0) + 1 +
                                    (jsum ? sr.jslots(b) : 0);
                bad += cnt > d.slots || poff[k] + cnt * nk[k] > end;
            }
        }
    }
    std::printf("rows %lld fits %lld refused %lld shrunk %lld failures %lld\n", rows_checked, fits,
                refused, shrunk, bad);
    return bad ? 1 : 0;
}
"""


def test_symmetric_rows_cover_pairs_and_bound_slots(tmp_path):
    from paper_1003_3896_gb300 import build
    lib = build.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "sym_rows.cu"
    src.write_text(SRC)
    exe = tmp_path / "sym_rows"
    subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-I", os.path.join(PKG, "csrc"),
                    "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe), "-L", os.path.dirname(lib), "-lnbsym",
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    f = dict(zip(r.stdout.split()[0::2], r.stdout.split()[1::2]))
    assert f["failures"] == "0"
    assert int(f["fits"]) > 1000 and int(f["refused"]) > 50 and int(f["shrunk"]) > 10
