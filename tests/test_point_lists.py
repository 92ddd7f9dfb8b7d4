"""Host-built lists of small children's entries (csrc/point_lists.cpp): compiled
with a program that makes random trees of fronts and compares every item's lists
with a stable sort of its points, on one thread and on several."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2508_04370_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include <utility>
#include "point_lists.h"
using namespace ipm;

// parents of the given sizes (large where flagged), each under children of 1 to
// `most` contribution rows
static Plan tree(std::mt19937 &g, const std::vector<std::pair<int, bool>> &parents, int most) {
    Plan P;
    P.child_ptr.push_back(0);
    std::vector<int> up;
    for (size_t p = 0; p < parents.size(); p++) {
        const int nch = (int)(g() % 9);
        for (int c = 0; c < nch; c++) {
            const int cc = 1 + (int)(g() % std::min(most, parents[p].first)), k = 1 + (int)(g() % 3);
            P.sn_k.push_back(k), P.sn_f.push_back(k + cc), P.sn_large.push_back(0);
            std::vector<int32_t> all(parents[p].first);
            for (size_t i = 0; i < all.size(); i++) all[i] = (int32_t)i;
            std::shuffle(all.begin(), all.end(), g);
            all.resize(cc);
            std::sort(all.begin(), all.end());
            P.map_off.push_back((int64_t)P.relmap.size());
            P.relmap.insert(P.relmap.end(), all.begin(), all.end());
            P.child_ptr.push_back(P.child_ptr.back());
            up.push_back((int)P.sn_k.size() - 1);
        }
        P.sn_k.push_back(1), P.sn_f.push_back(parents[p].first), P.sn_large.push_back(parents[p].second);
        P.map_off.push_back((int64_t)P.relmap.size());
        for (int c : up) P.child_list.push_back(c);
        P.child_ptr.push_back((int32_t)P.child_list.size());
        up.clear();
    }
    P.nsuper = (int32_t)P.sn_k.size();
    int64_t off = 0;
    for (int s = 0; s < P.nsuper; s++) {
        P.sn_ld.push_back((P.sn_f[s] + 3) & ~3);
        P.sn_off.push_back(off);
        off += (int64_t)P.sn_ld[s] * P.sn_f[s];
    }
    return P;
}

static int check(const Plan &P, const PointLists &L) {
    int64_t points = 0;
    if ((int64_t)L.seg.size() != L.first[P.nsuper] + 1) return 1;
    for (int s = 0; s < P.nsuper; s++) {
        const int f = P.sn_f[s], ld = P.sn_ld[s];
        int item = 0;
        for (int cb = 0; cb < (P.sn_large[s] ? (f + 31) / 32 : 1); cb++)
            for (int rb = 32 * cb / kAsmRows; P.sn_large[s] ? rb * kAsmRows < f : rb < 1; rb++, item++) {
                std::vector<std::pair<int32_t, int64_t>> want;
                for (int q = P.child_ptr[s]; q < P.child_ptr[s + 1]; q++) {
                    const int ch = P.child_list[q], k = P.sn_k[ch], cc = P.sn_f[ch] - k;
                    if (cc > kPointRows) continue;
                    const int32_t *m = P.relmap.data() + P.map_off[ch];
                    for (int j = 0; j < cc; j++)
                        for (int i = j; i < cc; i++) {
                            if (P.sn_large[s] && (m[j] / 32 != cb || m[i] / kAsmRows != rb)) continue;
                            want.push_back({P.sn_large[s] ? kAsmRows * (m[j] % 32) + m[i] % kAsmRows : m[j] * ld + m[i],
                                            P.sn_off[ch] + (int64_t)(k + j) * P.sn_ld[ch] + k + i});
                        }
                }
                std::stable_sort(want.begin(), want.end(), [](auto &x, auto &y) { return x.first < y.first; });
                std::vector<std::pair<int32_t, int64_t>> got;
                const int64_t d0 = L.seg[L.first[s] + item], d1 = L.seg[L.first[s] + item + 1];
                for (int64_t d = d0; d < d1; d++) {
                    if (d > d0 && L.dst[d] <= L.dst[d - 1]) return 2;
                    if (L.ptr[d] >= L.ptr[d + 1]) return 3;
                    for (int64_t q = L.ptr[d]; q < L.ptr[d + 1]; q++) got.push_back({L.dst[d], L.src[q]});
                }
                if (got != want) return 4;
                points += (int64_t)want.size();
            }
        if (item != (P.sn_large[s] ? asm_tiles(f) : 1)) return 5;
    }
    return points == L.nsrc ? 0 : 6;
}

int main() {
    // a child's place in a list of row blocks beyond 2^31
    for (int64_t rt : {int64_t(0), int64_t(1) << 31, (int64_t(1) << 40) + 5})
        for (int n : {1, 31, 32}) {
            const AsmChild c = asm_child_of(int64_t(1) << 35, int64_t(1) << 34, 200000, 100000, n, rt);
            if (c.rt() != rt || c.n() != n || c.a != 100000 || c.ldc != 200000) return 3;
        }
    std::mt19937 g(1);
    for (int round = 0; round < 20; round++) {
        std::vector<std::pair<int, bool>> parents;
        for (int f : {1, 2, 31, 32, 33, 64, 65, 100, 127, 128}) parents.push_back({f, false});
        for (int f : {66, 95, 96, 97, 128, 129, 191, 192, 193, 257, 320}) parents.push_back({f, true});
        std::shuffle(parents.begin(), parents.end(), g);
        const Plan P = tree(g, parents, round % 2 ? 64 : 70);
        for (int threads : {1, 2, 7, 60, 0}) {
            PointLists L;
            build_point_lists(P, L, threads);
            if (const int bad = check(P, L)) {
                std::printf("round %d threads %d: check %d\n", round, threads, bad);
                return 1;
            }
        }
    }
    PointLists L;
    build_point_lists(Plan(), L, 0);  // no fronts
    return L.nsrc == 0 && L.seg.size() == 1 ? 0 : 2;
}
"""


def test_lists_equal_a_stable_sort(tmp_path):
    src, exe = tmp_path / "lists.cpp", tmp_path / "lists"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-fsanitize=address,undefined", "-fno-sanitize-recover",
                    f"-I{CSRC}", str(src), os.path.join(CSRC, "point_lists.cpp"), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout + run.stderr
