// See point_lists.h.  A counting sort by destination (a bitmap of the ones met,
// their counts, one pass that places) instead of a comparison sort, fronts spread
// over threads: preparing a 64 x 64 grid (1.2 million points) sorted them
// for 17 ms of a set-up of 28.
#include "point_lists.h"

#include <algorithm>
#include <exception>
#include <system_error>
#include <thread>

namespace ipm {

namespace {

int64_t points_of(const Plan &P, int32_t s) {
    int64_t n = 0;
    for (int32_t q = P.child_ptr[s]; q < P.child_ptr[s + 1]; q++) {
        const int64_t cc = P.sn_f[P.child_list[q]] - P.sn_k[P.child_list[q]];
        if (cc <= kPointRows) n += cc * (cc + 1) / 2;
    }
    return n;
}

// The lists of fronts [s0, s1), their positions in src known beforehand.
struct Chunk {
    int32_t s0 = 0, s1 = 0;
    int64_t src0 = 0;            // the chunk's first position in src
    std::vector<int32_t> dst;
    std::vector<int64_t> ptr;    // start of each destination's list in src
    std::vector<int64_t> ends;   // per item: destinations of the chunk so far
    std::exception_ptr error;

    void build(const Plan &P, int64_t *src) {
        std::vector<int64_t> count(128 * 128, 0), ps, tile;
        std::vector<uint64_t> met(128 * 128 / 64, 0);
        std::vector<int32_t> pd;
        int64_t at = src0;
        // points [b, e) of pd / ps, destinations below range: one item's lists
        auto group = [&](int64_t b, int64_t e, int32_t range) {
            if (b < e) {
                const size_t d0 = dst.size();
                const int64_t base = at;
                for (int64_t u = b; u < e; u++)
                    if (count[pd[u]]++ == 0) met[pd[u] >> 6] |= uint64_t(1) << (pd[u] & 63);
                for (int32_t w = 0; 64 * w < range; w++) {
                    uint64_t m = met[w];
                    met[w] = 0;
                    for (; m; m &= m - 1) {
                        const int32_t d = 64 * w + __builtin_ctzll(m);
                        const int64_t n = count[d];
                        count[d] = at - base;
                        dst.push_back(d);
                        ptr.push_back(at);
                        at += n;
                    }
                }
                for (int64_t u = b; u < e; u++) src[base + count[pd[u]]++] = ps[u];
                for (size_t q = d0; q < dst.size(); q++) count[dst[q]] = 0;
            }
            ends.push_back((int64_t)dst.size());
        };
        for (int32_t s = s0; s < s1; s++) {
            const int64_t n = points_of(P, s);
            const int32_t f = P.sn_f[s], ld = P.sn_ld[s], nt = P.sn_large[s] ? asm_tiles(f) : 1;
            if (n == 0) {
                ends.insert(ends.end(), nt, (int64_t)dst.size());
                continue;
            }
            if ((int64_t)pd.size() < n) pd.resize(n), ps.resize(n);
            // each point's column and row in the front, and its arena position
            auto points = [&](auto &&column) {
                for (int32_t q = P.child_ptr[s]; q < P.child_ptr[s + 1]; q++) {
                    const int32_t ch = P.child_list[q], kc = P.sn_k[ch], cc = P.sn_f[ch] - kc, ldc = P.sn_ld[ch];
                    if (cc > kPointRows) continue;
                    const int32_t *m = P.relmap.data() + P.map_off[ch];
                    const int64_t cb0 = P.sn_off[ch] + (int64_t)kc * ldc + kc;
                    for (int32_t j = 0; j < cc; j++) column(m[j], m, j, cc, cb0 + (int64_t)j * ldc);
                }
            };
            if (!P.sn_large[s]) {
                int64_t u = 0;
                points([&](int32_t col, const int32_t *m, int32_t j, int32_t cc, int64_t pos) {
                    for (int32_t i = j; i < cc; i++, u++) pd[u] = col * ld + m[i], ps[u] = pos + i;
                });
                group(0, n, ld * f);
                continue;
            }
            // by item first
            tile.assign(nt + 1, 0);
            auto first = [&](int32_t col) { return asm_first_tile(f, col / 32) - 32 * (col / 32) / kAsmRows; };
            points([&](int32_t col, const int32_t *m, int32_t j, int32_t cc, int64_t) {
                int64_t *t = tile.data() + 1 + first(col);
                for (int32_t i = j; i < cc; i++) t[m[i] / kAsmRows]++;
            });
            for (int32_t t = 0; t < nt; t++) tile[t + 1] += tile[t];
            points([&](int32_t col, const int32_t *m, int32_t j, int32_t cc, int64_t pos) {
                int64_t *t = tile.data() + first(col);
                for (int32_t i = j; i < cc; i++) {
                    const int64_t u = t[m[i] / kAsmRows]++;
                    pd[u] = kAsmRows * (col % 32) + m[i] % kAsmRows, ps[u] = pos + i;
                }
            });
            // (tile[t] is now the end of item t)
            for (int32_t t = 0; t < nt; t++) group(t ? tile[t - 1] : 0, tile[t], 32 * kAsmRows);
        }
    }
};

}  // namespace

void build_point_lists(const Plan &P, PointLists &out, int threads) {
    const int32_t ns = P.nsuper;
    std::vector<int64_t> before(ns + 1, 0);  // points of the fronts before
    out.first.assign(ns + 1, 0);
    for (int32_t s = 0; s < ns; s++) {
        before[s + 1] = before[s] + points_of(P, s);
        out.first[s + 1] = out.first[s] + (P.sn_large[s] ? asm_tiles(P.sn_f[s]) : 1);
    }
    out.nsrc = before[ns];
    out.src.reset(new int64_t[out.nsrc]);
    if (threads <= 0)  // a thread costs about 50 us: 50,000 points
        threads = (int)std::min<int64_t>(std::min(8u, std::max(1u, std::thread::hardware_concurrency())),
                                         1 + out.nsrc / 50000);
    std::vector<Chunk> chunk(threads);
    for (int t = 0; t < threads; t++) {
        Chunk &c = chunk[t];
        c.s0 = t ? chunk[t - 1].s1 : 0;
        c.s1 = t + 1 == threads ? ns : (int32_t)(std::upper_bound(before.begin(), before.end(), out.nsrc * (t + 1) / threads) -
                                                 before.begin() - 1);
        c.s1 = std::min(std::max(c.s1, c.s0), ns);
        c.src0 = before[c.s0];
    }
    auto run = [&](Chunk &c) {
        try {
            c.build(P, out.src.get());
        } catch (...) {
            c.error = std::current_exception();
        }
    };
    std::vector<std::thread> workers;
    workers.reserve(threads);
    for (int t = 1; t < threads; t++) {
        try {
            workers.emplace_back(run, std::ref(chunk[t]));
        } catch (const std::system_error &) {  // no more threads: here
            run(chunk[t]);
        }
    }
    run(chunk[0]);
    for (std::thread &w : workers) w.join();
    for (Chunk &c : chunk)
        if (c.error) std::rethrow_exception(c.error);
    out.ndst = 0;
    for (const Chunk &c : chunk) out.ndst += (int64_t)c.dst.size();
    out.dst.reset(new int32_t[out.ndst]);
    out.ptr.reset(new int64_t[out.ndst + 1]);
    out.seg.assign(1, 0);
    out.seg.reserve(out.first[ns] + 1);
    int64_t d = 0;
    for (const Chunk &c : chunk) {
        std::copy(c.dst.begin(), c.dst.end(), out.dst.get() + d);
        std::copy(c.ptr.begin(), c.ptr.end(), out.ptr.get() + d);
        for (int64_t e : c.ends) out.seg.push_back(d + e);
        d += (int64_t)c.dst.size();
    }
    out.ptr[out.ndst] = out.nsrc;
}

}  // namespace ipm
