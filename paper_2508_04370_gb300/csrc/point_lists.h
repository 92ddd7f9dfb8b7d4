// Host-built lists of the entries that small children add to their parents'
// fronts: one list of arena positions per destination, children ascending.
#pragma once
#include <cstdint>
#include <memory>
#include <vector>

#include "ipm_plan.h"

#ifdef __CUDACC__
#define IPM_LIST_FN __host__ __device__ __forceinline__
#else
#define IPM_LIST_FN inline
#endif

namespace ipm {

constexpr int kAsmRows = 64;    // rows of an assembly item (its columns: a block of 32)
constexpr int kPointRows = 64;  // children of up to this many contribution rows go in as lists

inline int32_t asm_tiles(int32_t f) {  // items of a front of f rows, column blocks ascending
    const int32_t nc = (f + 31) / 32, nr = (f + kAsmRows - 1) / kAsmRows;
    return nc * nr - (nc - 1) * (nc - 1) / 4;  // block column i starts at block row i / 2
}
inline int32_t asm_first_tile(int32_t f, int32_t cb) {  // items of the column blocks before cb
    const int32_t nr = (f + kAsmRows - 1) / kAsmRows;
    return cb * nr - (cb - 1) * (cb - 1) / 4;
}

// A large child's part in a block of columns: its columns [a, a + n) land there, n <=
// 32; AsmLists::rt[rt + i] is where its rows of the front's i-th block of kAsmRows
// rows begin.  (Of a rank-one leaf cb is its column of L, row 1 first, and cb + ldc
// the column -u, u = L d: entry (i, j) of its contribution is l_i (-u_j).)
struct AsmChild {
    int64_t cb, map;  // its contribution block in the arena, its row map
    int64_t rt_n;     // 64 rt + n: a million children under a front of 140,000 rows pass 2^31 in rt
    int32_t ldc, a;
    IPM_LIST_FN int64_t rt() const { return rt_n >> 6; }
    IPM_LIST_FN int32_t n() const { return (int32_t)(rt_n & 63); }
};
inline AsmChild asm_child_of(int64_t cb, int64_t map, int32_t ldc, int32_t a, int32_t n, int64_t rt) {
    return {cb, map, rt * 64 + n, ldc, a};
}

// Item i of front s (a small front is one item, a large one asm_tiles(f)) has the
// destinations [seg[first[s] + i], seg[first[s] + i + 1]) of dst, ascending;
// destination d takes the arena positions src[ptr[d]] .. src[ptr[d + 1]].
// dst: 64 (column % 32) + row % 64 in a large front's item, column ld + row in a
// small front.
struct PointLists {
    std::vector<int64_t> first, seg;
    int64_t ndst = 0, nsrc = 0;
    std::unique_ptr<int32_t[]> dst;
    std::unique_ptr<int64_t[]> ptr, src;  // ndst + 1, nsrc
};
// threads: at most this many (0: by the work and the host's cores); the lists do
// not depend on it
void build_point_lists(const Plan &P, PointLists &out, int threads = 0);

}  // namespace ipm
