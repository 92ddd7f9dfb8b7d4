// Numeric multifrontal factorisation kernels (Zanetti & Gondzio,
// arXiv 2508.04370, Sec. 4.1, 4.4, 4.5), FP64.
//
// Every front s owns a resident f x f slab (column-major, leading dimension
// ld) in one device arena.  After its factorisation the first k columns hold
// L (strictly lower part; D on the diagonal) and the trailing (f-k) x (f-k)
// lower block holds the contribution block (Schur complement) that the
// parent pulls during its own assembly.  The strict upper part of a small
// front's slab holds scratch and is never read; that of a large front holds, for
// each row i below a panel, u_iq = l_iq d_q at (row q, column i), the FP64 updates'
// second operand (written by the triangular solve, read by no one after the
// panel's update).  A rank-one leaf holds -u in its second column instead of a
// contribution block.
//
// A front's entries are summed in one order whatever the schedule: the original
// entry, the children of up to kPointRows contribution rows ascending, the
// larger ones ascending, the rank-one leaves ascending (Sec. 4.3, determinism).
// The pivoting mode's fronts take all children ascending.
//
// Kernels: k_small_fronts (a whole front of f <= 128 in shared memory, one
// CTA per front); the large-front bodies (assembly, diagonal block,
// triangular solve, lookahead strip, trailing tile), run either one launch
// per kind and pivot block or as items of the persistent level kernel
// k_large_level; k_norm1 / k_set_b1 (||K||_1 and the lift floor) and
// k_factor_stats (inertia, lifts).  The tensor-core trailing update is in
// kernels_tc.cu.
//
// Pivot rule (Sec. 4.5, Prop. 3), applied to pivot p of the current pivot
// block [b0, b1) of nb fully-summed columns:
//   d   = F_pp + s_p * sigma_p          (static term after the pivot is computed)
//   b2  = max over j in (p, b1) with s_j = s_p and s_j F_jj > 0 of F_jp^2 / |F_jj|
//   d  <- s_p * max(s_p d, max(eps_piv ||K||_1, b2))
#include <cuda_runtime.h>

#include <cfloat>
#include <cstdint>

#include "ipm_dev.h"
#include "rows_common.cuh"
#include "sliced_common.cuh"

namespace ipm {

namespace {

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ double orig_value(const DevPlan &P, const DevVals &V, int64_t src) {
    if (src >= 0) return P.form == 1 ? V.Ax[src] : V.nev[src];
    const int64_t j = -1 - src;
    return -1.0 / V.theta[j];
}

// Pivot decision of Sec. 4.5 / Prop. 3 for pivot p of the block [0, w) held
// column-major in shared memory (one full warp, w <= 32):
//   d   = F_pp + s_p sigma_p          (static term after the pivot is computed)
//   b2  = max over j in (p, w) with s_j = s_p and s_j F_jj > 0 of F_jp^2 / |F_jj|
//   d  <- s_p max(s_p d, max(eps_piv ||K||_1, b2)).
// Every FP64 instruction costs this GPU about 64 cycles per warp whatever
// the number of active lanes, while integer instructions cost a few, so the
// common case is decided with integer arithmetic on the IEEE bit patterns:
// for non-negative doubles the bit pattern orders like the value, and
// bits(x) / 2^52 - 1023 is a lower bound of log2(x) that is within 0.0861 of
// it for normal x (and an upper-bound-preserving one for subnormal x).  A
// candidate j is screened out when 2 log2|F_jp| < log2|F_jj| + log2(t) - 0.0278
// with t = max(s_p d, eps_piv ||K||_1), which proves F_jp^2 / |F_jj| < t even
// after rounding, so b2 cannot change the pivot.  If any candidate survives
// the screen (rare: in exact arithmetic the same-sign block is definite and
// b2 <= |d|), the bound is evaluated exactly as written above.  Either way the
// result equals the plain evaluation of the rule.  Lane 0 records D, the
// lift and the status and returns the pivot and its reciprocal through
// shared memory.
constexpr long long kSignBit = (long long)0x8000000000000000ull;
constexpr long long kAbsMask = 0x7fffffffffffffffll;
constexpr long long kInfBits = 0x7ff0000000000000ll;
constexpr long long kBias = 0x3ff0000000000000ll;    // bits(1.0)
constexpr long long kScreen = 0x0003333333333333ll;  // 0.2 * 2^52
constexpr long long kTiny = 0x2000000000000000ll;    // bits(2^-511): squares stay normal above it
constexpr long long kHuge = 0x5fe0000000000000ll;    // bits(2^511): squares stay finite below it

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }

// 1 / x for a pivot: the hardware estimate (relative error below 2^-20 for
// normal x) refined by one third-order Newton-Raphson step for the
// reciprocal, r' = r (1 + e + e^2) with e = 1 - x r, whose error is about
// e^3 < 2^-60, below the rounding of the final fused multiply-add (so the
// result is within about half an ulp).  Three dependent FMAs instead of a
// full division on the pivot chain.  Outside [2^-1000, 2^1000] in magnitude
// (never the case for a pivot above the floor eps ||K||_1 of a sensible K)
// it divides.
__device__ __forceinline__ double recip_pivot(double x) {
    const long long a = __double_as_longlong(x) & 0x7fffffffffffffffll;
    if (a < 0x0170000000000000ll || a > 0x7e70000000000000ll) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// x > b for a non-negative, non-NaN b, with IEEE semantics (NaN > b is false).
__device__ __forceinline__ bool gt_nonneg(long long xb, long long bb) {
    return xb >= 0 && xb <= kInfBits && xb > bb;
}

// The exact evaluation of the rule for the lanes the integer screen could
// not settle (maybe).  For non-negative values the rule only takes maxima,
// so it runs on bit patterns: the result is max(s_p d, b1, b2) and a lane
// can change it only if its F_jp^2 / |F_jj| exceeds t = max(s_p d, b1).  A
// second screen decides that without dividing: with a = fl(F_jp^2) and
// b = fl(t |F_jj|), bits(a) < bits(b) - 16 gives a < b (1 - 2^-49) and so
// fl(a / |F_jj|) < t (for lanes inside the first screen's ranges, where no
// product over- or underflows in a way that could mislead it).  Only the
// lanes left over divide, as the rule is written.  Returns the bits of the
// signed pivot.
__device__ __forceinline__ long long pivot_exact_bits(bool maybe, bool screenable, double c, double g, long long tb,
                                                      long long sdb, long long b1b, int sp) {
    bool need = false;
    if (maybe) {
        need = true;
        if (screenable) {
            const long long a = dbits(c * c), b = dbits(__longlong_as_double(tb) * fabs(g));
            need = !(a < b - 16);
        }
    }
    long long b2b = 0;
    if (__any_sync(0xffffffffu, need)) {
        if (need) b2b = dbits(c * c / fabs(g));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long ov = __shfl_xor_sync(0xffffffffu, b2b, o);
            if (ov > b2b) b2b = ov;
        }
    }
    const long long bndb = b1b > b2b ? b1b : b2b;            // max(b1, b2), both >= 0
    const long long res = gt_nonneg(sdb, bndb) ? sdb : bndb;  // s_p d > bnd ? s_p d : bnd
    return sp < 0 ? res ^ kSignBit : res;
}

__device__ __forceinline__ void pivot_warp(const double *Fd, int LDD, int p, int w, const int8_t *sgn, double rho,
                                           double delta, double b1floor, double *dstat, double *piv_out) {
    const int lane = threadIdx.x & 31;
    const int sp = sgn[p];
    const double d = Fd[p * LDD + p] + (sp < 0 ? -rho : delta);
    const long long db = dbits(d);
    const long long sdb = sp < 0 ? db ^ kSignBit : db;  // bits of s_p d
    const long long b1b = dbits(b1floor);
    const long long tb = gt_nonneg(sdb, b1b) ? sdb : b1b;  // bits of t = max(s_p d, b1)
    const bool t_ok = tb > 0x000fffffffffffffll && tb < kInfBits;  // t normal and finite
    bool maybe = false, screenable = false;
    double c = 0.0, g = 0.0;
    const int j = p + 1 + lane;
    if (j < w && sgn[j] == sp) {
        g = Fd[j * LDD + j];
        const long long jb = dbits(g);
        const long long ja = jb & kAbsMask;
        const bool cand = ja != 0 && ja <= kInfBits && ((jb < 0) == (sp < 0));  // s_j F_jj > 0
        if (cand) {
            c = Fd[p * LDD + j];
            const long long ab = dbits(c) & kAbsMask;
            if (ab != 0) {
                screenable = t_ok && ab >= kTiny && ab < kHuge && ja > 0x000fffffffffffffll && ja < kInfBits;
                maybe = !screenable || 2 * (ab - kBias) >= (ja - kBias) + (tb - kBias) - kScreen;
            }
        }
    }
    // the common-case pivot and its reciprocal, started before the vote so
    // that the reciprocal's latency overlaps the screen
    const long long dnb_fast = sp < 0 ? tb ^ kSignBit : tb;
    const double rinv_fast = recip_pivot(__longlong_as_double(dnb_fast));
    long long dnb = dnb_fast;
    if (__any_sync(0xffffffffu, maybe)) dnb = pivot_exact_bits(maybe, screenable, c, g, tb, sdb, b1b, sp);
    if (lane == 0) {
        const double dn = __longlong_as_double(dnb);
        dstat[p] = d;  // the lift dn - d and the status are formed off the chain
        piv_out[0] = dn;
        piv_out[1] = dnb == dnb_fast ? rinv_fast : recip_pivot(dn);
    }
}

// Named barriers, the id chosen by parity so that it stays an immediate:
// sync/arrive on barrier base + (parity & 1) with kCount threads.
template <int kBase, int kCount = 128>
__device__ __forceinline__ void bar_sync_parity(int parity) {
    if (parity & 1) asm volatile("bar.sync %0, %1;" ::"n"(kBase + 1), "n"(kCount) : "memory");
    else asm volatile("bar.sync %0, %1;" ::"n"(kBase), "n"(kCount) : "memory");
}
template <int kBase, int kCount = 128>
__device__ __forceinline__ void bar_arrive_parity(int parity) {
    if (parity & 1) asm volatile("bar.arrive %0, %1;" ::"n"(kBase + 1), "n"(kCount) : "memory");
    else asm volatile("bar.arrive %0, %1;" ::"n"(kBase), "n"(kCount) : "memory");
}

// ------------------------------------------------------------ small fronts
// One CTA per front, the whole front in shared memory.  FP64 is scarce on
// this GPU (about 0.4 FP64 FMA per clock per SM sub-partition), so every
// pivot's work is spread over all warps: warp 0 decides the pivot
// (pivot_warp), all threads scale the pivot column with one reciprocal and
// apply the rank-1 update to the rest of the pivot block's columns (all rows
// below, which also performs the triangular solve of the rows under the
// block); after each block of 32 pivots all threads apply the block to the
// trailing lower part.  The children's entries come as lists per destination
// (children of more than kPointRows rows one by one): a front of 60 rows has up
// to 35 children, and each cost a chain of global reads and a barrier.
//
// Small children's entries, one thread per destination: T[d] += the arena
// values of d's list, children ascending.
__device__ __forceinline__ void sum_points(const AsmLists &A, int64_t g0, int64_t g1, int nthreads,
                                           const double *fronts, double *T) {
    for (int64_t g = g0 + threadIdx.x; g < g1; g += nthreads) {
        const int d = A.seg_dst[g];
        const int64_t e = A.seg_ptr[g + 1];
        double v = T[d];
        int64_t q = A.seg_ptr[g];
        for (; q + 4 <= e; q += 4) {
            double c[4];
#pragma unroll
            for (int u = 0; u < 4; u++) c[u] = __ldcg(fronts + A.src[q + u]);
#pragma unroll
            for (int u = 0; u < 4; u++) v += c[u];
        }
        for (; q < e; q++) v += __ldcg(fronts + A.src[q]);
        T[d] = v;
    }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_small_fronts(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                      double *__restrict__ Dg, double *__restrict__ Dig,
                                                      double *__restrict__ dyng, DevCtl *ctl, AsmLists A,
                                                      const int32_t *__restrict__ list, int nb) {
    extern __shared__ double smem[];
    __shared__ double wcol[128];  // fronts up to 128 rows use this kernel
    __shared__ double dq[32];
    __shared__ double dsm[32];  // statically regularised pivots of the block, before any lift
    __shared__ double piv[2];
    __shared__ int8_t sg[128];
    const int s = list[blockIdx.x];
    const int f = P.sn_f[s], k = P.sn_k[s], ld = P.sn_ld[s], c0 = P.sn_c0[s];
    double *F = smem;  // ld * f
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = NT / 32;
    const int sz = ld * f;
    for (int t = tid; t < sz; t += NT) F[t] = 0.0;
    __syncthreads();
    for (int64_t q = P.orig_ptr[s] + tid; q < P.orig_ptr[s + 1]; q += NT)
        F[P.orig_dst[q]] = orig_value(P, V, P.orig_src[q]);
    __syncthreads();
    sum_points(A, A.small[2 * s], A.small[2 * s + 1], NT, fronts, F);
    __syncthreads();
    for (int q = A.small_big[s]; q < P.child_ptr[s + 1]; q++) {
        const int c = P.child_list[q];
        const int kc = P.sn_k[c], ldc = P.sn_ld[c];
        const int cc = P.sn_f[c] - kc;
        const double *CB = fronts + P.sn_off[c] + (int64_t)kc * ldc + kc;
        const int32_t *map = P.relmap + P.map_off[c];
        for (int t = tid; t < cc * cc; t += NT) {
            const int jj = t / cc, ii = t - jj * cc;
            if (ii >= jj) F[map[jj] * ld + map[ii]] += CB[(int64_t)jj * ldc + ii];
        }
        __syncthreads();
    }
    for (int t = tid; t < k; t += NT) sg[t] = P.sign[c0 + t];
    __syncthreads();
    const int8_t *sgn = sg;
    const double b1floor = pivot_floor(P, ctl, c0);
    for (int b0 = 0; b0 < k; b0 += nb) {
        const int b1 = min(b0 + nb, k), w = b1 - b0;
        double *Fb = F + b0 * ld + b0;
        for (int p = 0; p < w; p++) {
            if (warp == 0) pivot_warp(Fb, ld, p, w, sgn + b0, V.rho, V.delta, b1floor, dsm, piv);
            __syncthreads();
            const double dn = piv[0], rinv = piv[1];
            const int pc = b0 + p;  // front column of the pivot
            for (int i = pc + 1 + tid; i < f; i += NT) {
                const double v = F[pc * ld + i];
                wcol[i] = v;
                F[pc * ld + i] = v * rinv;
            }
            if (tid == 0) {
                F[pc * ld + pc] = dn;
                dq[p] = dn;
                Dig[c0 + pc] = rinv;
            }
            __syncthreads();
            // rank-1 update of the block's remaining columns, all rows below
            for (int j = pc + 1 + warp; j < b0 + w; j += NW) {
                const double wj = wcol[j];
                for (int i = j + lane; i < f; i += 32) F[j * ld + i] -= F[pc * ld + i] * wj;
            }
            __syncthreads();
        }
        // the block's pivots, lifts and status (dq and dsm are rewritten only
        // after the barriers of the trailing update)
        if (tid < w) {
            const double dn = dq[tid], d = dsm[tid];
            const long long db = dbits(d), dnb = dbits(dn);
            Dg[c0 + b0 + tid] = dn;
            dyng[c0 + b0 + tid] = dnb == db ? 0.0 : dn - d;
            const bool fin = (db & kAbsMask) < kInfBits && (dnb & kAbsMask) < kInfBits && (dnb & kAbsMask) != 0;
            if (!fin) atomicOr(&ctl->status, kStatNonFinite);
        }
        // trailing update of columns [b1, f) by the block's pivots:
        // W_jq = L_jq d_q is formed once into the unused upper triangle
        // (row b0 + q of column j), then each entry takes one FMA per pivot
        for (int t = tid; t < w * (f - b1); t += NT) {
            const int q = t % w, j = b1 + t / w;
            F[j * ld + b0 + q] = F[(b0 + q) * ld + j] * dq[q];
        }
        __syncthreads();
        for (int j = b1 + warp; j < f; j += NW) {
            for (int i = j + lane; i < f; i += 32) {
                double acc = 0.0;
                for (int q = 0; q < w; q++) acc += F[(b0 + q) * ld + i] * F[j * ld + b0 + q];
                F[j * ld + i] -= acc;
            }
        }
        __syncthreads();
    }
    double *out = fronts + P.sn_off[s];
    for (int t = tid; t < sz; t += NT) out[t] = F[t];
}

// -------------------------------------------------------------- large fronts
// The work on a large front is cut into items (Sec. 4.4: per pivot block of
// nb = 32 columns, the diagonal block, the triangular solve of the rows below
// it and the trailing update), each written once as a CTA-wide body (256
// threads call it; bodies that need fewer leave the others idle).  The
// bodies serve both the one-launch-per-step kernels and the persistent
// level kernel below.  Front data are read through L2 (ld.global.cg)
// because in the persistent kernel other CTAs of the same launch wrote
// them.  All bodies share one shared-memory pool sized for the largest.
constexpr int kBodyThreads = 256;
constexpr int kPoolDoubles = 2 * 32 * 33 + 32;  // a 32 x 32 update tile's two operands; L_11, 1/d and a 32 x 33 tile

// Assembly of one block of 32 columns x 64 rows of a front: summed in shared
// memory and written once, so a front's assembly reads its children and writes
// itself, where zeroing and read-modify-write in the slab moved three times
// as much.  A front of an LP has a thousand children of a few entries (primal
// columns) and a handful of large ones: the small ones' entries are a list of
// positions per destination (one thread sums one destination; going through
// the children one by one cost a memory round trip and a CTA barrier for
// each), and of the large ones warp w adds the columns = w mod 8, in the
// children's order without CTA barriers, the next child's maps fetched
// while this one's entries arrive.  50-period staircase: the assembly launches
// of a factorisation take 5.6 ms instead of 23.7 (10.8 GB).
__device__ __forceinline__ void body_assemble(const DevPlan &P, const DevVals &V, double *fronts, const AsmLists &A,
                                              const AsmItem &ai, double *pool) {
    constexpr int NT = kBodyThreads, R = kAsmRows;
    static_assert(32 * R <= kPoolDoubles && NT / 32 == 8, "the block fits the pool, four columns per warp");
    double *T = pool;  // column c, row r at T[R (c - c_lo) + r % R]
    const int ld = P.sn_ld[ai.s];
    double *F = fronts + P.sn_off[ai.s];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c_lo = ai.c_lo, r_lo = ai.r_lo, r_hi = ai.r_hi, rbase = r_lo & ~(R - 1);
#pragma unroll
    for (int t = tid; t < 32 * R; t += NT) T[t] = 0.0;
    __syncthreads();
    for (int64_t q = ai.o0 + tid; q < ai.o1; q += NT) {
        const int32_t d = P.orig_dst[q];
        const int c = d / ld, r = d - c * ld;
        if (r >= r_lo && r < r_hi) T[R * (c - c_lo) + r - rbase] = orig_value(P, V, P.orig_src[q]);
    }
    __syncthreads();
    sum_points(A, ai.seg0, ai.seg1, NT, fronts, T);
    __syncthreads();
    // large children: lane j holds the front column of the child's column a + j,
    // and the front rows of the child's rows i0 and i0 + 32
    struct Maps {
        int64_t cb;
        int ldc, a, col, i0, r0, r1;
    };
    auto fetch = [&](int q) {
        const AsmChild C = A.child[q];
        Maps m;
        m.cb = C.cb;
        m.ldc = C.ldc;
        m.a = C.a;
        m.col = lane < C.n() ? __ldg(P.relmap + C.map + C.a + lane) - c_lo : -1;
        const int32_t *rt = A.rt + C.rt() + rbase / R;
        const int ilo = rt[0], ihi = rt[1];
        m.i0 = ilo + lane;
        m.r0 = m.i0 < ihi ? __ldg(P.relmap + C.map + m.i0) - rbase : -1;
        m.r1 = m.i0 + 32 < ihi ? __ldg(P.relmap + C.map + m.i0 + 32) - rbase : -1;
        return m;
    };
    if (ai.ch0 < ai.ch1) {
        Maps m = fetch(ai.ch0);
        for (int q = ai.ch0; q < ai.ch1; q++) {
            const Maps n = fetch(min(q + 1, ai.ch1 - 1));
            unsigned mine = __ballot_sync(0xffffffffu, m.col >= 0 && (m.col & 7) == warp);
            const double *CB = fronts + m.cb;
            double v[4][2];
            int c[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int j = mine ? __ffs(mine) - 1 : 0;
                c[u] = mine ? __shfl_sync(0xffffffffu, m.col, j) : -1;
                mine &= mine - 1;
                const int jj = m.a + j;
                const double *CBj = CB + (int64_t)jj * m.ldc;
                v[u][0] = (c[u] >= 0 && m.r0 >= 0 && m.i0 >= jj) ? __ldcg(CBj + m.i0) : 0.0;
                v[u][1] = (c[u] >= 0 && m.r1 >= 0 && m.i0 + 32 >= jj) ? __ldcg(CBj + m.i0 + 32) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (c[u] < 0) continue;  // uniform over the warp
                if (m.r0 >= 0) T[R * c[u] + m.r0] += v[u][0];
                if (m.r1 >= 0) T[R * c[u] + m.r1] += v[u][1];
            }
            __syncwarp();
            m = n;
        }
    }
    // rank-one leaves: formed here from their columns l and -u (the same
    // FP64 work as adding a stored block), the next child's on their way
    // while one is added
    struct Rank1 {
        double l0, l1, nu;
        int a, col, i0, r0, r1;
    };
    auto leaf = [&](int q) {
        const AsmChild C = A.child[min(q, ai.ch2 - 1)];
        Rank1 m;
        const int32_t *rt = A.rt + C.rt() + rbase / R;
        const int ilo = rt[0], ihi = rt[1];
        const int32_t *map = P.relmap + C.map;
        const double *L = fronts + C.cb;
        m.a = C.a;
        const bool in = lane < C.n();
        m.col = in ? __ldg(map + C.a + lane) - c_lo : -1;
        m.nu = in ? __ldcg(L + C.ldc + C.a + lane) : 0.0;
        m.i0 = ilo + lane;
        m.r0 = m.i0 < ihi ? __ldg(map + m.i0) - rbase : -1;
        m.r1 = m.i0 + 32 < ihi ? __ldg(map + m.i0 + 32) - rbase : -1;
        m.l0 = m.i0 < ihi ? __ldcg(L + m.i0) : 0.0;
        m.l1 = m.i0 + 32 < ihi ? __ldcg(L + m.i0 + 32) : 0.0;
        return m;
    };
    if (ai.ch1 < ai.ch2) {
        Rank1 m = leaf(ai.ch1);
        for (int q = ai.ch1; q < ai.ch2; q++) {
            const Rank1 n = leaf(q + 1);
            unsigned mine = __ballot_sync(0xffffffffu, m.col >= 0 && (m.col & 7) == warp);
            while (mine) {  // uniform over the warp
                const int j = __ffs(mine) - 1;
                mine &= mine - 1;
                const int jj = m.a + j;
                double *Tc = T + R * __shfl_sync(0xffffffffu, m.col, j);
                const double nu = __shfl_sync(0xffffffffu, m.nu, j);
                if (m.r0 >= 0 && m.i0 >= jj) Tc[m.r0] = fma(m.l0, nu, Tc[m.r0]);
                if (m.r1 >= 0 && m.i0 + 32 >= jj) Tc[m.r1] = fma(m.l1, nu, Tc[m.r1]);
            }
            __syncwarp();
            m = n;
        }
    }
    __syncthreads();
    for (int t = tid; t < 32 * R; t += NT) {
        const int c = c_lo + t / R, r = rbase + t % R;
        if (c < ai.c_hi && r >= r_lo && r < r_hi) F[(int64_t)c * ld + r] = T[t];
    }
}

// The nb x nb diagonal block of panel [p0, p0 + nb) of front s as a
// pipeline over the pivots spread over the SM's four sub-partitions (each
// FP64 instruction holds its sub-partition's FP64 pipe for tens of cycles,
// so the pivot chain is kept to as few FP64 instructions as possible on one
// of them).  Warp 0 owns the pivot chain: lane j keeps c = F_jp of the
// current pivot column, g = F_jj and gs = F_jj + s_j sigma_j (the static
// term) up to date; per pivot it screens the Prop. 3 candidates, scales the
// column (l_jp = F_jp / d_p, keeping the unscaled w_jp = F_jp), publishes p,
// and brings gs (first, for the next pivot), c and g to pivot p + 1.  Warp 5
// forms the reciprocal of each pivot's common case (the pivot or the lift
// floor, whichever is larger) from d, handed over through shared memory, while
// warp 0 screens; warp 0 recomputes it only when the exact rule moves the
// pivot.  Warps 2, 3, 6 and 7 apply pivot p to the strictly lower entries
// of columns >= p + 2 while warp 0 already works on pivot p + 1, which needs
// only column p + 1 and the diagonal; each of their threads holds up to four
// of these entries in registers for the whole block and stores one when its
// column has received its last update here.  Named barriers alternate by
// pivot parity (1-2 pivot published, 3-4 columns updated, 5-6 d ready, 7-8
// reciprocal ready), so no side runs more than one pivot ahead.  Every value
// is formed by the same operations as in a single warp, so the factor does
// not depend on the split.  The factorised block goes back to the slab (L
// strictly below the diagonal, D on it) together with D, 1/D and the lifts,
// and the panel workspace ws receives the rows of L_11 (row-major,
// ws[q * 33 + q'] = L_qq') and 1 / d_q for the triangular solve below.
constexpr int kPanelWs = 32 * 33 + 32;  // doubles of panel workspace per large front

__device__ __forceinline__ void body_diag(const DevPlan &P, const DevVals &V, double *__restrict__ fronts,
                                          double *__restrict__ Dg, double *__restrict__ Dig,
                                          double *__restrict__ dyng, DevCtl *ctl, int s, int p0, int nb,
                                          double *__restrict__ ws, double *pool) {
    // warp 0 (SM sub-partition 0) carries the chain, warp 5 (sub-partition 1)
    // forms each pivot's reciprocal, warps 2, 3, 6 and 7 (sub-partitions 2
    // and 3) apply the pivots to the later columns
    constexpr int LDD = 33, NU = 128, kOwn = 4;  // 4 x 128 >= 435 entries
    constexpr int kBarPub = 1, kBarUpd = 3, kBarD = 5, kBarR = 7;
    constexpr int kPubCount = 32 + NU;  // warp 0 and the update warps
    double *Fd = pool;                          // 32 x 33, column-major
    double(*wsv)[32] = reinterpret_cast<double(*)[32]>(pool + 32 * 33);  // [2][32]
    double *Dtmp = pool + 32 * 33 + 64, *dstat = Dtmp + 32, *rtmp = dstat + 32;
    int8_t *sg = reinterpret_cast<int8_t *>(rtmp + 32);
    double *shd = rtmp + 32 + 4, *shr = shd + 2;  // pivot d and its reciprocal, by pivot parity
    const int k = P.sn_k[s], ld = P.sn_ld[s], c0 = P.sn_c0[s];
    const int w = min(p0 + nb, k) - p0;
    if (w <= 0) return;  // uniform over the CTA
    double *F = fronts + P.sn_off[s];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {
        // all loads in flight before the shared-memory stores
        constexpr int U = 32 * 32 / kBodyThreads;
        double v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads, jj = t >> 5, ii = t & 31;
            v[u] = (jj < w && ii < w && ii >= jj) ? __ldcg(F + (int64_t)(p0 + jj) * ld + (p0 + ii)) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads;
            Fd[(t >> 5) * LDD + (t & 31)] = v[u];
        }
    }
    if (tid < 32) sg[tid] = tid < w ? P.sign[c0 + p0 + tid] : (int8_t)0;
    __syncthreads();
    if (warp == 0) {
        const double b1floor = pivot_floor(P, ctl, c0);
        const long long b1b = dbits(b1floor);
        const int sl = sg[lane];
        double g = lane < w ? Fd[lane * LDD + lane] : 0.0;   // F_jj of row j = lane
        double gs = g + (sl < 0 ? -V.rho : V.delta);
        double c = (lane > 0 && lane < w) ? Fd[lane] : 0.0;  // column 0
        double my_dn = 0.0, my_d = 0.0, my_r = 0.0;          // lane p keeps pivot p's values
        double d = __shfl_sync(0xffffffffu, gs, 0);
        if (lane == 0) shd[0] = d;
        __syncwarp();
        bar_arrive_parity<kBarD, 64>(0);
        for (int p = 0; p < w; p++) {
            const int sp = __shfl_sync(0xffffffffu, sl, p);
            // the Prop. 3 screen (on IEEE bit patterns) while warp 5 forms the
            // reciprocal of the common-case pivot
            const long long db = dbits(d);
            const long long sdb = sp < 0 ? db ^ kSignBit : db;
            const long long tb = gt_nonneg(sdb, b1b) ? sdb : b1b;
            const bool t_ok = tb > 0x000fffffffffffffll && tb < kInfBits;
            bool maybe = false, screenable = false;
            if (lane > p && lane < w && sl == sp) {
                const long long jb = dbits(g);
                const long long ja = jb & kAbsMask;
                const bool cand = ja != 0 && ja <= kInfBits && ((jb < 0) == (sp < 0));
                if (cand) {
                    const long long ab = dbits(c) & kAbsMask;
                    if (ab != 0) {
                        screenable = t_ok && ab >= kTiny && ab < kHuge && ja > 0x000fffffffffffffll && ja < kInfBits;
                        maybe = !screenable || 2 * (ab - kBias) >= (ja - kBias) + (tb - kBias) - kScreen;
                    }
                }
            }
            const long long dnb_fast = sp < 0 ? tb ^ kSignBit : tb;
            const bool any = __any_sync(0xffffffffu, maybe);
            bar_sync_parity<kBarR, 64>(p);
            double rinv = shr[p & 1];
            long long dnb = dnb_fast;
            if (any) {
                dnb = pivot_exact_bits(maybe, screenable, c, g, tb, sdb, b1b, sp);
                if (dnb != dnb_fast) rinv = recip_pivot(__longlong_as_double(dnb));
            }
            const double dn = __longlong_as_double(dnb);
            if (lane == p) {
                my_dn = dn;
                my_d = d;
                my_r = rinv;
            }
            const bool below = lane > p && lane < w;
            const double l = below ? c * rinv : 0.0;
            if (below) {
                Fd[p * LDD + lane] = l;
                wsv[p & 1][lane] = c;
            }
            __syncwarp();
            bar_arrive_parity<kBarPub, kPubCount>(p);
            if (p + 1 < w) {
                if (p >= 1) bar_sync_parity<kBarUpd, kPubCount>(p + 1);  // pivot p-1 applied to columns >= p+1
                const double wn = __shfl_sync(0xffffffffu, c, p + 1);  // w_{p+1,p}, unscaled
                const double fv = (lane > p + 1 && lane < w) ? Fd[(p + 1) * LDD + lane] : 0.0;
                // the next pivot first, so that its reciprocal starts early
                gs -= l * c;
                d = __shfl_sync(0xffffffffu, gs, p + 1);
                if (lane == 0) shd[(p + 1) & 1] = d;
                __syncwarp();
                bar_arrive_parity<kBarD, 64>(p + 1);
                const double cn = fv - l * wn;
                g -= l * c;
                c = lane > p + 1 ? cn : 0.0;
            }
        }
        // the pivots' values, off the chain (read only after the CTA barrier)
        if (lane < w) {
            Fd[lane * LDD + lane] = my_dn;
            Dtmp[lane] = my_dn;
            dstat[lane] = my_d;
            rtmp[lane] = my_r;
            const long long db = dbits(my_d), dnb = dbits(my_dn);
            const bool fin = (db & kAbsMask) < kInfBits && (dnb & kAbsMask) < kInfBits && (dnb & kAbsMask) != 0;
            if (!fin) atomicOr(&ctl->status, kStatNonFinite);
        }
    } else if (warp == 5) {
        // the reciprocal of each pivot's common case: the larger (as bit
        // patterns) of s_p d and the lift floor, with the sign s_p
        const long long b1b = dbits(pivot_floor(P, ctl, c0));
        for (int p = 0; p < w; p++) {
            const int sp = sg[p];
            bar_sync_parity<kBarD, 64>(p);
            const long long db = dbits(shd[p & 1]);
            const long long sdb = sp < 0 ? db ^ kSignBit : db;
            const long long tb = gt_nonneg(sdb, b1b) ? sdb : b1b;
            const double r = recip_pivot(__longlong_as_double(sp < 0 ? tb ^ kSignBit : tb));
            if (lane == 0) shr[p & 1] = r;
            __syncwarp();
            bar_arrive_parity<kBarR, 64>(p);
        }
    } else if (warp == 2 || warp == 3 || warp == 6 || warp == 7) {
        // this thread owns the strictly lower entries e = ut + 128 t of columns
        // >= 2, enumerated last column first: e = r (r + 1) / 2 + c  ->
        // column w-2-r, row w-1-r+c (0 <= c <= r)
        const int ut = ((warp & 3) - 2 + 2 * (warp >> 2)) * 32 + lane;
        const int nall = w >= 3 ? (w - 3) * (w - 2) / 2 : 0;
        int jo[kOwn], io[kOwn];
        double vo[kOwn];
#pragma unroll
        for (int t = 0; t < kOwn; t++) {
            const int e = ut + NU * t;
            jo[t] = 0;
            io[t] = 0;
            vo[t] = 0.0;
            if (e < nall) {
                int r = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
                while ((r + 1) * (r + 2) / 2 <= e) r++;
                while (r * (r + 1) / 2 > e) r--;
                jo[t] = w - 2 - r;
                io[t] = w - 1 - r + (e - r * (r + 1) / 2);
                vo[t] = Fd[jo[t] * LDD + io[t]];
            }
        }
        for (int q = 0; q < w; q++) {
            bar_sync_parity<kBarPub, kPubCount>(q);
            const int m = w - 3 - q;  // columns >= q + 2 have m (m + 1) / 2 such entries
            const int ne = m > 0 ? m * (m + 1) / 2 : 0;
            double lq[kOwn], wq[kOwn];
#pragma unroll
            for (int t = 0; t < kOwn; t++) {
                const bool on = ut + NU * t < ne;
                lq[t] = on ? Fd[q * LDD + io[t]] : 0.0;
                wq[t] = on ? wsv[q & 1][jo[t]] : 0.0;
            }
#pragma unroll
            for (int t = 0; t < kOwn; t++) {
                if (ut + NU * t < ne) {
                    vo[t] -= lq[t] * wq[t];
                    if (jo[t] == q + 2) Fd[jo[t] * LDD + io[t]] = vo[t];
                }
            }
            if (q <= w - 3) bar_arrive_parity<kBarUpd, kPubCount>(q);
        }
    }
    __syncthreads();
    for (int t = tid; t < 32 * 32; t += kBodyThreads) {
        const int jj = t >> 5, ii = t & 31;
        const bool in = jj < w && ii < w;
        if (in && ii >= jj) F[(int64_t)(p0 + jj) * ld + (p0 + ii)] = Fd[jj * LDD + ii];
        ws[ii * 33 + jj] = (in && ii > jj) ? Fd[jj * LDD + ii] : 0.0;  // L(row ii, column jj), row-major
    }
    if (tid < 32) {
        const int t = tid;
        ws[32 * 33 + t] = t < w ? rtmp[t] : 0.0;
        if (t < w) {
            const double dn = Dtmp[t], d = dstat[t];
            Dg[c0 + p0 + t] = dn;
            Dig[c0 + p0 + t] = rtmp[t];
            dyng[c0 + p0 + t] = dbits(dn) == dbits(d) ? 0.0 : dn - d;
        }
    }
}

// Rows [r0, r1) below the diagonal block of panel [p0, p0 + nb), one warp
// per row with one lane per pivot column q.  With u_iq = l_iq d_q the rows
// satisfy
//   u_iq = F_iq - sum_{q' < q} u_iq' L_qq',   l_iq = u_iq / d_q,
// so step q' broadcasts the finished u_iq' and every lane q > q' applies one
// FMA: 32 dependent steps per row instead of 528 per thread when a thread
// owns a whole row.  An item holds up to kTrsmItemRows rows (chunks of the
// level kernel hold kTrsmRows); warp w solves rows w, w + 8, w + 16 and
// w + 24 together, four independent chains on the same L_11, so a CTA costs
// about one chain's latency.
//
// The unscaled u_iq = l_iq d_q, which the FP64 updates take as their second
// operand, is left at the mirrored place (row p0 + q, column i of the front's
// unused upper part): a product per operand entry and tile was 3% of the updates'
// FP64 work, which bounds them.  A factorisation of the 10-period staircase in
// FP64 takes 74.2 ms instead of 77.0, of 64 random LPs at once 15.0 instead of
// 15.5.  (Not for rows that are sliced for the tensor cores.)
constexpr int kTrsmRows = 8;
constexpr int kTrsmItemRows = 32;
static_assert(kTrsmRows == kTrsmRowsHost && kTrsmItemRows == kTrsmItemRowsHost, "host and device row chunks differ");
static_assert(32 * kTrsmRows == kBodyThreads, "one warp per row");

// Where the triangular solve of a sliced front writes the digit slices of the
// rows it finishes (ws == nullptr: no slicing): block base + (row - p1) / 128,
// row (row - p1) % 128 of the step's work space.  pair = 0: one chunk, this
// panel's columns; pair = 1 (the second panel of a pair): two chunks with one
// row scale, the previous panel's 32 columns (final since the last step)
// and this panel's.
struct SliceOut {
    uint8_t *ws;
    int32_t *exps;
    int32_t base;
    int32_t pair;
    int32_t p1;
    const double *D;
    DevCtl *ctl;
};

template <int RW>  // rows per warp, solved together: items of up to 8 RW rows
__device__ __forceinline__ void body_trsm(const DevPlan &P, double *__restrict__ fronts, int s, int r0, int r1,
                                          int p0, int nb, const double *__restrict__ ws, double *pool,
                                          const SliceOut so = SliceOut{nullptr, nullptr, 0, 0, 0, nullptr, nullptr}) {
    constexpr int kRows = kTrsmRows * RW;
    constexpr int TP = kRows + 1;  // padded row count of the tile
    double *Wd = pool;                             // 32 x 33 + 32
    double(*T)[TP] = reinterpret_cast<double(*)[TP]>(pool + 32 * 33 + 32);  // [32 columns][rows]
    const int k = P.sn_k[s], ld = P.sn_ld[s];
    const int w = min(p0 + nb, k) - p0;
    const int nr = r1 - r0;  // <= kRows
    double *F = fronts + P.sn_off[s];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {
        // all loads in flight before the shared-memory stores
        constexpr int U = (32 * 33 + 32 + kBodyThreads - 1) / kBodyThreads;
        constexpr int V = 32 * kRows / kBodyThreads;
        double v[U], tv[V];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads;
            v[u] = t < 32 * 33 + 32 ? __ldcg(ws + t) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < V; u++) {
            const int t = tid + u * kBodyThreads, q = t / kRows, r = t % kRows;
            tv[u] = (q < w && r < nr) ? __ldcg(F + (int64_t)(p0 + q) * ld + r0 + r) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads;
            if (t < 32 * 33 + 32) Wd[t] = v[u];
        }
#pragma unroll
        for (int u = 0; u < V; u++) {
            const int t = tid + u * kBodyThreads;
            T[t / kRows][t % kRows] = tv[u];
        }
    }
    __syncthreads();
    if constexpr (RW == 4) {
        // rows warp, warp + 8, warp + 16 and warp + 24, eight lanes each: lane e of
        // a row holds columns e, e + 8, e + 16 and e + 24, so that a finished u is
        // applied to the columns after its block of eight only (79 FMAs per warp;
        // a lane per column and a row after the other takes 124, half of them on
        // columns that are finished)
        const int e = lane & 7, rr = warp + kTrsmRows * (lane >> 3);
        if (warp < nr) {
            double t[4];
#pragma unroll
            for (int b = 0; b < 4; b++) t[b] = T[8 * b + e][rr];
#pragma unroll
            for (int c = 0; c < 31; c++) {
                const double u = __shfl_sync(0xffffffffu, t[c >> 3], (lane & 24) | (c & 7));
#pragma unroll
                for (int b = c >> 3; b < 4; b++)
                    if (8 * b + e > c) t[b] -= u * Wd[(8 * b + e) * 33 + c];
            }
            double *U = F + (int64_t)(r0 + rr) * ld + p0;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                if (!so.ws && rr < nr && 8 * b + e < w) U[8 * b + e] = t[b];
                T[8 * b + e][rr] = t[b] * Wd[32 * 33 + 8 * b + e];
            }
        }
        __syncwarp();
    } else if (warp < nr) {
        // row warp, one lane per column
        double Lr[32];
#pragma unroll
        for (int c = 0; c < 32; c++) Lr[c] = Wd[lane * 33 + c];
        double t = T[lane][warp];
#pragma unroll
        for (int c = 0; c < 31; c++) {
            const double u = __shfl_sync(0xffffffffu, t, c);
            if (lane > c) t -= u * Lr[c];
        }
        if (!so.ws && lane < w) F[(int64_t)(r0 + warp) * ld + p0 + lane] = t;
        T[lane][warp] = t * Wd[32 * 33 + lane];
        __syncwarp();
    }
    if (so.ws) {
        // the finished rows, sliced for the tensor-core update
        const int c0 = P.sn_c0[s];
        const double dq = lane < w ? so.D[c0 + p0 + lane] : 0.0;
        for (int rr = warp; rr < nr; rr += kTrsmRows) {
            const int row = r0 + rr;
            const double lq = lane < w ? T[lane][rr] : 0.0;
            const int blk = so.base + (row - so.p1) / kSliceRows;
            uint8_t *bp = so.ws + (int64_t)blk * kSliceBlockBytes;
            int32_t *ep = so.exps + (int64_t)blk * kSliceRows * 2;
            bool bad;
            if (so.pair) {
                // the previous panel (always 32 columns) as chunk 0, this one as chunk 1
                const double l2[2] = {__ldcg(F + (int64_t)(p0 - 32 + lane) * ld + row), lq};
                const double d2[2] = {so.D[c0 + p0 - 32 + lane], dq};
                bad = sliced::slice_row_warp<2>(l2, d2, bp, ep, (row - so.p1) % kSliceRows);
            } else {
                const double l1[1] = {lq}, d1[1] = {dq};
                bad = sliced::slice_row_warp<1>(l1, d1, bp, ep, (row - so.p1) % kSliceRows);
            }
            if (bad && lane == 0) atomicOr(&so.ctl->status, kStatNonFinite);
        }
    }
    __syncthreads();
    for (int t = tid; t < 32 * kRows; t += kBodyThreads) {
        const int q = t / kRows, r = t % kRows;
        if (q < w && r < nr) F[(int64_t)(p0 + q) * ld + r0 + r] = T[q][r];
    }
}

// Trailing update of the lower part of columns [p1, f) by the panel
// [p0, p0+w): C(i, j) -= sum_q L(i,q) u(j,q), u = L d, one kUpdTile x kUpdTile
// tile at (i0, j0), 16 x 16 threads with 2 x 2 outputs each.  FP64 runs at
// about 2 FMA per clock per SM on this GPU, so tiles are small (32 x 32) to
// put every SM to work.
__device__ __forceinline__ void body_tile(const DevPlan &P, double *__restrict__ fronts,
                                          int s, int i0, int j0, int p0, int w,
                                          double *pool) {
    constexpr int T = kUpdTile;
    static_assert(T == 32, "16 x 16 threads, 2 x 2 outputs");
    double(*As)[T + 1] = reinterpret_cast<double(*)[T + 1]>(pool);
    double(*Bs)[T + 1] = reinterpret_cast<double(*)[T + 1]>(pool + 32 * (T + 1));
    const int f = P.sn_f[s], ld = P.sn_ld[s];
    w = min(w, P.sn_k[s] - p0);  // ragged last panel
    double *F = fronts + P.sn_off[s];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    // this thread's 2 x 2 outputs of the tile (lower part, columns from the
    // panel's end), fetched with the operands: their latency overlaps the
    // operand loads instead of following the products
    double cv[2][2];
#pragma unroll
    for (int b = 0; b < 2; b++) {
        const int j = j0 + ty + 16 * b;
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const int i = i0 + tx + 16 * a;
            cv[a][b] = (j < f && j >= p0 + w && i < f && i >= j) ? __ldcg(F + (int64_t)j * ld + i) : 0.0;
        }
    }
    {
        // all loads in flight before the shared-memory stores
        constexpr int U = 32 * T / kBodyThreads;
        double va[U], vb[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads, q = t / T, r = t % T;
            const int i = i0 + r, j = j0 + q;
            va[u] = (q < w && i < f) ? __ldcg(F + (int64_t)(p0 + q) * ld + i) : 0.0;
            // u_jr at its mirrored place (columns before the panel's end have none)
            vb[u] = (r < w && j < f && j >= p0 + w) ? __ldcg(F + (int64_t)j * ld + p0 + r) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads, q = t / T, r = t % T;
            As[q][r] = va[u];
            Bs[r][q] = vb[u];
        }
    }
    __syncthreads();
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    for (int q = 0; q < w; q++) {
        const double a0 = As[q][tx], a1 = As[q][tx + 16];
        const double b0 = Bs[q][ty], b1 = Bs[q][ty + 16];
        acc[0][0] += a0 * b0;
        acc[1][0] += a1 * b0;
        acc[0][1] += a0 * b1;
        acc[1][1] += a1 * b1;
    }
#pragma unroll
    for (int b = 0; b < 2; b++) {
        const int j = j0 + ty + 16 * b;
        if (j >= f || j < p0 + w) continue;  // a grid tile cut by a partial last panel
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const int i = i0 + tx + 16 * a;
            if (i < f && i >= j) F[(int64_t)j * ld + i] = cv[a][b] - acc[a][b];
        }
    }
}

// The same update for the next panel's columns, which lie on the critical
// path: a strip of kUpdTile rows x kStripCols columns at (i0, j0), one
// output per thread on threads 0..32 kStripCols - 1, summed over the panel's
// pivots in the same order as body_tile (so the results are identical).  A
// whole 32 x 32 tile is 32k FP64 FMAs, about 8 us on one SM of this GPU;
// strips spread those few tiles over eight times as many SMs.
__device__ __forceinline__ void body_strip(const DevPlan &P, double *__restrict__ fronts,
                                           int s, int i0, int j0, int p0, int w,
                                           double *pool) {
    constexpr int T = kUpdTile, C = kStripCols;
    static_assert(T == 32 && 32 * C <= kBodyThreads, "one row per lane, one column per warp");
    double(*As)[T + 1] = reinterpret_cast<double(*)[T + 1]>(pool);
    double(*Bs)[C] = reinterpret_cast<double(*)[C]>(pool + 32 * (T + 1));
    const int f = P.sn_f[s], ld = P.sn_ld[s];
    w = min(w, P.sn_k[s] - p0);
    double *F = fronts + P.sn_off[s];
    const int tid = threadIdx.x;
    {
        // all loads in flight before the shared-memory stores
        constexpr int U = 32 * T / kBodyThreads;
        double va[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads, q = t / T, r = t % T;
            va[u] = (q < w && i0 + r < f) ? __ldcg(F + (int64_t)(p0 + q) * ld + i0 + r) : 0.0;
        }
        double vb = 0.0;
        const int q = tid & 31, cc = tid >> 5, j = j0 + cc;
        if (cc < C && q < w && j < f && j >= p0 + w) vb = __ldcg(F + (int64_t)j * ld + p0 + q);
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int t = tid + u * kBodyThreads;
            As[t / T][t % T] = va[u];
        }
        if (cc < C) Bs[q][cc] = vb;
    }
    __syncthreads();
    const int r = tid & 31, cc = tid >> 5;
    const int i = i0 + r, j = j0 + cc;
    if (cc < C && i < f && j < f && i >= j && j >= p0 + w) {
        double acc = 0.0;
        for (int q = 0; q < w; q++) acc += As[q][r] * Bs[q][cc];
        double *e = F + (int64_t)j * ld + i;
        *e = __ldcg(e) - acc;
    }
}

// One launch per step: one item per CTA.
__global__ void __launch_bounds__(kBodyThreads) k_large_assemble(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                                  AsmLists A, int64_t first) {
    __shared__ double pool[32 * kAsmRows];
    const AsmItem ai = A.items[first + blockIdx.x];
    body_assemble(P, V, fronts, A, ai, pool);
}

__global__ void __launch_bounds__(kBodyThreads) k_panel_diag(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                              double *__restrict__ Dg, double *__restrict__ Dig,
                                                              double *__restrict__ dyng, DevCtl *ctl,
                                                              const PanelItem *__restrict__ items, int nb,
                                                              double *__restrict__ pws) {
    __shared__ double pool[kPoolDoubles];
    const PanelItem it = items[blockIdx.x];
    body_diag(P, V, fronts, Dg, Dig, dyng, ctl, it.s, it.p0, nb, pws + (int64_t)it.r1 * kPanelWs, pool);
}

template <int RW>
__global__ void __launch_bounds__(kBodyThreads) k_panel_trsm(DevPlan P, double *__restrict__ fronts,
                                                              const PanelItem *__restrict__ items,
                                                              const int32_t *slots, int nb,
                                                              const double *__restrict__ pws,
                                                              const int32_t *__restrict__ sbase, uint8_t *sws,
                                                              int32_t *sexp, const double *__restrict__ Dg,
                                                              DevCtl *ctl) {
    __shared__ double pool[kPoolDoubles];
    const PanelItem it = items[blockIdx.x];
    SliceOut so{nullptr, nullptr, 0, 0, 0, nullptr, nullptr};
    if (sws && sbase[blockIdx.x] >= 0)
        so = SliceOut{sws, sexp, sbase[blockIdx.x] >> 1, sbase[blockIdx.x] & 1, min(it.p0 + nb, P.sn_k[it.s]), Dg,
                      ctl};
    body_trsm<RW>(P, fronts, it.s, it.r0, it.r1, it.p0, nb, pws + (int64_t)slots[blockIdx.x] * kPanelWs, pool, so);
}

__global__ void __launch_bounds__(kBodyThreads) k_large_update(DevPlan P, double *__restrict__ fronts,
                                                                const TileItem *__restrict__ items, int w) {
    __shared__ double pool[kPoolDoubles];
    const TileItem it = items[blockIdx.x];
    body_tile(P, fronts, it.s, it.i0, it.j0, it.p0, w, pool);
}

__global__ void __launch_bounds__(kBodyThreads) k_large_update_strip(DevPlan P, double *__restrict__ fronts,
                                                                        const TileItem *__restrict__ items, int w) {
    __shared__ double pool[kPoolDoubles];
    const TileItem it = items[blockIdx.x];
    body_strip(P, fronts, it.s, it.i0, it.j0, it.p0, w, pool);
}

// A rank-one leaf: a large front of one column without children (a long
// column of an LP, eliminated first).  Its contribution -l d l' is not formed
// here: it would be f^2 / 2 numbers to write and read again, where the parent's
// assembly needs one FMA per entry from l and u = l d (the unscaled column) just
// as it needs one addition per stored entry.  So this kernel only scales the
// column by the pivot's reciprocal (the pivot rule of body_diag with no other
// candidate in the block) and leaves -u in the front's second column, and is
// bound by its loads.  7,702 leaves of 300 rows (40 block-angular blocks with 300
// dense rows): 33 us, and the assembly of their 40 parents no slower, where
// forming their 2.8 GB of blocks took 1.9 ms of the factorisation's 7.9.
constexpr int kRankOneThreads = 128;

__global__ void __launch_bounds__(kRankOneThreads) k_rank_one(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                              double *__restrict__ Dg, double *__restrict__ Dig,
                                                              double *__restrict__ dyng, DevCtl *ctl,
                                                              const int32_t *__restrict__ list) {
    __shared__ double sh_r;
    const int s = list[blockIdx.x];
    const int f = P.sn_f[s], ld = P.sn_ld[s], c0 = P.sn_c0[s];
    const int tid = threadIdx.x;
    double *F = fronts + P.sn_off[s];
    const int64_t o0 = P.orig_ptr[s], o1 = P.orig_ptr[s + 1];
    if (o1 - o0 < f) {
        for (int i = tid; i < f; i += kRankOneThreads) F[i] = 0.0;
        __syncthreads();
    }
    for (int64_t q = o0 + tid; q < o1; q += kRankOneThreads) F[P.orig_dst[q]] = orig_value(P, V, P.orig_src[q]);
    __syncthreads();
    if (tid == 0) {
        const int sp = P.sign[c0];
        const double d = F[0] + (sp < 0 ? -V.rho : V.delta);
        const long long db = dbits(d), b1b = dbits(pivot_floor(P, ctl, c0));
        const long long sdb = sp < 0 ? db ^ kSignBit : db;
        const long long tb = gt_nonneg(sdb, b1b) ? sdb : b1b;
        const long long dnb = sp < 0 ? tb ^ kSignBit : tb;
        const double dn = __longlong_as_double(dnb), r = recip_pivot(dn);
        const bool fin = (db & kAbsMask) < kInfBits && (dnb & kAbsMask) < kInfBits && (dnb & kAbsMask) != 0;
        if (!fin) atomicOr(&ctl->status, kStatNonFinite);
        F[0] = dn;
        Dg[c0] = dn;
        Dig[c0] = r;
        dyng[c0] = dnb == db ? 0.0 : dn - d;
        sh_r = r;
    }
    __syncthreads();
    const double r = sh_r;
    for (int i = 1 + tid; i < f; i += kRankOneThreads) {
        const double u = F[i];
        F[i] = u * r;
        F[ld + i] = __longlong_as_double(dbits(u) ^ kSignBit);
    }
}

// A thin leaf (a front without children, one pivot block, f <= kThinMaxF) whole
// in one CTA.  Every entry gets the operations of the per-step path in its
// order, so the front's values are those of that path bit for bit; what differs
// is what moves: the rows of L are kept in shared memory, the contribution block
// is formed and written in one pass (0 minus the products, where the steps zero
// it, read it and write it), and up to kThinCols pivot columns a thread solves a
// row by itself.  Bound by that write for a few columns, by the products
// (FP64, two per clock and SM) for many; where each side wins: thin_leaf.
constexpr int kThinPanel = 6144;  // doubles of L kept (three CTAs per SM fit)
__global__ void __launch_bounds__(kBodyThreads, 3) k_thin_fronts(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                               double *__restrict__ Dg, double *__restrict__ Dig,
                                                               double *__restrict__ dyng, DevCtl *ctl,
                                                               const int32_t *__restrict__ list,
                                                               const int32_t *__restrict__ slots,
                                                               double *__restrict__ pws, int nb) {
    extern __shared__ double panel[];
    __shared__ double pool[kPoolDoubles];
    const int s = list[blockIdx.x];
    const int f = P.sn_f[s], k = P.sn_k[s], ld = P.sn_ld[s];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double *F = fronts + P.sn_off[s];
    // originals lie in the pivot columns
    for (int c = warp; c < k; c += kBodyThreads / 32)
        for (int r = c + lane; r < f; r += 32) F[(int64_t)c * ld + r] = 0.0;
    __syncthreads();
    for (int64_t q = P.orig_ptr[s] + tid; q < P.orig_ptr[s + 1]; q += kBodyThreads)
        F[P.orig_dst[q]] = orig_value(P, V, P.orig_src[q]);
    __syncthreads();
    double *ws = pws + (int64_t)slots[blockIdx.x] * kPanelWs;
    body_diag(P, V, fronts, Dg, Dig, dyng, ctl, s, 0, nb, ws, pool);
    __syncthreads();
    if (k <= kThinCols) {
        // u_q = F_iq - sum_{q' < q} u_q' L_qq', l_q = u_q / d_q
        for (int i = k + tid; i < f; i += kBodyThreads) {
            double u[kThinCols];
#pragma unroll
            for (int q = 0; q < kThinCols; q++) {
                u[q] = q < k ? F[(int64_t)q * ld + i] : 0.0;
#pragma unroll
                for (int c = 0; c < q; c++)
                    if (q < k) u[q] -= u[c] * ws[q * 33 + c];
            }
#pragma unroll
            for (int q = 0; q < kThinCols; q++)
                if (q < k) {
                    F[(int64_t)i * ld + q] = u[q];
                    F[(int64_t)q * ld + i] = u[q] * ws[32 * 33 + q];
                }
        }
        __syncthreads();
    } else {
        for (int r0 = k; r0 < f; r0 += kTrsmRows) {
            body_trsm<1>(P, fronts, s, r0, min(r0 + kTrsmRows, f), 0, nb, ws, pool);
            __syncthreads();
        }
    }
    // the rows of L: in shared memory where they fit
    const bool kept = k * f <= kThinPanel;
    const double *Lp = kept ? panel : F;
    const int ls = kept ? f : ld;
    if (kept) {
        for (int q = 0; q < k; q++)
            for (int i = k + tid; i < f; i += kBodyThreads) panel[q * f + i] = F[(int64_t)q * ld + i];
        __syncthreads();
    }
    auto u_of = [&](int j) { return j < f && lane < k ? __ldcg(F + (int64_t)j * ld + lane) : 0.0; };
    double bn = u_of(k + warp);
    for (int j = k + warp; j < f; j += kBodyThreads / 32) {
        const double b = bn;
        bn = u_of(j + kBodyThreads / 32);
        constexpr int U = 4;  // rows a lane carries together
        for (int i0 = j + lane; i0 - lane < f; i0 += 32 * U) {
            double acc[U];
#pragma unroll
            for (int u = 0; u < U; u++) acc[u] = 0.0;
            for (int q = 0; q < k; q++) {
                const double bq = __shfl_sync(0xffffffffu, b, q);
                const double *Lq = Lp + q * ls + i0;
#pragma unroll
                for (int u = 0; u < U; u++)
                    if (i0 - lane + 32 * u < f) acc[u] += (i0 + 32 * u < f ? Lq[32 * u] : 0.0) * bq;
            }
            double *e = F + (int64_t)j * ld + i0;
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (i0 + 32 * u >= f) continue;
                // 0 - acc without an FP64 instruction (0 - 0 is +0)
                const long long bits = dbits(acc[u]);
                e[32 * u] = (bits & kAbsMask) ? __longlong_as_double(bits ^ kSignBit) : 0.0;
            }
        }
    }
}

// Persistent level kernel: all large-front items of one tree level in one
// launch.  CTAs take tickets in the host's order, wait (thread 0, bounded
// spin on acquire loads) until the item's counters reach their thresholds,
// run the item's body, and add the item's increment to its completion
// counter (release: thread 0 fences after the CTA barrier).
// Every item waits only on items with smaller tickets, which were taken by
// running CTAs, so the launch completes whatever the grid size.  A wait
// that runs out sets kStatTimeout and the item proceeds (its results are
// then wrong, but the launch still ends).
__device__ __forceinline__ int ld_acquire_i32(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Once some wait of the launch has given up, the others stop at their next
// check of the status word, so a failed launch ends after one wait limit.
__device__ __forceinline__ void wait_counter(const int32_t *cnt, int need, DevCtl *ctl, long long limit) {
    long long spins = 0;
    while (ld_acquire_i32(cnt) < need) {
        if (++spins > limit) {
            atomicOr(&ctl->status, kStatTimeout);
            break;
        }
        if ((spins & 1023) == 0 && (*(volatile int32_t *)&ctl->status & kStatTimeout)) break;
        __nanosleep(64);
    }
}

__global__ void __launch_bounds__(kBodyThreads) k_large_level(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                               double *__restrict__ Dg, double *__restrict__ Dig,
                                                               double *__restrict__ dyng, DevCtl *ctl,
                                                               const FactorItem *__restrict__ items, int nitems,
                                                               int32_t *sync, AsmLists A,
                                                               double *__restrict__ pws, int nb, long long limit) {
    __shared__ double pool[kPoolDoubles];
    __shared__ FactorItem sh_it;
    int32_t *cnt = sync + 1;
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) {
            const int t = atomicAdd(sync, 1);
            FactorItem a;
            a.kind = -1;
            if (t < nitems) a = items[t];
            sh_it = a;
        }
        __syncthreads();
        const FactorItem it = sh_it;  // (rewritten after the barriers below)
        if (it.kind < 0) break;
        if (tid == 0) {
            if (it.wait0 >= 0) wait_counter(cnt + it.wait0, it.need0, ctl, limit);
            if (it.wait1 >= 0) wait_counter(cnt + it.wait1, it.need1, ctl, limit);
        }
        __syncthreads();
        switch (it.kind) {
            case kItemAssemble: {
                const AsmItem ai = A.items[it.aux];
                body_assemble(P, V, fronts, A, ai, pool);
                break;
            }
            case kItemDiag:
                body_diag(P, V, fronts, Dg, Dig, dyng, ctl, it.s, it.t * nb, nb, pws + (int64_t)it.aux * kPanelWs,
                          pool);
                break;
            case kItemTrsm:
                body_trsm<1>(P, fronts, it.s, it.a, it.b, it.t * nb, nb, pws + (int64_t)it.aux * kPanelWs, pool);
                break;
            case kItemStrip: body_strip(P, fronts, it.s, it.a, it.b, it.t * nb, nb, pool); break;
            default: body_tile(P, fronts, it.s, it.a, it.b, it.t * nb, nb, pool); break;
        }
        // publish: the CTA barrier orders every thread's stores before thread 0's
        // fence, which makes them visible device-wide before the counter
        // (cumulativity); a fence in every thread cost the chain more
        __syncthreads();
        if (tid == 0 && it.sig >= 0) {
            __threadfence();
            atomicAdd(cnt + it.sig, it.add);
        }
    }
}

// The entries' values of the regularised matrix (the augmented K with its
// static terms, or M + delta I), |K|e and ||K||_1 = max_i (|K|e)_i; also checks
// that Theta is positive and finite.  The residuals of the refinement read the
// values and the row sums from here instead of forming them again.
__device__ __forceinline__ double k_entry(const DevPlan &P, const DevVals &V, int i, int64_t p, bool &bad) {
    const int64_t src = P.ksrc[p];
    if (P.form == 2) return V.nev[src] + (P.kj[p] == i ? V.delta : 0.0);
    if (src >= 0) return V.Ax[src];
    if (src == kDualDiag) return V.delta;
    const double th = V.theta[-1 - src];
    if (!(th > 0.0) || !isfinite(th)) bad = true;
    return -(1.0 / th + V.rho);
}

__global__ void __launch_bounds__(rows::kThreads) k_norm1(DevPlan P, DevVals V, DevCtl *ctl) {
    __shared__ double sh[rows::kThreads / 32][1];
    const rows::Part w = rows::part(P.nmid, P.nlong);
    const int lane = threadIdx.x & 31;
    double mx = 0.0;
    bool bad = false;
    auto put = [&](int i, double sum) {
        P.kabs[i] = sum;
        mx = fmax(mx, sum);
        if (P.inst)
            atomicMax((unsigned long long *)&P.inst_norm1[P.inst[i]], (unsigned long long)__double_as_longlong(sum));
    };
    auto strided = [&](int i, int t, int nt) {
        double sum = 0.0;
        const int64_t p1 = P.kp[i + 1];
#pragma unroll 4
        for (int64_t p = P.kp[i] + t; p < p1; p += nt) {
            const double v = k_entry(P, V, i, p, bad);
            P.kval[p] = v;
            sum += fabs(v);
        }
        return sum;
    };
    if (w.cta >= 0) {
        const int i = P.long_cols[w.cta];
        double a[1] = {strided(i, threadIdx.x, rows::kThreads)};
        rows::cta_add(a, sh);
        if (threadIdx.x == 0) put(i, a[0]);
    } else if (w.mid >= 0) {
        if (w.mid < P.nmid) {
            const int i = P.mid_cols[w.mid];
            double a[1] = {strided(i, lane, 32)};
            rows::warp_add(a);
            if (lane == 0) put(i, a[0]);
        }
    } else {
        for (int i = w.first; i < P.N; i += w.stride)
            if (P.kp[i + 1] - P.kp[i] <= kWarpRow) put(i, strided(i, 0, 1));
    }
    mx = warp_max(mx);
    if (lane == 0) atomicMax((unsigned long long *)&ctl->norm1, (unsigned long long)__double_as_longlong(mx));
    if (bad) atomicOr(&ctl->status, kStatNonFinite);
}

__global__ void k_set_b1(DevPlan P, DevCtl *ctl, double eps_piv) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->b1 = eps_piv * ctl->norm1;
    if (P.inst)
        for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.batch_count; b += gridDim.x * blockDim.x)
            P.inst_b1[b] = eps_piv * P.inst_norm1[b];
}

// Statistics of the factorisation: inertia, number and size of lifts.
__global__ void k_factor_stats(const double *__restrict__ D, const double *__restrict__ dyn, int N, double large_reg,
                               DevCtl *ctl) {
    int npos = 0, nneg = 0, ndyn = 0;
    double mx = 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        const double d = D[j];
        npos += d > 0.0;
        nneg += d < 0.0;
        const double a = fabs(dyn[j]);
        ndyn += a != 0.0;
        mx = fmax(mx, a);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        npos += __shfl_xor_sync(0xffffffffu, npos, o);
        nneg += __shfl_xor_sync(0xffffffffu, nneg, o);
        ndyn += __shfl_xor_sync(0xffffffffu, ndyn, o);
    }
    mx = warp_max(mx);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&ctl->npos, npos);
        atomicAdd(&ctl->nneg, nneg);
        atomicAdd(&ctl->ndyn, ndyn);
        atomicMax((unsigned long long *)&ctl->max_dyn, (unsigned long long)__double_as_longlong(mx));
        if (ndyn) atomicOr(&ctl->status, kStatDynReg);
        if (mx > large_reg) atomicOr(&ctl->status, kStatLargeReg);
    }
}

// ---------------------------------------------------------------------------
// Pivoting of Sec. 4.5 (the Bunch-Kaufman variation) for matrices that are not
// quasi-definite: one CTA per front assembles it (original entries, then the
// children's contribution blocks in ascending order), adds the static terms
// to its fully-summed diagonal and factorises its k fully-summed columns in
// pivot blocks of nb columns, with 1x1 and 2x2 pivots chosen inside the
// block: pre-swap of the largest remaining block diagonal, gamma_p = the
// largest magnitude below the pivot in the block (row r), a lift of the pivot
// to sign(M_pp) eps_piv ||K||_1 when max(|M_pp|, gamma_p) is not above it,
// else a 1x1 pivot at p when |M_pp| >= alpha gamma_p or
// |M_pp| gamma_r >= alpha gamma_p^2, a 1x1 pivot at r when
// |M_rr| >= alpha gamma_r, otherwise the 2x2 pivot (p, r).  Interchanges stay
// among the fully-summed columns, so the structure of the front is unchanged;
// every pivot updates the whole trailing part of the front (the contribution
// block included).  Each product and sum is rounded as written (no fused
// multiply-add), so the arithmetic is that of a plain evaluation of the rule.
// The front lives in its slab (lower triangle); a symmetric interchange of
// positions a < b moves entries of the lower triangle only.
constexpr int kBkThreads = 256;

__device__ void bk_swap(double *F, int ld, int f, int a, int b, int32_t *lperm) {
    if (a == b) return;
#define FE(i, j) F[(int64_t)(j) * ld + (i)]
    for (int i = threadIdx.x; i < f; i += kBkThreads) {
        if (i < a) {
            const double t = FE(a, i);
            FE(a, i) = FE(b, i);
            FE(b, i) = t;
        } else if (i == a) {
            const double t = FE(a, a);
            FE(a, a) = FE(b, b);
            FE(b, b) = t;
        } else if (i < b) {
            const double t = FE(i, a);
            FE(i, a) = FE(b, i);
            FE(b, i) = t;
        } else if (i > b) {
            const double t = FE(i, a);
            FE(i, a) = FE(i, b);
            FE(i, b) = t;
        }
    }
    if (threadIdx.x == 0) {
        const int32_t t = lperm[a];
        lperm[a] = lperm[b];
        lperm[b] = t;
    }
#undef FE
}

// argmax over lanes of v (first index on ties, -1 when every v is 0 and zero_is_none)
__device__ __forceinline__ int warp_argmax_first(double v, int idx) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
        if (ov > v || (ov == v && oi < idx)) {
            v = ov;
            idx = oi;
        }
    }
    return idx;
}

__global__ void __launch_bounds__(kBkThreads) k_front_bk(DevPlan P, DevVals V, double *__restrict__ fronts,
                                                         double *__restrict__ D, double *__restrict__ Doff,
                                                         int32_t *__restrict__ bsz, int32_t *__restrict__ lperm,
                                                         double *__restrict__ dyn, DevCtl *ctl,
                                                         const int32_t *__restrict__ list, int nb, double alpha) {
    __shared__ int sh_q, sh_two, sh_swap_a, sh_swap_b;
    const int s = list[blockIdx.x];
    const int f = P.sn_f[s], k = P.sn_k[s], ld = P.sn_ld[s], c0 = P.sn_c0[s];
    double *F = fronts + P.sn_off[s];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#define FE(i, j) F[(int64_t)(j) * ld + (i)]
    // assembly, in the order of the plain multifrontal method
    for (int64_t t = tid; t < (int64_t)f * ld; t += kBkThreads) F[t] = 0.0;
    __syncthreads();
    for (int64_t q = P.orig_ptr[s] + tid; q < P.orig_ptr[s + 1]; q += kBkThreads)
        F[P.orig_dst[q]] = orig_value(P, V, P.orig_src[q]);
    __syncthreads();
    for (int q = P.child_ptr[s]; q < P.child_ptr[s + 1]; q++) {
        const int c = P.child_list[q];
        const int kc = P.sn_k[c], ldc = P.sn_ld[c], cc = P.sn_f[c] - kc;
        const double *CB = fronts + P.sn_off[c] + (int64_t)kc * ldc + kc;
        const int32_t *map = P.relmap + P.map_off[c];
        for (int jj = warp; jj < cc; jj += kBkThreads / 32)
            for (int ii = jj + lane; ii < cc; ii += 32)
                F[(int64_t)map[jj] * ld + map[ii]] += CB[(int64_t)jj * ldc + ii];
        __syncthreads();
    }
    // static terms on the fully-summed diagonal; interchanges start from the identity
    for (int t = tid; t < k; t += kBkThreads) {
        const int sg = P.sign[c0 + t];
        const double sigma = sg < 0 ? V.rho : V.delta;
        FE(t, t) = __dadd_rn(FE(t, t), (double)sg * sigma);
        lperm[c0 + t] = t;
        Doff[c0 + t] = 0.0;
        dyn[c0 + t] = 0.0;
    }
    __syncthreads();
    const double b1 = ctl->b1;
    int32_t *lp = lperm + c0;
    for (int b0 = 0; b0 < k; b0 += nb) {
        const int b1c = min(b0 + nb, k);
        int p = b0;
        while (p < b1c) {
            // pre-swap: the largest remaining block diagonal to position p
            if (warp == 0) {
                const int t = p + lane;
                const double v = t < b1c ? fabs(FE(t, t)) : -1.0;
                const int q = warp_argmax_first(v, t < b1c ? t : 0x7fffffff);
                if (lane == 0) sh_q = q;
            }
            __syncthreads();
            bk_swap(F, ld, f, p, sh_q, lp);
            __syncthreads();
            // gamma_p and r within the block; the pivot decision
            if (warp == 0) {
                const int i = p + 1 + lane;
                const double v = i < b1c ? fabs(FE(i, p)) : -1.0;
                const int r0 = warp_argmax_first(v, i < b1c ? i : 0x7fffffff);
                const double gp_all = __shfl_sync(0xffffffffu, v, (r0 - p - 1) & 31);
                if (lane == 0) {
                    const double gp = (r0 < b1c && gp_all > 0.0) ? gp_all : 0.0;
                    const int r = gp > 0.0 ? r0 : -1;
                    const double app = FE(p, p);
                    int two = 0, sa = -1, sb = -1;
                    if ((fabs(app) > gp ? fabs(app) : gp) <= b1) {
                        const double dn = app < 0.0 ? -b1 : b1;
                        dyn[c0 + p] = __dsub_rn(dn, app);
                        FE(p, p) = dn;
                    } else if (fabs(app) < __dmul_rn(alpha, gp)) {
                        double gr = 0.0;
                        for (int t = p; t < b1c; t++) {
                            if (t == r) continue;
                            const double a = t < r ? fabs(FE(r, t)) : fabs(FE(t, r));
                            if (a > gr) gr = a;
                        }
                        if (__dmul_rn(fabs(app), gr) >= __dmul_rn(__dmul_rn(alpha, gp), gp)) {
                            // 1x1 at p
                        } else if (fabs(FE(r, r)) >= __dmul_rn(alpha, gr)) {
                            sa = p;
                            sb = r;
                        } else {
                            sa = p + 1;
                            sb = r;
                            two = 1;
                        }
                    }
                    sh_two = two;
                    sh_swap_a = sa;
                    sh_swap_b = sb;
                }
            }
            __syncthreads();
            if (sh_swap_a >= 0) {
                bk_swap(F, ld, f, sh_swap_a, sh_swap_b, lp);
                __syncthreads();
            }
            if (!sh_two) {
                const double d = FE(p, p);
                if (tid == 0) {
                    D[c0 + p] = d;
                    bsz[c0 + p] = 1;
                    if (!isfinite(d) || d == 0.0) atomicOr(&ctl->status, kStatNonFinite);
                }
                for (int i = p + 1 + tid; i < f; i += kBkThreads) FE(i, p) = __ddiv_rn(FE(i, p), d);
                __syncthreads();
                for (int j = p + 1 + warp; j < f; j += kBkThreads / 32) {
                    const double ljp = FE(j, p);
                    for (int i = j + lane; i < f; i += 32)
                        FE(i, j) = __dsub_rn(FE(i, j), __dmul_rn(__dmul_rn(FE(i, p), d), ljp));
                }
                __syncthreads();
                p += 1;
            } else {
                const double e11 = FE(p, p), e21 = FE(p + 1, p), e22 = FE(p + 1, p + 1);
                const double det = __dsub_rn(__dmul_rn(e11, e22), __dmul_rn(e21, e21));
                if (tid == 0) {
                    D[c0 + p] = e11;
                    D[c0 + p + 1] = e22;
                    Doff[c0 + p] = e21;
                    bsz[c0 + p] = 2;
                    bsz[c0 + p + 1] = 0;
                    if (!isfinite(det) || det == 0.0) atomicOr(&ctl->status, kStatNonFinite);
                }
                for (int i = p + 2 + tid; i < f; i += kBkThreads) {
                    const double x = FE(i, p), y = FE(i, p + 1);
                    FE(i, p) = __ddiv_rn(__dsub_rn(__dmul_rn(x, e22), __dmul_rn(y, e21)), det);
                    FE(i, p + 1) = __ddiv_rn(__dsub_rn(__dmul_rn(y, e11), __dmul_rn(x, e21)), det);
                }
                __syncthreads();
                for (int j = p + 2 + warp; j < f; j += kBkThreads / 32) {
                    const double l0 = FE(j, p), l1 = FE(j, p + 1);
                    const double w0 = __dadd_rn(__dmul_rn(e11, l0), __dmul_rn(e21, l1));
                    const double w1 = __dadd_rn(__dmul_rn(e21, l0), __dmul_rn(e22, l1));
                    for (int i = j + lane; i < f; i += 32)
                        FE(i, j) = __dsub_rn(FE(i, j), __dadd_rn(__dmul_rn(FE(i, p), w0), __dmul_rn(FE(i, p + 1), w1)));
                }
                __syncthreads();
                if (tid == 0) FE(p + 1, p) = 0.0;  // L is unit lower triangular: the 2x2 block lives in D
                __syncthreads();
                p += 2;
            }
        }
    }
#undef FE
}

// Inertia and lift statistics of a factorisation with 1x1 and 2x2 blocks: a
// 2x2 block holds one positive and one negative eigenvalue when its
// determinant is negative, else two of the sign of its trace.
__global__ void k_factor_stats_bk(const double *__restrict__ D, const double *__restrict__ Doff,
                                  const int32_t *__restrict__ bsz, const double *__restrict__ dyn, int N,
                                  double large_reg, DevCtl *ctl) {
    int npos = 0, nneg = 0, ndyn = 0;
    double mx = 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        const double a = fabs(dyn[j]);
        ndyn += a != 0.0;
        mx = fmax(mx, a);
        if (bsz[j] == 2) {
            const double det = __dsub_rn(__dmul_rn(D[j], D[j + 1]), __dmul_rn(Doff[j], Doff[j]));
            if (det < 0.0) {
                npos++;
                nneg++;
            } else if (det > 0.0) {
                if (__dadd_rn(D[j], D[j + 1]) > 0.0) npos += 2;
                else nneg += 2;
            }
        } else if (bsz[j] == 1) {
            npos += D[j] > 0.0;
            nneg += D[j] < 0.0;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        npos += __shfl_xor_sync(0xffffffffu, npos, o);
        nneg += __shfl_xor_sync(0xffffffffu, nneg, o);
        ndyn += __shfl_xor_sync(0xffffffffu, ndyn, o);
    }
    mx = warp_max(mx);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&ctl->npos, npos);
        atomicAdd(&ctl->nneg, nneg);
        atomicAdd(&ctl->ndyn, ndyn);
        atomicMax((unsigned long long *)&ctl->max_dyn, (unsigned long long)__double_as_longlong(mx));
        if (ndyn) atomicOr(&ctl->status, kStatDynReg);
        if (mx > large_reg) atomicOr(&ctl->status, kStatLargeReg);
    }
}

}  // namespace

void launch_small_fronts(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                         DevCtl *ctl, const AsmLists &A, const int32_t *list, int32_t count, int32_t nb, int32_t maxf,
                         int32_t threads, cudaStream_t st) {
    if (count <= 0) return;
    const int ldmax = (maxf + 3) & ~3;
    const size_t smem = (size_t)ldmax * maxf * sizeof(double);
    static uint64_t attr = 0;
    if (first_on_device(attr)) {
        cudaFuncSetAttribute(k_small_fronts<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_small_fronts<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_small_fronts<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_small_fronts<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    }
    switch (threads) {
        case 32: k_small_fronts<32><<<count, 32, smem, st>>>(P, V, fronts, D, Dinv, dyn, ctl, A, list, nb); break;
        case 64: k_small_fronts<64><<<count, 64, smem, st>>>(P, V, fronts, D, Dinv, dyn, ctl, A, list, nb); break;
        case 256: k_small_fronts<256><<<count, 256, smem, st>>>(P, V, fronts, D, Dinv, dyn, ctl, A, list, nb); break;
        default: k_small_fronts<128><<<count, 128, smem, st>>>(P, V, fronts, D, Dinv, dyn, ctl, A, list, nb); break;
    }
}

void launch_large_assemble(const DevPlan &P, const DevVals &V, double *fronts, const AsmLists &A, int64_t first,
                           int32_t count, cudaStream_t st) {
    if (count <= 0) return;
    k_large_assemble<<<count, kBodyThreads, 0, st>>>(P, V, fronts, A, first);
}

void launch_panel_diag(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                       DevCtl *ctl,
                       const PanelItem *items, int32_t count, int32_t nb, double *pws, cudaStream_t st) {
    if (count <= 0) return;
    k_panel_diag<<<count, kBodyThreads, 0, st>>>(P, V, fronts, D, Dinv, dyn, ctl, items, nb, pws);
}

void launch_panel_trsm(const DevPlan &P, double *fronts, const PanelItem *items, const int32_t *slots, int32_t count,
                       int32_t rows, int32_t nb, const double *pws, cudaStream_t st, const int32_t *sbase,
                       uint8_t *sws, int32_t *sexp, const double *D, DevCtl *ctl) {
    if (count <= 0) return;
    if (rows > kTrsmRows)
        k_panel_trsm<kTrsmItemRows / kTrsmRows>
            <<<count, kBodyThreads, 0, st>>>(P, fronts, items, slots, nb, pws, sbase, sws, sexp, D, ctl);
    else
        k_panel_trsm<1><<<count, kBodyThreads, 0, st>>>(P, fronts, items, slots, nb, pws, sbase, sws, sexp, D, ctl);
}

void launch_large_update(const DevPlan &P, double *fronts, const TileItem *items, int32_t count,
                         int32_t w, cudaStream_t st) {
    if (count <= 0) return;
    k_large_update<<<count, kBodyThreads, 0, st>>>(P, fronts, items, w);
}

void launch_large_update_strip(const DevPlan &P, double *fronts, const TileItem *items,
                               int32_t count, int32_t w, cudaStream_t st) {
    if (count <= 0) return;
    k_large_update_strip<<<count, kBodyThreads, 0, st>>>(P, fronts, items, w);
}

void launch_rank_one(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                     DevCtl *ctl, const int32_t *list, int32_t count, cudaStream_t st) {
    if (count <= 0) return;
    k_rank_one<<<count, kRankOneThreads, 0, st>>>(P, V, fronts, D, Dinv, dyn, ctl, list);
}

void launch_thin_fronts(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                        DevCtl *ctl, const int32_t *list, const int32_t *slots, double *pws, int32_t count, int32_t nb,
                        cudaStream_t st) {
    if (count <= 0) return;
    static uint64_t attr = 0;
    constexpr int smem = kThinPanel * (int)sizeof(double);
    if (first_on_device(attr))
        cudaFuncSetAttribute(k_thin_fronts, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k_thin_fronts<<<count, kBodyThreads, smem, st>>>(P, V, fronts, D, Dinv, dyn, ctl, list, slots, pws, nb);
}

void launch_large_level(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                        DevCtl *ctl, const FactorItem *items, int32_t count, int32_t *sync, int32_t ncounters,
                        const AsmLists &A, double *pws, int32_t nb, int32_t grid, long long spin_limit,
                        cudaStream_t st) {
    if (count <= 0) return;
    cudaMemsetAsync(sync, 0, sizeof(int32_t) * (size_t)(ncounters + 1), st);
    k_large_level<<<grid < count ? grid : count, kBodyThreads, 0, st>>>(P, V, fronts, D, Dinv, dyn, ctl, items, count,
                                                                        sync, A, pws, nb, spin_limit);
}

const void *large_level_kernel() { return reinterpret_cast<const void *>(k_large_level); }

// The pivot reciprocal of the factorisation beside CUDA's correctly rounded
// division, element by element (a test hook: the factorisation scales every
// column of L by this reciprocal, Sec. 4.4-4.5).
__global__ void k_test_recip(const double *__restrict__ x, double *__restrict__ rcp, double *__restrict__ quo,
                             int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        rcp[i] = recip_pivot(v);
        quo[i] = 1.0 / v;
    }
}

void launch_front_bk(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Doff, int32_t *bsz,
                     int32_t *lperm, double *dyn, DevCtl *ctl, const int32_t *list, int32_t count, int32_t nb,
                     cudaStream_t st) {
    if (count <= 0) return;
    k_front_bk<<<count, kBkThreads, 0, st>>>(P, V, fronts, D, Doff, bsz, lperm, dyn, ctl, list, nb,
                                            0.125 + 0.125 * sqrt(17.0));
}

void launch_factor_stats_bk(const double *D, const double *Doff, const int32_t *bsz, const double *dyn, int N,
                            double large_reg, DevCtl *ctl, cudaStream_t st) {
    k_factor_stats_bk<<<152, 256, 0, st>>>(D, Doff, bsz, dyn, N, large_reg, ctl);
}

void launch_test_recip(const double *x, double *rcp, double *quo, int64_t n, cudaStream_t st) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_test_recip<<<(int)(blocks < 1216 ? blocks : 1216), 256, 0, st>>>(x, rcp, quo, n);
}

void launch_norm1(const DevPlan &P, const DevVals &V, DevCtl *ctl, double eps_piv, cudaStream_t st) {
    if (P.inst) cudaMemsetAsync(P.inst_norm1, 0, sizeof(double) * P.batch_count, st);
    k_norm1<<<rows::grid(P.N, P.nmid, P.nlong), rows::kThreads, 0, st>>>(P, V, ctl);
    k_set_b1<<<P.inst ? (P.batch_count + 255) / 256 : 1, 256, 0, st>>>(P, ctl, eps_piv);
}

void launch_factor_stats(const double *D, const double *dyn, int N, double large_reg, DevCtl *ctl, cudaStream_t st) {
    k_factor_stats<<<152, 256, 0, st>>>(D, dyn, N, large_reg, ctl);
}

}  // namespace ipm
