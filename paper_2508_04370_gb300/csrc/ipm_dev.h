// Device-side view of the analysis plan and kernel entry points of the
// multifrontal factorise/solve (Zanetti & Gondzio, arXiv 2508.04370, Sec. 4).
#pragma once
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

#include "point_lists.h"

namespace ipm {

// Status bits written by kernels (never traps): OR-ed into DevCtl::status.
enum : int32_t {
    kStatNonFinite = 1,    // NaN / Inf in Theta, a pivot or a residual
    kStatDynReg = 2,       // a pivot was lifted
    kStatLargeReg = 4,     // a lift exceeded opt.large_reg
    kStatTimeout = 8,      // a bounded wait expired
    kStatRefineFail = 16,  // refinement did not reach the target
    kStatWaitCopy = 32,    // with kStatTimeout: a tensor-core kernel's wait for its bulk copies gave up
    kStatWaitMma = 64,     // with kStatTimeout: a wait for the completion of MMAs gave up
};

// Dynamic shared memory the per-level solve sweeps may use (one front's
// gathered vector, f doubles): fronts above 25,600 rows do not fit.
constexpr int64_t kSweepSmemLimit = 200 * 1024;

// Kernel attributes such as the dynamic shared-memory limit belong to one
// device: true the first time it is asked for the current device, so the
// attribute is set once per device and kernel (mask: one bit per device).
inline bool first_on_device(uint64_t &mask) {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= 64) {
        cudaGetLastError();
        return true;
    }
    const uint64_t bit = (uint64_t)1 << d;
    if (mask & bit) return false;
    mask |= bit;
    return true;
}

// Small control block in device memory.
struct DevCtl {
    int32_t status;
    int32_t ndyn;
    int32_t npos, nneg;
    double max_dyn;
    double norm1;          // ||K||_1 (or ||M||_1) of the current factorisation
    double b1;             // eps_piv * norm1
    // refinement
    double omega;          // backward error of the current iterate
    double omega_best;
    double dinf;           // ||d||_inf of the current iterate (as ordered bits >= 0)
    int32_t done;          // refinement finished
    int32_t steps;
    double omega_hist[16];
    int32_t gmres_iters;   // GMRES iterations of a graph-resident refinement
    int32_t best;          // graph-resident refinement: which of its two iterates is the best
};

// Read-only plan arrays on the device (all indices in factorisation order).
struct DevPlan {
    int32_t N, n, m, nsuper, form;
    const int32_t *sn_c0, *sn_k, *sn_f, *sn_ld;
    const int64_t *sn_off;        // slab offset (doubles)
    const int64_t *sn_rptr;       // row list offset
    const int32_t *sn_rows;       // global row indices
    const int32_t *child_ptr, *child_list;
    const int32_t *sn_parent;     // parent supernode or -1
    const int64_t *map_off;
    const int32_t *relmap;
    const int64_t *orig_ptr;
    const int32_t *orig_dst;
    const int64_t *orig_src;
    const int8_t *sign;           // expected pivot sign per row (-1 / +1)
    const int32_t *perm;          // perm[new] = old
    const int64_t *upd_off;       // solve: contribution-vector offsets
    // regularised matrix in factorisation order, full symmetric CSR (for
    // residuals): value source per entry (>= 0: A index, -1-j: primal
    // diagonal of old column j, kDualDiag: delta)
    const int64_t *kp;
    const int32_t *kj;
    const int64_t *ksrc;
    // the entries' values and the row sums |K|e of the latest factorisation's
    // matrix, written with its norm and read by every residual
    double *kval, *kabs;
    // rows of K with more than kLongColumn (a CTA each) and more than kWarpRow
    // (a warp each) stored entries
    const int32_t *long_cols, *mid_cols;
    int32_t nlong, nmid;
    // batches of independent problems: instance of each unknown (factorisation
    // order) and, per instance, ||K_b||_1 and eps_piv ||K_b||_1; null otherwise
    int32_t batch_count;
    const int32_t *inst;
    double *inst_norm1, *inst_b1;
};

// eps_piv ||K||_1 of the problem that owns column c (Sec. 4.5); the norm is
// per instance when independent problems are factorised together.
__device__ __forceinline__ double pivot_floor(const DevPlan &P, const DevCtl *ctl, int c) {
    return P.inst ? P.inst_b1[P.inst[c]] : ctl->b1;
}

constexpr int64_t kDualDiag = INT64_MIN;

// Numeric values for one factorisation.
struct DevVals {
    const double *Ax;      // A values (CSC order of the pattern)
    const double *theta;   // n
    const double *nev;     // normal equations: lower entries of M (or null)
    double rho, delta;
    double large_reg;
};

// Rows of a panel handled by one CTA of the panel kernel (one thread per row).
constexpr int kPanelRows = 128;
// Output tile of the FP64 trailing-update kernel.
constexpr int kUpdTile = 32;
// Lookahead (next panel) columns of the trailing update are cut into strips
// of kUpdTile rows x kStripCols columns, one output per thread.
constexpr int kStripCols = 4;
// Output tile of the tensor-core trailing update (M = N).
constexpr int kTcTile = 128;

// Device data of the normal-equations path.
struct NeView {
    int32_t n, m;
    int64_t nnz;                 // lower entries of M
    const int64_t *tptr;         // contributor pairs per entry
    const int32_t *ta, *tb, *tj;
    double *tt;                  // Theta~ (n)
    double *nev;                 // formed entries of M (nnz)
    const int64_t *Arp;          // A by rows: pointer, column, position in Ax
    const int32_t *Aci, *Apos;
    const int64_t *Acp;          // A by columns
    const int32_t *Ari;
    // the sums over more than kLongColumn (a CTA each) and more than kWarpRow
    // (a warp each) terms: entries of M by contributor pairs, columns of A,
    // and rows of A (as positions in the factorisation order)
    const int32_t *elong, *emid, *clong, *cmid, *rlong, *rmid;
    int32_t nelong, nemid, nclong, ncmid, nrlong, nrmid;
};

// Dependency-driven solve schedule, built once per pattern.  A supernode
// with k > 32 or a large rectangular part L21 is split into one item per
// 32-column block of L11 and row-chunk items (kRectRows rows of L21 each),
// which run on other SMs.
struct SolveNode {
    int64_t off;    // slab offset (doubles)
    int64_t upd;    // offset of its contribution vector
    int64_t rptr;   // first entry in sn_rows and gat_rp
    int64_t inv;    // inverses of its diagonal blocks in SolveSched::Linv, -1: none (layout: block_slot)
    int64_t part;   // its row chunks' sums in SolveSched::rpart (32 per block and chunk)
    int32_t f, k, ld, c0;
    int32_t parent, nchild, nrect, nblk;  // nblk: items of L11 (32-column blocks; 1 when unsplit)
    int32_t nback;  // row chunks of L21 in the backward sweep (0: the blocks take all rows themselves)
};
struct SolveItem {
    // r < 0: block -1-r of L11; else forward: row chunk r of L21, backward: row
    // chunk r % nback of L21 for the columns of block r / nback
    int32_t s, r;
};
struct SolveSched {
    const SolveNode *node;
    const int32_t *sn_rows;
    const int64_t *gat_rp;   // per front row: range in gat_src
    const int64_t *gat_src;  // contribution-vector positions summed into the row, children ascending
    const SolveItem *fwd, *bwd;
    int32_t nfwd, nbwd, nsuper;
    long long spin_limit;    // polls before a dependency wait gives up (kStatTimeout)
    // Per sweep (0 forward, 1 backward): ticket + 2 x nsuper counters (forward:
    // children done, items done; backward: done flag, blocks done) and the values
    // split supernodes' blocks pass along their chain (y forward, z backward),
    // an unset pattern before the sweep.  Each sweep resets the other's at its
    // start, so a pair of sweeps needs no reset launches.
    int32_t *sync[2];
    double *yv[2];
    int32_t nyv;
    double *rpart;           // backward sweep: the row chunks' sums, reset like yv
    int64_t nrpart;
    const int32_t *fwd_leaf, *bwd_leaf;  // leaf groups: 8 childless single-item supernodes with f <= 32
                                         // per ticket (-1 pads), one warp each
    const double *Linv;                  // inverse unit-lower diagonal blocks, column-major 32 x 32
};
// One diagonal block to invert after a factorisation: block b of supernode s
// into Linv + dst.
struct InvItem {
    int32_t s, b;
    int64_t dst;
};
constexpr int32_t kLeafGroup = INT32_MIN;  // SolveItem.r of a leaf group (s = group index)
constexpr int kRectRows = 32;
constexpr int64_t kRectSplit = 8192;  // split when k (f - k) reaches this
// Backward sweep: a block of 32 columns with more than kBackSplit rows below
// leaves them to items of kBackRows rows.  A block's 1,400 rows are 45,000 FMAs, 11 us
// of one SM's FP64 rate on the path from the root; chunks of 256 rows are 2 us.
constexpr int kBackRows = 256;
constexpr int kBackSplit = 384;

// Work item of the large-front path.
struct PanelItem {
    int32_t s;       // supernode
    int32_t r0, r1;  // row range (local) handled by this block
    int32_t p0;      // first column of the item's panel (diagonal blocks, triangular solves)
};
// An assembly item: columns [c_lo, c_hi) (a block of 32), rows [r_lo, r_hi) (a
// block of kAsmRows, from the columns' first: the upper part is never read) of
// large front s.  Its terms, in the order they are added: the original entries
// among [o0, o1) (those of the columns) that lie in its rows; the entries of
// the small children (contribution blocks of up to kPointRows rows) as one list
// of arena positions per destination, [seg0, seg1) of AsmLists; the large
// children [ch0, ch1); the rank-one leaves [ch1, ch2).  Device child lists hold the small children before the
// large ones, so every path adds in this order.
struct AsmItem {
    int64_t o0, o1, seg0, seg1;
    int32_t ch0, ch1, ch2, s, c_lo, c_hi, r_lo, r_hi;
};
struct AsmLists {
    const AsmItem *items;
    const int32_t *seg_dst;  // destination within the item: 64 (column - c_lo) + row % 64
    const int64_t *seg_ptr;  // its arena positions, children ascending
    const int64_t *src;
    const AsmChild *child;
    const int32_t *rt;
    // small fronts (k_small_fronts): segments [small[2 s], small[2 s + 1]), with
    // destinations column * ld + row, and the front's first large child
    const int64_t *small;
    const int32_t *small_big;
};
struct TileItem {
    int32_t s;
    int32_t i0, j0;  // first local row / column of a kUpdTile x kUpdTile output tile
                     // (kUpdTile x kStripCols for the lookahead strips)
    int32_t p0;      // first column of the panel whose update the tile applies
};

// Sliced tensor-core update (FP64-accurate Schur complement on bf16 tensor
// cores).  Panels of a large front are taken in pairs: after the first panel
// of a pair only the second panel's columns are updated; after the second,
// every trailing row r >= p1 of both panel operands over both panels' 64
// columns, L(r, q) and L(r, q) d_q, is scaled by one power of two per row
// and split into kSlices balanced 7-bit digits, and the whole trailing part
// receives the two panels' update at once (K = 64).  One slice block holds
// 128 rows: one chunk of digit images per 32 columns.
constexpr int kSlices = 8;                           // 8 x 7 = 56 bits per operand
constexpr int kSliceRows = 128;                      // rows per slice block (the MMA's M)
constexpr int kSliceCols = 32;                       // output columns per tile (the MMA's N), columns per chunk
constexpr int kSliceChunks = 2;                      // chunks of 32 columns per slice block (K <= 64)
constexpr int64_t kSlicePairBytes = 128 * 128;       // two slices of 128 rows x 32 bf16, one swizzled image
constexpr int64_t kSliceOperandBytes = 4 * kSlicePairBytes;
constexpr int64_t kSliceChunkBytes = 2 * kSliceOperandBytes;  // operand A (L), then operand B (L d)
constexpr int64_t kSliceBlockBytes = kSliceChunks * kSliceChunkBytes;

// A run of output tiles: rows i0 .. i0+127 (one slice block), nt tiles of 32
// columns from j0 (lower part only).  A CTA works through the runs
// [first, last) of its segment.
struct SlicedRun {
    int32_t s;
    int32_t i0, j0, nt;
    int32_t base, p1;  // slice block of rows p1 ..
    int32_t kc;        // chunks of the product: 1 (one panel, K <= 32) or 2 (a pair of panels, K <= 64)
};
struct SlicedSeg {
    int32_t first, last;
};
// SMs the launch of a pair's trailing update leaves to the next panels' kernels
// (50-period staircase, factorisation: 61.1 ms with 0, 60.3 with 8, 60.6 with 16,
// 66.8 with 48).
constexpr int kSliceFreeSms = 8;

// One item of the persistent level kernel (large fronts of one tree level):
// it waits until counter wait0 >= need0 and counter wait1 >= need1 (-1: no
// wait), runs, then adds `add` to counter sig.  Counters are per level,
// zeroed before the launch; the host orders the items so that every wait
// refers to items with smaller positions.
enum : int32_t { kItemAssemble = 0, kItemDiag = 1, kItemTrsm = 2, kItemStrip = 3, kItemTile = 4 };
struct FactorItem {
    int32_t kind;
    int32_t s, t;  // front, pivot block (panel) index
    int32_t a, b;  // trsm: rows [a, b); strip / tile: first row, first column
    int32_t aux;   // assemble: AsmItem index; diag / trsm: panel workspace slot
    int32_t wait0, need0, wait1, need1;
    int32_t sig, add;
};

// ---------------------------------------------------------------- launches
// factorisation (kernels_factor.cu)
void launch_norm1(const DevPlan &P, const DevVals &V, DevCtl *ctl, double eps_piv, cudaStream_t st);
// Threads per CTA of a small-front launch (32, 64, 128 or 256; the same arithmetic
// per entry whatever the width).  By default one warp per front up to f = 32, two
// up to 64, four beyond, and more where the launch leaves SMs idle (at most four
// fronts per SM, at most one): a front's pivots then run on all four
// sub-partitions' FP64 pipes (factorisation of a 31 x 31 grid with 12 levels of
// 10 to 600 fronts 0.86 -> 0.72 ms; a 64 x 64 grid, whose lower levels fill the
// chip, loses 1% with the wide CTAs there, so the autotuner tries the fixed
// widths too).
constexpr int32_t kSmallBaseWidth[3] = {32, 64, 128};  // by size class f <= 32, 64, 128
inline int32_t small_front_threads(int32_t cls, int32_t count, int32_t sms) {
    const int32_t w = kSmallBaseWidth[cls] * (count <= sms ? 4 : count <= 4 * sms ? 2 : 1);
    return w < 256 ? w : 256;
}
void launch_small_fronts(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                         DevCtl *ctl, const AsmLists &A, const int32_t *list, int32_t count, int32_t nb, int32_t maxf,
                         int32_t threads, cudaStream_t st);
void launch_large_assemble(const DevPlan &P, const DevVals &V, double *fronts, const AsmLists &A, int64_t first,
                           int32_t count, cudaStream_t st);
// panel step 1 (diagonal block of the panel [item.p0, item.p0 + nb), one item
// per front; item.r1 = workspace slot)
void launch_panel_diag(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                       DevCtl *ctl, const PanelItem *items, int32_t count, int32_t nb, double *pws, cudaStream_t st);
// panel step 2 (rows below, up to `rows` rows per item; slots[i] = workspace slot of item i)
// sbase[i] >= 0 (with sws non-null): item i also writes the digit slices of
// its rows into the sliced update's work space (slice blocks from
// sbase[i] >> 1; bit 0 set: the second panel of a pair, two chunks)
void launch_panel_trsm(const DevPlan &P, double *fronts, const PanelItem *items, const int32_t *slots, int32_t count,
                       int32_t rows, int32_t nb, const double *pws, cudaStream_t st, const int32_t *sbase = nullptr,
                       uint8_t *sws = nullptr, int32_t *sexp = nullptr, const double *D = nullptr,
                       DevCtl *ctl = nullptr);
constexpr int kTrsmRowsHost = 8;       // rows of a triangular-solve chunk of the level kernel
constexpr int kTrsmItemRowsHost = 32;  // rows of a triangular-solve item of the one-launch-per-step kernel,
constexpr int32_t kTrsmFewRows = 16;   // or of a chunk where the step has no more rows per SM than this (two chunks)
constexpr int kPanelWsHost = 32 * 33 + 32;
void launch_large_update_strip(const DevPlan &P, double *fronts, const TileItem *items,
                               int32_t count, int32_t w, cudaStream_t st);
constexpr int64_t kLongColumn = 2048;  // longer sums over a sparse row take a CTA each
constexpr int64_t kWarpRow = 32;       // and longer than this a warp each (rows_common.cuh)
// Thin leaves: large fronts without children of one pivot block and f <=
// kThinMaxF rows, whole in one CTA each (k_thin_fronts: list[i] the front,
// slots[i] its panel workspace slot) where a level has kThinMin of them; fewer
// leave SMs idle where the steps spread a front's blocks over the chip.  Only
// up to kThinCols columns, or kThinWide rows: factorisations with 1,024 leaves
// and 4,000 leaves as thin fronts and through the steps take (ms)
//   k = 2:  130 dense rows 1.65 / 1.82 and 6.4 / 7.1, 300 rows 2.48 / 2.85 and
//           9.2 / 10.6, 450 rows 3.06 / 3.55 and 11.1 / 13.2;
//   k = 4:  1.70 / 1.90 and 6.6 / 7.4, 2.67 / 3.04 and 10.2 / 11.6, 3.47 / 3.97 and
//           12.7 / 14.8;
//   k = 9:  2.11 / 2.02 and 7.88 / 7.84, 3.73 / 3.48 and 13.9 / 13.2, 5.3 / 5.0 and
//           19.7 / 18.7;
//   k = 32: 2.81 / 2.82 and 9.8 / 10.3, 6.9 / 5.6 and 22.5 / 21.6, 12.4 / 9.7 and
//           39.0 / 37.0.
// Fronts with children go through the steps (300 to 2,200 of them per level with 1
// to 30 columns over 2 to 6 children: whole in a CTA 5% faster to 17% slower;
// the 981 of a 200-block LP 20.4 against 19.5 for its factorisation).
constexpr int kThinMaxF = 512, kThinMin = 1024, kThinCols = 4, kThinWide = 224;
inline bool thin_leaf(int32_t k, int32_t f, int32_t nb) {
    return k <= nb && f <= kThinMaxF && (k <= kThinCols || f <= kThinWide);
}
// rank-one leaves (large fronts of one column without children under a large front)
void launch_rank_one(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                     DevCtl *ctl, const int32_t *list, int32_t count, cudaStream_t st);
void launch_thin_fronts(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                        DevCtl *ctl, const int32_t *list, const int32_t *slots, double *pws, int32_t count, int32_t nb,
                        cudaStream_t st);
void launch_large_level(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Dinv, double *dyn,
                        DevCtl *ctl, const FactorItem *items, int32_t count, int32_t *sync, int32_t ncounters,
                        const AsmLists &A, double *pws, int32_t nb, int32_t grid, long long spin_limit,
                        cudaStream_t st);
const void *large_level_kernel();
void launch_large_update(const DevPlan &P, double *fronts, const TileItem *items, int32_t count,
                         int32_t w, cudaStream_t st);
void launch_large_update_tc(const DevPlan &P, double *fronts, const double *D, const TileItem *items, int32_t count,
                            int32_t w, DevCtl *ctl, cudaStream_t st);
void launch_update_sliced(const DevPlan &P, double *fronts, const SlicedRun *runs, const SlicedSeg *segs, int32_t count,
                          const uint8_t *ws, const int32_t *ws_exp, DevCtl *ctl, cudaStream_t st);
int measure_fp64_peaks(double *out, int blocks, int iters, int reps, cudaStream_t st, double *dfma_tflops,
                       double *dmma_tflops);
void launch_front_bk(const DevPlan &P, const DevVals &V, double *fronts, double *D, double *Doff, int32_t *bsz,
                     int32_t *lperm, double *dyn, DevCtl *ctl, const int32_t *list, int32_t count, int32_t nb,
                     cudaStream_t st);
void launch_factor_stats_bk(const double *D, const double *Doff, const int32_t *bsz, const double *dyn, int N,
                            double large_reg, DevCtl *ctl, cudaStream_t st);
void launch_forward_bk(const DevPlan &P, const double *fronts, const double *D, const double *Doff,
                       const int32_t *bsz, const int32_t *lperm, double *x, double *upd, const int32_t *list,
                       int32_t count, int32_t maxf, cudaStream_t st);
void launch_backward_bk(const DevPlan &P, const double *fronts, const int32_t *lperm, double *x,
                        const int32_t *list, int32_t count, int32_t maxf, cudaStream_t st);
void launch_test_recip(const double *x, double *rcp, double *quo, int64_t n, cudaStream_t st);
void launch_factor_stats(const double *D, const double *dyn, int N, double large_reg, DevCtl *ctl, cudaStream_t st);
// solves and refinement (kernels_solve.cu)
void launch_forward(const DevPlan &P, const double *fronts, const double *D, double *x, double *upd,
                    const int32_t *list, int32_t count, int32_t maxf, cudaStream_t st);
void launch_backward(const DevPlan &P, const double *fronts, double *x, const int32_t *list, int32_t count,
                     int32_t maxf, cudaStream_t st);
void launch_diag_inverse(const SolveSched &S, const double *fronts, double *Linv, const InvItem *items,
                         int32_t count, const InvItem *pairs, int32_t npairs, cudaStream_t st);
// b: the right-hand side (not x); always followed by the backward sweep on x
void launch_forward_persistent(const SolveSched &S, const double *fronts, const double *Dinv, const double *b, double *x,
                               double *upd, int32_t maxf, int32_t grid, DevCtl *ctl, cudaStream_t st,
                               const int32_t *skip = nullptr);
// (also clears ctl->dinf and ctl->omega for the residual that follows)
void launch_backward_persistent(const SolveSched &S, const double *fronts, double *x, int32_t grid, DevCtl *ctl,
                                cudaStream_t st, const int32_t *skip = nullptr);
// both sweeps' counters and chain values to their state before a sweep
void launch_sweep_reset(const SolveSched &S, cudaStream_t st);
// GMRES refinement vectors (kernels_krylov.cu)
constexpr int kMaxDots = 16;  // vectors per dot-product launch (restart length + 1 at most)
constexpr int kGmresM = 8;    // GMRES restart length

// Device-side state of the GMRES refinement inside a captured graph: the
// Hessenberg matrix and its Givens rotations, and the flags the kernels of the
// section test at entry.
struct GmDev {
    double H[(kGmresM + 1) * kGmresM];  // H(i, j) at i * kGmresM + j
    double cs[kGmresM], sn[kGmresM], g[kGmresM + 1], y[kGmresM];
    double h[kMaxDots];                 // output of the dot products
    double beta, inv, eta, wbest;
    int32_t stop;        // GMRES finished: every kernel of the section returns at entry
    int32_t skip_inner;  // stop, or the current cycle has converged
    int32_t improved;    // the last cycle improved the best iterate
    int32_t jdone, iters;
};
struct GmresCoef {
    double c[kMaxDots];
};
void launch_dots(const double *w, const double *V, int64_t N, int32_t cnt, double *part, double *out,
                 cudaStream_t st, const int32_t *skip = nullptr);
// graph-resident GMRES (control kernels and device-parameter vector kernels)
void launch_gm_begin(DevCtl *ctl, GmDev *gm, double target, unsigned long long cond_handle, cudaStream_t st);
void launch_gm_cycle(DevCtl *ctl, GmDev *gm, double target, int32_t cycle, int32_t last, cudaStream_t st);
void launch_gm_init(DevCtl *ctl, GmDev *gm, double target, cudaStream_t st);
void launch_gm_hacc(GmDev *gm, int32_t j, cudaStream_t st);
void launch_gm_arnoldi(GmDev *gm, int32_t j, cudaStream_t st);
void launch_gm_ls(GmDev *gm, cudaStream_t st);
void launch_gm_end(DevCtl *ctl, GmDev *gm, cudaStream_t st);
void launch_gs_update_dev(double *w, const double *V, const GmDev *gm, int64_t N, int32_t cnt, cudaStream_t st);
void launch_scale_dev(double *dst, const double *src, const GmDev *gm, double factor, int64_t N,
                      const int32_t *skip, cudaStream_t st);
void launch_combine_dev(double *x, const double *Z, const GmDev *gm, int64_t N, cudaStream_t st);
void launch_gs_update(double *w, const double *V, const double *h, int64_t N, int32_t cnt, cudaStream_t st);
void launch_scale(double *dst, const double *src, double alpha, int64_t N, cudaStream_t st);
void launch_combine(double *x, const double *Z, const GmresCoef &y, int64_t N, int32_t cnt, cudaStream_t st);
int32_t dots_partial_size();
// normal equations (kernels_ne.cu)
void launch_ne_form(const NeView &E, const double *Ax, const double *theta, double rho, DevCtl *ctl, cudaStream_t st);
void launch_ne_rhs(const NeView &E, const int32_t *perm, const double *Ax, const double *r7, const double *r1,
                   double *f, cudaStream_t st);
void launch_ne_dx(const NeView &E, const double *Ax, const double *dy, const double *r7, double *dx, cudaStream_t st);
void launch_residual_K(const NeView &E, const int32_t *perm, const double *Ax, const double *theta, double rho, double delta,
                       const double *r7, const double *r1, const double *dx, const double *dy, double *f, double *r,
                       double *ad, double *ae, DevCtl *ctl, cudaStream_t st);
// backward error from precomputed r, |K||d|, |K|e, f (ctl->dinf set)
void launch_omega_only(int32_t N, const double *r, const double *ad, const double *ae, const double *f, DevCtl *ctl,
                       cudaStream_t st);
// CTAs per SM of the persistent sweeps (maxf: the widest front that is one forward item)
int32_t solve_ctas_per_sm(int32_t maxf);
void launch_permute_in(const DevPlan &P, const double *r7, const double *r1, double *f, cudaStream_t st);
// x1, sel: take x1 where *sel != 0
void launch_permute_out(const DevPlan &P, const double *x, double *dx, double *dy, cudaStream_t st,
                        const double *x1 = nullptr, const int32_t *sel = nullptr);
// skip != nullptr: the kernels return at entry while *skip != 0 (graph-captured refinement)
// r = f - K (x + c), xn = x + c (c, xn null: r = f - K x); clear: not after a
// backward sweep, which clears the norms
void launch_residual_omega(const DevPlan &P, const double *f, const double *x, const double *c, double *xn, double *r,
                           double *ad, DevCtl *ctl, cudaStream_t st, const int32_t *skip = nullptr, bool clear = false);
void launch_axpy(double *x, const double *c, int32_t N, cudaStream_t st, const int32_t *skip = nullptr);
void launch_refine_init(DevCtl *ctl, double target, int32_t max_steps, cudaStream_t st);
// handle != 0: also sets a graph's conditional node to run while not done
void launch_refine_step(DevCtl *ctl, double target, int32_t step, int32_t max_steps, cudaStream_t st,
                        unsigned long long handle = 0);
void launch_refine_finish(DevCtl *ctl, double target, cudaStream_t st);
// both of a graph's iterates = the best one
void launch_best_both(double *x0, double *x1, int32_t N, const DevCtl *ctl, cudaStream_t st);
// dst = src when flag == nullptr or (*flag != 0) != invert
void launch_copy_if(double *dst, const double *src, int32_t N, const int32_t *flag, int32_t invert, cudaStream_t st);

}  // namespace ipm
