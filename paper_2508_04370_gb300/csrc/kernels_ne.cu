// Normal-equations path (Zanetti & Gondzio, arXiv 2508.04370, Eq. normeq with
// the regularisation of Eq. regul_matrix):
//   Theta~ = (Theta^-1 + rho I)^-1
//   M      = A Theta~ A^T            (formed every iteration; delta enters at the pivot)
//   r8     = r1 + A Theta~ r7,   M_reg dy = r8,   dx = Theta~ (A^T dy - r7).
// Formation is deterministic (no atomics): every lower entry (r, i) of M sums its
// own contributor pairs a_rj Theta~_j a_ij, up to kWarpRow of them in ascending
// column j, more of them strided over the lanes of a warp or a CTA and the lanes'
// sums in a fixed tree (rows_common.cuh).
#include <cuda_runtime.h>

#include <cstdint>

#include "ipm_dev.h"
#include "rows_common.cuh"

namespace ipm {

namespace {

constexpr int kThreads = rows::kThreads;

inline int grid_for(int64_t work) {
    int64_t g = (work + kThreads - 1) / kThreads;
    return (int)(g < 1 ? 1 : (g > 1216 ? 1216 : g));
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__global__ void k_theta_tilde(const double *__restrict__ theta, double rho, int n, double *__restrict__ tt,
                              DevCtl *ctl) {
    bool bad = false;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double th = theta[j];
        if (!(th > 0.0) || !isfinite(th)) bad = true;
        tt[j] = 1.0 / (1.0 / th + rho);
    }
    if (bad) atomicOr(&ctl->status, kStatNonFinite);
}

// One sum per item over its terms [b, e): `range` gives the terms and what the
// sums start from (the first lane's), `term` adds term t to the NA sums of its
// lane, `put` stores the finished sums of an item.  Items of at most
// kWarpRow terms run one per thread in term order, longer ones a warp or a
// CTA each (rows_common.cuh).  On 37 blocks of 60 x 160 with 8 dense rows
// (sums of 5,920 terms) forming M takes 12 us instead of 1,750 and the
// residual on K 10 us instead of 1,180.
template <int NA, class Range, class Term, class Put>
__device__ __forceinline__ void row_sums(int64_t shorts, const int32_t *mid, int nmid, const int32_t *lng, int nlong,
                                         Range range, Term term, Put put) {
    __shared__ double sh[rows::kThreads / 32][NA];
    const rows::Part w = rows::part(nmid, nlong);
    auto strided = [&](int64_t b, int64_t e, int t, int nt, double (&a)[NA]) {
        if (t > 0)
#pragma unroll
            for (int c = 0; c < NA; c++) a[c] = 0.0;
#pragma unroll 4
        for (int64_t p = b + t; p < e; p += nt) term(p, a);
    };
    int64_t b, e;
    double a[NA];
    if (w.cta >= 0) {
        range(lng[w.cta], b, e, a);
        strided(b, e, threadIdx.x, rows::kThreads, a);
        rows::cta_add(a, sh);
        if (threadIdx.x == 0) put(lng[w.cta], a);
    } else if (w.mid >= 0) {
        if (w.mid < nmid) {
            range(mid[w.mid], b, e, a);
            strided(b, e, threadIdx.x & 31, 32, a);
            rows::warp_add(a);
            if ((threadIdx.x & 31) == 0) put(mid[w.mid], a);
        }
    } else {
        for (int64_t i = w.first; i < shorts; i += w.stride) {
            range(i, b, e, a);
            if (e - b > kWarpRow) continue;
            strided(b, e, 0, 1, a);
            put(i, a);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_ne_form(NeView E, const double *__restrict__ Ax) {
    row_sums<1>(
        E.nnz, E.emid, E.nemid, E.elong, E.nelong,
        [&](int64_t i, int64_t &b, int64_t &e, double (&a)[1]) { b = E.tptr[i], e = E.tptr[i + 1], a[0] = 0.0; },
        [&](int64_t t, double (&a)[1]) { a[0] += Ax[E.ta[t]] * (Ax[E.tb[t]] * E.tt[E.tj[t]]); },
        [&](int64_t i, const double (&a)[1]) { E.nev[i] = a[0]; });
}

// r8 in the factorisation order: f[i] = r1[o] + sum_j a_oj (Theta~_j r7_j), o = perm[i]
__global__ void __launch_bounds__(kThreads) k_ne_rhs(NeView E, const int32_t *__restrict__ perm,
                                                     const double *__restrict__ Ax, const double *__restrict__ r7,
                                                     const double *__restrict__ r1, double *__restrict__ f) {
    row_sums<1>(
        E.m, E.rmid, E.nrmid, E.rlong, E.nrlong,
        [&](int64_t i, int64_t &b, int64_t &e, double (&a)[1]) {
            const int o = perm[i];
            b = E.Arp[o], e = E.Arp[o + 1], a[0] = r1[o];
        },
        [&](int64_t p, double (&a)[1]) {
            const int j = E.Aci[p];
            a[0] += Ax[E.Apos[p]] * (E.tt[j] * r7[j]);
        },
        [&](int64_t i, const double (&a)[1]) { f[i] = a[0]; });
}

// dx_j = Theta~_j (sum_i a_ij dy_i - r7_j)
__global__ void __launch_bounds__(kThreads) k_ne_dx(NeView E, const double *__restrict__ Ax,
                                                    const double *__restrict__ dy, const double *__restrict__ r7,
                                                    double *__restrict__ dx) {
    row_sums<1>(
        E.n, E.cmid, E.ncmid, E.clong, E.nclong,
        [&](int64_t j, int64_t &b, int64_t &e, double (&a)[1]) { b = E.Acp[j], e = E.Acp[j + 1], a[0] = 0.0; },
        [&](int64_t p, double (&a)[1]) { a[0] += Ax[p] * dy[E.Ari[p]]; },
        [&](int64_t j, const double (&a)[1]) { dx[j] = E.tt[j] * (a[0] - r7[j]); });
}

// Residual of the regularised augmented system in the original order (for
// reporting the backward error on K of a normal-equations solve):
// r = [r7; r1] - K [dx; dy], ad = |K||d|, ae = |K|e, running max |d|.  Two
// launches: the columns of A, then its rows.
struct KResidual {
    double *f, *r, *ad, *ae;
};
__device__ __forceinline__ void start_residual(double dg, double di, double (&a)[3]) {
    a[0] = dg * di;
    a[1] = fabs(dg) * fabs(di);
    a[2] = fabs(dg);
}
__device__ __forceinline__ void put_residual(const KResidual &R, int64_t i, double fi, const double (&a)[3]) {
    R.f[i] = fi;
    R.r[i] = fi - a[0];
    R.ad[i] = a[1];
    R.ae[i] = a[2];
}
__device__ __forceinline__ void add_term(double (&a)[3], double v, double x) {
    a[0] += v * x;
    a[1] += fabs(v) * fabs(x);
    a[2] += fabs(v);
}
__device__ __forceinline__ void max_abs(DevCtl *ctl, double xm) {
    xm = warp_max(xm);
    if ((threadIdx.x & 31) == 0)
        atomicMax((unsigned long long *)&ctl->dinf, (unsigned long long)__double_as_longlong(xm));
}

__global__ void __launch_bounds__(kThreads) k_residual_K_cols(NeView E, const double *__restrict__ Ax,
                                                              const double *__restrict__ theta, double rho,
                                                              const double *__restrict__ r7,
                                                              const double *__restrict__ dx,
                                                              const double *__restrict__ dy, KResidual R, DevCtl *ctl) {
    double xm = 0.0;
    row_sums<3>(
        E.n, E.cmid, E.ncmid, E.clong, E.nclong,
        [&](int64_t j, int64_t &b, int64_t &e, double (&a)[3]) {
            b = E.Acp[j], e = E.Acp[j + 1];
            start_residual(-(1.0 / theta[j] + rho), dx[j], a);
        },
        [&](int64_t p, double (&a)[3]) { add_term(a, Ax[p], dy[E.Ari[p]]); },
        [&](int64_t j, const double (&a)[3]) {
            put_residual(R, j, r7[j], a);
            xm = fmax(xm, fabs(dx[j]));
        });
    max_abs(ctl, xm);
}

__global__ void __launch_bounds__(kThreads) k_residual_K_rows(NeView E, const int32_t *__restrict__ perm,
                                                              const double *__restrict__ Ax, double delta,
                                                              const double *__restrict__ r1,
                                                              const double *__restrict__ dx,
                                                              const double *__restrict__ dy, KResidual R, DevCtl *ctl) {
    double xm = 0.0;
    row_sums<3>(
        E.m, E.rmid, E.nrmid, E.rlong, E.nrlong,
        [&](int64_t i, int64_t &b, int64_t &e, double (&a)[3]) {
            const int o = perm[i];
            b = E.Arp[o], e = E.Arp[o + 1];
            start_residual(delta, dy[o], a);
        },
        [&](int64_t p, double (&a)[3]) { add_term(a, Ax[E.Apos[p]], dx[E.Aci[p]]); },
        [&](int64_t i, const double (&a)[3]) {
            const int o = perm[i];
            put_residual(R, (int64_t)E.n + o, r1[o], a);
            xm = fmax(xm, fabs(dy[o]));
        });
    max_abs(ctl, xm);
}

}  // namespace

void launch_ne_form(const NeView &E, const double *Ax, const double *theta, double rho, DevCtl *ctl,
                    cudaStream_t st) {
    k_theta_tilde<<<grid_for(E.n), kThreads, 0, st>>>(theta, rho, E.n, E.tt, ctl);
    const int32_t shorts = (int32_t)(E.nnz < (int64_t(1) << 30) ? E.nnz : (int64_t(1) << 30));  // sizes the grid only
    k_ne_form<<<rows::grid(shorts, E.nemid, E.nelong), kThreads, 0, st>>>(E, Ax);
}

void launch_ne_rhs(const NeView &E, const int32_t *perm, const double *Ax, const double *r7, const double *r1,
                   double *f, cudaStream_t st) {
    k_ne_rhs<<<rows::grid(E.m, E.nrmid, E.nrlong), kThreads, 0, st>>>(E, perm, Ax, r7, r1, f);
}

void launch_ne_dx(const NeView &E, const double *Ax, const double *dy, const double *r7, double *dx,
                  cudaStream_t st) {
    k_ne_dx<<<rows::grid(E.n, E.ncmid, E.nclong), kThreads, 0, st>>>(E, Ax, dy, r7, dx);
}

void launch_residual_K(const NeView &E, const int32_t *perm, const double *Ax, const double *theta, double rho,
                       double delta, const double *r7, const double *r1, const double *dx, const double *dy, double *f,
                       double *r, double *ad, double *ae, DevCtl *ctl, cudaStream_t st) {
    cudaMemsetAsync(&ctl->dinf, 0, sizeof(double), st);
    cudaMemsetAsync(&ctl->omega, 0, sizeof(double), st);
    const KResidual R{f, r, ad, ae};
    k_residual_K_cols<<<rows::grid(E.n, E.ncmid, E.nclong), kThreads, 0, st>>>(E, Ax, theta, rho, r7, dx, dy, R, ctl);
    k_residual_K_rows<<<rows::grid(E.m, E.nrmid, E.nrlong), kThreads, 0, st>>>(E, perm, Ax, delta, r1, dx, dy, R, ctl);
}

}  // namespace ipm
