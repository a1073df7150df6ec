// Approximate Jacobian J0 of App. B.2 and its solve, one filament per warp.
//
// Per filament, J0 = [[I, 0, J13], [0, J22, J23], [I, J32, J33]] acting on
// (Y_1, u_0..u_{N-1}, Lam_0..Lam_{N-2}) (0-based segments; Lam_j joins segments
// j and j+1). Its blocks are those of App. B.2 (J13, J33 as in App. B.1):
//   J13 = -c_t I on Lam_0;  J33: c_t (Lam_{s-1} - Lam_s) in the row of segment s;
//   J32: (dL/2) w [x t_n] with w = 1 at the ends of the cumulative sum, 2 inside;
//   J22, J23 from the Taylor-truncated dexpinv and the frame-vector moments;
//   c_t = b dt/(6 pi eta a), c_r = b dt/(8 pi eta a^3), b = 2/3 (BDF2) or 1.
//
// The paper factors each 6N x 6N block densely (O(N^3)). Here the same linear
// system is solved exactly in O(N): row 1 gives Y_1 = b1 + c_t Lam_0; subtracting
// consecutive constraint rows (row_{s+1} - row_s, and row_1 - row of Y_1) removes
// Y_1 and turns the cumulative J32 into two neighbour terms. With the unknowns
// interleaved as (u_0, Lam_0, u_1, Lam_1, ..., Lam_{N-2}, u_{N-1}) the remaining
// (6N-3) x (6N-3) matrix is block-pentadiagonal in 3x3 blocks, i.e. banded with
// 8 sub- and 8 super-diagonals, and is factored by Gaussian elimination with
// partial pivoting inside the band (U gains up to 8 more super-diagonals).
//
// Band storage: row-major windows, A(i, c) at band[i * kBandW + (c - i + kBandKL)]
// for c - i in [-8, 16]; filament f starts at row 6 off[f] - 3 f.
#include <cuda_runtime.h>

#include <algorithm>

#include "approx64.cuh"
#include "fil_internal.cuh"
#include "j0_common.cuh"
#include "quat.cuh"

namespace fil {
namespace {

template <typename TO>
__device__ __forceinline__ void put_block(TO *band, int64_t row_block, int64_t col_block,
                                          const M33 &B) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int64_t i = 3 * row_block + r;
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            const int64_t col = 3 * col_block + cc;
            band[i * kBandW + (col - i + kBandKL)] = (TO)B.m[3 * r + cc];
        }
    }
}

// Assemble the band of each filament (one warp per filament), computed in
// FP64 and stored in the precision TO of the factors.
template <typename TO>
__global__ void j0_build_kernel(Layout lay, const double *__restrict__ X,
                                const double *__restrict__ qc, const double *__restrict__ Tint,
                                J0Params p, TO *__restrict__ band_all) {
    const int warp = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (warp >= lay.M) return;
    const int s0 = lay.off[warp];
    const int N = lay.off[warp + 1] - s0;
    const int64_t nrow = 6 * (int64_t)N - 3;
    TO *band = band_all + (6 * (int64_t)s0 - 3 * (int64_t)warp) * kBandW;
    for (int64_t i = lane; i < nrow * kBandW; i += 32) band[i] = TO(0);
    __syncwarp();
    const double *Xf = X + 6 * (int64_t)s0;
    const double *Lam = Xf + 3 + 3 * N;
    const M33 I3 = meye();
    for (int s = lane; s < N; s += 32) {
        const int64_t g = s0 + s;
        const Q4 qs = ld4(qc + 4 * g);
        const V3 ts = frame_t(qs);
        const V3 u = ld3(Xf + 3 + 3 * s);
        const V3 T = ld3(Tint + 3 * g);
        const V3 Lsum = ((s <= N - 2) ? ld3(Lam + 3 * s) : v3(0, 0, 0)) +
                        ((s >= 1) ? ld3(Lam + 3 * (s - 1)) : v3(0, 0, 0));
        M33 Da_r, Db_r, Da_l, Db_l;   // joint s (right) and joint s-1 (left)
        if (s <= N - 2) moment_derivs(p, qs, ld4(qc + 4 * (g + 1)), Da_r, Db_r);
        if (s >= 1) moment_derivs(p, ld4(qc + 4 * (g - 1)), qs, Da_l, Db_l);
        const M33 ux = skew(u);
        const M33 ux2 = mmul(ux, ux);
        // A_s = I - [u x]/2 + [u x]^2/12
        const M33 A = madd(madd(I3, ux, -0.5), ux2, 1.0 / 12.0);
        // dT_s/du_s
        M33 dT = mscale(mmul(rskew(Lsum), rskew(ts)), 0.5 * p.dL);
        if (s <= N - 2) dT = madd(dT, Da_r);
        if (s >= 1) dT = madd(dT, Db_l, -1.0);
        // J22_ss = I - c_r { dT - ([x T] + [u x] dT)/2 + ([x (u x T)] + [u x][x T] + [u x]^2 dT)/12 }
        const M33 xT = rskew(T);
        M33 inner = madd(dT, madd(xT, mmul(ux, dT)), -0.5);
        M33 third = madd(madd(rskew(cross(u, T)), mmul(ux, xT)), mmul(ux2, dT));
        inner = madd(inner, third, 1.0 / 12.0);
        const int64_t rb = 2 * s;   // block row of the rotation rows of segment s
        put_block(band, rb, 2 * s, madd(I3, inner, -p.cr));
        if (s <= N - 2) put_block(band, rb, 2 * s + 2, mscale(mmul(A, Db_r), -p.cr));
        if (s >= 1) put_block(band, rb, 2 * s - 2, mscale(mmul(A, Da_l), p.cr));
        // J23: -c_r A (dL/2) [t_s x] on Lam_{s-1} and Lam_s
        const M33 G = mscale(mmul(A, skew(ts)), -p.cr * 0.5 * p.dL);
        if (s >= 1) put_block(band, rb, 2 * s - 1, G);
        if (s <= N - 2) put_block(band, rb, 2 * s + 1, G);
        // differenced constraint rows of joint j = s:
        // (dL/2)([x t_s] u_s + [x t_{s+1}] u_{s+1}) + c_t(-Lam_{s-1} + 2 Lam_s - Lam_{s+1})
        if (s <= N - 2) {
            const int64_t cb = 2 * s + 1;
            const V3 tn = frame_t(ld4(qc + 4 * (g + 1)));
            put_block(band, cb, 2 * s, mscale(rskew(ts), 0.5 * p.dL));
            put_block(band, cb, 2 * s + 2, mscale(rskew(tn), 0.5 * p.dL));
            put_block(band, cb, 2 * s + 1, mscale(I3, 2.0 * p.ct));
            if (s >= 1) put_block(band, cb, 2 * s - 1, mscale(I3, -p.ct));
            if (s + 1 <= N - 2) put_block(band, cb, 2 * s + 3, mscale(I3, -p.ct));
        }
    }
}

constexpr int kJ0Threads = 128;
constexpr int kLuRing = 16;    // band rows a warp keeps in shared memory
constexpr int kLuAhead = 13;   // column j requests row j + kLuAhead

// One element of a band row, global -> shared, asynchronously (cp.async).
template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst, const T *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

// In-place banded LU with partial pivoting (one warp per filament), in the
// precision T of the stored factors. Column j reads and writes rows j .. j+8
// only, and row j is final once column j is done, so each warp keeps a ring
// of kLuRing band rows in shared memory: row j + kLuAhead is requested with
// cp.async at column j (into the slot of row j - 3, already written back),
// waited for five columns later, and row j is written back, with its pivot
// replaced by the reciprocal the solves multiply by, when column j is done.
template <typename T>
__global__ void __launch_bounds__(kJ0Threads)
band_lu_kernel(Layout lay, T *__restrict__ band_all, int *__restrict__ piv_all,
               int *__restrict__ flags) {
    static_assert(kLuAhead < kLuRing, "a requested row reuses the slot of a written-back row");
    __shared__ T ring_all[kJ0Threads / 32][kLuRing * kBandW];
    const int warp = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (warp >= lay.M) return;
    const int s0 = lay.off[warp];
    const int N = lay.off[warp + 1] - s0;
    const int n = 6 * N - 3;
    const int64_t row0 = 6 * (int64_t)s0 - 3 * (int64_t)warp;
    T *G = band_all + row0 * kBandW;
    T *R = ring_all[threadIdx.x >> 5];
    int *piv = piv_all + row0;
#define RB(i, c) R[((i) & (kLuRing - 1)) * kBandW + ((c) - (i) + kBandKL)]
    for (int r = 0; r < kLuAhead && r < n; ++r)
        if (lane < kBandW) cp_async_elem(&R[r * kBandW + lane], G + (int64_t)r * kBandW + lane);
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    for (int j = 0; j < n; ++j) {
        {
            const int r = j + kLuAhead;
            if (r < n && lane < kBandW)
                cp_async_elem(&R[(r & (kLuRing - 1)) * kBandW + lane], G + (int64_t)r * kBandW + lane);
            cp_async_commit();
        }
        // rows up to j + 8, requested at column j + 8 - kLuAhead or before, have landed
        cp_async_wait<kLuAhead - kBandKL>();
        __syncwarp();
        const int last = min(n - 1, j + kBandKL);
        // pivot: first row of maximal |A(i, j)|, i in [j, last]
        T v = T(-1);
        int idx = j;
        if (j + lane <= last && lane <= kBandKL) {
            v = fabs(RB(j + lane, j));
            idx = j + lane;
        }
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) {
            const T ov = __shfl_down_sync(0xffffffffu, v, d);
            const int oi = __shfl_down_sync(0xffffffffu, idx, d);
            if (ov > v || (ov == v && oi < idx)) {
                v = ov;
                idx = oi;
            }
        }
        const int p = __shfl_sync(0xffffffffu, idx, 0);
        const T pv = __shfl_sync(0xffffffffu, v, 0);
        if (lane == 0) piv[j] = p;
        const int cmax = min(n - 1, j + kBandKL + kBandKU);
        if (p != j) {
            const int c = j + lane;
            if (c <= cmax) {
                const T t = RB(j, c);
                RB(j, c) = RB(p, c);
                RB(p, c) = t;
            }
        }
        __syncwarp();
        if (pv == T(0)) {
            if (lane == 0) atomicOr(flags + 1, 1);
        } else {
            const T inv = T(1) / RB(j, j);
            if (lane >= 1 && j + lane <= last) RB(j + lane, j) = RB(j + lane, j) * inv;
            __syncwarp();
            // rank-1 update of rows j+1..last (lane / 16 + 2k), columns j+1..cmax (lane % 16)
            const int c = j + 1 + (lane & 15);
            if (c <= cmax) {
                const T ujc = RB(j, c);
#pragma unroll
                for (int k = 0; k < kBandKL / 2; ++k) {
                    const int i = j + 1 + (lane >> 4) + 2 * k;
                    if (i <= last) RB(i, c) -= RB(i, j) * ujc;
                }
            }
        }
        __syncwarp();
        // row j is final: write it back (the solves multiply by the reciprocal pivot)
        if (lane < kBandW) {
            T e = R[(j & (kLuRing - 1)) * kBandW + lane];
            if (lane == kBandKL) e = e != T(0) ? T(1) / e : T(0);
            G[(int64_t)j * kBandW + lane] = e;
        }
    }
#undef RB
}

constexpr int kLu64Threads = 128;

// The same elimination in FP64 for one system: a CTA per filament. A column is
// one chain (pivot search, reciprocal, multipliers, rank-1 update, next column)
// and a warp instruction on FP64 takes 64 cycles of its quarter of the SM, so
// what counts is the number of them in one warp's chain. Each of the 128
// threads updates one element (8 rows x 16 columns, one warp instruction on
// each quarter), the pivot search compares bit patterns as integers, the nine
// candidates' reciprocals are formed beside it by recip above, and rows are
// exchanged by reading from the other row. One 20-segment filament (117
// columns): 168 us with one warp's work as in band_lu_kernel, 75 us here.
// Ensembles keep band_lu_kernel: their iteration counts follow the last bit.
__global__ void __launch_bounds__(kLu64Threads)
band_lu64_kernel(Layout lay, double *__restrict__ band_all, int *__restrict__ piv_all,
                 int *__restrict__ flags) {
    static_assert(kLu64Threads == 16 * kBandKL && kBandKL + kBandKU == 16, "a thread per element");
    __shared__ double R[kLuRing * kBandW];
    const int f = blockIdx.x, t = threadIdx.x, lane = t & 31;
    const int s0 = lay.off[f];
    const int n = 6 * (lay.off[f + 1] - s0) - 3;
    const int64_t row0 = 6 * (int64_t)s0 - 3 * (int64_t)f;
    double *G = band_all + row0 * kBandW;
    int *piv = piv_all + row0;
#define RB(i, c) R[((i) & (kLuRing - 1)) * kBandW + ((c) - (i) + kBandKL)]
    for (int r = 0; r < kLuAhead && r < n; ++r)
        if (t < kBandW) cp_async_elem(&R[r * kBandW + t], G + (int64_t)r * kBandW + t);
    cp_async_commit();
    cp_async_wait<0>();
    for (int j = 0; j < n; ++j) {
        {
            const int r = j + kLuAhead;
            if (r < n && t < kBandW)
                cp_async_elem(&R[(r & (kLuRing - 1)) * kBandW + t], G + (int64_t)r * kBandW + t);
            cp_async_commit();
        }
        // rows up to j + 8, requested at column j + 8 - kLuAhead or before, have landed
        cp_async_wait<kLuAhead - kBandKL>();
        __syncthreads();
        const int last = min(n - 1, j + kBandKL);
        // pivot: first row of maximal |A(i, j)|, i in [j, last] (every warp finds it)
        const bool cand = lane <= kBandKL && j + lane <= last;
        const double v = cand ? RB(j + lane, j) : 0.0;
        const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
        const unsigned lo = (unsigned)__double2loint(v);
        const double rv = recip(cand && (hi | lo) ? v : 1.0);
        const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
        const unsigned mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
        const int pl = __ffs(__ballot_sync(0xffffffffu, cand && hi == mhi && lo == mlo)) - 1;
        const int p = j + pl;
        const bool zero = (mhi | mlo) == 0;
        const double inv = zero ? 0.0 : __shfl_sync(0xffffffffu, rv, pl);
        const int cmax = min(n - 1, j + kBandKL + kBandKU);
        // element (i, c) of the trailing window, from row j where the rows change places
        const int i = j + 1 + (t >> 4), c = j + 1 + (t & 15);
        const int src = i == p ? j : i;
        const bool in = i <= last && c <= cmax;
        double l = 0.0, a = 0.0;
        if (i <= last) l = RB(src, j) * inv;
        if (in) a = fma(-l, RB(p, c), RB(src, c));
        // row j is final: the multipliers that lie in it, the reciprocal pivot, U
        if (t < kBandW) {
            const int cj = j + t - kBandKL;
            G[(int64_t)j * kBandW + t] = t < kBandKL                 ? R[(j & (kLuRing - 1)) * kBandW + t]
                                         : t == kBandKL ? inv
                                         : cj <= cmax   ? RB(p, cj)
                                                        : 0.0;
        }
        if (t == 0) {
            piv[j] = p;
            if (zero) atomicOr(flags + 1, 1);
        }
        __syncthreads();
        if (!zero) {
            if (in) RB(i, c) = a;
            if ((t & 15) == 0 && i <= last) RB(i, j) = l;
        }
    }
#undef RB
}

constexpr int kSolvePf = 8;     // rows of factors loaded ahead by the band solve
constexpr int kSolveLanes = 16; // lanes per filament

// Forward and backward substitution in the banded factors for one right-hand
// side z (n entries in shared memory, in band order), by
// 16 lanes, half a warp; the two halves of a warp run the longer one's n_both
// steps together.
//
// A row step is a chain: the finished entry z_j, one multiply-add in each row
// it reaches, the next finished entry. The window of rows it reaches (j + 1 ..
// j + 8 forward, j - 1 .. j - 16 backward) therefore stays in registers, row i
// in lane i mod 16, and z_j goes to the lanes with a shuffle; shared memory
// holds only the entries that wait to enter the window. (With the window in
// shared memory a step was two loads, a store and a warp barrier long, ~40
// instructions of a whole warp. One 20-segment filament in FP64 41 -> 30 us,
// where the FP64 unit takes 64 cycles per warp instruction; the steps of 256
// ensemble systems in FP32 80.5 -> 77.7 ms. Same bits.)
template <typename T>
__device__ __forceinline__ void band_substitute(const T *__restrict__ A,
                                                const int *__restrict__ piv, T *z, int n,
                                                int n_both, int lane) {
#define BAND(i, c) A[(int64_t)(i) * kBandW + ((c) - (i) + kBandKL)]
    // The factors a row step needs do not depend on z, so each lane loads them
    // kSolvePf rows ahead into a register queue: the loads of the next block are
    // in flight while the current block's chain runs.
    // forward: L with row interchanges applied in elimination order; lane l holds
    // the row r in [j, j + 15] with r = l (mod 16)
    T w;
    {
        w = lane < n ? z[lane] : T(0);
    }
    {
        T lq[kSolvePf];
        int pq[kSolvePf];
        const auto fetch = [&](int j, T &l, int &p) {
            const int d = (lane - j) & (kSolveLanes - 1);        // row j + d
            l = (d >= 1 && d <= kBandKL && j + d < n) ? BAND(j + d, j) : T(0);
            p = j < n ? piv[j] : j;
        };
#pragma unroll
        for (int u = 0; u < kSolvePf; ++u) fetch(u, lq[u], pq[u]);
        for (int jb = 0; jb < n_both; jb += kSolvePf) {
            T ln[kSolvePf];
            int pn[kSolvePf];
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) fetch(jb + kSolvePf + u, ln[u], pn[u]);
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) {
                const int j = jb + u;
                const int p = pq[u];
                // the entry that enters the window when row j leaves it
                const int in = j + kSolveLanes;
                const T zin = (in & (kSolveLanes - 1)) == lane && in < n ? z[in] : T(0);
                // row j after the interchange with row p (p in j .. j+8)
                const T zold = __shfl_sync(0xffffffffu, w, j & (kSolveLanes - 1), kSolveLanes);
                const T zj = __shfl_sync(0xffffffffu, w, p & (kSolveLanes - 1), kSolveLanes);
                const int d = (lane - j) & (kSolveLanes - 1);
                if (d >= 1 && d <= kBandKL && j + d < n) w = ((j + d == p) ? zold : w) - lq[u] * zj;
                if (d == 0 && j < n) {
                    z[j] = zj;
                    w = zin;
                }
            }
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) {
                lq[u] = ln[u];
                pq[u] = pn[u];
            }
        }
    }
    __syncwarp();
    // backward, column by column: z_j *= 1/U_jj (stored reciprocal), then the
    // kl + ku rows above take their U_ij z_j; lane l holds the row r in [j - 15, j]
    // with r = l (mod 16), and row j - 16 once z_j is out
    {
        // (a shorter half starts when its last row comes up: k counts from n_both - 1)
        const int k0 = n_both - 1;
        {
            const int d = (n - 1 - lane) & (kSolveLanes - 1);   // row n - 1 - d
            w = n - 1 - d >= 0 ? z[n - 1 - d] : T(0);
        }
        T uq[kSolvePf], dq[kSolvePf];
        const auto fetch = [&](int j, T &uu, T &dd) {
            const bool in = j < n;
            int d = (j - lane) & (kSolveLanes - 1);             // row j - d, d = 16 for lane j mod 16
            if (d == 0) d = kSolveLanes;
            uu = (in && j - d >= 0) ? BAND(j - d, j) : T(0);
            dd = (in && j >= 0) ? BAND(j, j) : T(0);
        };
        static_assert(kBandKL + kBandKU == kSolveLanes, "a lane per row a backward step reaches");
#pragma unroll
        for (int u = 0; u < kSolvePf; ++u) fetch(k0 - u, uq[u], dq[u]);
        for (int jb = k0; jb >= 0; jb -= kSolvePf) {
            T un[kSolvePf], dn[kSolvePf];
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) fetch(jb - kSolvePf - u, un[u], dn[u]);
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) {
                const int j = jb - u;
                const bool mine = (j & (kSolveLanes - 1)) == lane;
                const T zin = mine && j < n && j >= kSolveLanes ? z[j - kSolveLanes] : T(0);
                const T zj = __shfl_sync(0xffffffffu, w, j & (kSolveLanes - 1), kSolveLanes) * dq[u];
                if (j >= 0 && j < n) {
                    if (mine) {
                        z[j] = zj;
                        w = zin;
                    }
                    int d = (j - lane) & (kSolveLanes - 1);
                    if (d == 0) d = kSolveLanes;
                    if (j - d >= 0) w -= uq[u] * zj;
                }
            }
#pragma unroll
            for (int u = 0; u < kSolvePf; ++u) {
                uq[u] = un[u];
                dq[u] = dn[u];
            }
        }
    }
    __syncwarp();
#undef BAND
}

// x = J0^{-1} b for every filament (b and x in the X / f layout; may alias),
// with the factors and the working vector in precision T, 16 lanes (half a
// warp) per filament.
template <typename T>
__global__ void band_solve_kernel(Layout lay, const T *__restrict__ band_all,
                                  const int *__restrict__ piv_all, double ct,
                                  const double *b, double *x, int zmax,
                                  const int *__restrict__ active, int fil_per_cta) {
    extern __shared__ __align__(16) unsigned char zraw[];
    pdl_enter();
    const int slot = threadIdx.x / kSolveLanes;        // filament within the CTA
    const int lane = threadIdx.x % kSolveLanes;
    const int f = blockIdx.x * fil_per_cta + slot;
    // (a half without a filament, or of a converged system, takes no rows)
    bool live = slot < fil_per_cta && f < lay.M;
    int s0 = 0, N = 0;
    if (live) {
        s0 = lay.off[f];
        N = lay.off[f + 1] - s0;
        if (active && !active[lay.sys_of[s0]]) live = false;
    }
    const int n = live ? 6 * N - 3 : 0;
    const int n_both = max(n, __shfl_xor_sync(0xffffffffu, n, kSolveLanes));
    if (n_both == 0) return;
    T *z = reinterpret_cast<T *>(zraw) + (int64_t)(live ? slot : 0) * zmax;
    const int64_t row0 = 6 * (int64_t)s0 - 3 * (int64_t)(live ? f : 0);
    const T *A = band_all + row0 * kBandW;
    const int *piv = piv_all + row0;
    const double *bf = b + 6 * (int64_t)s0;
    double *xf = x + 6 * (int64_t)s0;
    // gather the right-hand side in band order
    double b1x = 0.0, b1y = 0.0, b1z = 0.0;
    if (live) {
        for (int e = lane; e < 3 * N; e += kSolveLanes) {
            const int s = e / 3, r = e % 3;
            z[6 * s + r] = (T)bf[3 + 3 * s + r];   // rotation rows of segment s
            if (s <= N - 2) {
                const double b3n = bf[3 + 3 * N + 3 * s + r];                  // f3 of segment s+1
                const double b3p = (s == 0) ? bf[r] : bf[3 + 3 * N + 3 * (s - 1) + r];
                z[6 * s + 3 + r] = (T)(b3n - b3p);
            }
        }
        b1x = bf[0];
        b1y = bf[1];
        b1z = bf[2];
    }
    __syncwarp();
    band_substitute(A, piv, z, n, n_both, lane);
    if (!live) return;
    // scatter back: u_s, Lam_j, and Y_1 = b1 + c_t Lam_0
    for (int e = lane; e < 3 * N; e += kSolveLanes) {
        const int s = e / 3, r = e % 3;
        xf[3 + 3 * s + r] = (double)z[6 * s + r];
        if (s <= N - 2) xf[3 + 3 * N + 3 * s + r] = (double)z[6 * s + 3 + r];
    }
    if (lane == 0) {
        const double l0 = (N >= 2) ? (double)z[3] : 0.0, l1 = (N >= 2) ? (double)z[4] : 0.0,
                     l2 = (N >= 2) ? (double)z[5] : 0.0;
        xf[0] = b1x + ct * l0;
        xf[1] = b1y + ct * l1;
        xf[2] = b1z + ct * l2;
    }
}

// The solve of one FP64 system in blocks of kBlk rows. Substitution row by row is
// a serial chain of 2 (6N - 3) steps, and a chain step on FP64 (a multiply-add or
// two, each 64 cycles of a quarter of the SM, and the shuffle between) costs the
// same whether one row or 32 take part. So each factorization also forms, for
// every block of kBlk columns, what its steps do together to the rows they
// reach: forward, interchanges included, one dense map of the kBlk + 8 rows
// from the block's first on (F); backward one of the block's kBlk entries to
// the solution there and to the updates of the 16 rows above (B). A solve is
// then one small matrix-vector product per block and direction, whose columns
// spread over the lanes of four warps.
//
// The maps are made of the same factors. Against extended arithmetic a solve is as
// close as row by row: relative error 1.05e-15 and 1.23e-15 (rms, blocks and rows)
// at 20 segments, 2.09e-15 and 2.12e-15 at 40, 5.07e-15 and 5.16e-15 for 4 x 64; the
// full inverse of a filament's band, as quick to apply, was 1.3 to 2 times as far
// off. Blocks of 16 rows fill four warps (F: 24 x 24, B: 32 x 16); larger ones do
// more work per row (24: F 32 x 32, B 40 x 24).
//
// One 20-segment filament: a solve 33 -> 14.6 us, forming the maps 14.5 us once a
// factorization. The rule (block_solve_on) is two filaments for each SM, as long as
// the chains bound the solve and not the SMs' FP64 rate. Four time steps at drag
// mobility, rows and blocks: 1 x 20 segments 5.20 and 3.35 ms, 1 x 100 30.9 and 15.9,
// 20 x 32 14.9 and 11.4, 152 x 10 13.0 and 12.6, 304 x 10 43.2 and 42.4. Beyond, each
// filament added costs a block's 4x as many multiply-adds. kBlkMaxSeg bounds the maps'
// memory (3.3 KB a segment). Ensembles keep the rows: their iteration counts follow
// the last bit.
constexpr int kBlk = kBlkRows;
constexpr int kFwd = kBlk + kBandKL;                       // rows (and columns) of F
constexpr int kBwd = kBlk + kBandKL + kBandKU;             // rows of B
constexpr int kBlkThreads = 128;                           // 8 rows x 4 column groups a warp
constexpr int kFwdThreads = 4 * kFwd;
static_assert(4 * kBwd == kBlkThreads && kBwd == 32 && kFwd == 24, "the lanes' share of F and B");
static_assert(kFwd * kFwd + kBwd * kBlk == kBlkDoubles, "doubles of a block's maps");

// Position of (row, column) of F or B in the order the solve's threads read them:
// thread (row / 8) 32 + (column mod 4) 8 + row mod 8 takes columns 4 k + column mod 4.
__device__ __forceinline__ int map_pos(int r, int c, int threads) {
    return (c >> 2) * threads + (r >> 3) * 32 + (c & 3) * 8 + (r & 7);
}

// F (blockIdx.z = 0) and B (1) of one block, by one warp: the block's steps
// applied to unit vectors, a lane per column (F) or two (B, half the rows each).
__global__ void __launch_bounds__(32)
band_block_kernel(Layout lay, const int64_t *__restrict__ bofs, const double *__restrict__ band_all,
                  const int *__restrict__ piv_all, double *__restrict__ maps) {
    __shared__ double rows[kBwd * kBandW];     // the band rows the block reaches
    __shared__ double w[kBwd][32];             // the vectors: [row of the window][lane]
    pdl_enter();
    const int f = blockIdx.x, lane = threadIdx.x;
    const int s0 = lay.off[f];
    const int n = 6 * (lay.off[f + 1] - s0) - 3;
    const int jb = kBlk * blockIdx.y;
    if (jb >= n) return;
    const int64_t row0 = 6 * (int64_t)s0 - 3 * (int64_t)f;
    double *out = maps + (bofs[f] + blockIdx.y) * kBlkDoubles;
    const int steps = min(kBlk, n - jb);
    const bool forward = blockIdx.z == 0;
    const int i0 = forward ? jb : jb - (kBandKL + kBandKU);     // first row of the window
    const int ni = forward ? kFwd : kBwd;
    for (int e = lane; e < ni * kBandW; e += 32) {
        const int i = i0 + e / kBandW;
        rows[e] = i >= 0 && i < n ? band_all[(row0 + i0) * kBandW + e] : 0.0;
    }
#define BAND(i, c) rows[((i) - i0) * kBandW + ((c) - (i) + kBandKL)]
    if (forward) {
        for (int r = 0; r < kFwd; ++r) w[r][lane] = r == lane ? 1.0 : 0.0;
        int pv = lane < steps ? piv_all[row0 + jb + lane] - jb : 0;
        __syncwarp();
        for (int jj = 0; jj < steps; ++jj) {
            const int p = __shfl_sync(0xffffffffu, pv, jj);
            const double z = w[p][lane];
            w[p][lane] = w[jj][lane];
            w[jj][lane] = z;
#pragma unroll
            for (int d = 1; d <= kBandKL; ++d)       // (rows past the last hold zeros)
                w[jj + d][lane] = fma(-BAND(jb + jj + d, jb + jj), z, w[jj + d][lane]);
        }
        if (lane < kFwd)
            for (int r = 0; r < kFwd; ++r) out[map_pos(r, lane, kFwdThreads)] = w[r][lane];
    } else {
        const int c = lane & (kBlk - 1), half = lane / kBlk;
        for (int r = half; r < kBwd; r += 2) w[r][c] = r == c + kBwd - kBlk ? 1.0 : 0.0;
        __syncwarp();
        for (int jj = steps - 1; jj >= 0; --jj) {
            const int j = jb + jj, rj = jj + kBwd - kBlk;
            const double z = w[rj][c] * BAND(j, j);
            __syncwarp();
            if (half == 0) w[rj][c] = z;
#pragma unroll
            for (int d = 0; d < (kBandKL + kBandKU) / 2; ++d) {
                const int r = jj + half * (kBandKL + kBandKU) / 2 + d;      // row i0 + r
                w[r][c] = fma(-BAND(i0 + r, j), z, w[r][c]);                // (zeros above row 0)
            }
            __syncwarp();
        }
        out += kFwd * kFwd;
        for (int r = half; r < kBwd; r += 2) out[map_pos(r, c, kBlkThreads)] = w[r][c];
    }
#undef BAND
}

// x = J0^{-1} b with those maps, a CTA per filament (b and x may alias: b is read
// before x is written). Each step reads the block's input from one of two small
// buffers and leaves the next block's in the other, one barrier a step; the maps
// of the next step are loaded during it.
__global__ void __launch_bounds__(kBlkThreads)
band_block_solve_kernel(Layout lay, const int64_t *__restrict__ bofs,
                        const double *__restrict__ maps, double ct, int zmax, const double *b,
                        double *x) {
    extern __shared__ __align__(16) unsigned char zraw[];
    __shared__ double next[2][kBlk];
    pdl_enter();
    const int f = blockIdx.x, t = threadIdx.x;
    const int s0 = lay.off[f];
    const int N = lay.off[f + 1] - s0;
    const int n = 6 * N - 3;
    const int nb = (n + kBlk - 1) / kBlk;
    double *z = reinterpret_cast<double *>(zraw);     // the right-hand side, in band order
    double *y = z + zmax;                             // after the forward pass, then x
    const double *bf = b + 6 * (int64_t)s0;
    double *xf = x + 6 * (int64_t)s0;
    const double *mf = maps + bofs[f] * kBlkDoubles + t;
    const int row = (t >> 5) * 8 + (t & 7), g = (t >> 3) & 3;     // row of the map, column group
    constexpr int kF = kFwd / 4, kB = kBlk / 4;
    double m[kF];
    if (t < kFwdThreads) {
#pragma unroll
        for (int k = 0; k < kF; ++k) m[k] = mf[k * kFwdThreads];
    }
    for (int i = t; i < nb * kBlk + kBandKL; i += kBlkThreads) {
        const int s = i / 6, q = i % 6;
        double v = 0.0;                               // (rows past the last)
        if (i < n) {
            if (q < 3) {
                v = bf[3 + 3 * s + q];                // rotation rows of segment s
            } else {                                  // f3 of segment s + 1, less that of s
                const int r = q - 3;
                v = bf[3 + 3 * N + 3 * s + r] -
                    (s == 0 ? bf[r] : bf[3 + 3 * N + 3 * (s - 1) + r]);
            }
        }
        z[i] = v;
        if (i < kBandKL) next[0][i] = v;
    }
    const double b1 = t < 3 ? bf[t] : 0.0;
    __syncthreads();
    for (int k0 = 0; k0 < nb; ++k0) {
        const int jb = k0 * kBlk, now = k0 & 1;
        double a = 0.0, mn[kF];
        if (t < kFwdThreads) {
            if (k0 + 1 < nb) {
#pragma unroll
                for (int k = 0; k < kF; ++k)
                    mn[k] = mf[(int64_t)(k0 + 1) * kBlkDoubles + k * kFwdThreads];
            }
#pragma unroll
            for (int k = 0; k < kF; ++k)
                a = fma(m[k], 4 * k < kBandKL ? next[now][4 * k + g] : z[jb + 4 * k + g], a);
            a += __shfl_xor_sync(0xffffffffu, a, 8);
            a += __shfl_xor_sync(0xffffffffu, a, 16);
            if (g == 0) {
                if (row < kBlk)
                    y[jb + row] = a;
                else
                    next[now ^ 1][row - kBlk] = a;
            }
#pragma unroll
            for (int k = 0; k < kF; ++k) m[k] = mn[k];
        }
        if (k0 + 1 < nb) __syncthreads();
    }
    mf += kFwd * kFwd;
#pragma unroll
    for (int k = 0; k < kB; ++k) m[k] = mf[(int64_t)(nb - 1) * kBlkDoubles + k * kBlkThreads];
    __syncthreads();
    if (t < kBlk) next[0][t] = y[(nb - 1) * kBlk + t];
    __syncthreads();
    for (int k0 = nb - 1, now = 0; k0 >= 0; --k0, now ^= 1) {
        const int jb = k0 * kBlk;
        double mn[kB];
        if (k0 > 0) {
#pragma unroll
            for (int k = 0; k < kB; ++k)
                mn[k] = mf[(int64_t)(k0 - 1) * kBlkDoubles + k * kBlkThreads];
        }
        double a = 0.0;
#pragma unroll
        for (int k = 0; k < kB; ++k) a = fma(m[k], next[now][4 * k + g], a);
        a += __shfl_xor_sync(0xffffffffu, a, 8);
        a += __shfl_xor_sync(0xffffffffu, a, 16);
        if (g == 0) {
            if (row >= kBlk)
                y[jb + row - kBlk] = a;
            else if (k0 > 0)
                next[now ^ 1][row] = y[jb - kBlk + row] + a;
        }
#pragma unroll
        for (int k = 0; k < kB; ++k) m[k] = mn[k];
        __syncthreads();
    }
    // scatter: u_s, Lam_j, and Y_1 = b1 + c_t Lam_0
    for (int i = t; i < n; i += kBlkThreads) {
        const int s = i / 6, q = i % 6;
        xf[q < 3 ? 3 + 3 * s + q : 3 + 3 * N + 3 * s + q - 3] = y[i];
    }
    if (t < 3) xf[t] = b1 + ct * (N >= 2 ? y[3 + t] : 0.0);
}

size_t block_solve_smem(const fil_ctx *c) {
    return 2 * sizeof(double) * (size_t)(6 * c->lay.maxN + 2 * kBlk);
}

J0Params make_params(const fil_ctx *c) {
    const double beta = c->have_prev ? 2.0 / 3.0 : 1.0;
    return J0Params{c->dL, c->KB, c->KT, c->g0, c->kmu, c->knu,
                    beta * c->dt / (6.0 * kPi * c->eta * c->a),
                    beta * c->dt / (8.0 * kPi * c->eta * c->a * c->a * c->a)};
}

}  // namespace

bool block_solve_on(const fil_ctx *c) {
    return c->n_sys == 1 && !fast_mixed(c) && c->lay.M <= 2 * c->num_sms && c->lay.S <= kBlkMaxSeg &&
           block_solve_smem(c) <= kSolveSmemMax;
}

cudaError_t j0_build_factor(fil_ctx *c, const double *X) {
    const unsigned grid = (unsigned)(((int64_t)c->lay.M * 32 + kJ0Threads - 1) / kJ0Threads);
    const J0Params p = make_params(c);
    if (c->band32) {
        // mixed precision: the band is stored, factored and solved in FP32 (J0 is an
        // approximation of the Jacobian far coarser than FP32 rounding; FP64 issues at
        // 1/64 of the FP32 rate on this GPU); its entries are still computed in FP64
        j0_build_kernel<float><<<grid, kJ0Threads, 0, c->stream>>>(c->lay, X, c->qc, c->Tint, p,
                                                                   c->band32);
        band_lu_kernel<float><<<grid, kJ0Threads, 0, c->stream>>>(c->lay, c->band32, c->piv,
                                                                  c->d_flags);
    } else {
        j0_build_kernel<double><<<grid, kJ0Threads, 0, c->stream>>>(c->lay, X, c->qc, c->Tint, p,
                                                                    c->band);
        if (c->n_sys == 1)
            band_lu64_kernel<<<c->lay.M, kLu64Threads, 0, c->stream>>>(c->lay, c->band, c->piv,
                                                                       c->d_flags);
        else
            band_lu_kernel<double><<<grid, kJ0Threads, 0, c->stream>>>(c->lay, c->band, c->piv,
                                                                       c->d_flags);
    }
    c->n_launches += 2;
    if (c->bmaps) {
        const unsigned blocks = (unsigned)((6 * c->lay.maxN - 3 + kBlk - 1) / kBlk);
        c->n_launches += 1;
        return launch_pdl(band_block_kernel, dim3((unsigned)c->lay.M, blocks, 2), 32, 0, c->stream,
                          c->lay, c->jofs, c->band, c->piv, c->bmaps);
    }
    return cudaGetLastError();
}

cudaError_t j0_solve(fil_ctx *c, const double *b, double *x, const int *active) {
    // in blocks of rows (one system, which no list of active ones narrows), else half a
    // warp per filament; up to 4 warps per CTA, fewer for long filaments so that each
    // filament's right-hand side fits in shared memory
    const double ct = make_params(c).ct;
    if (c->bmaps) {
        const size_t smem = block_solve_smem(c);
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(band_block_solve_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
        }
        c->n_launches += 1;
        // Early (launch_dep) while its CTAs find SMs of their own. Three steps at drag
        // mobility, early and plainly, FIL_FP64: 1.83 and 1.89 ms with 5 filaments, 3.23 and
        // 3.41 with 20, 5.0 and 5.2 with 38, 10.9 and 11.0 with 76, 57.6 and 57.4 with 200;
        // FIL_PAIR32: 4.95 and 5.03 with 60, 6.38 and 6.18 with 100, 19.7 and 17.7 with 300.
        return launch_dep(c->lay.M <= c->num_sms / 2, band_block_solve_kernel, c->lay.M,
                          kBlkThreads, smem, c->stream, c->lay, c->jofs, c->bmaps, ct,
                          6 * c->lay.maxN + 2 * kBlk, b, x);
    }
    const int zmax = 6 * c->lay.maxN;
    const size_t per = (size_t)zmax * sizeof(double);
    const int fils = (int)std::min<size_t>(8, kSolveSmemMax / per);
    if (fils < 1) return cudaErrorInvalidValue;
    const size_t smem = fils * per;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(band_solve_kernel<double>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(band_solve_kernel<float>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int threads = (kSolveLanes * fils + 31) / 32 * 32;
    const unsigned grid = (unsigned)((c->lay.M + fils - 1) / fils);
    c->n_launches += 1;
    // Early (launch_dep) up to one filament per SM: the kernel is one wave, each SM bound
    // by its chains, and waits for the fullest SM. Two steps of ensembles, early and
    // plainly: 3.46 and 3.53 ms with 51 filaments, 4.77 and 4.36 with 232, 6.42 and 5.47
    // with 336, 10.40 and 9.37 with 1 460, 74.9 and 74.7 with 8 192.
    const bool early = c->lay.M <= c->num_sms;
    return c->band32 ? launch_dep(early, band_solve_kernel<float>, grid, threads, smem, c->stream,
                                  c->lay, c->band32, c->piv, ct, b, x, zmax, active, fils)
                     : launch_dep(early, band_solve_kernel<double>, grid, threads, smem, c->stream,
                                  c->lay, c->band, c->piv, ct, b, x, zmax, active, fils);
}

}  // namespace fil
