// Rotne-Prager-Yamakawa mobility apply on sm_103a (paper Sec. 2.7.1).
//
//   V_n     = sum_m Mtt_nm F_m + Mtr_nm T_m
//   Omega_n = sum_m Mrt_nm F_m + Mrr_nm T_m      over all S^2 ordered pairs.
//
// With d = Y_n - Y_m, r = |d| and every block scaled by 8 pi eta, a pair adds
//   V     += A F + B (d.F) d + G (T x d)
//   Omega += C T + D (d.T) d + G (F x d)
// far form (r >= 2a):  A = 1/r + (2a^2/3)/r^3, B = 1/r^3 - 2a^2/r^5,
//                      C = -1/(2 r^3), D = 3/(2 r^5), G = 1/r^3;
// overlapping spheres (r < 2a, equal-radius form of Wajnryb et al., which the
// paper cites for this case):
//                      A = (4/(3a)) (1 - 9r/(32a)),  B = 1/(8 a^2 r),
//                      C = (1 - 27r/(32a) + 5r^3/(64a^3)) / a^3,
//                      D = (9/(32 a r) - 3r/(64 a^3)) / a^3,
//                      G = (1 - 3r/(8a)) / (2 a^3);
// at r = 0 (the self pair, or coincident distinct segments) the d-terms vanish
// and A, C give the self mobilities 1/(6 pi eta a), 1/(8 pi eta a^3).
//
// Kernel design (GB300, one GPU):
//  * No tensor cores: the pair sum is not a dense contraction (forming its two
//    contracted coefficients and splitting them into BF16 pieces costs as many
//    FP32-pipe cycles as the sums it would save). The bound is the FP32 (or
//    FP64) FMA pipe.
//  * Packed FP32x2 arithmetic. One system (rpy_pair32_warp_kernel): a thread
//    evaluates two targets against one source at once, lane x and lane y of every
//    float2 (pair32_far2). Ensembles and other schedules (rpy_pair32_kernel):
//    one target against two sources, whose records are stored interleaved so that
//    each loaded float2 is an operand (pair32_far).
//  * Each thread owns two targets in registers (one in the 128-target
//    schedules) and all lanes read the same source from shared memory
//    (broadcast).
//  * One system's sources come in groups of 32 relative to the group's centre, and
//    the pair terms are summed in that frame, but for Omega at the targets inside a
//    group that spans several filaments (wide_radius2).
//  * Stream-K persistent grid: the work units (tile of targets, group of
//    sources) are split evenly over the grid; who touches a tile only in part
//    writes one partial of it, and the CTA that completes a tile (a counter
//    per tile) sums its partials in a fixed order and writes the tile's rows,
//    in the same launch. The order of the sums never depends on timing:
//    results are bitwise reproducible.
//  * Mixed precision: FP32 pair terms, 32 of them summed in FP32 and folded
//    into a (hi, lo) compensated accumulator (TwoSum); groups in which a warp
//    met a pair closer than R_c = 4a are evaluated again with hi/lo position
//    differences, and with the exact far / overlap coefficients where a pair
//    overlaps.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <vector>
#include <mutex>
#include <type_traits>
#include <utility>

#include "approx64.cuh"
#include "fil_internal.cuh"

namespace fil {
namespace {

constexpr float kFarPad = 1.0e5f;   // position of padding sources (they carry no load)

struct RpyConst32 {
    float near2;       // (2a)^2
    float over2;       // (2a)^2 (1 + 1e-3): a far pass that meets a pair this close may hold an overlap
    float close2;      // R_c^2 = (4a)^2: groups with a pair this close use hi/lo differences
    float k23a2;       // 2a^2/3
    float k2a2;        // 2a^2
    float ov_A0, ov_A1;          // A = ov_A0 - ov_A1 r
    float ov_B;                  // B = ov_B / r
    float ov_C0, ov_C1, ov_C3;   // C = ov_C0 - ov_C1 r + ov_C3 r^3
    float ov_D0, ov_D1;          // D = ov_D0 / r - ov_D1 r
    float ov_G0, ov_G1;          // G = ov_G0 - ov_G1 r
};

struct RpyConst64 {
    double near2, k23a2, k2a2;
    double ov_A0, ov_A1, ov_B, ov_C0, ov_C1, ov_C3, ov_D0, ov_D1, ov_G0, ov_G1;
};

template <typename T, typename K>
__host__ K make_const(double a) {
    K k;
    k.near2 = (T)(4.0 * a * a);
    if constexpr (sizeof(T) == 4) {
        k.close2 = (T)(16.0 * a * a);
        k.over2 = (T)(4.004 * a * a);
    }
    k.k23a2 = (T)(2.0 * a * a / 3.0);
    k.k2a2 = (T)(2.0 * a * a);
    k.ov_A0 = (T)(4.0 / (3.0 * a));
    k.ov_A1 = (T)(4.0 / (3.0 * a) * 9.0 / (32.0 * a));
    k.ov_B = (T)(1.0 / (8.0 * a * a));
    double ia3 = 1.0 / (a * a * a);
    k.ov_C0 = (T)ia3;
    k.ov_C1 = (T)(ia3 * 27.0 / (32.0 * a));
    k.ov_C3 = (T)(ia3 * 5.0 / (64.0 * a * a * a));
    k.ov_D0 = (T)(ia3 * 9.0 / (32.0 * a));
    k.ov_D1 = (T)(ia3 * 3.0 / (64.0 * a * a * a));
    k.ov_G0 = (T)(0.5 * ia3);
    k.ov_G1 = (T)(0.5 * ia3 * 3.0 / (8.0 * a));
    return k;
}

// ---------------------------------------------------------------------------
// Ensembles of independent systems: every system is padded to a multiple of
// kRpyPad positions in the source/target layout, so that a work unit (tile,
// source chunk) never mixes systems and the apply stays one persistent launch.
// System s owns padded positions [pad_off[s], pad_off[s+1]); its tiles come
// in order, each with ceil(S_s / unit_sources) units, and
// padding records sit far away with zero load. With null tables there is one
// system whose padded position equals the segment index (tile = u / n_units).
// ---------------------------------------------------------------------------
struct SysMap {
    const int64_t *tile_unit_off;  // [n_tiles + 1] first unit of each listed tile
    const int64_t *tile_src;       // [n_tiles] padded position of the tile's first source
    const int64_t *tile_nsrc;      // [n_tiles] real sources of the tile's system (null: n_src)
    const int *tile_id;            // [n_tiles] padded tile of each listed tile (null: same)
    const int *pad_map;            // [Spad] segment at a padded position, or -1
    int64_t n_tiles, n_units;      // listed tiles; n_units: units per tile, the one-system case
    int64_t n_src;                 // real sources of the one-system case
    // non-null: {listed tiles, work units} read on the device, so that a captured
    // launch stays valid when the list of active tiles is rewritten
    const int64_t *dyn = nullptr;
};

// Sources of a work unit: one group where the sources are in frames (the automatic
// schedule of one FP32 system), else whole 128-source chunks.
constexpr int unit_sources(bool frames) { return frames ? kRpyComp : kRpyChunk; }

// The listed tiles and the unit count of a launch (from the device when dynamic).
__device__ __forceinline__ void resolve_dyn(SysMap &m, int64_t &W) {
    if (m.dyn) {
        m.n_tiles = m.dyn[0];
        W = m.dyn[1];
    }
}

__device__ __forceinline__ int64_t tile_unit_begin(const SysMap &m, int64_t tile) {
    return m.tile_unit_off ? m.tile_unit_off[tile] : tile * m.n_units;
}

// Tile of work unit u, the tile's first unit and unit count, and its first source.
__device__ __forceinline__ void locate_unit(const SysMap &m, int64_t u, int64_t &tile,
                                            int64_t &ubeg, int64_t &nun, int64_t &src0) {
    if (!m.tile_unit_off) {
        tile = u / m.n_units;
        ubeg = tile * m.n_units;
        nun = m.n_units;
        src0 = 0;
        return;
    }
    int64_t lo = 0, hi = m.n_tiles;      // tile_unit_off[lo] <= u < tile_unit_off[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (m.tile_unit_off[mid] <= u) lo = mid;
        else hi = mid;
    }
    tile = lo;
    ubeg = m.tile_unit_off[lo];
    nun = m.tile_unit_off[lo + 1] - ubeg;
    src0 = m.tile_src[lo];
}

__device__ __forceinline__ int64_t segment_at(const SysMap &m, int64_t P, int64_t S) {
    return m.pad_map ? (int64_t)m.pad_map[P] : (P < S ? P : -1);
}

// Error-free transformation s + e = a + b (Knuth's TwoSum), with the adds
// kept out of FMA contraction and reassociation.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// a b - c d to within 1.5 ulp of the exact value (Kahan).
__device__ __forceinline__ float diff_of_products(float a, float b, float c, float d) {
    const float w = __fmul_rn(c, d);
    return __fadd_rn(__fmaf_rn(a, b, -w), __fmaf_rn(-c, d, w));
}

// ---------------------------------------------------------------------------
// Pack: FP64 (Y, FT) -> FP32 source groups of kRpyComp = 32 padded positions.
// A group is Rec::kGroupF4 float4: first its centre (c_x, c_y, c_z, w), the mean of
// its real positions relative to the first segment of the apply (the apply is
// translation invariant, and FP32 rounding then depends on the extent of the
// suspension, not on where it sits), rounded to FP32; then 16 source pairs of
// kRpyPairF4 float4. With s' = Y - Y_0 - c a source has 18 values
//   -s'(hi) 3 | F 3 | T 3 | -T x s' 3 | -(2/3) F x s' 3 | -s'(lo) 3
// and value c of source h (0 even, 1 odd) of a pair sits at float 2c + h, so
// that each float2 holds one component of both; the far-form loop reads the
// first 15. One warp packs one group. Padding records sit far away with zero
// load, so they add exactly zero. w is the squared radius within which targets take
// the cross products per pair (wide_radius2; 0: none).
// Ensembles, and one system in another schedule than the automatic one, have records
// without a frame (kFrames false): 12 values per source
//   -y(hi) 3 | F 3 | T 3 | -y(lo) 3,   y = Y - Y_0 = hi + lo.
// The ensembles' systems with the drag J0 take tens of Broyden iterations whose path
// follows the last bits of the pair sums (a system's count moves by one or two
// with any other rounding, and its multipliers with it, by ~1e-3), so their
// pair arithmetic, work units and order of sums stay those their trajectories
// were made with.
// ---------------------------------------------------------------------------
template <bool kFrames>
struct Rec {
    static constexpr int kPairF4 = kFrames ? kRpyPairF4 : 6;      // float4 per source pair
    static constexpr int kLo = kFrames ? 7 : 4;                   // the lo parts: float4 kLo, half 1 on
    static constexpr int kHead = kFrames ? 1 : 0;                 // float4 before the pairs (centre)
    static constexpr int kGroupF4 = kHead + kPairF4 * kRpyComp / 2;
};

// Order of the n groups' records for the automatic schedule: 16 runs of neighbouring
// groups dealt out in turn, so that the groups whose close pairs cost a tile up to
// three times a far unit (its own and the next ones of its filaments) go to
// different warps. spread_group: the group at place i; spread_place: its inverse.
// spread_count: n where the order pays, else 0, the groups' own. Whole applies, own
// order and spread, filaments of 32, of 20, of 16 to 48 segments: 960 segments 20.9 and
// 21.7 us, 21.9 and 23.3, 22.5 and 23.6 (a unit per warp: nothing to spread); 1 536 26.6 and
// 28.2, 28.3 and 30.2, 33.4 and 31.4; 1 920 33.5 and 35.3, 36.4 and 37.5, 40.7 and 37.4;
// 3 200 46.7 and 45.0, 52.8 and 47.9, 53.3 and 48.2; 6 400 86 and 85, 98 and 93, 106 and
// 100; 12 288 240 and 243, 270 and 265, 265 and 265; 16 000 384 and 388, 423 and 429, 422
// and 421.
__host__ __device__ __forceinline__ int spread_count(int64_t n) {
    return n >= 48 && n <= 384 ? (int)n : 0;
}
__device__ __forceinline__ int spread_group(int i, int n) {
    const int r = i & 15, q = n >> 4, rem = n & 15;
    return i < n ? r * q + min(r, rem) + (i >> 4) : i;
}
__device__ __forceinline__ int spread_place(int g, int n) {
    const int q = n >> 4, head = (n & 15) * (q + 1);       // groups in the longer runs
    if (g >= n) return g;
    const int r = g < head ? g / (q + 1) : (n & 15) + (g - head) / q;
    return 16 * (g < head ? g % (q + 1) : (g - head) % q) + r;
}

// The squared radius around a group's centre within which its targets are summed
// with the cross products formed per pair (w of the group), 0 for none. The sums in
// the group's frame (pair32_far) leave a cross product as the difference of two sums,
// (sum G F) x t - sum G (F x s), which cancel where |t| and |s| are large against the
// distance: at the targets inside the ball a group spans when its segments are not
// neighbours of one another. A group whose consecutive segments lie within R_c is a
// piece of one filament and keeps the sums in its frame at any extent, as does one
// within 16a. Error of Omega against 64 bits (2%, 32 000 segments), with the cross
// products per pair everywhere, in the frames everywhere, and by this rule: single
// segments 1.81e-7, 2.43e-7, 1.65e-7; filaments of 8 1.62, 1.77, 1.56; of 16 to 48
// 1.63, 1.68, 1.60; of 32 1.63, 1.62, 1.60. Whole applies in the frames everywhere and
// by the rule: 1515 and 1671 us, 1436 and 1592, 1421 and 1516, 1426 and 1435. (A ball of
// half that squared radius would be 1-3% faster and no longer as close for filaments of 16.)
constexpr float kCompact = 16.f, kChainGap = 4.f;
__device__ __forceinline__ float wide_radius2(const float *sp, bool live, float a) {
    const unsigned all = 0xffffffffu;
    float gap2 = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float d = sp[c] - __shfl_up_sync(all, sp[c], 1);       // (lane 0: its own)
        gap2 = fmaf(d, d, gap2);
    }
    float ext2 = live ? fmaf(sp[0], sp[0], fmaf(sp[1], sp[1], sp[2] * sp[2])) : 0.f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) ext2 = fmaxf(ext2, __shfl_xor_sync(all, ext2, d));
    const bool chain = !__any_sync(all, live && gap2 > kChainGap * kChainGap * a * a);
    return chain || ext2 <= kCompact * kCompact * a * a ? 0.f : ext2;
}

// (two warps per CTA: a small system's groups then spread over the SMs)
constexpr int kPackThreads = 64;
template <bool kFrames>
__global__ void __launch_bounds__(kPackThreads)
pack32_kernel(const double *__restrict__ Y, const double *__restrict__ FT, int64_t S, int64_t Spad,
              SysMap sm, int n_spread, float a, float4 *__restrict__ src) {
    pdl_enter();
    const int64_t P = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (P >= Spad) return;             // Spad is a multiple of 32: whole warps leave
    const int lane = threadIdx.x & 31;
    // (the first n_spread groups in the order of spread_group, the rest in their own)
    const int64_t i = segment_at(
        sm, n_spread ? 32 * (int64_t)spread_group((int)(P >> 5), n_spread) + lane : P, S);
    double y[3] = {0.0, 0.0, 0.0};
    float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i >= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) y[c] = Y[3 * i + c] - Y[c];
#pragma unroll
        for (int c = 0; c < 6; ++c) f[c] = __double2float_rn(FT[6 * i + c]);
    }
    using R = Rec<kFrames>;
    float v[2 * R::kPairF4];
#pragma unroll
    for (int c = 0; c < 2 * R::kPairF4; ++c) v[c] = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) v[3 + c] = f[c];
    float4 *g = src + R::kGroupF4 * (P >> 5);
    if constexpr (kFrames) {
        const unsigned live = __ballot_sync(0xffffffffu, i >= 0);
        const float inv = live ? 1.f / (float)__popc(live) : 0.f;
        float cen[3], sp[3], yh[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float m = yh[c] = __double2float_rn(y[c]);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) m += __shfl_xor_sync(0xffffffffu, m, d);
            cen[c] = m * inv;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // s' = y - c from the FP32 parts of y (the FP64 unit has 1/64 of the rate)
            const float l = __double2float_rn(y[c] - (double)yh[c]);
            float u, e;
            two_sum(yh[c], -cen[c], u, e);
            e = __fadd_rn(e, l);
            two_sum(u, e, sp[c], e);
            v[c] = -sp[c];
            v[15 + c] = -e;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // -(T x s')_c and -(2/3)(F x s')_c, the differences of products with the
            // rounding of one product carried along (one FMA each)
            const int p = (c + 1) % 3, q = (c + 2) % 3;
            v[9 + c] = -diff_of_products(f[3 + p], sp[q], f[3 + q], sp[p]);
            v[12 + c] = (-2.f / 3.f) * diff_of_products(f[p], sp[q], f[q], sp[p]);
        }
        const float w2 = wide_radius2(sp, i >= 0, a);
        if (lane == 0) g[0] = make_float4(cen[0], cen[1], cen[2], w2);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float h = __double2float_rn(y[c]);
            v[c] = -h;
            v[9 + c] = -__double2float_rn(y[c] - (double)h);
        }
    }
    if (i < 0) {
#pragma unroll
        for (int c = 0; c < 2 * R::kPairF4; ++c) v[c] = c < 3 ? -kFarPad : 0.f;
    }
    float *o = reinterpret_cast<float *>(g + R::kHead + R::kPairF4 * (lane >> 1)) + (lane & 1);
#pragma unroll
    for (int c = 0; c < 2 * R::kPairF4; ++c) o[2 * c] = v[c];
}

// FP64 records: 9 doubles per segment (Y, F, T); padding far away, no load.
__global__ void pack64_kernel(const double *__restrict__ Y, const double *__restrict__ FT,
                              int64_t S, int64_t Spad, SysMap sm, double *__restrict__ src) {
    pdl_enter();
    const int64_t P = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (P >= Spad) return;
    const int64_t i = segment_at(sm, P, S);
    double *o = src + 9 * P;
    if (i >= 0) {
        o[0] = Y[3 * i];
        o[1] = Y[3 * i + 1];
        o[2] = Y[3 * i + 2];
        for (int k = 0; k < 6; ++k) o[3 + k] = FT[6 * i + k];
    } else {
        o[0] = o[1] = o[2] = (double)kFarPad;
        for (int k = 0; k < 6; ++k) o[3 + k] = 0.0;
    }
}

// 1/sqrt(x): one MUFU operation (PTX rsqrt.approx.ftz.f32, max relative error
// 2^-22.9 for normal x). Its results are kept only for r^2 >= (2a)^2.
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

// sqrt(x) and 1/x: one MUFU operation each (PTX sqrt.approx.ftz.f32,
// rcp.approx.ftz.f32; a few ulp at most, no slow path).
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Exact coefficients of one pair (one lane): the far form for r^2 >= (2a)^2,
// the overlapping-sphere form below it and the self values at r = 0, chosen
// without a branch (both are evaluated; this runs in recomputed groups only).
__device__ __forceinline__ void coef_exact(float r2, const RpyConst32 &k, float &A, float &B,
                                           float &C, float &D, float &G) {
    const bool ov = r2 < k.near2;
    const float rinv = rsqrt_approx(fmaxf(r2, k.near2));   // the far form's, finite everywhere
    const float r = sqrt_approx(r2);
    const float ri = r > 0.f ? rcp_approx(r) : 0.f;
    const float rinv2 = rinv * rinv;
    const float rinv3 = rinv * rinv2;
    const float rinv5 = rinv3 * rinv2;
    A = ov ? fmaf(-k.ov_A1, r, k.ov_A0) : fmaf(k.k23a2, rinv3, rinv);
    B = ov ? k.ov_B * ri : fmaf(-k.k2a2, rinv5, rinv3);
    C = ov ? fmaf(k.ov_C3 * r2, r, fmaf(-k.ov_C1, r, k.ov_C0)) : -0.5f * rinv3;
    D = ov ? fmaf(k.ov_D0, ri, -k.ov_D1 * r) : 1.5f * rinv5;
    G = ov ? fmaf(-k.ov_G1, r, k.ov_G0) : rinv3;
}

// (V, Omega) sums of a pair with the coefficients A..G and the difference d,
// the cross products formed for the pair (negated operands fold into the
// packed FMA).
__device__ __forceinline__ void add_pair(float2 dx, float2 dy, float2 dz, float2 Fx, float2 Fy,
                                         float2 Fz, float2 Tx, float2 Ty, float2 Tz, float2 A,
                                         float2 B, float2 C, float2 D, float2 G, float2 *acc) {
    const float2 bF = __fmul2_rn(B, __ffma2_rn(dx, Fx, __ffma2_rn(dy, Fy, __fmul2_rn(dz, Fz))));
    const float2 dT = __fmul2_rn(D, __ffma2_rn(dx, Tx, __ffma2_rn(dy, Ty, __fmul2_rn(dz, Tz))));
    const float2 ex = __fmul2_rn(G, dx), ey = __fmul2_rn(G, dy), ez = __fmul2_rn(G, dz);
    const float2 nTx = neg2(Tx), nTy = neg2(Ty), nTz = neg2(Tz);
    const float2 nFx = neg2(Fx), nFy = neg2(Fy), nFz = neg2(Fz);
    acc[0] = __ffma2_rn(A, Fx, __ffma2_rn(bF, dx, __ffma2_rn(Ty, ez, __ffma2_rn(nTz, ey, acc[0]))));
    acc[1] = __ffma2_rn(A, Fy, __ffma2_rn(bF, dy, __ffma2_rn(Tz, ex, __ffma2_rn(nTx, ez, acc[1]))));
    acc[2] = __ffma2_rn(A, Fz, __ffma2_rn(bF, dz, __ffma2_rn(Tx, ey, __ffma2_rn(nTy, ex, acc[2]))));
    acc[3] = __ffma2_rn(C, Tx, __ffma2_rn(dT, dx, __ffma2_rn(Fy, ez, __ffma2_rn(nFz, ey, acc[3]))));
    acc[4] = __ffma2_rn(C, Ty, __ffma2_rn(dT, dy, __ffma2_rn(Fz, ex, __ffma2_rn(nFx, ez, acc[4]))));
    acc[5] = __ffma2_rn(C, Tz, __ffma2_rn(dT, dz, __ffma2_rn(Fx, ey, __ffma2_rn(nFy, ex, acc[5]))));
}

// The loads of a record's two sources.
__device__ __forceinline__ void add_pair(const float4 *q, float2 dx, float2 dy, float2 dz, float2 A,
                                         float2 B, float2 C, float2 D, float2 G, float2 *acc) {
    const float4 q1 = q[1], q2 = q[2], q3 = q[3];
    const float2 Tz = reinterpret_cast<const float2 *>(q + 4)[0];
    add_pair(dx, dy, dz, f2(q1.z, q1.w), f2(q2.x, q2.y), f2(q2.z, q2.w), f2(q3.x, q3.y),
             f2(q3.z, q3.w), Tz, A, B, C, D, G, acc);
}

// Far-form coefficients.
__device__ __forceinline__ void far_coef(float2 rinv, const RpyConst32 &k, float2 &A, float2 &B,
                                         float2 &C, float2 &D, float2 &G) {
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    G = __fmul2_rn(rinv, rinv2);
    const float2 rinv5 = __fmul2_rn(G, rinv2);
    A = __ffma2_rn(f2(k.k23a2, k.k23a2), G, rinv);
    B = __ffma2_rn(f2(-k.k2a2, -k.k2a2), rinv5, G);
    C = __fmul2_rn(f2(-0.5f, -0.5f), G);
    D = __fmul2_rn(f2(1.5f, 1.5f), rinv5);
}

// The inner loop without frames: the pair terms of one target (position t relative to
// the apply's first segment, both lanes) and the two sources of a packed record q, lane
// x = even source, lane y = odd source, in the far form, branch-free; whatever it
// produces for close, overlapping or coincident pairs (Inf or NaN at r = 0) is
// discarded by the caller, which evaluates such groups again. rmin2 tracks the
// smallest r^2. 48 FP32 operations a pair, acc[0..2] += V terms, acc[3..5] += Omega
// terms.
__device__ __forceinline__ void pair32_far(const float2 *t, const float4 *q, const RpyConst32 &k,
                                           float2 *acc, float &rmin2) {
    const float4 q0 = q[0], q1 = q[1];
    const float2 dx = __fadd2_rn(t[0], f2(q0.x, q0.y));
    const float2 dy = __fadd2_rn(t[1], f2(q0.z, q0.w));
    const float2 dz = __fadd2_rn(t[2], f2(q1.x, q1.y));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    rmin2 = fminf(rmin2, fminf(r2.x, r2.y));
    float2 A, B, C, D, G;
    far_coef(f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y)), k, A, B, C, D, G);
    add_pair(q, dx, dy, dz, A, B, C, D, G, acc);
}

// The inner loop in the group's frame: the same for two targets, lane x and lane y of t,
// and source H (0 even, 1 odd) of the record.
//
// With d = t - s in the group's frame the cross products split,
//   sum G (T x d) = (sum G T) x t - sum G (T x s),
// and likewise for F x d, so that a pair needs no G d: 12 sums take
//   acc[0..2] += (1/r) F + B (d.F) d - G (T x s)   (V without its G F part)
//   acc[3..5] += r^-5 (d.T) d - (2/3) G (F x s)    (2/3 of Omega's d-terms)
//   acc[6..8] += G T,  acc[9..11] += G F           (see combine_group2)
// in 39 FP32 operations a pair, 9 fewer than with the cross products formed
// for every pair. What bounds the loop is register operands: a packed FMA
// with three distinct register operands issues every third cycle, one with
// two every second, and this form drops 3-operand FMAs (24 -> 21 sums) as
// well as multiplies. Both targets take a source's values from single registers, so a
// packed FMA reads one register fewer than with two sources in the lanes.
// Measured (32 000 segments in filaments of 32, pair kernel): 1700 us with the cross
// products formed per pair, 1491 us with two sources in the lanes (whole apply 1477),
// 1426 (whole apply) in this form, unrolled in full; by 8 1484, as iterations of the loop
// do not overlap. Error against 64 bits of V 1.85e-7 and 1.55e-7 (the frames make the
// differences finer), of Omega 1.63e-7 and 1.60e-7: that gains nothing where a group spans
// more than its neighbourhood, see wide_radius2.
constexpr int kFarSums = 12;
template <int H>
__device__ __forceinline__ float2 both(const float4 &v, int half) {
    const float x = half ? (H ? v.w : v.z) : (H ? v.y : v.x);
    return f2(x, x);
}
template <int H>
__device__ __forceinline__ void pair32_far2(const float2 *t, const float4 *q, const RpyConst32 &k,
                                            float2 *acc, float2 &rmin2) {
    const float2 nk2 = f2(-k.k2a2, -k.k2a2);
    const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3], q4 = q[4], q5 = q[5], q6 = q[6];
    const float q7 = reinterpret_cast<const float *>(q + 7)[H];
    const float2 dx = __fadd2_rn(t[0], both<H>(q0, 0));
    const float2 dy = __fadd2_rn(t[1], both<H>(q0, 1));
    const float2 dz = __fadd2_rn(t[2], both<H>(q1, 0));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float2 rinv = f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
    rmin2 = f2(fminf(rmin2.x, r2.x), fminf(rmin2.y, r2.y));
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    const float2 G = __fmul2_rn(rinv, rinv2);
    const float2 rinv5 = __fmul2_rn(G, rinv2);
    const float2 B = __ffma2_rn(nk2, rinv5, G);
    const float2 Fx = both<H>(q1, 1), Fy = both<H>(q2, 0), Fz = both<H>(q2, 1);
    const float2 Tx = both<H>(q3, 0), Ty = both<H>(q3, 1), Tz = both<H>(q4, 0);
    const float2 bF = __fmul2_rn(B, __ffma2_rn(dx, Fx, __ffma2_rn(dy, Fy, __fmul2_rn(dz, Fz))));
    const float2 dT =
        __fmul2_rn(rinv5, __ffma2_rn(dx, Tx, __ffma2_rn(dy, Ty, __fmul2_rn(dz, Tz))));
    acc[0] = __ffma2_rn(rinv, Fx, __ffma2_rn(G, both<H>(q4, 1), __ffma2_rn(bF, dx, acc[0])));
    acc[1] = __ffma2_rn(rinv, Fy, __ffma2_rn(G, both<H>(q5, 0), __ffma2_rn(bF, dy, acc[1])));
    acc[2] = __ffma2_rn(rinv, Fz, __ffma2_rn(G, both<H>(q5, 1), __ffma2_rn(bF, dz, acc[2])));
    acc[3] = __ffma2_rn(G, both<H>(q6, 0), __ffma2_rn(dT, dx, acc[3]));
    acc[4] = __ffma2_rn(G, both<H>(q6, 1), __ffma2_rn(dT, dy, acc[4]));
    acc[5] = __ffma2_rn(G, f2(q7, q7), __ffma2_rn(dT, dz, acc[5]));
    acc[6] = __ffma2_rn(G, Tx, acc[6]);
    acc[7] = __ffma2_rn(G, Ty, acc[7]);
    acc[8] = __ffma2_rn(G, Tz, acc[8]);
    acc[9] = __ffma2_rn(G, Fx, acc[9]);
    acc[10] = __ffma2_rn(G, Fy, acc[10]);
    acc[11] = __ffma2_rn(G, Fz, acc[11]);
}

// Two targets against source H, for the targets inside a wide group (wide_radius2): as
// pair32_far2, but Omega's cross product formed for the pair,
//   acc[0..2] += A F + B (d.F) d - G (T x s)   (V without P x t)
//   acc[3..5] += D (d.T) d + G (F x d)         (Omega without -P/2)
//   acc[6..8] += G T = P
// V keeps its frame: dominated by A F, it is closer to 64 bits there. 44 operations a pair
// (48 with V's cross product per pair too: 32 000 single segments 1741 us, 1673 in this
// form). The loop is unrolled by 2 only: a warp changes between it and the far loop, and
// both must fit in the instruction cache (9 651 segments in ragged filaments by 2 180 us,
// by 4 185; with 48 operations by 8 205, by 16 236).
constexpr int kCrossSums = 9;
template <int H>
__device__ __forceinline__ void pair32_cross2(const float2 *t, const float4 *q, const RpyConst32 &k,
                                              float2 *acc, float2 &rmin2) {
    const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3], q4 = q[4], q5 = q[5];
    const float2 dx = __fadd2_rn(t[0], both<H>(q0, 0));
    const float2 dy = __fadd2_rn(t[1], both<H>(q0, 1));
    const float2 dz = __fadd2_rn(t[2], both<H>(q1, 0));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    rmin2 = f2(fminf(rmin2.x, r2.x), fminf(rmin2.y, r2.y));
    float2 A, B, C, D, G;
    far_coef(f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y)), k, A, B, C, D, G);
    const float2 Fx = both<H>(q1, 1), Fy = both<H>(q2, 0), Fz = both<H>(q2, 1);
    const float2 Tx = both<H>(q3, 0), Ty = both<H>(q3, 1), Tz = both<H>(q4, 0);
    const float2 bF = __fmul2_rn(B, __ffma2_rn(dx, Fx, __ffma2_rn(dy, Fy, __fmul2_rn(dz, Fz))));
    const float2 dT = __fmul2_rn(D, __ffma2_rn(dx, Tx, __ffma2_rn(dy, Ty, __fmul2_rn(dz, Tz))));
    const float2 ex = __fmul2_rn(G, dx), ey = __fmul2_rn(G, dy), ez = __fmul2_rn(G, dz);
    acc[0] = __ffma2_rn(A, Fx, __ffma2_rn(G, both<H>(q4, 1), __ffma2_rn(bF, dx, acc[0])));
    acc[1] = __ffma2_rn(A, Fy, __ffma2_rn(G, both<H>(q5, 0), __ffma2_rn(bF, dy, acc[1])));
    acc[2] = __ffma2_rn(A, Fz, __ffma2_rn(G, both<H>(q5, 1), __ffma2_rn(bF, dz, acc[2])));
    acc[3] = __ffma2_rn(dT, dx, __ffma2_rn(Fy, ez, __ffma2_rn(neg2(Fz), ey, acc[3])));
    acc[4] = __ffma2_rn(dT, dy, __ffma2_rn(Fz, ex, __ffma2_rn(neg2(Fx), ez, acc[4])));
    acc[5] = __ffma2_rn(dT, dz, __ffma2_rn(Fx, ey, __ffma2_rn(neg2(Fy), ex, acc[5])));
    acc[6] = __ffma2_rn(G, Tx, acc[6]);
    acc[7] = __ffma2_rn(G, Ty, acc[7]);
    acc[8] = __ffma2_rn(G, Tz, acc[8]);
}

__device__ __forceinline__ void combine_cross2(const float2 (&acc)[2][kCrossSums], const float2 *t,
                                               float2 *out) {
    float2 s[kCrossSums];
#pragma unroll
    for (int c = 0; c < kCrossSums; ++c) s[c] = __fadd2_rn(acc[0][c], acc[1][c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int p = (c + 1) % 3, q = (c + 2) % 3;
        out[c] = __ffma2_rn(s[6 + p], t[q], __ffma2_rn(neg2(s[6 + q]), t[p], s[c]));
        out[3 + c] = __ffma2_rn(f2(-0.5f, -0.5f), s[6 + c], s[3 + c]);
    }
}

// The (V, Omega) terms of a group for two targets, from the twelve sums of pair32_far2
// over the even and the odd sources: with P = sum G T and Q = sum G F,
//   V     = acc[0..2] + (2a^2/3) Q + P x t
//   Omega = 3/2 acc[3..5] - P/2 + Q x t.
__device__ __forceinline__ void combine_group2(const float2 (&acc)[2][kFarSums],
                                               const float2 *t, float k23, float2 *out) {
    float2 s[kFarSums];
#pragma unroll
    for (int c = 0; c < kFarSums; ++c) s[c] = __fadd2_rn(acc[0][c], acc[1][c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int p = (c + 1) % 3, q = (c + 2) % 3;
        out[c] = __ffma2_rn(f2(k23, k23), s[9 + c],
                            __ffma2_rn(s[6 + p], t[q], __ffma2_rn(neg2(s[6 + q]), t[p], s[c])));
        out[3 + c] = __ffma2_rn(
            f2(1.5f, 1.5f), s[3 + c],
            __ffma2_rn(f2(-0.5f, -0.5f), s[6 + c],
                       __ffma2_rn(s[9 + p], t[q], __fmul2_rn(neg2(s[9 + q]), t[p]))));
    }
}

// How a close group is evaluated again (pair32_near's MODE).
enum PairMode { kFarHiLo = 1, kExact = 2 };

// The pair terms of one target and the two sources of a record with the
// differences d = (t_hi - s_hi) + (t_lo - s_lo), which keep ~2 ulp of relative
// accuracy, and the cross products formed per pair.
//  kFarHiLo: far form; source jx (jx + 1 for lane y) equal to self_j is the
//    target itself: its term is zero (d = 0 and 1/r taken as 0) and it is left
//    out of the smallest r^2.
//  kExact: the exact coefficients of every pair (coef_exact; the self pair
//    takes the self values).
template <bool kFrames, int MODE>
__device__ __forceinline__ void pair32_near(const float *th, const float *tl, const float4 *q,
                                            const RpyConst32 &k, float2 *acc, float &rmin2,
                                            int self_j = -1, int jx = 0) {
    constexpr int kLo = Rec<kFrames>::kLo;
    const float4 q0 = q[0], ql = q[kLo + 1];
    const float2 z = reinterpret_cast<const float2 *>(q + 1)[0];
    const float2 lx = reinterpret_cast<const float2 *>(q + kLo)[1];
    const float2 dx = __fadd2_rn(__fadd2_rn(f2(th[0], th[0]), f2(q0.x, q0.y)),
                                 __fadd2_rn(f2(tl[0], tl[0]), lx));
    const float2 dy = __fadd2_rn(__fadd2_rn(f2(th[1], th[1]), f2(q0.z, q0.w)),
                                 __fadd2_rn(f2(tl[1], tl[1]), f2(ql.x, ql.y)));
    const float2 dz = __fadd2_rn(__fadd2_rn(f2(th[2], th[2]), z),
                                 __fadd2_rn(f2(tl[2], tl[2]), f2(ql.z, ql.w)));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    float2 A, B, C, D, G;
    if (MODE == kFarHiLo) {
        float2 rinv = f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
        const bool sx = (jx == self_j), sy = (jx + 1 == self_j);
        rinv.x = sx ? 0.f : rinv.x;
        rinv.y = sy ? 0.f : rinv.y;
        rmin2 = fminf(rmin2, fminf(sx ? k.close2 : r2.x, sy ? k.close2 : r2.y));
        far_coef(rinv, k, A, B, C, D, G);
    } else {
        coef_exact(r2.x, k, A.x, B.x, C.x, D.x, G.x);
        coef_exact(r2.y, k, A.y, B.y, C.y, D.y, G.y);
    }
    add_pair(q, dx, dy, dz, A, B, C, D, G, acc);
}

// Position of a target relative to the apply's first segment, y = th + tl, from
// its own group's record (target P of the padded layout).
template <bool kFrames>
__device__ __forceinline__ void load_target(const float4 *src, int64_t P, float *th, float *tl) {
    using R = Rec<kFrames>;
    const float4 *g = src + R::kGroupF4 * (P >> 5);
    const int lane = (int)(P & 31);
    const float *f =
        reinterpret_cast<const float *>(g + R::kHead + R::kPairF4 * (lane >> 1)) + (lane & 1);
    constexpr int kL = 2 * (2 * R::kLo + 1);      // first lo value
    if constexpr (kFrames) {
        const float4 c = g[0];
        const float cc[3] = {c.x, c.y, c.z};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            float e;
            two_sum(cc[x], -f[2 * x], th[x], e);
            tl[x] = __fadd_rn(e, -f[kL + 2 * x]);
        }
    } else {
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            th[x] = -f[2 * x];
            tl[x] = -f[kL + 2 * x];
        }
    }
}

// The target in the frame of the group with records q, as hi + lo parts.
__device__ __forceinline__ void to_frame_hl(const float4 *q, const float *th, const float *tl,
                                            float *uh, float *ul) {
    const float4 c = q[-1];
    const float cc[3] = {c.x, c.y, c.z};
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        float e;
        two_sum(th[x], -cc[x], uh[x], e);
        ul[x] = __fadd_rn(e, tl[x]);
    }
}

// One pair in FP64 (record layout: Y, F, T).
__device__ __forceinline__ void pair64(double tx, double ty, double tz, const double *s,
                                       const RpyConst64 &k, double *acc) {
    const double dx = tx - s[0], dy = ty - s[1], dz = tz - s[2];
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    double A, B, C, D, G;
    if (__builtin_expect(r2 < k.near2, 0)) {
        const double r = sqrt(r2);
        const double rinv = r > 0.0 ? 1.0 / r : 0.0;
        A = fma(-k.ov_A1, r, k.ov_A0);
        B = k.ov_B * rinv;
        C = fma(k.ov_C3 * r2, r, fma(-k.ov_C1, r, k.ov_C0));
        D = fma(k.ov_D0, rinv, -k.ov_D1 * r);
        G = fma(-k.ov_G1, r, k.ov_G0);
    } else {
        const double rinv = rsqrt(r2);
        const double rinv2 = rinv * rinv;
        const double rinv3 = rinv * rinv2;
        const double rinv5 = rinv3 * rinv2;
        A = fma(k.k23a2, rinv3, rinv);
        B = fma(-k.k2a2, rinv5, rinv3);
        C = -0.5 * rinv3;
        D = 1.5 * rinv5;
        G = rinv3;
    }
    const double Fx = s[3], Fy = s[4], Fz = s[5], Tx = s[6], Ty = s[7], Tz = s[8];
    const double bF = B * fma(dx, Fx, fma(dy, Fy, dz * Fz));
    const double dT = D * fma(dx, Tx, fma(dy, Ty, dz * Tz));
    const double ex = G * dx, ey = G * dy, ez = G * dz;
    acc[0] = fma(A, Fx, fma(bF, dx, fma(Ty, ez, fma(-Tz, ey, acc[0]))));
    acc[1] = fma(A, Fy, fma(bF, dy, fma(Tz, ex, fma(-Tx, ez, acc[1]))));
    acc[2] = fma(A, Fz, fma(bF, dz, fma(Tx, ey, fma(-Ty, ex, acc[2]))));
    acc[3] = fma(C, Tx, fma(dT, dx, fma(Fy, ez, fma(-Fz, ey, acc[3]))));
    acc[4] = fma(C, Ty, fma(dT, dy, fma(Fz, ex, fma(-Fx, ez, acc[4]))));
    acc[5] = fma(C, Tz, fma(dT, dz, fma(Fx, ey, fma(-Fy, ex, acc[5]))));
}

// One lane's share of the asynchronous copy of a group of sources from global to
// shared memory (16 bytes per cp.async, one commit group): a warp streams its own
// groups, and waits with cp.async.wait_group and __syncwarp alone.
template <bool kFrames>
__device__ __forceinline__ void stage_group(float4 *dst, const float4 *__restrict__ g, int lane) {
    constexpr int kF4 = Rec<kFrames>::kGroupF4;
#pragma unroll
    for (int i = 0; i < (kF4 + 31) / 32; ++i) {
        const int e = lane + 32 * i;
        if (e < kF4) {
            const unsigned sa = (unsigned)__cvta_generic_to_shared(dst + e);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(g + e)
                         : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Unit range of CTA b in the stream-K split of W units over G CTAs.
__device__ __forceinline__ int64_t unit_start(int64_t b, int64_t W, int64_t G) {
    return (b * W) / G;
}

// ---------------------------------------------------------------------------
// Completion of a tile: the stream-K partials of its targets are summed and
// scaled by 1/(8 pi eta) inside the pair kernel, by the CTA that finishes the
// tile's last work unit, so that no separate reduce launch follows the pair
// kernel and the sums of early tiles overlap the pair work of late ones.
// Every CTA that wrote a partial of the tile adds the units it covered to the
// tile's counter (one acquire-release atomic after a barrier, which orders
// the whole CTA's stores before it); the CTA whose addition completes
// the tile's unit count reads the partials of all the tile's CTAs (from L2),
// adds them in CTA order -- the same order whichever CTA came last, so results
// do not depend on timing -- writes the targets' rows of VW and sets the
// counter back to zero for the next launch.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cta_range_of_tile(const SysMap &sm, int64_t tile, int64_t W,
                                                  int64_t G, int64_t &u0, int64_t &u1,
                                                  int64_t &b0, int64_t &b1) {
    // CTA b owns units [floor(bW/G), floor((b+1)W/G)); the CTA that holds unit
    // u is ceil((u+1)G/W) - 1.
    u0 = tile_unit_begin(sm, tile);
    u1 = tile_unit_begin(sm, tile + 1) - 1;
    b0 = ((u0 + 1) * G + W - 1) / W - 1;
    b1 = ((u1 + 1) * G + W - 1) / W - 1;
}

// fetch-and-add with acquire-release semantics at GPU scope: its release
// covers the writes the CTA's threads made before the preceding barrier, its
// acquire the reads they make after the following one
__device__ __forceinline__ int fetch_add_acq_rel(int *p, int v) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;"
                 : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

template <typename PT, int NPART, int TPT>
__device__ __forceinline__ void finish_tile(const PT *part, const SysMap &smap, int64_t tile,
                                            int64_t ptile, int64_t units, int64_t n_units,
                                            int64_t W, int64_t G, int *__restrict__ cnt,
                                            double scale, double *__restrict__ VW,
                                            bool worker = true) {
    constexpr int kTile = kRpyThreads * TPT;
    __shared__ int s_last;
    const int tid = threadIdx.x;
    __syncthreads();   // the CTA's partial is written before it is counted
    if (tid == 0)
        s_last = fetch_add_acq_rel(cnt + tile, (int)units) + (int)units == (int)n_units;
    __syncthreads();
    // (`worker`: false for the second half of a source-split CTA, which holds no targets)
    if (!s_last || !worker) return;
    int64_t u0, u1, b0, b1;
    cta_range_of_tile(smap, tile, W, G, u0, u1, b0, b1);
    // With G > W (a fixed grid over a short active list) a CTA owns at most one
    // unit and some own none: the tile's CTAs are then the owners of its units.
    const bool by_unit = G > W;
    const int64_t n_parts = by_unit ? u1 - u0 + 1 : b1 - b0 + 1;
    // FP32 partials (hi, lo) are added in float-float arithmetic (TwoSum of the
    // hi parts, the lo parts added to its error, renormalised by a second
    // TwoSum: ~2^-44 relative, far below the 2^-24 of the pair terms) and
    // converted to FP64 once per target: the whole tile's sum runs on one SM,
    // and on GB300 the FP64 pipe has 1/64 of the FP32 rate.
    // FP64 partials are added in FP64.
    using Acc = typename std::conditional<NPART == 2, float, double>::type;
    Acc ah[TPT][6], al[TPT][6];
#pragma unroll
    for (int t = 0; t < TPT; ++t)
#pragma unroll
        for (int c = 0; c < 6; ++c) ah[t][c] = al[t][c] = (Acc)0;
#pragma unroll 4
    for (int64_t i = 0; i < n_parts; ++i) {
        const int64_t cb = by_unit ? ((u0 + i + 1) * G + W - 1) / W - 1 : b0 + i;
        const PT *p = part + (size_t)(cb + tile) * (6 * NPART) * kTile;
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            const int local = t * kRpyThreads + tid;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                if constexpr (NPART == 2) {
                    const float h = __ldcg(p + c * kTile + local);
                    const float l = __ldcg(p + (6 + c) * kTile + local);
                    float sh, e;
                    two_sum(ah[t][c], h, sh, e);
                    e = __fadd_rn(e, __fadd_rn(al[t][c], l));
                    two_sum(sh, e, ah[t][c], al[t][c]);
                } else {
                    ah[t][c] += (double)__ldcg(p + c * kTile + local);
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < TPT; ++t) {
        const int64_t n = segment_at(smap, ptile * kTile + t * kRpyThreads + tid, smap.n_src);
        if (n >= 0) {
#pragma unroll
            for (int c = 0; c < 6; ++c)
                VW[6 * n + c] = ((double)ah[t][c] + (double)al[t][c]) * scale;
        }
    }
    if (tid == 0) cnt[tile] = 0;
}

// ---------------------------------------------------------------------------
// Mixed-precision pair kernel. A CTA owns a tile of kRpyThreads * TPT targets,
// TPT per thread; their pair terms are summed in registers over groups of
// kRpyComp sources with the branch-free far form (pair32_far) and the group
// sums folded (TwoSum) into (hi, lo) accumulators.
//  * A group in which the warp met a pair closer than R_c = 4a is evaluated
//    again with hi/lo differences. TPT = 2, 256-target tiles (large systems):
//    with the exact coefficients at once. TPT = 1, 128-target tiles (a warp's
//    own segments sit in one of every few dozen groups): the group holding the
//    warp's own segments is recognised by index and evaluated once with hi/lo
//    differences and the self pair masked, other close groups again with hi/lo
//    differences in the far form, and exactly only when distinct segments
//    overlap.
// SPLIT = 2 (128-target tiles only) gives a CTA twice the warps on the same
// targets: the two sets of four warps take alternate 32-source groups
// and their sums are added (float-float, in set order) before the
// partial is written.
// Each warp streams its groups through two buffers of its own and meets the others
// only at the tile's end, so that one that evaluates a close group again (its own
// filaments': every few groups in a system of some hundred segments, where they
// took a quarter of the apply) delays nobody. Measured, 256 systems of about 1000
// segments, with chunks of four groups shared by the CTA between barriers: 965 us an
// apply; close groups' loop unrolled by 4 942; streams of their own 930; an empty
// second slot left out 910, all with the same bits. By 8 the loop spills: 1037.
// These kernels run ensembles, and one system in another schedule than the automatic
// one, which runs rpy_pair32_warp_kernel below. (One system in the groups' frames here
// too was 5-8% faster at 32 000 segments in most of these schedules, 1541 and 1738 us
// with 256-target tiles at 3 CTAs per SM, and slower with few warps: 3026 and 2538 with
// 128-target tiles at one; the automatic schedule is faster than any, 1435.)
// ---------------------------------------------------------------------------
constexpr int min_blocks(int tpt, int split) {
    return split == 2 ? kRpyMinBlocksSplit2 : tpt == 2 ? kRpyMinBlocksTpt2 : kRpyMinBlocksTpt1;
}

template <int TPT, int SPLIT = 1>
__global__ void __launch_bounds__(kRpyThreads * SPLIT, min_blocks(TPT, SPLIT))
rpy_pair32_kernel(const float4 *__restrict__ src, SysMap smap, int64_t W, int G, RpyConst32 k,
                  float *__restrict__ part, int *__restrict__ cnt, double scale,
                  double *__restrict__ VW) {
    constexpr int kGroupF4 = Rec<false>::kGroupF4, kPairF4 = Rec<false>::kPairF4;
    constexpr int kUnitGroups = unit_sources(false) / kRpyComp;   // groups per work unit
    constexpr int kWarps = kRpyThreads * SPLIT / 32;
    constexpr int kT = TPT;                               // targets per thread
    constexpr int kTile = kRpyThreads * TPT;              // targets per tile
    static_assert(SPLIT == 1 || (SPLIT == 2 && TPT == 1), "source split: 128-target tiles only");
    __shared__ float4 sm[kWarps][2][kGroupF4];            // two groups of each warp
    // target slot, and which of the SPLIT sets of source groups the thread takes
    const int tid = SPLIT == 1 ? (int)threadIdx.x : (int)(threadIdx.x % kRpyThreads);
    const int set = SPLIT == 1 ? 0 : (int)(threadIdx.x / kRpyThreads);
    const int lane = tid & 31;
    float4(*buf)[kGroupF4] = sm[threadIdx.x >> 5];
    pdl_enter();
    const int64_t b = blockIdx.x;
    resolve_dyn(smap, W);
    int64_t u = unit_start(b, W, G);
    const int64_t u_end = unit_start(b + 1, W, G);

    while (u < u_end) {
        int64_t tile, ubeg, n_units, src0;
        locate_unit(smap, u, tile, ubeg, n_units, src0);
        const int64_t u_last = min(ubeg + n_units, u_end);      // this CTA's units of the tile
        const float4 *srcs = src + kGroupF4 * (src0 / kRpyComp);   // this tile's system
        const int64_t ptile = smap.tile_id ? smap.tile_id[tile] : tile;   // padded tile
        const int64_t nsrc = smap.tile_nsrc ? smap.tile_nsrc[tile] : smap.n_src;
        // their groups (the padding-only groups of a system's last unit are left out)
        const int64_t c_begin = (u - ubeg) * kUnitGroups;
        const int64_t c_end = min((u_last - ubeg) * kUnitGroups, (nsrc + kRpyComp - 1) / kRpyComp);

        // first target of this warp (slot 0)
        const int64_t wbase = ptile * kTile + (tid & ~31);
        // a warp whose targets are all padding (in a system's last tile) computes
        // nothing; the tile's sum never reads those rows
        // and one whose second slot is all padding leaves that out
        const bool both = kT == 1 || wbase + kRpyThreads - src0 < nsrc;
        const int64_t g_end = wbase - src0 < nsrc ? c_end : c_begin;
        int64_t grp = c_begin + set;
        if (grp < g_end) stage_group<false>(buf[0], srcs + kGroupF4 * grp, lane);
        float th[kT][3], tl[kT][3];
#pragma unroll
        for (int t = 0; t < kT; ++t)
            load_target<false>(src, ptile * kTile + t * kRpyThreads + tid, th[t], tl[t]);
        float hi[kT][6], lo[kT][6];
#pragma unroll
        for (int t = 0; t < kT; ++t)
#pragma unroll
            for (int c = 0; c < 6; ++c) hi[t][c] = lo[t][c] = 0.f;

#pragma unroll 1
        for (int cur = 0; grp < g_end; grp += SPLIT, cur ^= 1) {
            if (grp + SPLIT < g_end) {
                stage_group<false>(buf[cur ^ 1], srcs + kGroupF4 * (grp + SPLIT), lane);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                cp_async_wait_all();
            }
            __syncwarp();
            const float4 *qg = buf[cur];
            float out[kT][6];
            // the group that holds this warp's own segments
            const bool own =
                TPT == 1 && src0 + grp * kRpyComp == wbase;
            bool near = own;
            if (!own) {
                float2 t2[kT][3], acc[kT][6];
#pragma unroll
                for (int t = 0; t < kT; ++t) {
#pragma unroll
                    for (int x = 0; x < 3; ++x) t2[t][x] = f2(th[t][x], th[t][x]);
#pragma unroll
                    for (int c = 0; c < 6; ++c) acc[t][c] = f2(0.f, 0.f);
                }
                float rmin2 = k.close2;
                if (both) {
#pragma unroll (kRpyUnroll / 2)
                    for (int jp = 0; jp < kRpyComp / 2; ++jp) {
#pragma unroll
                        for (int t = 0; t < kT; ++t)
                            pair32_far(t2[t], qg + kPairF4 * jp, k, acc[t], rmin2);
                    }
                } else {
#pragma unroll (kRpyUnroll / 2)
                    for (int jp = 0; jp < kRpyComp / 2; ++jp)
                        pair32_far(t2[0], qg + kPairF4 * jp, k, acc[0], rmin2);
                }
                // (where slot 1 is left out: in a group with padding sources its padding
                // targets would have met them at r = 0)
                near = __any_sync(0xffffffffu, rmin2 < k.close2) ||
                       (!both && (grp + 1) * kRpyComp > nsrc);
#pragma unroll
                for (int t = 0; t < kT; ++t)
#pragma unroll
                    for (int c = 0; c < 6; ++c) out[t][c] = __fadd_rn(acc[t][c].x, acc[t][c].y);
            }
            if (near) {
                // (one target at a time: fewer live registers)
#pragma unroll
                for (int t = 0; t < kT; ++t) {
                    if (t == 1 && !both) continue;
                    float2 acc[6];
                    float rmin2 = k.close2;
                    bool exact = TPT == 2;
                    if constexpr (TPT == 1) {
                        const int self_j = own ? lane : -1;
#pragma unroll
                        for (int c = 0; c < 6; ++c) acc[c] = f2(0.f, 0.f);
#pragma unroll 1
                        for (int jp = 0; jp < kRpyComp / 2; ++jp)
                            pair32_near<false, kFarHiLo>(th[t], tl[t], qg + kPairF4 * jp, k, acc,
                                                           rmin2, self_j, 2 * jp);
                        // overlapping distinct segments (r < 2a): the exact coefficients
                        exact = __any_sync(0xffffffffu, rmin2 < k.near2);
                    }
                    if (exact) {
#pragma unroll
                        for (int c = 0; c < 6; ++c) acc[c] = f2(0.f, 0.f);
#pragma unroll 4
                        for (int jp = 0; jp < kRpyComp / 2; ++jp)
                            pair32_near<false, kExact>(th[t], tl[t], qg + kPairF4 * jp, k, acc, rmin2);
                    }
#pragma unroll
                    for (int c = 0; c < 6; ++c) out[t][c] = __fadd_rn(acc[c].x, acc[c].y);
                    if (own && !exact) {
                        // the self term, left out of the far-form pass above:
                        // 4/(3a) F_n and T_n / a^3
                        const float *f = reinterpret_cast<const float *>(
                                             qg + kPairF4 * (lane >> 1)) + (lane & 1);
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            out[t][c] = fmaf(k.ov_A0, f[2 * (3 + c)], out[t][c]);
                            out[t][3 + c] = fmaf(k.ov_C0, f[2 * (6 + c)], out[t][3 + c]);
                        }
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < kT; ++t)
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    float sh, e;
                    two_sum(hi[t][c], out[t][c], sh, e);
                    hi[t][c] = sh;
                    lo[t][c] = __fadd_rn(lo[t][c], e);
                }
            __syncwarp();     // every lane is done with this buffer before it is refilled
        }

        if constexpr (SPLIT > 1) {
            // the other sets' sums join the first's in set order (TwoSum of the hi
            // parts, the lo parts into its error, renormalised), through the group
            // buffers, which are next written after the barrier in finish_tile
            float *xs = reinterpret_cast<float *>(&sm[0][0][0]);
            static_assert((SPLIT - 1) * 12 * kRpyThreads * sizeof(float) <= sizeof(sm),
                          "the sets' sums fit in the group buffers");
            __syncthreads();          // every warp is done with its groups
            if (set > 0) {
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    xs[((set - 1) * 12 + c) * kRpyThreads + tid] = hi[0][c];
                    xs[((set - 1) * 12 + 6 + c) * kRpyThreads + tid] = lo[0][c];
                }
            }
            __syncthreads();
            if (set == 0) {
#pragma unroll
                for (int o = 0; o < SPLIT - 1; ++o)
#pragma unroll
                    for (int c = 0; c < 6; ++c) {
                        float sh, e;
                        two_sum(hi[0][c], xs[(o * 12 + c) * kRpyThreads + tid], sh, e);
                        e = __fadd_rn(e, __fadd_rn(lo[0][c],
                                                   xs[(o * 12 + 6 + c) * kRpyThreads + tid]));
                        two_sum(sh, e, hi[0][c], lo[0][c]);
                    }
            }
        }
        // partial of this CTA for this tile -> slot (b + tile)
        if (set == 0) {
            float *p = part + (size_t)(b + tile) * 12 * kTile;
#pragma unroll
            for (int t = 0; t < kT; ++t) {
                const int local = t * kRpyThreads + tid;
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    p[c * kTile + local] = hi[t][c];
                    p[(6 + c) * kTile + local] = lo[t][c];
                }
            }
        }
        finish_tile<float, 2, TPT>(part, smap, tile, ptile, u_last - u, n_units, W, G, cnt, scale,
                                   VW, set == 0);
        u = u_last;
    }
}

// ---------------------------------------------------------------------------
// The pair kernel of the automatic schedule: warps that share nothing. A tile
// is 64 targets, two per lane of one warp; a work unit is (tile, group of 32
// sources), and the units are split evenly over all warps of the grid (one
// CTA of 12 warps per SM). Each warp streams its groups through two
// private shared-memory buffers (cp.async) and never waits for another warp,
// so that a warp that has to evaluate a close group again delays nobody, and
// the split is even to one unit of 64 x 32 pairs. A tile that a single warp
// covers is written from registers; the others leave one partial per warp in
// slot (warp + tile), and when a CTA's warps are done it counts its units of
// each such tile; the CTA that completes a tile sums its partials in warp
// order (float-float) and writes the rows.
// Measured, whole applies, against 256-target tiles of four warps with a barrier
// per 128 sources: 9 651 segments in ragged filaments 224 -> 181 us, 3200
// segments 73 -> 50 us, 32 000 1504 -> 1491 us (at the close groups' loop
// unrolled by 2; by 4 its registers cost the far loop 7%). One system only. With the
// two targets of a lane packed (pair32_far2) and the spread order 9 651 took 160 us,
// 3200 44 and 32 000 1426, of which 36 us are the compensated fold and 10 the close
// groups; with Omega's cross products per pair inside wide groups 173, 45 and 1435.
// ---------------------------------------------------------------------------
constexpr int kWarpTile = kRpyMinTile;          // targets per tile
constexpr int kWarpPart = 12 * kWarpTile;       // floats of a partial
constexpr int kWarpCta = 12;                    // warps per CTA (168 registers a thread)
constexpr int kGroupF4 = Rec<true>::kGroupF4, kPairF4 = Rec<true>::kPairF4;
constexpr size_t kWarpSmem = sizeof(float4) * 2 * kGroupF4 * kWarpCta;

// Warps that W units are split over, on n_ctas CTAs: as many as leave no warp
// with more units than another by more than the last one's remainder (with
// every warp of the grid at work some would have ceil(W / warps) units and the
// rest one less, and the same end). Never more than W, so every one of them
// owns a unit.
__host__ __device__ __forceinline__ int64_t warp_count(int64_t W, int64_t n_ctas) {
    const int64_t most = n_ctas * kWarpCta;
    const int64_t m = (W + most - 1) / most;
    return (W + m - 1) / m;
}

// The tiles that the CTA's units (those of warps [w0, w1)) lie in, once its
// warps are done. Not inlined: its registers would be taken from the main loop.
__device__ __noinline__ void finish_warp_tiles(const SysMap &smap, int64_t W, int64_t G,
                                               int64_t w0, int64_t w1, const float *part,
                                               int *cnt, double scale, double *VW) {
    constexpr int kThreads = 32 * kWarpCta;
    __shared__ int s_done[kThreads];
    if (w0 >= w1) return;                       // the whole CTA leaves
    const int64_t c_beg = unit_start(w0, W, G), c_end = unit_start(w1, W, G);
    const int64_t t_first = c_beg / smap.n_units, t_last = (c_end - 1) / smap.n_units;
    for (int64_t tb = t_first; tb <= t_last; tb += kThreads) {
        __syncthreads();      // the CTA's partials are written (and s_done is free)
        {
            const int64_t t = tb + threadIdx.x;
            int done = 0;
            if (t <= t_last) {
                const int64_t b0 = tile_unit_begin(smap, t), b1 = tile_unit_begin(smap, t + 1);
                const int64_t o0 = ((b0 + 1) * G + W - 1) / W - 1, o1 = (b1 * G + W - 1) / W - 1;
                if (o0 != o1) {
                    const int units = (int)(min(b1, c_end) - max(b0, c_beg));
                    done = fetch_add_acq_rel(cnt + t, units) + units == (int)(b1 - b0);
                }
            }
            s_done[threadIdx.x] = done;
        }
        __syncthreads();
        const int nt = (int)min((int64_t)kThreads, t_last - tb + 1);
        for (int i = 0; i < nt; ++i) {
            if (!s_done[i]) continue;
            const int64_t t = tb + i;
            const int64_t b0 = tile_unit_begin(smap, t), b1 = tile_unit_begin(smap, t + 1);
            const int64_t o0 = ((b0 + 1) * G + W - 1) / W - 1, o1 = (b1 * G + W - 1) / W - 1;
            const int n_parts = (int)(o1 - o0 + 1);
            static_assert(kThreads == 6 * kWarpTile, "a thread per (component, target)");
            const int c = threadIdx.x / kWarpTile, l = threadIdx.x % kWarpTile;
            const float *p0 = part + (size_t)(o0 + t) * kWarpPart + c * kWarpTile + l;
            float ah = 0.f, al = 0.f;
            // a batch of loads in flight before its sums (one part at a time, each sum
            // waiting for its load, took 450 cycles a part: 17 us for the 37 parts of
            // a tile at 3200 segments, half of the kernel)
            constexpr int kBatch = 24;
            for (int j0 = 0; j0 < n_parts; j0 += kBatch) {
                float h[kBatch], lw[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    // (parts past the last read it again and add zero)
                    const float *p = p0 + min(j0 + j, n_parts - 1) * kWarpPart;
                    h[j] = __ldcg(p);
                    lw[j] = __ldcg(p + 6 * kWarpTile);
                }
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    const bool in = j0 + j < n_parts;
                    float sh, e;
                    two_sum(ah, in ? h[j] : 0.f, sh, e);
                    e = __fadd_rn(e, __fadd_rn(al, in ? lw[j] : 0.f));
                    two_sum(sh, e, ah, al);
                }
            }
            const int64_t n = segment_at(smap, t * kWarpTile + l, smap.n_src);
            if (n >= 0) VW[6 * n + c] = ((double)ah + (double)al) * scale;
            if (threadIdx.x == 0) cnt[t] = 0;
        }
    }
}

template <bool kSpread>
__global__ void __launch_bounds__(32 * kWarpCta, 1)
rpy_pair32_warp_kernel(const float4 *__restrict__ src, SysMap smap, int64_t W, int n_ctas,
                       RpyConst32 k, float *__restrict__ part, int *__restrict__ cnt,
                       double scale, double *__restrict__ VW) {
    extern __shared__ float4 wsm[];             // [kWarpCta][2][kGroupF4]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t G = warp_count(W, n_ctas);
    const int64_t w0 = unit_start(blockIdx.x, G, n_ctas);        // this CTA's warps
    const int64_t w1 = unit_start((int64_t)blockIdx.x + 1, G, n_ctas);
    const int64_t w = w0 + wid;
    int64_t u = 0, u_end = 0;
    if (w < w1) {
        u = unit_start(w, W, G);
        u_end = unit_start(w + 1, W, G);
    }
    float4 *buf = wsm + 2 * kGroupF4 * wid;
    const int64_t n_units = smap.n_units;
    int64_t tile = 0, ubeg = 0;
    if (u < u_end) {
        tile = u / n_units;
        ubeg = tile * n_units;
    }
    pdl_enter();
    if (u < u_end) {
        stage_group<true>(buf, src + kGroupF4 * (u - ubeg), lane);
    }
    int cur = 0;
    while (u < u_end) {
        const int64_t base = tile * kWarpTile;              // the tile's first target
        const int64_t s_end = min(u_end, ubeg + n_units);  // this warp's units of the tile
        const bool whole = u == ubeg && s_end == ubeg + n_units;
        float th[2][3], tl[2][3];
        float2 hi[6], lo[6];                               // lane x: slot 0, lane y: slot 1
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            int64_t P = base + 32 * t;
            if constexpr (kSpread) P = 32 * (int64_t)spread_place((int)(P >> 5), (int)n_units);
            load_target<true>(src, P + lane, th[t], tl[t]);
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) hi[c] = lo[c] = f2(0.f, 0.f);
#pragma unroll 1
        for (; u < s_end; ++u, cur ^= 1) {
            if (u + 1 < u_end) {
                // the next group, or the first one for the next tile
                const int64_t gn = u + 1 < s_end ? u + 1 - ubeg : 0;
                stage_group<true>(buf + kGroupF4 * (cur ^ 1), src + kGroupF4 * gn, lane);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                cp_async_wait_all();
            }
            __syncwarp();
            const float4 *qg = buf + kGroupF4 * cur + Rec<true>::kHead;
            float2 out[6], rmin2 = f2(k.close2, k.close2);
            {
                const float4 ce = qg[-1];
                const float cc[3] = {ce.x, ce.y, ce.z};
                float2 t2[3];
#pragma unroll
                for (int x = 0; x < 3; ++x)
                    t2[x] = f2(__fadd_rn(__fsub_rn(th[0][x], cc[x]), tl[0][x]),
                               __fadd_rn(__fsub_rn(th[1][x], cc[x]), tl[1][x]));
                const float2 tt =
                    __ffma2_rn(t2[0], t2[0], __ffma2_rn(t2[1], t2[1], __fmul2_rn(t2[2], t2[2])));
                if (!__any_sync(0xffffffffu, fminf(tt.x, tt.y) < ce.w)) {
                    float2 acc[2][kFarSums];
#pragma unroll
                    for (int c = 0; c < kFarSums; ++c) acc[0][c] = acc[1][c] = f2(0.f, 0.f);
#pragma unroll
                    for (int jp = 0; jp < kRpyComp / 2; ++jp) {
                        pair32_far2<0>(t2, qg + kPairF4 * jp, k, acc[0], rmin2);
                        pair32_far2<1>(t2, qg + kPairF4 * jp, k, acc[1], rmin2);
                    }
                    combine_group2(acc, t2, k.k23a2, out);
                } else {
                    float2 acc[2][kCrossSums];
#pragma unroll
                    for (int c = 0; c < kCrossSums; ++c) acc[0][c] = acc[1][c] = f2(0.f, 0.f);
#pragma unroll 2
                    for (int jp = 0; jp < kRpyComp / 2; ++jp) {
                        pair32_cross2<0>(t2, qg + kPairF4 * jp, k, acc[0], rmin2);
                        pair32_cross2<1>(t2, qg + kPairF4 * jp, k, acc[1], rmin2);
                    }
                    combine_cross2(acc, t2, out);
                }
            }
            // slots in which a pair came closer than R_c, one at a time through one copy of
            // the code: with hi/lo differences in the far form, or with the exact
            // coefficients where a pair overlaps (the group that holds the slot's own
            // segments counts as one: it has the self pairs)
            unsigned close = 0;
            if (__any_sync(0xffffffffu, rmin2.x < k.close2)) close |= 1u;
            if (__any_sync(0xffffffffu, rmin2.y < k.close2)) close |= 2u;
            while (close) {
                const bool t1 = close == 2u;
                close &= 2u * (close == 3u);
                const bool exact = __any_sync(0xffffffffu, (t1 ? rmin2.y : rmin2.x) < k.over2);
                float ph[3], pl[3], uh[3], ul[3];
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    ph[x] = t1 ? th[1][x] : th[0][x];
                    pl[x] = t1 ? tl[1][x] : tl[0][x];
                }
                to_frame_hl(qg, ph, pl, uh, ul);
                float2 acc[6];
                float rm = 0.f;
#pragma unroll
                for (int c = 0; c < 6; ++c) acc[c] = f2(0.f, 0.f);
                if (exact) {
#pragma unroll 2
                    for (int jp = 0; jp < kRpyComp / 2; ++jp)
                        pair32_near<true, kExact>(uh, ul, qg + kPairF4 * jp, k, acc, rm);
                } else {
#pragma unroll 2
                    for (int jp = 0; jp < kRpyComp / 2; ++jp)
                        pair32_near<true, kFarHiLo>(uh, ul, qg + kPairF4 * jp, k, acc, rm);
                }
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    const float v = __fadd_rn(acc[c].x, acc[c].y);
                    if (t1) out[c].y = v;
                    else out[c].x = v;
                }
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                float2 sh, e;
                two_sum(hi[c].x, out[c].x, sh.x, e.x);
                two_sum(hi[c].y, out[c].y, sh.y, e.y);
                hi[c] = sh;
                lo[c] = __fadd2_rn(lo[c], e);
            }
            __syncwarp();     // every lane is done with this buffer before it is refilled
        }
        if (whole) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int64_t n = segment_at(smap, base + 32 * t + lane, smap.n_src);
                if (n >= 0) {
#pragma unroll
                    for (int c = 0; c < 6; ++c)
                        VW[6 * n + c] = (t ? (double)hi[c].y + (double)lo[c].y
                                           : (double)hi[c].x + (double)lo[c].x) * scale;
                }
            }
        } else {
            float *p = part + (size_t)(w + tile) * kWarpPart;
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    p[c * kWarpTile + 32 * t + lane] = t ? hi[c].y : hi[c].x;
                    p[(6 + c) * kWarpTile + 32 * t + lane] = t ? lo[c].y : lo[c].x;
                }
        }
        tile += 1;
        ubeg += n_units;
    }

    finish_warp_tiles(smap, W, G, w0, w1, part, cnt, scale, VW);
}

// ---------------------------------------------------------------------------
// FP64 pair kernel (same stream-K scaffolding).
// ---------------------------------------------------------------------------
template <int TPT>
__global__ void __launch_bounds__(kRpyThreads)
rpy_pair64_kernel(const double *__restrict__ src, SysMap smap, int64_t W, int G, RpyConst64 k,
                  double *__restrict__ part, int *__restrict__ cnt, double scale,
                  double *__restrict__ VW) {
    constexpr int kRec = 9 * kRpyChunk;
    constexpr int kTile = kRpyThreads * TPT;
    __shared__ double sm[2][kRec];
    const int tid = threadIdx.x;
    pdl_enter();
    const int64_t b = blockIdx.x;
    resolve_dyn(smap, W);
    int64_t u = unit_start(b, W, G);
    const int64_t u_end = unit_start(b + 1, W, G);

    while (u < u_end) {
        int64_t tile, ubeg, n_units, src0;
        locate_unit(smap, u, tile, ubeg, n_units, src0);
        const int64_t c_begin = u - ubeg;
        const int64_t c_end = min(n_units, c_begin + (u_end - u));
        const double *srcs = src + 9 * src0;
        const int64_t ptile = smap.tile_id ? smap.tile_id[tile] : tile;
        // real sources of the tile's system (its padding follows them): padded
        // sources carry no load and padded targets are never read, so both are
        // left out (a small system would otherwise cost a whole padded tile x
        // chunk at the FP64 rate)
        const int64_t nsrc = smap.tile_nsrc ? smap.tile_nsrc[tile] : smap.n_src;
        // A tile whose real targets fit in one warp (a system of <= 32 segments)
        // would leave three of the four warps idle, and one warp issues FP64
        // only through its own sub-partition's share of the SM's small FP64
        // rate: then every warp takes the first warp's targets and every fourth
        // source, and the four sums are added in warp order before the partial.
        const bool narrow = nsrc - (ptile * kTile - src0) <= 32;
        const int wid = tid >> 5;

        double ty[TPT][3];
        bool live[TPT];
        bool any = false;
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            const int64_t n = ptile * kTile + t * kRpyThreads + (narrow ? (tid & 31) : tid);
            ty[t][0] = src[9 * n];
            ty[t][1] = src[9 * n + 1];
            ty[t][2] = src[9 * n + 2];
            live[t] = (!narrow || t == 0) && n - src0 < nsrc;
            any = any || live[t];
        }
        double acc[TPT][6];
#pragma unroll
        for (int t = 0; t < TPT; ++t)
#pragma unroll
            for (int c = 0; c < 6; ++c) acc[t][c] = 0.0;

        {
            const double *g = srcs + 9 * (c_begin * kRpyChunk);
            for (int i = tid; i < kRec; i += kRpyThreads) sm[0][i] = g[i];
        }
        __syncthreads();
        for (int64_t ch = c_begin; ch < c_end; ++ch) {
            const int buf = (int)((ch - c_begin) & 1);
            double pre[(kRec + kRpyThreads - 1) / kRpyThreads];
            const bool has_next = (ch + 1 < c_end);
            if (has_next) {
                const double *g = srcs + 9 * ((ch + 1) * kRpyChunk);
#pragma unroll
                for (int r = 0; r < (kRec + kRpyThreads - 1) / kRpyThreads; ++r) {
                    const int i = tid + r * kRpyThreads;
                    pre[r] = (i < kRec) ? g[i] : 0.0;
                }
            }
            const double *s = sm[buf];
            const int jmax = any ? (int)min((int64_t)kRpyChunk, nsrc - ch * kRpyChunk) : 0;
            const int jstep = narrow ? kRpyThreads / 32 : 1;
#pragma unroll 2
            for (int j = narrow ? wid : 0; j < jmax; j += jstep) {
#pragma unroll
                for (int t = 0; t < TPT; ++t)
                    if (live[t]) pair64(ty[t][0], ty[t][1], ty[t][2], s + 9 * j, k, acc[t]);
            }
            if (has_next) {
#pragma unroll
                for (int r = 0; r < (kRec + kRpyThreads - 1) / kRpyThreads; ++r) {
                    const int i = tid + r * kRpyThreads;
                    if (i < kRec) sm[buf ^ 1][i] = pre[r];
                }
            }
            __syncthreads();
        }
        if (narrow) {
            // the other warps' sums join the first warp's; their own slots (and
            // the second slot of every thread) are padding and stay zero. The
            // buffer is next written after the next segment's first barrier.
            __shared__ double red64[kRpyThreads / 32 - 1][6][32];
            if (wid > 0) {
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    red64[wid - 1][c][tid & 31] = acc[0][c];
                    acc[0][c] = 0.0;
                }
            }
            __syncthreads();
            if (wid == 0) {
                for (int w = 0; w < kRpyThreads / 32 - 1; ++w)
#pragma unroll
                    for (int c = 0; c < 6; ++c) acc[0][c] += red64[w][c][tid];
            }
        }
        double *p = part + (size_t)(b + tile) * 6 * kTile;
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            const int local = t * kRpyThreads + tid;
#pragma unroll
            for (int c = 0; c < 6; ++c) p[c * kTile + local] = acc[t][c];
        }
        finish_tile<double, 1, TPT>(part, smap, tile, ptile, c_end - c_begin, n_units, W, G, cnt,
                                    scale, VW);
        u = ubeg + c_end;
    }
}

// ---------------------------------------------------------------------------
// FP64 applies of one system without packed records: two kernels that read the
// caller's arrays. The FP64 unit is the bound (2 lanes per clock and SM: a warp
// instruction takes 64 cycles of its sub-partition, whatever its lanes do), so
// shuffles, shared memory and integer work cost nothing beside it, and what
// counts is the FP64 instructions per pair and how evenly they are spread.
// ---------------------------------------------------------------------------

// Coefficients of a pair at r^2. The comparisons are on the bits (r^2 >= 0), so
// they take no FP64 instruction; the overlapping form runs only in warps that
// hold such a pair, from the same 1/r.
__device__ __forceinline__ void coef64(double r2, const RpyConst64 &k, double &A, double &B,
                                       double &C, double &D, double &G) {
    const long long bits = __double_as_longlong(r2);
    // 1/r taken as 0 where r = 0 and where r^2 overflows
    const bool none = bits < __double_as_longlong(1e-290) || bits >= 0x7ff0000000000000ll;
    const double rinv = none ? 0.0 : rsqrt_iter(r2);
    const double rinv2 = rinv * rinv;
    G = rinv * rinv2;
    const double rinv5 = G * rinv2;
    A = fma(k.k23a2, G, rinv);
    B = fma(-k.k2a2, rinv5, G);
    C = -0.5 * G;
    D = 1.5 * rinv5;
    if (bits < __double_as_longlong(k.near2)) {
        const double r = r2 * rinv;
        A = fma(-k.ov_A1, r, k.ov_A0);
        B = k.ov_B * rinv;
        C = fma(k.ov_C3 * r2, r, fma(-k.ov_C1, r, k.ov_C0));
        D = fma(k.ov_D0, rinv, -k.ov_D1 * r);
        G = fma(-k.ov_G1, r, k.ov_G0);
    }
}

// acc += the (V, Omega) terms of loads (F, T) = f at difference d, with e = sg G d
// (sg = -1 for the source of the pair: its difference is -d).
__device__ __forceinline__ void add64(const double *f, const double *d, const double *e, double A,
                                      double B, double C, double D, double *acc) {
    const double bF = B * fma(d[0], f[0], fma(d[1], f[1], d[2] * f[2]));
    const double dT = D * fma(d[0], f[3], fma(d[1], f[4], d[2] * f[5]));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int p = (c + 1) % 3, q = (c + 2) % 3;
        acc[c] = fma(A, f[c], fma(bF, d[c], fma(f[3 + p], e[q], fma(-f[3 + q], e[p], acc[c]))));
        acc[3 + c] = fma(C, f[3 + c], fma(dT, d[c], fma(f[p], e[q], fma(-f[q], e[p], acc[3 + c]))));
    }
}

// Small systems: a warp per target, its lanes over the sources, one warp per
// CTA, so that the few hundred pairs of a single filament spread over the SMs.
// The lane sums are combined by halving: at each step a lane keeps some of its
// components and gives the others away, 8 FP64 adds instead of 30.
// Measured (apply on the device, packed kernel -> this): 20 segments 25 -> 9 us,
// 256 segments 523 -> 22 us, 1024 segments 525 -> 109 us (the packed kernel gives a
// small system's few 256 x 128 units to as few SMs).
__global__ void __launch_bounds__(32)
rpy_direct64_kernel(const double *__restrict__ Y, const double *__restrict__ FT, int S,
                    RpyConst64 k, double scale, double *__restrict__ VW) {
    pdl_enter();
    const int n = blockIdx.x, lane = threadIdx.x;
    const double t0 = Y[3 * (int64_t)n], t1 = Y[3 * (int64_t)n + 1], t2 = Y[3 * (int64_t)n + 2];
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int m = lane; m < S; m += 32) {
        const double *y = Y + 3 * (int64_t)m, *f = FT + 6 * (int64_t)m;
        const double d[3] = {t0 - y[0], t1 - y[1], t2 - y[2]};
        const double ft[6] = {f[0], f[1], f[2], f[3], f[4], f[5]};
        double A, B, C, D, G;
        coef64(fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2])), k, A, B, C, D, G);
        const double e[3] = {G * d[0], G * d[1], G * d[2]};
        add64(ft, d, e, A, B, C, D, v);
    }
    const unsigned all = 0xffffffffu;
    double w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {          // V in lanes 0-15, Omega in lanes 16-31
        const double keep = lane & 16 ? v[3 + c] : v[c], give = lane & 16 ? v[c] : v[3 + c];
        w[c] = keep + __shfl_xor_sync(all, give, 16);
    }
    // components 0, 1 where lane bit 3 is clear, component 2 where it is set
    const double g0 = __shfl_xor_sync(all, lane & 8 ? w[0] : w[2], 8);
    const double g1 = __shfl_xor_sync(all, w[1], 8);
    double a = (lane & 8 ? w[2] : w[0]) + g0;
    const double b = w[1] + g1;
    // lane bit 2 splits components 0 and 1; component 2 is summed by both halves
    const double g = __shfl_xor_sync(all, lane & 8 ? a : (lane & 4 ? a : b), 4);
    a = (lane & 8 ? a : (lane & 4 ? b : a)) + g;
    a += __shfl_xor_sync(all, a, 2);
    a += __shfl_xor_sync(all, a, 1);
    const int c = (lane & 16 ? 3 : 0) + (lane & 8 ? 2 : (lane & 4 ? 1 : 0));
    if ((lane & 3) == 0 && (lane & 12) != 12) VW[6 * (int64_t)n + c] = a * scale;
}

// Medium systems: every unordered pair once. A CTA of four warps takes a pair of
// 64-segment tiles (I <= J), a warp one 32 x 32 block: a lane keeps one segment
// of the row block; the segments of the column block go round the lanes, their
// sums travelling with them by shuffles, so that after 32 steps both sides of
// every pair were added. 85 FP64 instructions for the two ordered pairs instead
// of 106 (the difference, 1/r and the coefficients are shared). A block on the
// diagonal takes its pairs at distance 1 .. 16 round the block, and the self
// terms. The CTA's sums go to the rows of its two tiles in slots named by the
// other tile, and sum64_kernel adds a row's slots in order. The CTAs are handed
// out by the hardware as SMs come free (the cost of a block depends on its
// overlapping pairs), the diagonal ones last.
// Measured: 3200 segments 1476 -> 827 us (a warp per target: 1012), 4000 1976 ->
// 1258; at 1024 both small forms take 108 us. Error against 64 bits 7e-16 -> 5e-16.
constexpr int kSymTile = 64;
constexpr int kSymThreads = 128;
constexpr int64_t kSymMaxSeg = 8192;          // slots: (S / 64) x 6 S doubles
constexpr int64_t kDirectMaxSeg = 1024;       // up to here a warp per target is faster
// The FP32 modes take it too while it is faster than packing and the FP32 kernel,
// whose chain of a few units alone is 11-15 us: at 32 segments 5.1 and 11.1 us, at 96 7.8
// and 15.0, at 160 11.5 and 14.4; at 192 13.5 and 14.3, at 224 15.4 and 14.3. (FP64
// throughout, so closer than the FP32 sums; the line stays at the 160 that fil.h states.)
constexpr int64_t kDirect32MaxSeg = 160;
inline int64_t direct_max(bool pair32) { return pair32 ? kDirect32MaxSeg : kDirectMaxSeg; }

__global__ void __launch_bounds__(kSymThreads)
rpy_sym64_kernel(const double *__restrict__ Y, const double *__restrict__ FT, int S, int tiles,
                 RpyConst64 k, double *__restrict__ slots) {
    __shared__ double sf[2][9][kSymTile];     // positions and loads of the two tiles
    __shared__ double sums[2][2][6][kSymTile];   // [side][which of the two blocks added][...]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // CTA -> (I, J): off-diagonal pairs row by row, then the diagonal tiles
    const int off = tiles * (tiles - 1) / 2;
    int I, J;
    if ((int)blockIdx.x >= off) {
        I = J = (int)blockIdx.x - off;
    } else {
        // pairs of row J (I < J) start at J (J - 1) / 2
        J = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)blockIdx.x)) * 0.5f);
        while (J * (J - 1) / 2 > (int)blockIdx.x) --J;
        while ((J + 1) * J / 2 <= (int)blockIdx.x) ++J;
        I = (int)blockIdx.x - J * (J - 1) / 2;
    }
    pdl_enter();
    {
        const int side = threadIdx.x >> 6, l = threadIdx.x & 63;
        const int n = (side ? J : I) * kSymTile + l;
        const bool in = n < S;
        // (past the end: no load, and a place of its own far away)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            sf[side][c][l] = in ? Y[3 * (int64_t)n + c] : (double)kFarPad * (double)(2 + l + 64 * side);
#pragma unroll
        for (int c = 0; c < 6; ++c) sf[side][3 + c][l] = in ? FT[6 * (int64_t)n + c] : 0.0;
    }
    __syncthreads();
    const int a = wid >> 1, b = wid & 1;      // blocks of I and J
    const bool diag = I == J;
    const bool self = diag && a == b;
    double vt[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, vs[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (!(diag && a > b)) {
        double t[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) t[c] = sf[0][c][32 * a + lane];
        if (self) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                vt[c] = k.ov_A0 * t[3 + c];
                vt[3 + c] = k.ov_C0 * t[6 + c];
            }
        }
        const int first = self ? 1 : 0, last = self ? 16 : 31;
        for (int st = first; st <= last; ++st) {
            if (st > 0) {                     // the sums of segment (lane + st) mod 32 arrive
#pragma unroll
                for (int c = 0; c < 6; ++c)
                    vs[c] = __shfl_sync(0xffffffffu, vs[c], (lane + 1) & 31);
            }
            const int j = 32 * b + ((lane + st) & 31);
            double f[6];
            const double d[3] = {t[0] - sf[1][0][j], t[1] - sf[1][1][j], t[2] - sf[1][2][j]};
#pragma unroll
            for (int c = 0; c < 6; ++c) f[c] = sf[1][3 + c][j];
            // (at distance 16 in a diagonal block each pair comes up twice)
            if (!(self && st == 16 && lane >= 16)) {
                double A, B, C, D, G;
                coef64(fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2])), k, A, B, C, D, G);
                const double e[3] = {G * d[0], G * d[1], G * d[2]};
                const double ne[3] = {-e[0], -e[1], -e[2]};
                add64(f, d, e, A, B, C, D, vt);
                add64(t + 3, d, ne, A, B, C, D, vs);
            }
        }
        // home: after `last` steps the sums of segment (lane + last) mod 32 are here
#pragma unroll
        for (int c = 0; c < 6; ++c) vs[c] = __shfl_sync(0xffffffffu, vs[c], (lane - last) & 31);
    }
    // rows of I: blocks (a, 0) and (a, 1); rows of J: blocks (0, b) and (1, b)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        sums[0][b][c][32 * a + lane] = vt[c];
        sums[1][a][c][32 * b + lane] = vs[c];
    }
    __syncthreads();
    const int64_t rows = (int64_t)tiles * kSymTile;
    for (int i = threadIdx.x; i < 6 * kSymTile; i += kSymThreads) {
        const int c = i / kSymTile, l = i % kSymTile;
        const double x = sums[0][0][c][l] + sums[0][1][c][l];
        const double y = sums[1][0][c][l] + sums[1][1][c][l];
        if (diag) {
            slots[((int64_t)I * 6 + c) * rows + I * kSymTile + l] = x + y;
        } else {
            slots[((int64_t)J * 6 + c) * rows + I * kSymTile + l] = x;
            slots[((int64_t)I * 6 + c) * rows + J * kSymTile + l] = y;
        }
    }
}

// Row sums over the slots, in order.
__global__ void __launch_bounds__(64)
sum64_kernel(const double *__restrict__ slots, int S, int tiles, double scale,
             double *__restrict__ VW) {
    pdl_enter();
    const int n = blockIdx.x * 64 + threadIdx.x, c = blockIdx.y;
    if (n >= S) return;
    const int64_t rows = (int64_t)tiles * kSymTile;
    const double *p = slots + c * rows + n;
    double a = 0.0;
#pragma unroll 16
    for (int t = 0; t < tiles; ++t) a += p[(int64_t)t * 6 * rows];
    VW[6 * (int64_t)n + c] = a * scale;
}

// Bytes of [p, p + n) and [q, q + m) overlap.
bool overlaps(const double *p, int64_t n, const double *q, int64_t m) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
    return a < b + 8 * (uintptr_t)m && b < a + 8 * (uintptr_t)n;
}

// Source groups in their own frames: the automatic schedule of one FP32 system.
bool frames_on(const fil_ctx *c) { return pair32_on(c) && c->rpy_auto; }

SysMap sys_map(const fil_ctx *c, bool active_only) {
    SysMap m{};
    m.n_src = c->lay.S;
    if (c->n_sys == 1 && !active_only) {
        // one system: tiles and groups in order, no table
        m.n_tiles = c->rpy_tiles;
        const int per = unit_sources(frames_on(c));
        m.n_units = (c->lay.S + per - 1) / per;
        return m;
    }
    m.pad_map = c->pad_map_d;
    if (active_only) {
        m.tile_unit_off = c->act_unit_off_d;
        m.tile_src = c->act_src_d;
        m.tile_nsrc = c->act_nsrc_d;
        m.tile_id = c->act_tile_d;
        m.n_tiles = c->act_tiles;
        m.dyn = c->act_dyn_d;
    } else {
        m.tile_unit_off = c->tile_unit_off_d;
        m.tile_src = c->tile_src_d;
        m.tile_nsrc = c->tile_nsrc_d;
        m.tile_id = c->tile_id_d;
        m.n_tiles = c->rpy_tiles;
    }
    return m;
}

constexpr int kRpyPad = 256;   // systems start at multiples of this in the padded layout

int64_t count_tiles(const fil_ctx *c, int T) {
    int64_t n = 0;
    for (int s = 0; s < c->n_sys; ++s)
        n += (c->sys_seg_off_h[s + 1] - c->sys_seg_off_h[s] + T - 1) / T;
    return n;
}

cudaError_t allow_warp_smem() {
    for (const auto kernel : {rpy_pair32_warp_kernel<false>, rpy_pair32_warp_kernel<true>}) {
        const cudaError_t e = cudaFuncSetAttribute(
            kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Tiles of T targets of every system (only tiles that hold real targets),
// each with ceil(S_s / unit) units.
void build_tiles(fil_ctx *c) {
    const int T = frames_on(c) ? kWarpTile : rpy_tile(c);
    const int per = unit_sources(frames_on(c));
    c->tile_unit_off_h.assign(1, 0);
    c->tile_src_h.clear();
    c->tile_nsrc_h.clear();
    c->tile_sys_h.clear();
    c->tile_id_h.clear();
    for (int s = 0; s < c->n_sys; ++s) {
        const int64_t Ss = c->sys_seg_off_h[s + 1] - c->sys_seg_off_h[s];
        const int64_t tiles = (Ss + T - 1) / T;
        const int64_t units = (Ss + per - 1) / per;
        for (int64_t t = 0; t < tiles; ++t) {
            c->tile_unit_off_h.push_back(c->tile_unit_off_h.back() + units);
            c->tile_src_h.push_back(c->sys_pad_off_h[s]);
            c->tile_nsrc_h.push_back(Ss);
            c->tile_sys_h.push_back(s);
            c->tile_id_h.push_back((int)(c->sys_pad_off_h[s] / T + t));
        }
    }
    c->rpy_tiles = (int64_t)c->tile_src_h.size();
    c->rpy_units = c->tile_unit_off_h.back();
}

template <typename K>
int occupancy(K kernel, int threads = kRpyThreads) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, 0) != cudaSuccess)
        return 1;
    return std::max(1, occ);
}


// Resident CTAs per SM of the pair kernel of a schedule (targets per thread,
// source split; the split exists for the FP32 kernel with one target per thread).
int pair_occupancy(const fil_ctx *c, int tpt, int split) {
    if (!pair32_on(c))
        return tpt == 1 ? occupancy(rpy_pair64_kernel<1>) : occupancy(rpy_pair64_kernel<2>);
    return min_blocks(tpt, split);
}

// The grid of the current schedule, and whether it fills the SMs. One that does not
// is launched plainly: an early launch (launch_dep) would put two CTAs on some SMs and
// none on others (32 000 segments, 256-target tiles at one CTA per SM: 1786 us plainly,
// 3091 early).
void set_grids(fil_ctx *c) {
    c->rpy_grid32 = c->rpy_ctas * c->num_sms;
    c->rpy_grid64 = c->rpy_ctas * c->num_sms;
    c->rpy_full = c->rpy_ctas >= pair_occupancy(c, c->rpy_tpt, c->rpy_split);
}

}  // namespace

// The automatic schedule of one system goes by the values a new context reports, so that
// a schedule that was read and is set again is the one that ran.
static int automatic_schedule(const fil_ctx *c, int tpt, int ctas, int split) {
    return c->n_sys == 1 && tpt == kRpyTargetsPerThread && split == 1 &&
           ctas == pair_occupancy(c, kRpyTargetsPerThread, 1);
}

cudaError_t rpy_setup(fil_ctx *c) {
    c->rpy_tpt = kRpyTargetsPerThread;
    c->rpy_threads = kRpyThreads;
    const int occ = pair_occupancy(c, kRpyTargetsPerThread, 1);
    c->rpy_ctas = occ;
    c->rpy_split = 1;
    c->rpy_ctas_max = std::max({occ, kRpyMinBlocksTpt1, kRpyMinBlocksTpt2,
                                occupancy(rpy_pair64_kernel<1>), occupancy(rpy_pair64_kernel<2>)});
    set_grids(c);
    // padded layout: system s occupies [pad_off[s], pad_off[s+1]), a multiple of kRpyPad
    const int ns = c->n_sys;
    c->sys_pad_off_h.assign(ns + 1, 0);
    c->pairs_all = 0.0;
    for (int s = 0; s < ns; ++s) {
        const int64_t Ss = c->sys_seg_off_h[s + 1] - c->sys_seg_off_h[s];
        c->sys_pad_off_h[s + 1] = c->sys_pad_off_h[s] + (Ss + kRpyPad - 1) / kRpyPad * kRpyPad;
        c->pairs_all += (double)Ss * (double)Ss;
    }
    c->pairs_act = c->pairs_all;
    c->Spad = c->sys_pad_off_h[ns];
    c->pad_map_h.assign(c->Spad, -1);
    for (int s = 0; s < ns; ++s)
        for (int64_t g = c->sys_seg_off_h[s]; g < c->sys_seg_off_h[s + 1]; ++g) {
            const int64_t P = c->sys_pad_off_h[s] + (g - c->sys_seg_off_h[s]);
            c->pad_map_h[P] = (int)g;
        }
    c->rpy_tiles_max = count_tiles(c, kWarpTile);
    c->rpy_auto = automatic_schedule(c, c->rpy_tpt, c->rpy_ctas, c->rpy_split);
    if (frames_on(c)) {
        const cudaError_t e = allow_warp_smem();
        if (e != cudaSuccess) return e;
    }
    build_tiles(c);
    return cudaSuccess;
}

// Tile tables of the current tile size (after the arena exists, and after a retune).
cudaError_t upload_tiles(fil_ctx *c) {
    cudaError_t e = cudaMemcpyAsync(c->tile_unit_off_d, c->tile_unit_off_h.data(),
                                    sizeof(int64_t) * c->tile_unit_off_h.size(),
                                    cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->tile_src_d, c->tile_src_h.data(), sizeof(int64_t) * c->tile_src_h.size(),
                            cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->tile_nsrc_d, c->tile_nsrc_h.data(),
                            sizeof(int64_t) * c->tile_nsrc_h.size(), cudaMemcpyHostToDevice,
                            c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->tile_id_d, c->tile_id_h.data(), sizeof(int) * c->tile_id_h.size(),
                            cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return e;
}

cudaError_t rpy_upload_tables(fil_ctx *c) {
    cudaError_t e = upload_tiles(c);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->pad_map_d, c->pad_map_h.data(), sizeof(int) * c->pad_map_h.size(),
                            cudaMemcpyHostToDevice, c->stream);
    return e;
}

size_t rpy_partial_bytes(const fil_ctx *c) {
    // slots b + tile for b < G and listed tiles; 12 floats = 6 doubles per target;
    // the largest over the tile sizes and grids the autotuner may choose
    const int64_t G = (int64_t)c->rpy_ctas_max * c->num_sms;
    size_t most = 0;
    for (int tpt = 1; tpt <= 2; ++tpt) {
        const int T = kRpyThreads * tpt;
        const size_t b = (size_t)(G + count_tiles(c, T)) * T * 12 * sizeof(float);
        most = std::max(most, b);
    }
    if (pair32_on(c) && c->n_sys == 1)
        most = std::max(most, (size_t)((int64_t)c->num_sms * kWarpCta + c->rpy_tiles_max) *
                                  kWarpPart * sizeof(float));
    else if (c->n_sys == 1 && c->lay.S > kDirectMaxSeg && c->lay.S <= kSymMaxSeg) {
        const size_t tiles = (size_t)(c->lay.S + kSymTile - 1) / kSymTile;
        most = std::max(most, tiles * 6 * tiles * kSymTile * sizeof(double));
    }
    return most;
}

// The tiles of the systems still iterating (c->active_h), listed for the
// stream-K split of the next applies with active_only.
cudaError_t rpy_set_active(fil_ctx *c) {
    std::vector<int64_t> uoff(1, 0), src, nsrc;
    std::vector<int> tid;
    for (int64_t t = 0; t < c->rpy_tiles; ++t) {
        if (!c->active_h[c->tile_sys_h[t]]) continue;
        tid.push_back(c->tile_id_h[t]);
        src.push_back(c->tile_src_h[t]);
        nsrc.push_back(c->tile_nsrc_h[t]);
        uoff.push_back(uoff.back() + (c->tile_unit_off_h[t + 1] - c->tile_unit_off_h[t]));
    }
    c->act_tiles = (int64_t)tid.size();
    c->act_units = uoff.back();
    c->pairs_act = 0.0;
    for (int s = 0; s < c->n_sys; ++s)
        if (c->active_h[s]) {
            const double Ss = (double)(c->sys_seg_off_h[s + 1] - c->sys_seg_off_h[s]);
            c->pairs_act += Ss * Ss;
        }
    cudaError_t e = cudaMemcpyAsync(c->act_unit_off_d, uoff.data(), sizeof(int64_t) * uoff.size(),
                                    cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess && !tid.empty())
        e = cudaMemcpyAsync(c->act_src_d, src.data(), sizeof(int64_t) * src.size(),
                            cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess && !tid.empty())
        e = cudaMemcpyAsync(c->act_nsrc_d, nsrc.data(), sizeof(int64_t) * nsrc.size(),
                            cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess && !tid.empty())
        e = cudaMemcpyAsync(c->act_tile_d, tid.data(), sizeof(int) * tid.size(),
                            cudaMemcpyHostToDevice, c->stream);
    const int64_t dyn[2] = {c->act_tiles, c->act_units};
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->act_dyn_d, dyn, sizeof(dyn), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);   // host vectors go out of scope
    return e;
}

namespace {

// A timing event on the context stream; while the stream is being captured the
// record becomes an event-record node of the graph, so that the events hold
// the kernel's times of each replay.
void prof_record(fil_ctx *c, cudaEvent_t ev) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &cs) != cudaSuccess) cs = cudaStreamCaptureStatusNone;
    cudaEventRecordWithFlags(ev, c->stream, cs == cudaStreamCaptureStatusActive
                                                ? cudaEventRecordExternal
                                                : cudaEventRecordDefault);
}

}  // namespace

// CTAs of the warp kernel: one per SM, fewer when there are not as many units.
static int warp_grid(int64_t W, int sms) { return (int)std::min<int64_t>(sms, W); }

cudaError_t rpy_apply(fil_ctx *c, const double *Y, const double *FT, double *VW,
                      bool active_only) {
    const int64_t S = c->lay.S;
    const double scale = 1.0 / (8.0 * kPi * c->eta);
    const int pb = 256;
    const unsigned pgrid = (unsigned)((c->Spad + pb - 1) / pb);
    const bool timed = c->prof_on && c->prof_n < kProfMax;
    const SysMap sm = sys_map(c, active_only);
    const int64_t W = active_only ? c->act_units : c->rpy_units;
    if (W == 0) return cudaSuccess;
    // (with tune_pair set the first event is recorded again after the packing)
    if (c->tune_ev) cudaEventRecord(c->tune_ev[0], c->stream);
    // The stream-K kernels start early (launch_dep) where the grid is full, and in ensembles
    // has a unit for every CTA, or too small to crowd. Ensembles' applies, early and
    // plainly: 25 systems of 6 780 segments (about 100 units) 86.2 and 45.5 us, 9 of 5 460
    // 71.0 and 45.5, 64 small ones 66.3 and 55.5, 5 of 2 059 (40 units) 41.5 and 45.4. One
    // system in 128-target tiles, 3 CTAs per SM: 320 segments, 30 units, 16.0 and 18.5; 960,
    // 240 units, 27.9 and 26.7. 256 systems in such tiles 1519 and 855.
    // The FP64 kernel only where it is too small to crowd: its few units a CTA wait for the
    // fullest SM, and early placement makes that a matter of luck (one system of 8 193
    // segments 7.46 ms early and 7.16 plainly, 9 000 9.1 and 9.5, 10 000 10.7 and 11.3, 12 000
    // 14.6 and 14.5; three systems in 8 193 3.2 and 2.9, in 16 000 9.1 and 8.9).
    const bool small = W <= (c->n_sys == 1 ? c->num_sms : c->num_sms / 3);
    const bool early = small || (c->rpy_full && (c->n_sys == 1 || W >= c->rpy_grid32));
    // the active-tile list changes between applies: its launches keep a fixed grid
    // (and read the unit count from the device), so captured graphs stay valid
    if (c->rpy_auto && S <= direct_max(pair32_on(c)) && !overlaps(VW, 6 * S, Y, 3 * S) &&
        !overlaps(VW, 6 * S, FT, 6 * S)) {
        // Early (launch_dep) while each SM partition has at most one target's warp. One
        // FP64 time step of a 32-segment filament cloud, early and plainly: 1.57 and 1.61
        // ms at 320 segments, 2.40 and 2.40 at 640, 3.91 and 3.55 at 960.
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n]);
        launch_dep(S <= 4 * c->num_sms, rpy_direct64_kernel, (unsigned)S, 32, 0, c->stream, Y, FT,
                   (int)S, make_const<double, RpyConst64>(c->a), scale, VW);
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n + 1]);
        if (c->tune_ev) cudaEventRecord(c->tune_ev[1], c->stream);
        if (timed) c->prof_n += 1;
        c->n_launches += 1;
        c->n_applies += 1;
        c->n_pairs += c->pairs_all;
        return cudaGetLastError();
    }
    if (pair32_on(c)) {
        const auto pack = c->rpy_auto ? pack32_kernel<true> : pack32_kernel<false>;
        const int n_spread = c->rpy_auto ? spread_count((S + kRpyComp - 1) / kRpyComp) : 0;
        launch_pdl(pack, (unsigned)(c->Spad / kPackThreads), kPackThreads, 0, c->stream, Y, FT, S,
                   c->Spad, sm, n_spread, (float)c->a, c->src32);
        if (c->tune_ev && c->tune_pair) cudaEventRecord(c->tune_ev[0], c->stream);
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n]);
        const RpyConst32 k = make_const<float, RpyConst32>(c->a);
        if (c->rpy_auto) {
            const int G = warp_grid(W, c->num_sms);
            launch_pdl(n_spread ? rpy_pair32_warp_kernel<true> : rpy_pair32_warp_kernel<false>, G,
                       32 * kWarpCta, kWarpSmem, c->stream, c->src32, sm, W, G, k,
                       (float *)c->partials, c->tile_cnt, scale, VW);
        } else {
            const int G = (int)(active_only ? c->rpy_grid32 : std::min<int64_t>(c->rpy_grid32, W));
            const bool split = c->rpy_tpt == 1 && c->rpy_split == 2;
            const auto pair = split             ? rpy_pair32_kernel<1, 2>
                              : c->rpy_tpt == 1 ? rpy_pair32_kernel<1>
                                                : rpy_pair32_kernel<2>;
            launch_dep(early, pair, G, kRpyThreads * (split ? 2 : 1), 0, c->stream, c->src32,
                       sm, W, G, k, (float *)c->partials, c->tile_cnt, scale, VW);
        }
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n + 1]);
        if (c->tune_ev) cudaEventRecord(c->tune_ev[1], c->stream);
    } else {
        const RpyConst64 k = make_const<double, RpyConst64>(c->a);
        // one system on the automatic schedule: straight from the caller's arrays, unless
        // the result overwrites them (or is too large for the slots)
        if (c->rpy_auto && S <= kSymMaxSeg && !overlaps(VW, 6 * S, Y, 3 * S) &&
            !overlaps(VW, 6 * S, FT, 6 * S)) {
            if (timed) prof_record(c, c->prof_ev[2 * c->prof_n]);
            // (a plain launch: one FP64 time step of a 32-segment filament cloud took 10.7 ms
            // with the early one and 9.5 without at 1 920 segments, see launch_dep)
            const int tiles = (int)((S + kSymTile - 1) / kSymTile);
            launch_dep(false, rpy_sym64_kernel, (unsigned)(tiles * (tiles + 1) / 2), kSymThreads, 0,
                       c->stream, Y, FT, (int)S, tiles, k, (double *)c->partials);
            launch_pdl(sum64_kernel, dim3((unsigned)((S + 63) / 64), 6), 64, 0, c->stream,
                       (const double *)c->partials, (int)S, tiles, scale, VW);
            c->n_launches += 2;
            if (timed) prof_record(c, c->prof_ev[2 * c->prof_n + 1]);
            if (c->tune_ev) cudaEventRecord(c->tune_ev[1], c->stream);
            if (timed) c->prof_n += 1;
            c->n_applies += 1;
            c->n_pairs += c->pairs_all;
            return cudaGetLastError();
        }
        const int G = (int)(active_only ? c->rpy_grid64 : std::min<int64_t>(c->rpy_grid64, W));
        launch_pdl(pack64_kernel, pgrid, pb, 0, c->stream, Y, FT, S, c->Spad, sm, c->src64);
        if (c->tune_ev && c->tune_pair) cudaEventRecord(c->tune_ev[0], c->stream);
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n]);
        launch_dep(small, c->rpy_tpt == 1 ? rpy_pair64_kernel<1> : rpy_pair64_kernel<2>, G,
                   kRpyThreads, 0, c->stream, c->src64, sm, W, G, k, (double *)c->partials,
                   c->tile_cnt, scale, VW);
        if (timed) prof_record(c, c->prof_ev[2 * c->prof_n + 1]);
        if (c->tune_ev) cudaEventRecord(c->tune_ev[1], c->stream);
    }
    if (timed) c->prof_n += 1;
    c->n_applies += 1;
    c->n_pairs += active_only ? c->pairs_act : c->pairs_all;
    c->n_launches += 2;
    return cudaGetLastError();
}


// Autotuner of the pair kernel: times every (targets per thread, resident CTAs
// per SM) candidate on `reps` applies of (Y, FT) and keeps the fastest. What is
// compared are whole applies, as some schedules pack their sources in a launch of
// their own, and an event between the two launches would keep the second from
// starting early; the choice's pair kernel alone is timed at the end, for the
// report. An FP32 system small enough for the direct FP64 sums has no other
// candidate, so that tuning does not change its accuracy. An idle
// GPU runs at a low clock for some tens of milliseconds after work arrives, so
// the applies first run for kSpinUpMs of wall time, and the candidates are then
// swept twice, each keeping the faster of its two times: a candidate measured
// while the clock still climbs is not chosen against or for that reason.
cudaError_t rpy_autotune(fil_ctx *c, const double *Y, const double *FT, double *VW, int reps,
                         double *best_ms) {
    constexpr double kSpinUpMs = 50.0;
    constexpr int kSweeps = 2;
    const int64_t a0 = c->n_applies, l0 = c->n_launches;
    const double p0 = c->n_pairs;
    // each rep's pair kernel is timed by its own pair of events, so
    // that host launch gaps between applies (which dominate tiny problems) do not
    // enter the comparison
    std::vector<cudaEvent_t> ev(2 * (size_t)std::max(1, reps), nullptr);
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < ev.size() && e == cudaSuccess; ++i) e = cudaEventCreate(&ev[i]);
    struct cand { int tpt, split, ctas; float ms; };
    std::vector<cand> cands;
    const bool direct = c->n_sys == 1 && pair32_on(c) && c->lay.S <= kDirect32MaxSeg;
    for (int tpt = 1; tpt <= 2 && !direct; ++tpt) {
        for (int split = 1; split <= (tpt == 1 && pair32_on(c) ? 2 : 1); ++split) {
            const int occ = pair_occupancy(c, tpt, split);
            for (int ctas = 1; ctas <= std::min(occ, c->rpy_ctas_max); ++ctas)
                cands.push_back({tpt, split, ctas, 1e30f});
        }
    }
    if (direct) cands.push_back({kRpyTargetsPerThread, 1, pair_occupancy(c, 2, 1), 1e30f});
    const auto t0 = std::chrono::steady_clock::now();
    while (e == cudaSuccess) {
        for (int r = 0; r < 4 && e == cudaSuccess; ++r) e = rpy_apply(c, Y, FT, VW);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        const std::chrono::duration<double, std::milli> dt = std::chrono::steady_clock::now() - t0;
        if (dt.count() >= kSpinUpMs) break;
    }
    const auto use = [&](const cand &k) {
        return rpy_set_schedule(c, k.tpt, kRpyThreads, k.ctas, k.split);
    };
    // the time of `reps` applies, or of their pair kernels, in the schedule in use
    const auto time = [&](bool pair, float &ms) {
        cudaError_t er = rpy_apply(c, Y, FT, VW);       // warm-up
        c->tune_pair = pair;
        for (int r = 0; r < reps && er == cudaSuccess; ++r) {
            c->tune_ev = &ev[2 * r];
            er = rpy_apply(c, Y, FT, VW);
            c->tune_ev = nullptr;
        }
        if (er == cudaSuccess) er = cudaStreamSynchronize(c->stream);
        ms = 0.f;
        for (int r = 0; r < reps && er == cudaSuccess; ++r) {
            float one = 0.f;
            er = cudaEventElapsedTime(&one, ev[2 * r], ev[2 * r + 1]);
            ms += one;
        }
        return er;
    };
    cand best{c->rpy_tpt, c->rpy_split, c->rpy_ctas, 1e30f};
    for (int sweep = 0; sweep < kSweeps && e == cudaSuccess; ++sweep) {
        for (cand &k : cands) {
            float ms = 0.f;
            e = use(k);
            if (e == cudaSuccess) e = time(false, ms);
            if (e != cudaSuccess) break;
            k.ms = std::min(k.ms, ms);
        }
    }
    for (const cand &k : cands)
        if (k.ms < best.ms) best = k;
    const cudaError_t eu = use(best);       // (a valid schedule also where a launch failed)
    if (e == cudaSuccess) e = eu;
    for (int sweep = 0; sweep < kSweeps && e == cudaSuccess; ++sweep) {
        float ms = 0.f;
        e = time(true, ms);
        best.ms = sweep ? std::min(best.ms, ms) : ms;
    }
    for (cudaEvent_t x : ev)
        if (x) cudaEventDestroy(x);
    c->n_applies = a0;
    c->n_launches = l0;
    c->n_pairs = p0;
    if (best_ms) *best_ms = best.ms / std::max(1, reps);
    return e;
}

// A given pair schedule (targets per thread, threads per CTA, resident CTAs per
// SM for the stream-K grid); false if the kernel has no such schedule or the
// CTA count exceeds its occupancy.
bool rpy_schedule_valid(const fil_ctx *c, int tpt, int threads, int ctas, int split) {
    if (threads != kRpyThreads || (tpt != 1 && tpt != 2)) return false;
    if (split != 1 && !(split == 2 && tpt == 1 && pair32_on(c))) return false;
    const int occ = pair_occupancy(c, tpt, split);
    return ctas >= 1 && ctas <= std::min(occ, c->rpy_ctas_max);
}

cudaError_t rpy_set_schedule(fil_ctx *c, int tpt, int threads, int ctas, int split) {
    c->rpy_auto = automatic_schedule(c, tpt, ctas, split);
    c->rpy_tpt = tpt;
    c->rpy_split = split;
    c->rpy_threads = threads;
    c->rpy_ctas = ctas;
    set_grids(c);
    build_tiles(c);
    return upload_tiles(c);
}

// ---------------------------------------------------------------------------
// Allocation-free mobility apply (fil_rpy_apply_noalloc).
//
// For callers that cannot allocate device memory themselves -- code running
// where cudaMalloc is unavailable or forbidden, e.g. inside another
// framework's memory pool or a process whose allocations are owned by
// someone else -- this variant of the mixed-precision apply uses no context
// and allocates nothing: its scratch (packed FP32 sources, the stream-K
// partial sums and the tiles' completion counters) is the file-scope arrays
// below, which every GPU that loads the library holds until the process exits.
// The caller passes the inputs and the output in device memory.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t kNoAllocMaxSeg = 32768;     // largest S accepted
// The context path runs the stream-K split over (resident CTAs per SM) x SMs
// CTAs. The scratch holds the partial sums of at most kNoAllocMaxSMs SMs at
// the pair kernel's compiled residency (GB300 has 152 SMs); on a larger part
// the grid is capped here, and the results then differ from
// fil_mobility_apply's in rounding only (another summation order).
constexpr int kNoAllocMaxSMs = 152;
constexpr int64_t kNoAllocMaxTiles = (kNoAllocMaxSeg + kWarpTile - 1) / kWarpTile;
constexpr int64_t kNoAllocMaxSpad = kNoAllocMaxTiles * kWarpTile;
constexpr size_t kNoAllocSrcBytes =
    (size_t)Rec<true>::kGroupF4 * (kNoAllocMaxSpad / kRpyComp) * sizeof(float4);
constexpr size_t kNoAllocPartBytes =
    (size_t)(kNoAllocMaxSMs * kWarpCta + kNoAllocMaxTiles) * kWarpPart * sizeof(float);
constexpr size_t kNoAllocBytes = kNoAllocSrcBytes + kNoAllocPartBytes;   // ~9.6 MB

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];
// per-tile completion counters of the pair kernel: zero at load, and every
// launch leaves them zero
static __device__ int g_noalloc_cnt[kNoAllocMaxTiles] = {0};

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
unsigned char *g_noalloc_ptr[kNoAllocMaxDevices];   // device address of the array, per device
int *g_noalloc_cnt_ptr[kNoAllocMaxDevices];         // and of the counters
int g_noalloc_grid[kNoAllocMaxDevices];

// Once per device, with that device current: the device addresses of the
// arrays (their names are only host-side stand-ins) and the stream-K grid size.
cudaError_t noalloc_setup(int dev, unsigned char **ptr, int **cnt, int *grid) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr, *q = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        e = cudaGetSymbolAddress(&q, g_noalloc_cnt);
        if (e != cudaSuccess) return e;
        g_noalloc_cnt_ptr[dev] = static_cast<int *>(q);
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        e = allow_warp_smem();
        if (e != cudaSuccess) return e;
        g_noalloc_grid[dev] = std::max(1, std::min(kNoAllocMaxSMs, sms));
        g_noalloc_ptr[dev] = static_cast<unsigned char *>(p);
    }
    *ptr = g_noalloc_ptr[dev];
    *cnt = g_noalloc_cnt_ptr[dev];
    *grid = g_noalloc_grid[dev];
    return cudaSuccess;
}

// Memory the kernels may read on device `dev`: device memory of that device,
// or managed memory. Host memory and memory of another GPU (which these
// kernels could only reach through peer access) are rejected.
bool on_device(const void *p, int dev) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();   // the error of this query only
        return false;
    }
    if (at.type == cudaMemoryTypeManaged) return true;
    return at.type == cudaMemoryTypeDevice && at.device == dev;
}

// A launch whose own status is returned (cudaGetLastError would also report
// an earlier, unrelated failure of the caller's).
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem,
                   cudaStream_t st, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = nullptr;
    cfg.numAttrs = 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace

}  // namespace fil

extern "C" fil_status fil_rpy_apply_noalloc(int64_t n_seg, const double *Y, const double *FT,
                                            double *VW, double a, double eta, void *stream) {
    using namespace fil;
    if (n_seg < 1 || n_seg > kNoAllocMaxSeg) return FIL_EINVAL;
    if (!(a > 0) || !(eta > 0) || !Y || !FT || !VW) return FIL_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return FIL_ECUDA;
    if (!on_device(Y, dev) || !on_device(FT, dev) || !on_device(VW, dev)) return FIL_EINVAL;
    unsigned char *base = nullptr;
    int *cnt = nullptr;
    int grid_max = 1;
    if (noalloc_setup(dev, &base, &cnt, &grid_max) != cudaSuccess) return FIL_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (n_seg <= kDirect32MaxSeg && !overlaps(VW, 6 * n_seg, Y, 3 * n_seg) &&
        !overlaps(VW, 6 * n_seg, FT, 6 * n_seg)) {       // as fil_mobility_apply
        const cudaError_t e = launch(rpy_direct64_kernel, (unsigned)n_seg, 32, 0, st,
                                     Y, FT, (int)n_seg, make_const<double, RpyConst64>(a),
                                     1.0 / (8.0 * kPi * eta), VW);
        return e == cudaSuccess ? FIL_OK : FIL_ECUDA;
    }
    const int64_t tiles = (n_seg + kWarpTile - 1) / kWarpTile;
    const int64_t Spad = tiles * kWarpTile;
    const int64_t n_units = (n_seg + kRpyComp - 1) / kRpyComp;   // source groups per tile
    const int64_t W = tiles * n_units;
    const int G = warp_grid(W, grid_max);
    float4 *src = reinterpret_cast<float4 *>(base);
    float *part = reinterpret_cast<float *>(base + kNoAllocSrcBytes);
    // every source record up to Spad and every partial slot a tile's sum reads
    // is written below; the tile counters are zero between launches
    SysMap sm{};                       // one system, no tables
    sm.n_tiles = tiles;
    sm.n_units = n_units;
    sm.n_src = n_seg;
    const int n_spread = spread_count(n_units);
    cudaError_t e = launch(pack32_kernel<true>, (unsigned)(Spad / kPackThreads), kPackThreads, 0,
                           st, Y, FT, n_seg, Spad, sm, n_spread, (float)a, src);
    if (e == cudaSuccess)
        e = launch(n_spread ? rpy_pair32_warp_kernel<true> : rpy_pair32_warp_kernel<false>,
                   (unsigned)G, 32 * kWarpCta, kWarpSmem, st, (const float4 *)src, sm, W, G,
                   make_const<float, RpyConst32>(a), part, cnt, 1.0 / (8.0 * kPi * eta), VW);
    return e == cudaSuccess ? FIL_OK : FIL_ECUDA;
}
