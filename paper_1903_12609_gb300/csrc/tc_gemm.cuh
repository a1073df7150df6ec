// BF16 GEMM on the 5th-generation tensor cores (tcgen05, sm_100 family):
//   C[M x N] = A[M x K] . B[N x K]^T      (A, B row-major BF16, K contiguous)
// with FP32 accumulation in tensor memory and a fused epilogue. It is the
// contraction of the per-filament warm-start MLP (inference and training).
//
// One launch runs up to kMaxProblems products. One CTA computes a 128 x nt
// tile (nt a multiple of 32, at most 256, the same for the launch):
//   * K is consumed in stages of 64 (one 128-byte swizzle atom of BF16): 128
//     threads copy the A and B stage tiles from global memory with cp.async
//     into the 128-byte-swizzled K-major layout (16-byte chunk c of row r
//     stored at chunk c ^ (r % 8), 1024-byte aligned tiles), `stages` - 1
//     stages ahead of the one being multiplied;
//   * one thread issues four tcgen05.mma (M = 128, N = nt, K = 16 each, the
//     shared-memory descriptors advanced by 32 bytes inside the atom) into an
//     FP32 accumulator in tensor memory, then tcgen05.commit to the stage's
//     mbarrier; a stage is refilled once its mbarrier completed (every wait is
//     bounded);
//   * the epilogue reads the accumulator with tcgen05.ld (warp w owns rows
//     32w..32w+31, i.e. tensor-memory lanes 32w..) and applies bias, ReLU or
//     a ReLU mask and an output scale, storing FP32 and/or BF16 (row-major and
//     transposed) and the column sums of its 128 rows.
// Rows past M read as zero and are not stored; N must be a multiple of 32 and
// K a multiple of 64 (callers pad with zeros).
//
// What bounds it: these products are small (0.1-0.4 GFLOP, 2-8 row tiles), so
// the latency of a CTA's serial chain of K stages and the number of CTAs, not
// the tensor rate. nt is the smallest that keeps the launch within one CTA per
// SM (pick_tile_n), and the copies run several stages ahead. Measured on one
// batch of 1024 (cold, per product): 57 us with 256-column tiles and each stage
// loaded, multiplied and waited for in turn; about 6 us in this form.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fil {
namespace tc {

constexpr int kTileM = 128;
constexpr int kTileK = 64;
constexpr int kMaxTileN = 256;
constexpr int kThreads = 128;
constexpr int kMaxProblems = 4;
constexpr int kMaxStages = 8;
// stages in flight and dynamic shared memory by tile width (A and B tiles of
// every stage, and alignment slack): one CTA per SM
__host__ __device__ constexpr int stages_for(int nt) {
    return nt <= 32 ? 8 : nt <= 64 ? 7 : nt <= 128 ? 5 : 4;
}
__host__ __device__ constexpr int stage_bytes(int nt) { return (kTileM + nt) * 128; }
constexpr int smem_bytes(int nt) { return stages_for(nt) * stage_bytes(nt) + 1024; }

struct Epilogue {
    float *c_f32;              // [M x ldc] FP32 out (nullable)
    int ldc;
    __nv_bfloat16 *c_bf16;     // [M x ldh] BF16 out (nullable)
    int ldh;
    __nv_bfloat16 *c_bf16_t;   // [N x ldt] BF16 out, transposed (nullable)
    int ldt;
    int t_rows;                // its columns M .. t_rows - 1 are set to zero
    const float *bias;         // [N] added before the activation (nullable)
    int relu;                  // 1: max(x, 0)
    const __nv_bfloat16 *mask; // [M x ldm]: x *= (mask > 0) (nullable; ReLU derivative)
    int ldm;
    const float *shift, *scale;   // [N]: the FP32 out is shift + scale x (nullable, together)
    float *col_sums;           // [row tiles x N] sums over each tile's rows (nullable)
    int n_valid;               // columns >= n_valid are not stored (multiples of 32)
};

struct Problem {
    const __nv_bfloat16 *A, *B;
    int lda, ldb, M, N, K;
    int tiles_n, cta0;         // column tiles, first CTA (set by plan)
    int b_ready;               // B was complete before the launch's predecessor (weights)
    Epilogue ep;
};

struct Batch {
    Problem p[kMaxProblems];
    int count, nt;
    int *err;
};

// Tile width of a launch: the narrowest that needs at most one CTA per SM.
inline int pick_tile_n(const Batch &b, int sms) {
    for (int nt = 32; nt < kMaxTileN; nt *= 2) {
        int64_t ctas = 0;
        for (int i = 0; i < b.count; ++i)
            ctas += (int64_t)((b.p[i].M + kTileM - 1) / kTileM) * ((b.p[i].N + nt - 1) / nt);
        if (ctas <= sms) return nt;
    }
    return kMaxTileN;
}

// Tile width and CTA ranges of the batch; returns the number of CTAs.
inline int64_t plan(Batch &b, int sms) {
    b.nt = pick_tile_n(b, sms);
    int64_t ctas = 0;
    for (int i = 0; i < b.count; ++i) {
        Problem &p = b.p[i];
        p.tiles_n = (p.N + b.nt - 1) / b.nt;
        p.cta0 = (int)ctas;
        ctas += (int64_t)((p.M + kTileM - 1) / kTileM) * p.tiles_n;
    }
    return ctas;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), leading byte offset unused (16 B).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);          // start address, 16-byte units
    d |= (uint64_t)(16 >> 4) << 16;                      // leading byte offset
    d |= (uint64_t)(1024 >> 4) << 32;                    // stride byte offset
    d |= (uint64_t)1 << 46;                              // descriptor version (tcgen05)
    d |= (uint64_t)2 << 61;                              // swizzle: 128 B
    return d;
}

// Instruction descriptor, kind::f16: BF16 A and B (K-major), FP32 D, M = 128.
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
    return (1u << 4)                        // D format F32
           | (1u << 7)                      // A format BF16
           | (1u << 10)                     // B format BF16
           | ((uint32_t)(n >> 3) << 17)     // N / 8
           | ((uint32_t)(kTileM >> 4) << 24);   // M / 16
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :
        : "r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :
                 : "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" : : "r"(mbar), "r"(count) : "memory");
}

// Bounded wait for phase `parity` of the mbarrier (try_wait suspends for a
// bounded time per call): false if it did not complete within the limit.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// One 16-byte chunk, global -> shared, asynchronously (zeros if !valid).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 :
                 : "r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch: the next kernel of the stream may start its
// prologue now / wait here until the previous kernel is complete and its writes
// are visible. Nothing before the wait may read what that kernel writes.
__device__ __forceinline__ void pdl_launch_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int kNt>
__global__ void __launch_bounds__(kThreads)
gemm_bf16_kernel(const __grid_constant__ Batch g) {
    constexpr int kStages = stages_for(kNt), kStage = stage_bytes(kNt);
    constexpr int kCols = kNt < 32 ? 32 : kNt;       // tensor-memory columns (a power of two)
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t mbar[kStages];
    __shared__ uint32_t tmem_slot;
    __shared__ float csum[kThreads / 32][kNt];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const uint32_t sbase = smem_u32(base);           // per stage: A 128 rows x 128 B, then B
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int pi = 0;
    while (pi + 1 < g.count && (int)blockIdx.x >= g.p[pi + 1].cta0) ++pi;
    const Problem &p = g.p[pi];
    const Epilogue &ep = p.ep;
    const int local = (int)blockIdx.x - p.cta0;
    const int mt = local / p.tiles_n, m0 = mt * kTileM;
    const int n0 = (local - mt * p.tiles_n) * kNt;
    const int M = p.M, nt = min(kNt, p.N - n0);
    const int kb_n = p.K / kTileK;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_u32(&tmem_slot)), "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) mbar_init(smem_u32(&mbar[i]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // this thread's chunks of a stage: rows (tid / 8) + 16 i, chunk tid % 8
    const int r0 = tid >> 3, ch = tid & 7;
    const uint32_t s0 = (uint32_t)(r0 * 128 + ((ch ^ (r0 & 7)) << 4));   // row r0 + 16 i: + 2048 i
    const __nv_bfloat16 *Ap = p.A + (size_t)(m0 + r0) * p.lda + 8 * ch;
    const __nv_bfloat16 *Bp = p.B + (size_t)(n0 + r0) * p.ldb + 8 * ch;
    const auto load_a = [&](int kb) {
        const uint32_t d = sbase + (uint32_t)((kb % kStages) * kStage) + s0;
        const int k0 = kb * kTileK;
#pragma unroll
        for (int i = 0; i < kTileM / 16; ++i) {
            const bool in = m0 + r0 + 16 * i < M;
            cp_async16(d + 2048 * i, in ? Ap + (size_t)(16 * i) * p.lda + k0 : p.A, in);
        }
    };
    const auto load_b = [&](int kb) {
        const uint32_t d = sbase + (uint32_t)((kb % kStages) * kStage) + s0 + kTileM * 128;
        const int k0 = kb * kTileK;
#pragma unroll
        for (int i = 0; i < kNt / 16; ++i) {
            const bool in = r0 + 16 * i < nt;
            cp_async16(d + 2048 * i, in ? Bp + (size_t)(16 * i) * p.ldb + k0 : p.B, in);
        }
    };
    // the first stages; weights are copied while the previous kernel still runs
    pdl_launch_next();
    if (p.b_ready)
        for (int kb = 0; kb < min(kStages - 1, kb_n); ++kb) load_b(kb);
    pdl_wait_previous();
#pragma unroll
    for (int kb = 0; kb < kStages - 1; ++kb) {
        if (kb < kb_n) {
            load_a(kb);
            if (!p.b_ready) load_b(kb);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_slot;
    const uint32_t idesc = idesc_bf16(nt);

    bool bad = false, failed = false;
    int issued = 0;                        // K blocks whose products were committed
    for (int kb = 0; kb < kb_n; ++kb) {
        cp_async_wait<kStages - 2>();      // this thread's part of stage kb has landed
        fence_proxy_async();
        if (__syncthreads_or(bad)) {
            failed = true;
            break;
        }
        const int st = kb % kStages;
        if (tid == 0) {
            fence_after();
            const uint32_t sa = sbase + (uint32_t)(st * kStage), sb = sa + kTileM * 128;
#pragma unroll
            for (int kk = 0; kk < kTileK / 16; ++kk)
                mma_bf16(tmem, sw128_desc(sa + 32 * kk), sw128_desc(sb + 32 * kk), idesc,
                         (kb > 0 || kk > 0) ? 1u : 0u);
            mma_commit(smem_u32(&mbar[st]));
        }
        issued = kb + 1;
        // stage kb - 1 is refilled with block kb - 1 + kStages once its products are done
        const int next = kb + kStages - 1;
        if (next < kb_n) {
            if (kb > 0)
                bad = !mbar_wait(smem_u32(&mbar[(kb - 1) % kStages]),
                                 (uint32_t)(((kb - 1) / kStages) & 1));
            if (!bad) {
                load_a(next);
                load_b(next);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    cp_async_wait<0>();
    if (!failed) {
        bad = !mbar_wait(smem_u32(&mbar[(kb_n - 1) % kStages]),
                         (uint32_t)(((kb_n - 1) / kStages) & 1));
        fence_after();
        failed = __syncthreads_or(bad);
    }
    if (failed) {
        if (tid == 0) atomicExch(g.err, 1);
        // the products in flight, bounded (the last commit covers them all)
        if (issued > 0)
            mbar_wait(smem_u32(&mbar[(issued - 1) % kStages]),
                      (uint32_t)(((issued - 1) / kStages) & 1));
    } else {
        // epilogue: thread = row m0 + 32 warp + lane
        const int row = m0 + 32 * warp + lane;
        const bool live = row < M;
        const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
        for (int c0 = 0; c0 < nt; c0 += 32) {
            float v[32];
            tmem_ld32(trow + (uint32_t)c0, v);
            const int nb = n0 + c0;
            if (nb >= ep.n_valid) continue;
            if (ep.bias) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += ep.bias[nb + j];
            }
            if (ep.relu) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j], 0.f);
            }
            if (ep.mask && live) {
                const uint4 *mp = reinterpret_cast<const uint4 *>(ep.mask + (size_t)row * ep.ldm + nb);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 m4 = mp[q];
                    const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        // (a BF16 is the upper half of an FP32)
                        if (!(__uint_as_float(mw[h] << 16) > 0.f)) v[8 * q + 2 * h] = 0.f;
                        if (!(__uint_as_float(mw[h] & 0xffff0000u) > 0.f)) v[8 * q + 2 * h + 1] = 0.f;
                    }
                }
            }
            if (live && ep.c_f32) {
                float4 *o = reinterpret_cast<float4 *>(ep.c_f32 + (size_t)row * ep.ldc + nb);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float4 w = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    if (ep.scale) {
                        w.x = ep.shift[nb + 4 * j] + ep.scale[nb + 4 * j] * w.x;
                        w.y = ep.shift[nb + 4 * j + 1] + ep.scale[nb + 4 * j + 1] * w.y;
                        w.z = ep.shift[nb + 4 * j + 2] + ep.scale[nb + 4 * j + 2] * w.z;
                        w.w = ep.shift[nb + 4 * j + 3] + ep.scale[nb + 4 * j + 3] * w.w;
                    }
                    o[j] = w;
                }
            }
            if (ep.c_bf16 || ep.c_bf16_t) {
                uint32_t h[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                    h[j] = *reinterpret_cast<const uint32_t *>(&b2);
                }
                if (live && ep.c_bf16) {
                    uint4 *o = reinterpret_cast<uint4 *>(ep.c_bf16 + (size_t)row * ep.ldh + nb);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        o[j] = make_uint4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
                }
                if (ep.c_bf16_t && row < ep.t_rows) {
                    unsigned short *o = reinterpret_cast<unsigned short *>(ep.c_bf16_t) +
                                        (size_t)nb * ep.ldt + row;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        o[(size_t)j * ep.ldt] =
                            live ? (unsigned short)(h[j >> 1] >> (16 * (j & 1))) : (unsigned short)0;
                }
            }
            if (ep.col_sums) {
                // lane l ends with the sum of column nb + l over the warp's 32 rows:
                // at each step a lane keeps the half of its columns named by its bit
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = live ? v[j] : 0.f;
#pragma unroll
                for (int d = 16; d > 0; d >>= 1)
#pragma unroll
                    for (int j = 0; j < d; ++j) {
                        const float keep = (lane & d) ? v[j + d] : v[j];
                        const float give = (lane & d) ? v[j] : v[j + d];
                        v[j] = keep + __shfl_xor_sync(0xffffffffu, give, d);
                    }
                csum[warp][c0 + lane] = v[0];
            }
        }
        if (ep.col_sums) {
            __syncthreads();
            for (int c = tid; c < nt; c += kThreads)
                ep.col_sums[(size_t)mt * p.N + n0 + c] =
                    (csum[0][c] + csum[1][c]) + (csum[2][c] + csum[3][c]);
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :
                     : "r"(tmem), "r"(kCols)
                     : "memory");
    }
}

}  // namespace tc
}  // namespace fil
