// Per-filament warm-start MLP (include/fil_mlp.h): inference and training on
// the tensor cores (tc_gemm.cuh), FP32 master weights with Adam.
//
// Layer l maps in_l -> out_l: (800 padded to 832) -> 256 -> 256 -> 256 -> 192.
// Forward (rows = batch b):
//   X^  = BF16((x - in_mean) / in_std)                 [B x 832] (+ transposed)
//   H_l = BF16(relu(H_{l-1} W_l^T + b_l)), l = 1..3     [B x 256] (+ transposed)
//   Y^  = H_3 W_4^T + b_4 (FP32)                        [B x 192]
// Backward of L = sum (Y^ - T^)^2 / (2B):
//   dY = (Y^ - T^) / B;  dH_3 = (dY W_4) * [H_3 > 0];  dH_{l-1} = (dH_l W_l) * [H_{l-1} > 0]
//   dW_l = dZ_l^T H_{l-1} (K = batch), db_l = column sums of dZ_l (FP32)
// Every product is C = A . B^T with both operands K-major: the weights are
// kept in BF16 both as [out x in] and transposed, and activations and
// gradients are stored both row-major and transposed by the GEMM epilogues.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "../../include/fil_mlp.h"
#include "tc_gemm.cuh"

using bf16 = __nv_bfloat16;

namespace fil {
namespace {

constexpr int kLayers = 4;
constexpr int kIn = FIL_MLP_IN, kInP = (FIL_MLP_IN + 63) / 64 * 64, kHid = FIL_MLP_HIDDEN, kOut = FIL_MLP_OUT;
constexpr int kDimIn[kLayers] = {kIn, kHid, kHid, kHid};
constexpr int kDimInP[kLayers] = {kInP, kHid, kHid, kHid};
constexpr int kDimOut[kLayers] = {kHid, kHid, kHid, kOut};

// offsets of W_l and b_l in the packed parameter vector
struct Offsets {
    int64_t w[kLayers], b[kLayers];
};
Offsets param_offsets() {
    Offsets o;
    int64_t p = 0;
    for (int l = 0; l < kLayers; ++l) {
        o.w[l] = p;
        p += (int64_t)kDimOut[l] * kDimIn[l];
        o.b[l] = p;
        p += kDimOut[l];
    }
    return o;
}

int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

tc::Epilogue epi() {
    tc::Epilogue e{};
    e.n_valid = 1 << 30;
    return e;
}

tc::Problem product(const bf16 *A, int lda, const bf16 *B, int ldb, int M, int N, int K,
                    const tc::Epilogue &ep, bool weights = false) {
    return tc::Problem{A, B, lda, ldb, M, N, K, 0, 0, weights ? 1 : 0, ep};
}

// A launch whose prologue may overlap the kernel before it in the stream (both
// call pdl_wait_previous / pdl_launch_next): the calls are chains of 5 and 11
// kernels of a few microseconds, and each gap between two costs about as much.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem,
                       cudaStream_t st, Args &&...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <int kNt>
cudaError_t launch_gemm(const tc::Batch &b, int64_t ctas, cudaStream_t st) {
    const cudaError_t e = cudaFuncSetAttribute(tc::gemm_bf16_kernel<kNt>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               tc::smem_bytes(kNt));
    if (e != cudaSuccess) return e;
    return launch_pdl(tc::gemm_bf16_kernel<kNt>, dim3((unsigned)ctas), tc::kThreads,
                      tc::smem_bytes(kNt), st, b);
}

// The products of a batch in one launch.
cudaError_t gemm(tc::Batch &b, int sms, cudaStream_t st) {
    const int64_t ctas = tc::plan(b, sms);
    if (ctas > 0x7fffffff) return cudaErrorInvalidValue;
    switch (b.nt) {
        case 32: return launch_gemm<32>(b, ctas, st);
        case 64: return launch_gemm<64>(b, ctas, st);
        case 128: return launch_gemm<128>(b, ctas, st);
        default: return launch_gemm<256>(b, ctas, st);
    }
}

// Batch rows per CTA of the input and loss kernels, which give a thread one
// column: its 32 rows are 64 contiguous bytes of the transposed BF16 copy.
constexpr int kRows = 32;
constexpr int kInThreads = kInP / 4;     // four CTAs across the padded inputs
static_assert(kInP % 4 == 0 && kInThreads <= 1024, "input kernel covers the padded inputs");

// Thread c's column of the transposed copy, batch rows b0 .. b0 + 31, written up
// to row `rows` (a multiple of 8).
__device__ __forceinline__ void store_column(bf16 *t, int64_t b0, int64_t rows,
                                             const uint32_t (&h)[kRows / 2]) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (b0 + 8 * j < rows)
            reinterpret_cast<uint4 *>(t + b0)[j] =
                make_uint4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
}

// x^ = (x - mean) / std in BF16, row-major [B x kInP] (zero padding) and, for
// training, transposed [kInP x ldt] with columns B .. Kb - 1 zero.
__global__ void __launch_bounds__(kInThreads)
input_kernel(const float *__restrict__ x, int64_t B, const float *__restrict__ mean,
             const float *__restrict__ stdv, bf16 *__restrict__ X, bf16 *__restrict__ Xt,
             int64_t ldt, int64_t Kb) {
    tc::pdl_launch_next();
    // (one dimension, the only one with more than 65 535 blocks. Addresses are a base a
    // thread and small offsets: with the 64-bit row index in each of them the kernel took
    // 100 registers and a forward pass of 100 000 rows 545 us; 55 and 483 in this form)
    const int c = (int)(blockIdx.x % 4) * kInThreads + threadIdx.x;
    const int64_t b0 = (int64_t)(blockIdx.x / 4) * kRows;
    const int rows = (int)min((int64_t)kRows, B - b0);       // (0 or less: padding only)
    const float *xp = x + b0 * kIn + c;
    bf16 *Xp = X + b0 * kInP + c;
    const bool in = c < kIn;
    const float mu = in ? mean[c] : 0.f, sd = in ? stdv[c] : 1.f;
    float v[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
        v[r] = in && r < rows ? xp[r * kIn] : mu;
    uint32_t h[kRows / 2];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const bf16 q = __float2bfloat16_rn((v[r] - mu) / sd);
        const uint32_t bits = r < rows ? *reinterpret_cast<const unsigned short *>(&q) : 0u;
        if (r & 1) h[r >> 1] |= bits << 16;
        else h[r >> 1] = bits;
        if (r < rows) Xp[r * kInP] = q;
    }
    if (Xt) store_column(Xt + (int64_t)c * ldt, b0, Kb, h);
}

// y = mean + std y^ (an output array the last product cannot store to).
__global__ void output_kernel(const float *__restrict__ yhat, int64_t n, const float *__restrict__ mean,
                              const float *__restrict__ stdv, float *__restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % kOut);
    y[i] = mean[c] + stdv[c] * yhat[i];
}

// dY = (y^ - t^) / B in BF16 (row-major, and transposed with columns B .. Kb - 1
// zero), its FP32 column sums over each CTA's 32 rows, and each CTA's part of
// the loss: squares and their sum in float-float (TwoSum), FP64 once per thread
// (one CTA over the whole batch in FP64 took 234 us at 1024 rows). Where a square or
// the sum would leave FP32's range (or is infinite or NaN), and where the squares'
// rounding errors would, a thread sums its squares in FP64.
constexpr float kSquareMax = 1e38f, kSquareMin = 1e-12f;
constexpr int kLossThreads = kOut;

// hi + lo += x, the error of the addition (TwoSum) into lo.
__device__ __forceinline__ void add_two(float &hi, float &lo, float x) {
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
}

__global__ void __launch_bounds__(kLossThreads)
loss_kernel(const float *__restrict__ yhat, const float *__restrict__ t, int64_t B,
            const float *__restrict__ mean, const float *__restrict__ stdv, bf16 *__restrict__ dY,
            bf16 *__restrict__ dYt, int64_t ldt, int64_t Kb, float *__restrict__ col_sums,
            double *__restrict__ part, int n_part) {
    __shared__ double red[kLossThreads / 32];
    tc::pdl_launch_next();
    tc::pdl_wait_previous();
    const int c = threadIdx.x;
    const int64_t b0 = (int64_t)blockIdx.x * kRows;
    const float inv = 1.f / (float)B, mu = mean[c], sd = stdv[c];
    float y[kRows], g[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const bool in = b0 + r < B;
        y[r] = in ? yhat[(b0 + r) * kOut + c] : 0.f;
        g[r] = in ? t[(b0 + r) * kOut + c] : mu;
    }
    float hi = 0.f, lo = 0.f, sum = 0.f, sum_lo = 0.f, most = 0.f;
    uint32_t h[kRows / 2];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const bool in = b0 + r < B;
        const float d = in ? y[r] - (g[r] - mu) / sd : 0.f;
        most = fmaxf(most, fabsf(d));
        const float sq = __fmul_rn(d, d);
        add_two(hi, lo, sq);
        lo = __fadd_rn(lo, __fmaf_rn(d, d, -sq));
        const float gr = d * inv;
        add_two(sum, sum_lo, gr);
        const bf16 q = __float2bfloat16_rn(gr);
        const uint32_t bits = in ? *reinterpret_cast<const unsigned short *>(&q) : 0u;
        if (r & 1) h[r >> 1] |= bits << 16;
        else h[r >> 1] = bits;
        if (in) dY[(b0 + r) * kOut + c] = q;
    }
    store_column(dYt + (int64_t)c * ldt, b0, Kb, h);
    if ((int)blockIdx.x >= n_part) return;      // rows of the zero padding only
    col_sums[(int64_t)blockIdx.x * kOut + c] = __fadd_rn(sum, sum_lo);
    double acc = 0.5 * ((double)hi + (double)lo);
    if (!(hi < kSquareMax && (most > kSquareMin || most == 0.f))) {
        acc = 0.0;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const double d = b0 + r < B ? (double)(y[r] - (g[r] - mu) / sd) : 0.0;
            acc = fma(0.5 * d, d, acc);
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    if ((c & 31) == 0) red[c >> 5] = acc;
    __syncthreads();
    if (c == 0) {
        for (int w = 1; w < kLossThreads / 32; ++w) acc += red[w];
        part[blockIdx.x] = acc;
    }
}

// db_l[c] = sum of the column sums' parts (l < 3: one per row tile of the
// product that formed dZ_l; l = 3: one per CTA of the loss kernel), and the
// loss. Parts in order, compensated (TwoSum), eight loads in flight.
struct BiasParts {
    const float *p[kLayers];
    int n[kLayers];
    float *db[kLayers];
};
__global__ void finish_kernel(BiasParts bp, const double *__restrict__ part, int n_part, double B,
                              float *__restrict__ loss) {
    tc::pdl_wait_previous();
    const int l = blockIdx.y, c = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = l < 3 ? kHid : kOut;
    if (c < N) {
        float s = 0.f, lo = 0.f;
        const float *p = bp.p[l] + c;
#pragma unroll 8
        for (int i = 0; i < bp.n[l]; ++i) add_two(s, lo, p[(int64_t)i * N]);
        bp.db[l][c] = __fadd_rn(s, lo);
    }
    if (l == 0 && blockIdx.x == 0 && threadIdx.x < 32) {
        double a = 0.0;
        for (int i = threadIdx.x; i < n_part; i += 32) a += part[i];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
        if (threadIdx.x == 0) *loss = (float)(a / B);
    }
}

// BF16 copies of W_l: [out x inP] (zero-padded columns) and [inP x out].
__global__ void pack_weights_kernel(const float *__restrict__ w, int out, int in, int inP,
                                    bf16 *__restrict__ W, bf16 *__restrict__ Wt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)out * inP) return;
    const int o = (int)(i / inP), c = (int)(i - (int64_t)o * inP);
    const bf16 h = __float2bfloat16_rn(c < in ? w[(int64_t)o * in + c] : 0.f);
    W[i] = h;
    Wt[(int64_t)c * out + o] = h;
}

__global__ void adam_kernel(int64_t n, const float *__restrict__ g, float *__restrict__ p,
                            float *__restrict__ m, float *__restrict__ v, float lr, float c1,
                            float c2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

__device__ int g_tc_err;   // wait-limit flag of the standalone GEMM entry point

int device_sms() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n;
}

bool dev_ptr(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace fil

using namespace fil;

struct fil_mlp {
    cudaStream_t stream;
    int sms;                         // of the device it was created on
    int64_t max_batch, ldt;          // ldt: padded batch (K of the weight gradients)
    Offsets off;
    float *params, *grad, *adam_m, *adam_v;
    int64_t adam_t;
    bf16 *W[kLayers], *Wt[kLayers];
    float *in_mean, *in_std, *out_mean, *out_std;
    bf16 *X, *Xt, *H[3], *Ht[3], *dY, *dYt, *dH[3], *dHt[3];
    float *Y;
    float *sums[kLayers];            // column sums of dZ_l, by row tile (l < 3) or loss CTA
    double *loss_part;               // per loss CTA
    float *loss;                     // followed by err: read back together
    int *err;
    void *arena;
};

namespace {

struct Carver {
    char *base;
    size_t used = 0;
    template <typename T>
    T *take(size_t n) {
        size_t off = (used + 255) & ~(size_t)255;
        used = off + n * sizeof(T);
        return base ? reinterpret_cast<T *>(base + off) : nullptr;
    }
};

void carve(fil_mlp *m, Carver &c) {
    const int64_t B = m->max_batch, T = m->ldt;
    m->params = c.take<float>(FIL_MLP_NPARAM);
    m->grad = c.take<float>(FIL_MLP_NPARAM);
    m->adam_m = c.take<float>(FIL_MLP_NPARAM);
    m->adam_v = c.take<float>(FIL_MLP_NPARAM);
    for (int l = 0; l < kLayers; ++l) {
        m->W[l] = c.take<bf16>((size_t)kDimOut[l] * kDimInP[l]);
        m->Wt[l] = c.take<bf16>((size_t)kDimOut[l] * kDimInP[l]);
    }
    m->in_mean = c.take<float>(kIn);
    m->in_std = c.take<float>(kIn);
    m->out_mean = c.take<float>(kOut);
    m->out_std = c.take<float>(kOut);
    m->X = c.take<bf16>((size_t)B * kInP);
    m->Xt = c.take<bf16>((size_t)kInP * T);
    for (int l = 0; l < 3; ++l) {
        m->H[l] = c.take<bf16>((size_t)B * kHid);
        m->Ht[l] = c.take<bf16>((size_t)kHid * T);
        m->dH[l] = c.take<bf16>((size_t)B * kHid);
        m->dHt[l] = c.take<bf16>((size_t)kHid * T);
    }
    m->dY = c.take<bf16>((size_t)B * kOut);
    m->dYt = c.take<bf16>((size_t)kOut * T);
    m->Y = c.take<float>((size_t)B * kOut);
    for (int l = 0; l < 3; ++l)
        m->sums[l] = c.take<float>((size_t)((B + tc::kTileM - 1) / tc::kTileM) * kHid);
    m->sums[3] = c.take<float>((size_t)((B + kRows - 1) / kRows) * kOut);
    m->loss_part = c.take<double>((size_t)((B + kRows - 1) / kRows));
    m->loss = c.take<float>(2);
    m->err = m->loss ? reinterpret_cast<int *>(m->loss + 1) : nullptr;
}

const float *to_device(fil_mlp *m, const float *p, size_t n, float *scratch, cudaError_t &e) {
    if (dev_ptr(p)) return p;
    e = cudaMemcpyAsync(scratch, p, n * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    return scratch;
}

cudaError_t refresh_weights(fil_mlp *m) {
    for (int l = 0; l < kLayers; ++l) {
        const int64_t n = (int64_t)kDimOut[l] * kDimInP[l];
        pack_weights_kernel<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(
            m->params + m->off.w[l], kDimOut[l], kDimIn[l], kDimInP[l], m->W[l], m->Wt[l]);
    }
    return cudaGetLastError();
}

cudaError_t one_product(fil_mlp *m, const tc::Problem &p) {
    tc::Batch b{};
    b.p[0] = p;
    b.count = 1;
    b.err = m->err;
    return gemm(b, m->sms, m->stream);
}

// Forward pass on normalised inputs; `train` also writes the transposed
// activations, `y` (FP32, 16-byte aligned) takes the outputs in raw units;
// without it m->Y takes the normalised ones.
cudaError_t forward(fil_mlp *m, const float *x, int64_t B, bool train, float *y) {
    const int64_t Kb = round_up(B, tc::kTileK);
    const dim3 grid(4 * (unsigned)(((train ? Kb : B) + kRows - 1) / kRows));
    input_kernel<<<grid, kInThreads, 0, m->stream>>>(x, B, m->in_mean, m->in_std, m->X,
                                                     train ? m->Xt : nullptr, m->ldt, Kb);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bf16 *act = m->X;
    int ld = kInP;
    for (int l = 0; l < 3; ++l) {
        tc::Epilogue ep = epi();
        ep.c_bf16 = m->H[l];
        ep.ldh = kHid;
        if (train) {
            ep.c_bf16_t = m->Ht[l];
            ep.ldt = (int)m->ldt;
            ep.t_rows = (int)Kb;
        }
        ep.bias = m->params + m->off.b[l];
        ep.relu = 1;
        e = one_product(m, product(act, ld, m->W[l], kDimInP[l], (int)B, kHid, kDimInP[l], ep,
                                   true));
        if (e != cudaSuccess) return e;
        act = m->H[l];
        ld = kHid;
    }
    tc::Epilogue ep = epi();
    ep.c_f32 = y ? y : m->Y;
    ep.ldc = kOut;
    ep.bias = m->params + m->off.b[3];
    if (y) {
        ep.shift = m->out_mean;
        ep.scale = m->out_std;
    }
    return one_product(m, product(act, ld, m->W[3], kHid, (int)B, kOut, kHid, ep, true));
}

// Outputs in raw units to y: straight from the last product where its 16-byte
// stores may (y aligned), through m->Y otherwise.
cudaError_t forward_raw(fil_mlp *m, const float *x, float *y, int64_t B) {
    const bool direct = (reinterpret_cast<uintptr_t>(y) & 15) == 0;
    cudaError_t e = forward(m, x, B, false, direct ? y : nullptr);
    if (e == cudaSuccess && !direct) {
        const int64_t n = B * kOut;
        output_kernel<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(m->Y, n, m->out_mean,
                                                                          m->out_std, y);
        e = cudaGetLastError();
    }
    return e;
}

// Loss and gradient into `grad` (16-byte aligned); the loss (device) in m->loss.
// Eleven launches: the input, four forward products, the loss, the three products
// that carry dZ back, all four weight gradients in one, and the bias gradients.
cudaError_t gradients(fil_mlp *m, const float *x, const float *t, int64_t B, float *grad) {
    const int64_t Kb = round_up(B, tc::kTileK);
    cudaError_t e = forward(m, x, B, true, nullptr);
    if (e != cudaSuccess) return e;
    const int loss_ctas = (int)((Kb + kRows - 1) / kRows);
    const int loss_parts = (int)((B + kRows - 1) / kRows);
    e = launch_pdl(loss_kernel, dim3((unsigned)loss_ctas), kLossThreads, 0, m->stream,
                   (const float *)m->Y, t, B, (const float *)m->out_mean, (const float *)m->out_std,
                   m->dY, m->dYt, m->ldt, Kb, m->sums[3], m->loss_part, loss_parts);
    if (e != cudaSuccess) return e;
    // dH_{l-1} = (dZ_l W_l) * [H_{l-1} > 0], with its column sums
    const bf16 *dZ = m->dY;
    int ldz = kOut;
    for (int l = 3; l > 0; --l) {
        tc::Epilogue eb = epi();
        eb.c_bf16 = l > 1 ? m->dH[l - 1] : nullptr;
        eb.ldh = kHid;
        eb.c_bf16_t = m->dHt[l - 1];
        eb.ldt = (int)m->ldt;
        eb.t_rows = (int)Kb;
        eb.mask = m->H[l - 1];
        eb.ldm = kHid;
        eb.col_sums = m->sums[l - 1];
        e = one_product(m, product(dZ, ldz, m->Wt[l], kDimOut[l], (int)B, kHid, kDimOut[l], eb,
                                   true));
        if (e != cudaSuccess) return e;
        dZ = m->dH[l - 1];
        ldz = kHid;
    }
    // dW_l = dZ_l^T H_{l-1} (H_{-1}: the inputs)
    tc::Batch b{};
    b.count = kLayers;
    b.err = m->err;
    for (int l = 0; l < kLayers; ++l) {
        tc::Epilogue eg = epi();
        eg.c_f32 = grad + m->off.w[l];
        eg.ldc = kDimIn[l];
        eg.n_valid = kDimIn[l];
        b.p[l] = product(l == 3 ? m->dYt : m->dHt[l], (int)m->ldt, l > 0 ? m->Ht[l - 1] : m->Xt,
                         (int)m->ldt, kDimOut[l], kDimInP[l], (int)Kb, eg);
    }
    e = gemm(b, m->sms, m->stream);
    if (e != cudaSuccess) return e;
    BiasParts bp;
    for (int l = 0; l < kLayers; ++l) {
        bp.p[l] = m->sums[l];
        bp.n[l] = l < 3 ? (int)((B + tc::kTileM - 1) / tc::kTileM) : loss_parts;
        bp.db[l] = grad + m->off.b[l];
    }
    return launch_pdl(finish_kernel, dim3(kHid / 64, kLayers), 64, 0, m->stream, bp,
                      (const double *)m->loss_part, loss_parts, (double)B, m->loss);
}

// Waits for the stream; FIL_ECUDA if a wait in a product ran out. The loss, when
// asked for, comes back with the same copy.
fil_status finish_call(fil_mlp *m, float *loss) {
    struct {
        float loss;
        int err;
    } h;
    static_assert(sizeof(h) == 8, "loss and err are adjacent");
    if (cudaMemcpyAsync(&h, m->loss, sizeof(h), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return FIL_ECUDA;
    if (loss) *loss = h.loss;
    return h.err ? FIL_ECUDA : FIL_OK;
}

}  // namespace

namespace fil {

cudaError_t mlp_forward_async(fil_mlp *m, const float *x, float *y, int64_t batch,
                              cudaStream_t st, int64_t *launches) {
    const cudaStream_t own = m->stream;
    m->stream = st;
    const cudaError_t e = forward_raw(m, x, y, batch);
    m->stream = own;
    if (launches) *launches += 5;
    return e;
}

int64_t mlp_max_batch(const fil_mlp *m) { return m->max_batch; }

}  // namespace fil

extern "C" {

fil_status fil_mlp_create(int64_t max_batch, void *stream, fil_mlp **out) {
    if (!out || max_batch < 1 || max_batch > (1 << 24)) return FIL_EINVAL;
    *out = nullptr;
    fil_mlp *m = new fil_mlp();
    m->stream = (cudaStream_t)stream;
    m->max_batch = max_batch;
    m->ldt = round_up(max_batch, tc::kTileK);
    m->off = param_offsets();
    m->sms = device_sms();
    Carver sizing{nullptr};
    carve(m, sizing);
    if (cudaMalloc(&m->arena, sizing.used) != cudaSuccess) {
        cudaGetLastError();
        delete m;
        return FIL_ENOMEM;
    }
    Carver c{static_cast<char *>(m->arena)};
    carve(m, c);
    cudaError_t e = cudaMemsetAsync(m->arena, 0, sizing.used, m->stream);
    std::vector<float> ones(std::max(kIn, kOut), 1.f);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->in_std, ones.data(), kIn * sizeof(float), cudaMemcpyHostToDevice,
                            m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->out_std, ones.data(), kOut * sizeof(float), cudaMemcpyHostToDevice,
                            m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        cudaFree(m->arena);
        delete m;
        return FIL_ECUDA;
    }
    *out = m;
    return FIL_OK;
}

void fil_mlp_destroy(fil_mlp *m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->arena);
    delete m;
}

fil_status fil_mlp_set_params(fil_mlp *m, const float *params) {
    if (!m || !params) return FIL_EINVAL;
    cudaError_t e = cudaSuccess;
    const float *p = to_device(m, params, FIL_MLP_NPARAM, m->params, e);
    if (e == cudaSuccess && p != m->params)
        e = cudaMemcpyAsync(m->params, p, FIL_MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToDevice,
                            m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->adam_m, 0, FIL_MLP_NPARAM * sizeof(float), m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->adam_v, 0, FIL_MLP_NPARAM * sizeof(float), m->stream);
    m->adam_t = 0;
    if (e == cudaSuccess) e = refresh_weights(m);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? FIL_OK : FIL_ECUDA;
}

fil_status fil_mlp_get_params(fil_mlp *m, float *params) {
    if (!m || !params) return FIL_EINVAL;
    cudaError_t e = cudaMemcpyAsync(params, m->params, FIL_MLP_NPARAM * sizeof(float),
                                    cudaMemcpyDefault, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? FIL_OK : FIL_ECUDA;
}

fil_status fil_mlp_set_norm(fil_mlp *m, const float *in_mean, const float *in_std,
                            const float *out_mean, const float *out_std) {
    if (!m || !in_mean || !in_std || !out_mean || !out_std) return FIL_EINVAL;
    cudaError_t e = cudaMemcpyAsync(m->in_mean, in_mean, kIn * sizeof(float), cudaMemcpyDefault,
                                    m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->in_std, in_std, kIn * sizeof(float), cudaMemcpyDefault, m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->out_mean, out_mean, kOut * sizeof(float), cudaMemcpyDefault,
                            m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->out_std, out_std, kOut * sizeof(float), cudaMemcpyDefault, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? FIL_OK : FIL_ECUDA;
}

fil_status fil_mlp_forward(fil_mlp *m, const float *x, float *y, int64_t batch) {
    if (!m || !x || !y || batch < 1 || batch > m->max_batch) return FIL_EINVAL;
    if (!dev_ptr(x) || !dev_ptr(y)) return FIL_EINVAL;
    if (forward_raw(m, x, y, batch) != cudaSuccess) return FIL_ECUDA;
    return finish_call(m, nullptr);
}

fil_status fil_mlp_gradients(fil_mlp *m, const float *x, const float *target, int64_t batch,
                             float *grad, float *loss) {
    if (!m || !x || !target || !grad || batch < 1 || batch > m->max_batch) return FIL_EINVAL;
    if (!dev_ptr(x) || !dev_ptr(target) || !dev_ptr(grad)) return FIL_EINVAL;
    // (the products store 16 bytes at a time)
    const bool direct = (reinterpret_cast<uintptr_t>(grad) & 15) == 0;
    cudaError_t e = gradients(m, x, target, batch, direct ? grad : m->grad);
    if (e == cudaSuccess && !direct)
        e = cudaMemcpyAsync(grad, m->grad, FIL_MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToDevice,
                            m->stream);
    if (e != cudaSuccess) return FIL_ECUDA;
    return finish_call(m, loss);
}

fil_status fil_mlp_train_step(fil_mlp *m, const float *x, const float *target, int64_t batch,
                              float lr, float *loss) {
    if (!m || !x || !target || batch < 1 || batch > m->max_batch || !(lr > 0.f)) return FIL_EINVAL;
    if (!dev_ptr(x) || !dev_ptr(target)) return FIL_EINVAL;
    cudaError_t e = gradients(m, x, target, batch, m->grad);
    m->adam_t += 1;
    const float c1 = 1.f - std::pow(0.9f, (float)m->adam_t);
    const float c2 = 1.f - std::pow(0.999f, (float)m->adam_t);
    if (e == cudaSuccess) {
        adam_kernel<<<(FIL_MLP_NPARAM + 255) / 256, 256, 0, m->stream>>>(
            FIL_MLP_NPARAM, m->grad, m->params, m->adam_m, m->adam_v, lr, c1, c2);
        e = refresh_weights(m);
    }
    if (e != cudaSuccess) return FIL_ECUDA;
    return loss ? finish_call(m, loss) : FIL_OK;
}

fil_status fil_tc_gemm_bf16(const uint16_t *A, int64_t lda, const uint16_t *B, int64_t ldb,
                            float *C, int64_t ldc, int64_t M, int64_t N, int64_t K, void *stream) {
    if (!A || !B || !C || M < 1 || N < 32 || N % 32 || K < 64 || K % 64 || lda % 8 || ldb % 8 ||
        ldc % 4 || lda < K || ldb < K || ldc < N || M > (1 << 24) || N > (1 << 16) ||
        K > (1 << 24))
        return FIL_EINVAL;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) |
         reinterpret_cast<uintptr_t>(C)) & 15)
        return FIL_EINVAL;
    if (!dev_ptr(A) || !dev_ptr(B) || !dev_ptr(C)) return FIL_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int *err = nullptr;
    if (cudaGetSymbolAddress((void **)&err, g_tc_err) != cudaSuccess) return FIL_ECUDA;
    if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) return FIL_ECUDA;
    tc::Epilogue ep = epi();
    ep.c_f32 = C;
    ep.ldc = (int)ldc;
    tc::Batch b{};
    b.p[0] = product(reinterpret_cast<const bf16 *>(A), (int)lda, reinterpret_cast<const bf16 *>(B),
                     (int)ldb, (int)M, (int)N, (int)K, ep);
    b.count = 1;
    b.err = err;
    if (gemm(b, device_sms(), st) != cudaSuccess) return FIL_ECUDA;
    int h = 0;
    if (cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return FIL_ECUDA;
    return h ? FIL_ECUDA : FIL_OK;
}

}  // extern "C"
