// Surrogate of the tuning search (Sec. 4.4 tunes the method's hyper-parameters
// by scoring many configurations; a regression network trained on scores of
// full runs ranks candidates so that only the most promising ones are run).
//
// Network: 30 standardised inputs -> 256 ReLU -> 256 ReLU -> 1, trained with
// the mean squared error and Adam. FP32 master weights; every product reads
// the bfloat16 rounding of the weights and accumulates in FP32.
//
// Two passes per batch of B rows: the row pass (forward, dL/dz2, dL/dz1) and the
// weight pass (gradients as sums over the batch in row order, so they are
// deterministic). Training runs both, with Adam, for whole epochs in one
// cooperative launch; prediction is the row pass's forward alone.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "common.cuh"
#include "runtime.h"

namespace lne {

namespace {

constexpr int kIn = kSurrogateInputs;
constexpr int kHid = kSurrogateHidden;
constexpr int64_t kW1 = 0, kB1 = kW1 + kIn * kHid, kW2 = kB1 + kHid, kB2 = kW2 + kHid * kHid, kW3 = kB2 + kHid,
                  kB3 = kW3 + kHid;
static_assert(kB3 + 1 == kSurrogateParams, "parameter layout");

__device__ __forceinline__ float bf(__nv_bfloat16 x) { return __bfloat162float(x); }

// He-uniform initial weights (U(-a, a), a = sqrt(6 / fan_in)) from Philox
// (counter = parameter index, key = seed); zero biases.
__global__ void sur_init_kernel(float *__restrict__ w, uint32_t k0, uint32_t k1) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < kSurrogateParams;
         i += (int64_t)gridDim.x * blockDim.x) {
        float a = 0.f;
        if (i < kB1) a = sqrtf(6.0f / kIn);
        else if (i >= kW2 && i < kB2) a = sqrtf(6.0f / kHid);
        else if (i >= kW3 && i < kB3) a = sqrtf(6.0f / kHid);
        const u32x4 r = philox10(u32x4{(uint32_t)i, 0x5u, 0u, 0u}, k0, k1);
        const float u = ((float)(r.x >> 8) + 0.5f) * (1.0f / 16777216.0f);
        w[i] = (2.0f * u - 1.0f) * a;
    }
}

__global__ void sur_cast_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < kSurrogateParams;
         i += (int64_t)gridDim.x * blockDim.x)
        wb[i] = __float2bfloat16_rn(w[i]);
}

// Per-feature mean and population standard deviation (two passes, FP64, one
// CTA per feature, fixed-order reduction); std < 1e-6 becomes 1.
__global__ void __launch_bounds__(256) sur_scaling_kernel(const float *__restrict__ X, int64_t rows,
                                                          float *__restrict__ mean, float *__restrict__ std) {
    __shared__ double red[256];
    const int f = blockIdx.x, tid = threadIdx.x;
    double s = 0.0;
    for (int64_t r = tid; r < rows; r += blockDim.x) s += (double)X[r * kIn + f];
    red[tid] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (tid < h) red[tid] += red[tid + h];
        __syncthreads();
    }
    const double mu = red[0] / (double)rows;
    __syncthreads();
    double q = 0.0;
    for (int64_t r = tid; r < rows; r += blockDim.x) {
        const double d = (double)X[r * kIn + f] - mu;
        q += d * d;
    }
    red[tid] = q;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (tid < h) red[tid] += red[tid + h];
        __syncthreads();
    }
    if (tid == 0) {
        const double sd = sqrt(red[0] / (double)rows);
        mean[f] = (float)mu;
        std[f] = sd < 1e-6 ? 1.0f : (float)sd;
    }
}

// ---------------------------------------------------------------------------
// The row pass: forward, and in training dL/dz2 and dL/dz1, for groups of R
// rows. Rows are independent and a row's work is three dependent chains of 30,
// 256 and 256 FMAs, so a CTA takes few rows (enough CTAs to fill the GPU) and
// keeps the whole network in shared memory: W2 is copied in once with
// cp.async (rows padded to 264 entries), read by columns in the forward
// (two adjacent units a thread, one 4-byte load a k) and by rows in the
// backward (eight units of one row per 16-byte load, conflict-free by the
// padding). Each output is summed over k in ascending order from the bias.
// Measured: 256 rows (2 a CTA, 128 CTAs) 115 -> 8 us; the pass before it took
// 32 rows a CTA and one shared-memory load per FMA, which bound it.
// ---------------------------------------------------------------------------
constexpr int kThreads = 256;
constexpr int kW2Pitch = kHid + 8;                                  // bf16 entries
constexpr int kSmW1 = kHid * kW2Pitch * 2;                          // byte offsets in shared memory
constexpr int kSmVec = kSmW1 + (kIn * kHid + kHid) * 2;             // b2, w3
constexpr int kSmRows = kSmVec + 2 * kHid * 2;
static_assert(kThreads == kHid && kSmRows % 16 == 0, "thread j owns unit j; row buffers are 16-byte aligned");

// Shared-memory row buffers of a group of R rows (after the weights).
template <int R>
struct RowBufs {
    float *x, *h1, *h2, *dz2, *dys;
    __device__ explicit RowBufs(char *sm) {
        x = reinterpret_cast<float *>(sm + kSmRows);
        h1 = x + R * 32;
        h2 = h1 + R * kHid;
        dz2 = h2 + R * kHid;
        dys = dz2 + R * kHid;
    }
};
constexpr int rows_smem(int R, bool train) {
    return kSmRows + (R * 32 + (train ? 3 : 2) * R * kHid + (train ? R : 0)) * 4;
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float2 bf2(uint32_t w) {   // a bfloat16 is the upper half of the FP32 with its value
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// Starts the copies of the network into shared memory: five groups, W1 with
// the vectors and then W2 by quarters, so that layer 2 starts on the first.
__device__ __forceinline__ void load_network(char *sm, const __nv_bfloat16 *wb) {
    const int tid = threadIdx.x;
    const char *g = reinterpret_cast<const char *>(wb);
    constexpr int c1 = (kIn * kHid + kHid) * 2 / 16, c2 = 2 * kHid * 2 / 16;
    for (int e = tid; e < c1; e += kThreads) cp_async16(sm + kSmW1 + 16 * e, g + 16 * e);
    for (int e = tid; e < c2; e += kThreads) cp_async16(sm + kSmVec + 16 * e, g + kB2 * 2 + 16 * e);
    cp_async_commit();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {   // 64 rows of 32 16-byte chunks
            const int e = t * kThreads + tid, row = q * 64 + (e >> 5), ch = e & 31;
            cp_async16(sm + row * (kW2Pitch * 2) + 16 * ch, g + kW2 * 2 + row * (kHid * 2) + 16 * ch);
        }
        cp_async_commit();
    }
}

// acc[i] += in[i][k] (w[k][j], w[k][j + 1]) for k in [k0, k1), ascending;
// k1 - k0 is a multiple of 4. w points at column j, pitch in 32-bit words.
template <int RPT>
__device__ __forceinline__ void layer_chain(const uint32_t *w, int pitch, const float *in, int ld, int k0, int k1,
                                            float2 (&acc)[RPT]) {
#pragma unroll(RPT <= 4 ? 4 : 1)
    for (int k = k0; k < k1; k += 4) {
        const float2 w0 = bf2(w[k * pitch]), w1 = bf2(w[(k + 1) * pitch]), w2 = bf2(w[(k + 2) * pitch]),
                     w3 = bf2(w[(k + 3) * pitch]);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const float4 a = *reinterpret_cast<const float4 *>(in + i * ld + k);
            f2_add_prod(acc[i], make_float2(a.x, a.x), w0);
            f2_add_prod(acc[i], make_float2(a.y, a.y), w1);
            f2_add_prod(acc[i], make_float2(a.z, a.z), w2);
            f2_add_prod(acc[i], make_float2(a.w, a.w), w3);
        }
    }
}

struct RowArgs {
    const float *X, *t;           // inputs, targets (t: training only)
    const int32_t *idx;           // batch row -> X row (NULL: the same)
    int64_t B;                    // rows of the batch
    const float *mean, *std;
    const __nv_bfloat16 *wb;
    float *y;                     // [B]
    float *Xs, *H1, *H2;          // training: [B][32], [B][256], [B][256]
    float *dy, *dZ1, *dZ2;        // training: [B], [B][256], [B][256]
};

// Standardised inputs of rows r0 .. r0 + R - 1 into shared memory (zeros past
// the batch's end; columns 30 and 31 are zeros) and, in training, into Xs.
template <int R, bool TRAIN>
__device__ __forceinline__ void load_rows(const RowArgs &A, const RowBufs<R> &b, int64_t r0) {
    for (int e = threadIdx.x; e < R * 32; e += kThreads) {
        const int r = e >> 5, i = e & 31;
        float v = 0.f;
        if (r0 + r < A.B) {
            if (i < kIn) {
                const int64_t row = A.idx ? (int64_t)A.idx[r0 + r] : r0 + r;
                v = (A.X[row * kIn + i] - A.mean[i]) / A.std[i];
            }
            if (TRAIN) A.Xs[(r0 + r) * 32 + i] = v;
        }
        b.x[e] = v;
    }
}

// One group of R rows whose inputs are in shared memory (or being written by
// this CTA's threads). fresh: the network's copies are still in flight.
template <int R, bool TRAIN>
__device__ __forceinline__ void row_group(const RowArgs &A, char *sm, const RowBufs<R> &b, int64_t r0, bool fresh) {
    constexpr int RPT = R / 2;
    const int tid = threadIdx.x, half = tid >> 7, j = 2 * (tid & 127);
    const int nr = (int)imin64(R, A.B - r0);
    const __nv_bfloat16 *b1 = reinterpret_cast<const __nv_bfloat16 *>(sm + kSmW1) + kB1;
    const __nv_bfloat16 *b2 = reinterpret_cast<const __nv_bfloat16 *>(sm + kSmVec), *w3 = b2 + kHid;
    if (fresh) cp_async_wait<4>();
    __syncthreads();
    float2 acc[RPT];
    {
        const float2 bias = bf2(*reinterpret_cast<const uint32_t *>(b1 + j));
#pragma unroll
        for (int i = 0; i < RPT; ++i) acc[i] = bias;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(sm + kSmW1) + (j >> 1);
        const float *in = b.x + half * RPT * 32;
        layer_chain<RPT>(w, kHid / 2, in, 32, 0, 28, acc);
        static_assert(kIn == 30, "the last two inputs");
#pragma unroll
        for (int k = 28; k < kIn; ++k) {
            const float2 wk = bf2(w[k * (kHid / 2)]);
#pragma unroll
            for (int i = 0; i < RPT; ++i) f2_add_prod(acc[i], make_float2(in[i * 32 + k], in[i * 32 + k]), wk);
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = half * RPT + i;
            const float2 h = make_float2(fmaxf(acc[i].x, 0.f), fmaxf(acc[i].y, 0.f));
            *reinterpret_cast<float2 *>(b.h1 + r * kHid + j) = h;
            if (TRAIN && r < nr) *reinterpret_cast<float2 *>(A.H1 + (r0 + r) * kHid + j) = h;
        }
    }
    {
        const float2 bias = bf2(*reinterpret_cast<const uint32_t *>(b2 + j));
#pragma unroll
        for (int i = 0; i < RPT; ++i) acc[i] = bias;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(sm) + (j >> 1);
        const float *in = b.h1 + half * RPT * kHid;
        if (fresh) cp_async_wait<3>();
        __syncthreads();
        layer_chain<RPT>(w, kW2Pitch / 2, in, kHid, 0, 64, acc);
        if (fresh) {
            cp_async_wait<2>();
            __syncthreads();
        }
        layer_chain<RPT>(w, kW2Pitch / 2, in, kHid, 64, 128, acc);
        if (fresh) {
            cp_async_wait<1>();
            __syncthreads();
        }
        layer_chain<RPT>(w, kW2Pitch / 2, in, kHid, 128, 192, acc);
        if (fresh) {
            cp_async_wait<0>();
            __syncthreads();
        }
        layer_chain<RPT>(w, kW2Pitch / 2, in, kHid, 192, 256, acc);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = half * RPT + i;
            const float2 h = make_float2(fmaxf(acc[i].x, 0.f), fmaxf(acc[i].y, 0.f));
            *reinterpret_cast<float2 *>(b.h2 + r * kHid + j) = h;
            if (TRAIN && r < nr) *reinterpret_cast<float2 *>(A.H2 + (r0 + r) * kHid + j) = h;
        }
    }
    __syncthreads();
    // output: a warp per row, lanes over units, fixed shuffle tree. Training:
    // dy = 2 (y - t) / B
    const int warp = tid >> 5, lane = tid & 31;
    for (int r = warp; r < R; r += kThreads / 32) {
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < kHid / 32; ++t) s = fmaf(b.h2[r * kHid + lane + 32 * t], bf(w3[lane + 32 * t]), s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            // b3 is one entry past the staged vectors: read through L2, where
            // the training kernel's other CTAs update it
            const uint16_t raw = __ldcg(reinterpret_cast<const uint16_t *>(A.wb) + kB3);
            const float yr = s + __uint_as_float((uint32_t)raw << 16);
            if (r < nr) A.y[r0 + r] = yr;
            if (TRAIN) {
                float v = 0.f;
                if (r < nr) {
                    const int64_t row = A.idx ? (int64_t)A.idx[r0 + r] : r0 + r;
                    v = 2.0f * (yr - A.t[row]) / (float)A.B;
                    A.dy[r0 + r] = v;
                }
                b.dys[r] = v;
            }
        }
    }
    __syncthreads();
    if (!TRAIN) return;
    // dz2 = dy w3 [h2 > 0]; dz1 = (W2 dz2) [h1 > 0], thread k over row k of W2
    {
        const float w3j = bf(w3[tid]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float v = 0.f;
            if (r < nr && b.h2[r * kHid + tid] > 0.f) v = b.dys[r] * w3j;
            b.dz2[r * kHid + tid] = v;
            if (r < nr) A.dZ2[(r0 + r) * kHid + tid] = v;
        }
    }
    __syncthreads();
    float dz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) dz[r] = 0.f;
    const uint4 *wr = reinterpret_cast<const uint4 *>(sm + tid * (kW2Pitch * 2));
#pragma unroll 2
    for (int jj = 0; jj < kHid; jj += 8) {
        const uint4 q = wr[jj >> 3];
        const float2 w01 = bf2(q.x), w23 = bf2(q.y), w45 = bf2(q.z), w67 = bf2(q.w);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 lo = *reinterpret_cast<const float4 *>(b.dz2 + r * kHid + jj);
            const float4 hi = *reinterpret_cast<const float4 *>(b.dz2 + r * kHid + jj + 4);
            dz[r] = fmaf(lo.x, w01.x, dz[r]);
            dz[r] = fmaf(lo.y, w01.y, dz[r]);
            dz[r] = fmaf(lo.z, w23.x, dz[r]);
            dz[r] = fmaf(lo.w, w23.y, dz[r]);
            dz[r] = fmaf(hi.x, w45.x, dz[r]);
            dz[r] = fmaf(hi.y, w45.y, dz[r]);
            dz[r] = fmaf(hi.z, w67.x, dz[r]);
            dz[r] = fmaf(hi.w, w67.y, dz[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (r < nr) A.dZ1[(r0 + r) * kHid + tid] = b.h1[r * kHid + tid] > 0.f ? dz[r] : 0.f;
    __syncthreads();   // the next group rewrites the row buffers
}

template <int R, bool TRAIN>
__global__ void __launch_bounds__(kThreads, 1) sur_rows_kernel(RowArgs A) {
    extern __shared__ __align__(16) char sm[];
    const RowBufs<R> b(sm);
    load_network(sm, A.wb);
    bool fresh = true;
    for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < A.B; r0 += (int64_t)gridDim.x * R) {
        load_rows<R, TRAIN>(A, b, r0);
        row_group<R, TRAIN>(A, sm, b, r0, fresh);
        fresh = false;
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// The weight pass: gradients as sums over the batch in row order. 152 tiles,
// one CTA each: tiles 0..127 16 x 32 of dW2[k][j] = sum_r h1[r][k] dz2[r][j],
// tiles 128..143 the same of dW1[i][j] = sum_r x[r][i] dz1[r][j], tiles
// 144..151 32 columns of db1, db2 and dw3 (and db3). The tile's columns of the
// batch are staged in shared memory 256 rows at a time; four warps sum, a
// thread owning four adjacent entries (5 shared-memory wavefronts a row; two
// entries on each of eight warps: 16, and those bound the pass). `use(i, n, g)`
// takes the gradients g of parameters i .. i + n - 1 (n = 4 or 1), `fetch(i,
// n)` is called before the sums start.
// ---------------------------------------------------------------------------
constexpr int kWTiles = kHid / 16 * (kHid / 32) + 2 * (kHid / 32) + kHid / 32;
constexpr int kWChunk = 256;
constexpr int kWPitch = kWChunk + 4;   // floats a row of the transposed left operand
constexpr int kGradSmem = (3 * kWChunk * 32 + kWChunk) * 4;
static_assert((16 * kWPitch + kWChunk * 32) * 4 <= kGradSmem, "the matrix tiles' staging fits as well");

struct GradArgs {
    const float *Xs, *H1, *H2, *dy, *dZ1, *dZ2;
    int64_t B;
};

template <typename Fetch, typename Use>
__device__ __forceinline__ void weight_tile(const GradArgs &A, int tile, float *sm, Fetch fetch, Use use) {
    const int tid = threadIdx.x;
    if (tile < 144) {
        const bool l2 = tile < 128;
        const int t = l2 ? tile : tile - 128, k0 = (t >> 3) * 16, j0 = (t & 7) * 32;
        const float *P = l2 ? A.H1 : A.Xs, *D = l2 ? A.dZ2 : A.dZ1;
        const int ldp = l2 ? kHid : 32;
        float *ps = sm, *ds = sm + 16 * kWPitch;
        const int kk = tid >> 3, jq = 4 * (tid & 7);
        const bool sums = tid < 128, live = sums && (l2 || k0 + kk < kIn);
        const int64_t i = (l2 ? kW2 : kW1) + (int64_t)(k0 + kk) * kHid + j0 + jq;
        if (live) fetch(i, 4);
        float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
        for (int64_t c0 = 0; c0 < A.B; c0 += kWChunk) {
            const int nr = (int)imin64(kWChunk, A.B - c0);
            float4 p[4], d[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = q * kThreads + tid, r = e >> 2;
                if (r < nr) p[q] = __ldcg(reinterpret_cast<const float4 *>(P + (c0 + r) * ldp + k0) + (e & 3));
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = q * kThreads + tid, r = e >> 3;
                if (r < nr) d[q] = __ldcg(reinterpret_cast<const float4 *>(D + (c0 + r) * kHid + j0) + (e & 7));
            }
            __syncthreads();   // the last chunk's sums are done
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = q * kThreads + tid, r = e >> 2;
                if (r >= nr) continue;
                float *to = ps + 4 * (e & 3) * kWPitch + r;
                to[0] = p[q].x;
                to[kWPitch] = p[q].y;
                to[2 * kWPitch] = p[q].z;
                to[3 * kWPitch] = p[q].w;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = q * kThreads + tid;
                if ((e >> 3) < nr) reinterpret_cast<float4 *>(ds)[e] = d[q];
            }
            __syncthreads();
            if (sums) {
                const float *pk = ps + kk * kWPitch, *dj = ds + jq;
                auto add = [&](float pr, int r) {
                    const float4 x = *reinterpret_cast<const float4 *>(dj + r * 32);
                    f2_add_prod(acc0, make_float2(pr, pr), make_float2(x.x, x.y));
                    f2_add_prod(acc1, make_float2(pr, pr), make_float2(x.z, x.w));
                };
                int r = 0;
#pragma unroll 4
                for (; r + 4 <= nr; r += 4) {
                    const float4 pr = *reinterpret_cast<const float4 *>(pk + r);
                    add(pr.x, r);
                    add(pr.y, r + 1);
                    add(pr.z, r + 2);
                    add(pr.w, r + 3);
                }
                for (; r < nr; ++r) add(pk[r], r);
            }
        }
        if (live) use(i, 4, make_float4(acc0.x, acc0.y, acc1.x, acc1.y));
    } else {
        const int j0 = (tile - 144) * 32, warp = tid >> 5, lane = tid & 31;
        float *s1 = sm, *s2 = s1 + kWChunk * 32, *s3 = s2 + kWChunk * 32, *sy = s3 + kWChunk * 32;
        const bool live = warp < 3 || (warp == 3 && lane == 0 && j0 == 0);
        const int64_t i = warp == 0 ? kB1 + j0 + lane : warp == 1 ? kB2 + j0 + lane : warp == 2 ? kW3 + j0 + lane : kB3;
        if (live) fetch(i, 1);
        float s = 0.f;
        for (int64_t c0 = 0; c0 < A.B; c0 += kWChunk) {
            const int nr = (int)imin64(kWChunk, A.B - c0);
            float4 a[8], d[8], h[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = q * kThreads + tid, r = e >> 3;
                if (r >= nr) continue;
                const int64_t at = (c0 + r) * kHid + j0;
                a[q] = __ldcg(reinterpret_cast<const float4 *>(A.dZ1 + at) + (e & 7));
                d[q] = __ldcg(reinterpret_cast<const float4 *>(A.dZ2 + at) + (e & 7));
                h[q] = __ldcg(reinterpret_cast<const float4 *>(A.H2 + at) + (e & 7));
            }
            const float yv = tid < nr ? __ldcg(A.dy + c0 + tid) : 0.f;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = q * kThreads + tid;
                if ((e >> 3) >= nr) continue;
                reinterpret_cast<float4 *>(s1)[e] = a[q];
                reinterpret_cast<float4 *>(s2)[e] = d[q];
                reinterpret_cast<float4 *>(s3)[e] = h[q];
            }
            sy[tid] = yv;
            __syncthreads();
            if (warp == 0) {
#pragma unroll 8
                for (int r = 0; r < nr; ++r) s += s1[r * 32 + lane];
            } else if (warp == 1) {
#pragma unroll 8
                for (int r = 0; r < nr; ++r) s += s2[r * 32 + lane];
            } else if (warp == 2) {
#pragma unroll 8
                for (int r = 0; r < nr; ++r) s = fmaf(s3[r * 32 + lane], sy[r], s);
            } else if (warp == 3) {
#pragma unroll 8
                for (int r = 0; r < nr; ++r) s += sy[r];
            }
        }
        if (live) use(i, 1, make_float4(s, 0.f, 0.f, 0.f));
    }
}

__global__ void __launch_bounds__(kThreads) sur_weight_grad_kernel(GradArgs A, float *__restrict__ g) {
    extern __shared__ __align__(16) char sm[];
    for (int tile = blockIdx.x; tile < kWTiles; tile += gridDim.x) {
        weight_tile(A, tile, reinterpret_cast<float *>(sm), [](int64_t, int) {},
                    [&](int64_t i, int n, float4 gi) {
                        if (n == 4) *reinterpret_cast<float4 *>(g + i) = gi;
                        else g[i] = gi.x;
                    });
        __syncthreads();
    }
}

__device__ __forceinline__ uint32_t bf16_bits(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }

// Adam with bias correction (c1 = 1 - beta1^step, c2 = 1 - beta2^step). The
// roundings are written out: a last-bit change in one step grows into another
// trajectory over the thousands that follow.
struct AdamArgs {
    float *w, *m, *v;
    __nv_bfloat16 *wb;
    float lr, beta1, beta2, eps;
};
__device__ __forceinline__ float adam_step(const AdamArgs &A, float c1, float c2, float gi, float wi, float &mi,
                                           float &vi) {
    mi = __fmaf_rn(1.0f - A.beta1, gi, __fmul_rn(A.beta1, mi));
    vi = __fmaf_rn(__fmul_rn(1.0f - A.beta2, gi), gi, __fmul_rn(A.beta2, vi));
    return wi - A.lr * (mi / c1) / (sqrtf(vi / c2) + A.eps);
}

// Whole passes over the training rows in one cooperative launch: `epochs`
// orders of `rows` indices, mini-batches of `batch` rows, one Adam step each.
// A step is the row pass, a grid barrier, the weight pass with Adam applied to
// each parameter by the thread that summed its gradient, and a grid barrier.
// The next step's rows are fetched before that last barrier (Xs is
// double-buffered for it). corr[s] holds step s's bias corrections.
// Measured (8,192 rows, batches of 256, 3,200 steps): 254 us a step as four
// launches on 8 to 287 CTAs, 16 us here: 3.3 us the network's copies (147 KB
// into each CTA), 4 us the row pass' dependent chains, 5.5 us the weight pass,
// the rest the two barriers. The arithmetic (0.45 MFLOP a row) is 2 us of it.
struct TrainArgs {
    RowArgs rows;
    AdamArgs adam;
    const int32_t *order;
    const float2 *corr;
    int64_t n_rows, batch;
    int epochs;
    float *Xs2;
    uint64_t *bar;
    int *status;
};

template <int R>
__global__ void __launch_bounds__(kThreads, 1) sur_train_kernel(TrainArgs T) {
    extern __shared__ __align__(16) char sm[];
    const RowBufs<R> b(sm);
    uint64_t target = 0;
    const int64_t nb = (T.n_rows + T.batch - 1) / T.batch, steps = nb * T.epochs;
    const int64_t first = (int64_t)blockIdx.x * R;
    auto batch_of = [&](int64_t s) {
        RowArgs A = T.rows;
        const int64_t e = s / nb, b0 = (s - e * nb) * T.batch;
        A.idx = T.order + e * T.n_rows + b0;
        A.B = imin64(T.batch, T.n_rows - b0);
        if (s & 1) A.Xs = T.Xs2;
        return A;
    };
    RowArgs A = batch_of(0);
    if (first < A.B) load_rows<R, true>(A, b, first);
    for (int64_t s = 0; s < steps; ++s) {
        if (first < A.B) {
            load_network(sm, A.wb);
            bool fresh = true;
            for (int64_t r0 = first; r0 < A.B; r0 += (int64_t)gridDim.x * R) {
                if (!fresh) load_rows<R, true>(A, b, r0);
                row_group<R, true>(A, sm, b, r0, fresh);
                fresh = false;
            }
        }
        const float2 cc = __ldg(T.corr + s);
        if (!grid_barrier(T.bar, target, T.status)) return;
        const GradArgs G{A.Xs, A.H1, A.H2, A.dy, A.dZ1, A.dZ2, A.B};
        if (s + 1 < steps) {
            A = batch_of(s + 1);
            if (first < A.B) load_rows<R, true>(A, b, first);
        }
        for (int tile = blockIdx.x; tile < kWTiles; tile += gridDim.x) {
            float4 w = make_float4(0.f, 0.f, 0.f, 0.f), m = w, v = w;
            weight_tile(
                G, tile, reinterpret_cast<float *>(sm),
                [&](int64_t i, int n) {
                    if (n == 4) {
                        w = *reinterpret_cast<const float4 *>(T.adam.w + i);
                        m = *reinterpret_cast<const float4 *>(T.adam.m + i);
                        v = *reinterpret_cast<const float4 *>(T.adam.v + i);
                    } else {
                        w.x = T.adam.w[i];
                        m.x = T.adam.m[i];
                        v.x = T.adam.v[i];
                    }
                },
                [&](int64_t i, int n, float4 g) {
                    w.x = adam_step(T.adam, cc.x, cc.y, g.x, w.x, m.x, v.x);
                    if (n == 4) {
                        w.y = adam_step(T.adam, cc.x, cc.y, g.y, w.y, m.y, v.y);
                        w.z = adam_step(T.adam, cc.x, cc.y, g.z, w.z, m.z, v.z);
                        w.w = adam_step(T.adam, cc.x, cc.y, g.w, w.w, m.w, v.w);
                        *reinterpret_cast<float4 *>(T.adam.w + i) = w;
                        *reinterpret_cast<float4 *>(T.adam.m + i) = m;
                        *reinterpret_cast<float4 *>(T.adam.v + i) = v;
                        uint2 b4;
                        b4.x = bf16_bits(w.x) | (bf16_bits(w.y) << 16);
                        b4.y = bf16_bits(w.z) | (bf16_bits(w.w) << 16);
                        *reinterpret_cast<uint2 *>(T.adam.wb + i) = b4;
                    } else {
                        T.adam.w[i] = w.x;
                        T.adam.m[i] = m.x;
                        T.adam.v[i] = v.x;
                        T.adam.wb[i] = __float2bfloat16_rn(w.x);
                    }
                });
            __syncthreads();
        }
        if (s + 1 < steps && !grid_barrier(T.bar, target, T.status)) return;
    }
}

// Mean squared error of a batch (one CTA, FP64, fixed order); t row r is
// t[idx[r]] (or t[r]).
__global__ void __launch_bounds__(256) sur_mse_kernel(const float *__restrict__ y, const float *__restrict__ t,
                                                      const int32_t *__restrict__ idx, int64_t B,
                                                      double *__restrict__ out) {
    __shared__ double red[256];
    const int tid = threadIdx.x;
    double s = 0.0;
    for (int64_t r = tid; r < B; r += blockDim.x) {
        const double d = (double)y[r] - (double)t[idx ? (int64_t)idx[r] : r];
        s += d * d;
    }
    red[tid] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (tid < h) red[tid] += red[tid + h];
        __syncthreads();
    }
    if (tid == 0) *out = red[0] / (double)B;
}

inline int param_grid() { return 2 * num_sms(); }

}  // namespace

Surrogate::~Surrogate() {
    if (buf) cudaFree(buf);
}

int Surrogate::ensure() {
    if (buf) return 0;
    // master, m, v, grad (FP32), bf16 copy, mean, std
    const size_t f32 = sizeof(float) * (size_t)kSurrogateParams;
    const size_t b16 = sizeof(__nv_bfloat16) * (size_t)kSurrogateParams;
    auto pad = [](size_t n) { return (n + 255) / 256 * 256; };
    const size_t bytes =
        4 * pad(f32) + pad(b16) + 2 * pad(sizeof(float) * kIn);
    LNE_CUDA_TRY(cudaMalloc(&buf, bytes));
    char *p = static_cast<char *>(buf);
    auto take = [&](size_t n) {
        char *q = p;
        p += pad(n);
        return q;
    };
    w = reinterpret_cast<float *>(take(f32));
    m = reinterpret_cast<float *>(take(f32));
    v = reinterpret_cast<float *>(take(f32));
    g = reinterpret_cast<float *>(take(f32));
    wb = reinterpret_cast<__nv_bfloat16 *>(take(b16));
    mean = reinterpret_cast<float *>(take(sizeof(float) * kIn));
    std = reinterpret_cast<float *>(take(sizeof(float) * kIn));
    return 0;
}

namespace {

int refresh_copies(Surrogate &S, cudaStream_t st) {
    LNE_TRACE("sur_cast", st);
    sur_cast_kernel<<<param_grid(), 256, 0, st>>>(S.w, S.wb);
    LNE_LAUNCH_CHECK();
    return 0;
}

int reset_optimizer(Surrogate &S, cudaStream_t st) {
    LNE_CUDA_TRY(cudaMemsetAsync(S.m, 0, sizeof(float) * kSurrogateParams, st));
    LNE_CUDA_TRY(cudaMemsetAsync(S.v, 0, sizeof(float) * kSurrogateParams, st));
    S.step = 0;
    return 0;
}

struct BatchBufs {
    float *y = nullptr, *xs = nullptr, *h1 = nullptr, *h2 = nullptr, *dy = nullptr, *dz1 = nullptr, *dz2 = nullptr;
};

int batch_bufs(Workspace &ws, int64_t B, BatchBufs *b) {
    LNE_TRY(ws.get("sur.y", (size_t)B, &b->y));
    LNE_TRY(ws.get("sur.xs", (size_t)B * 32, &b->xs));
    LNE_TRY(ws.get("sur.h1", (size_t)B * kHid, &b->h1));
    LNE_TRY(ws.get("sur.h2", (size_t)B * kHid, &b->h2));
    LNE_TRY(ws.get("sur.dy", (size_t)B, &b->dy));
    LNE_TRY(ws.get("sur.dz1", (size_t)B * kHid, &b->dz1));
    LNE_TRY(ws.get("sur.dz2", (size_t)B * kHid, &b->dz2));
    return 0;
}

RowArgs row_args(const Surrogate &S, const float *X, const float *t, int64_t rows, float *y, const BatchBufs *train) {
    RowArgs A{};
    A.X = X;
    A.t = t;
    A.B = rows;
    A.mean = S.mean;
    A.std = S.std;
    A.wb = S.wb;
    A.y = y;
    if (train) {
        A.Xs = train->xs;
        A.H1 = train->h1;
        A.H2 = train->h2;
        A.dy = train->dy;
        A.dZ1 = train->dz1;
        A.dZ2 = train->dz2;
    }
    return A;
}

template <int R, bool TRAIN>
int launch_rows(const RowArgs &A, cudaStream_t st) {
    LNE_TRY(allow_dynamic_smem(sur_rows_kernel<R, TRAIN>));
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(A.B, R), num_sms());
    sur_rows_kernel<R, TRAIN><<<grid, kThreads, rows_smem(R, TRAIN), st>>>(A);
    LNE_LAUNCH_CHECK();
    return 0;
}

int forward(Surrogate &S, const float *X, int64_t rows, float *y, cudaStream_t st) {
    if (rows <= 0) return 0;
    LNE_TRACE("sur_forward", st);
    const RowArgs A = row_args(S, X, nullptr, rows, y, nullptr);
    // the smallest group that gives every row a CTA of its own wave: the pass
    // is latency-bound until each CTA has about 8 rows; then 32, so that one
    // weight load serves 16 rows a thread
    const int64_t per = ceil_div(rows, num_sms());
    if (per <= 2) return launch_rows<2, false>(A, st);
    if (per <= 8) return launch_rows<8, false>(A, st);
    return launch_rows<32, false>(A, st);
}

template <int R>
int launch_train(TrainArgs T, cudaStream_t st) {
    const int smem = std::max(rows_smem(R, true), kGradSmem);
    LNE_TRY(allow_dynamic_smem(sur_train_kernel<R>));
    const unsigned grid = (unsigned)std::min(kWTiles, num_sms());   // one CTA per SM (shared memory), all resident
    void *args[] = {&T};
    LNE_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(sur_train_kernel<R>), dim3(grid),
                                             dim3(kThreads), args, smem, st));
    LNE_LAUNCH_CHECK();
    return 0;
}

}  // namespace

int surrogate_init(Surrogate &S, uint64_t seed, cudaStream_t st) {
    LNE_TRY(S.ensure());
    {
        LNE_TRACE("sur_init", st);
        sur_init_kernel<<<param_grid(), 256, 0, st>>>(S.w, (uint32_t)seed, (uint32_t)(seed >> 32));
        LNE_LAUNCH_CHECK();
    }
    const std::vector<float> zero(kIn, 0.f), one(kIn, 1.f);
    LNE_CUDA_TRY(cudaMemcpyAsync(S.mean, zero.data(), sizeof(float) * kIn, cudaMemcpyHostToDevice, st));
    LNE_CUDA_TRY(cudaMemcpyAsync(S.std, one.data(), sizeof(float) * kIn, cudaMemcpyHostToDevice, st));
    LNE_TRY(reset_optimizer(S, st));
    LNE_TRY(refresh_copies(S, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));   // the host vectors above go out of scope
    S.ready = true;
    return 0;
}

int surrogate_fit_scaling(Surrogate &S, const float *X, int64_t rows, cudaStream_t st) {
    if (!S.ready) return fail(LNE_ERR_INVALID, "surrogate not initialised");
    LNE_TRACE("sur_scaling", st);
    sur_scaling_kernel<<<kIn, 256, 0, st>>>(X, rows, S.mean, S.std);
    LNE_LAUNCH_CHECK();
    return 0;
}

int surrogate_set(Surrogate &S, const float *w, const float *mean, const float *std, cudaStream_t st) {
    LNE_TRY(S.ensure());
    LNE_CUDA_TRY(cudaMemcpyAsync(S.w, w, sizeof(float) * kSurrogateParams, cudaMemcpyDefault, st));
    LNE_CUDA_TRY(cudaMemcpyAsync(S.mean, mean, sizeof(float) * kIn, cudaMemcpyDefault, st));
    LNE_CUDA_TRY(cudaMemcpyAsync(S.std, std, sizeof(float) * kIn, cudaMemcpyDefault, st));
    LNE_TRY(reset_optimizer(S, st));
    LNE_TRY(refresh_copies(S, st));
    S.ready = true;
    return 0;
}

int surrogate_get(Surrogate &S, float *w, float *mean, float *std, cudaStream_t st) {
    if (!S.ready) return fail(LNE_ERR_INVALID, "surrogate not initialised");
    if (w) LNE_CUDA_TRY(cudaMemcpyAsync(w, S.w, sizeof(float) * kSurrogateParams, cudaMemcpyDefault, st));
    if (mean) LNE_CUDA_TRY(cudaMemcpyAsync(mean, S.mean, sizeof(float) * kIn, cudaMemcpyDefault, st));
    if (std) LNE_CUDA_TRY(cudaMemcpyAsync(std, S.std, sizeof(float) * kIn, cudaMemcpyDefault, st));
    return 0;
}

int surrogate_predict(Surrogate &S, const float *X, int64_t rows, float *yhat, cudaStream_t st) {
    if (!S.ready) return fail(LNE_ERR_INVALID, "surrogate not initialised");
    return forward(S, X, rows, yhat, st);
}

int surrogate_grad(Surrogate &S, Workspace &ws, const float *X, const float *t, int64_t rows, float *grad,
                   double *loss, cudaStream_t st) {
    if (!S.ready) return fail(LNE_ERR_INVALID, "surrogate not initialised");
    BatchBufs b;
    LNE_TRY(batch_bufs(ws, rows, &b));
    {
        LNE_TRACE("sur_backward", st);
        const RowArgs A = row_args(S, X, t, rows, b.y, &b);
        if (ceil_div(rows, num_sms()) <= 2) LNE_TRY((launch_rows<2, true>(A, st)));
        else LNE_TRY((launch_rows<8, true>(A, st)));
        LNE_TRY(allow_dynamic_smem(sur_weight_grad_kernel));
        sur_weight_grad_kernel<<<kWTiles, kThreads, kGradSmem, st>>>(
            GradArgs{b.xs, b.h1, b.h2, b.dy, b.dz1, b.dz2, rows}, S.g);
        LNE_LAUNCH_CHECK();
    }
    if (grad) LNE_CUDA_TRY(cudaMemcpyAsync(grad, S.g, sizeof(float) * kSurrogateParams, cudaMemcpyDefault, st));
    if (loss) {
        double *d = nullptr;
        LNE_TRY(ws.get("sur.loss", 1, &d));
        sur_mse_kernel<<<1, 256, 0, st>>>(b.y, t, nullptr, rows, d);
        LNE_LAUNCH_CHECK();
        LNE_CUDA_TRY(cudaMemcpyAsync(loss, d, sizeof(double), cudaMemcpyDeviceToHost, st));
        LNE_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return 0;
}

int surrogate_train(Surrogate &S, Workspace &ws, const float *X, const float *t, int64_t rows, int epochs, int batch,
                    float lr, uint64_t seed, double *final_loss, cudaStream_t st) {
    if (!S.ready) return fail(LNE_ERR_INVALID, "surrogate not initialised");
    if (epochs < 1 || rows < 1) epochs = 0;
    const int64_t B = std::min<int64_t>(batch, std::max<int64_t>(rows, 1));
    const int64_t nb = ceil_div(std::max<int64_t>(rows, 1), B);
    BatchBufs b;
    LNE_TRY(batch_bufs(ws, B, &b));
    // Epochs per launch: the orders of a launch are drawn while the launch
    // before it runs, so the first ones are short; at most 2^22 indices.
    const int most = (int)std::max<int64_t>(1, std::min<int64_t>(8, (int64_t(1) << 22) / std::max<int64_t>(rows, 1)));
    int32_t *idx = nullptr;
    float2 *corr = nullptr;
    float *xs2 = nullptr;
    uint64_t *bar = nullptr;
    int *status = nullptr;
    LNE_TRY(ws.get("sur.idx", (size_t)rows * most, &idx));
    LNE_TRY(ws.get("sur.corr", (size_t)nb * most, &corr));
    LNE_TRY(ws.get("sur.xs2", (size_t)B * 32, &xs2));
    LNE_TRY(ws.get("sur.bar", 1, &bar));
    LNE_TRY(ws.get("sur.status", 2, &status));
    LNE_CUDA_TRY(cudaMemsetAsync(status, 0, 2 * sizeof(int), st));
    TrainArgs T{};
    T.rows = row_args(S, X, t, B, b.y, &b);
    T.adam = AdamArgs{S.w, S.m, S.v, S.wb, lr, 0.9f, 0.999f, 1e-8f};
    T.order = idx;
    T.corr = corr;
    T.n_rows = rows;
    T.batch = B;
    T.Xs2 = xs2;
    T.bar = bar;
    T.status = status;
    std::vector<int32_t> perms[2];
    std::vector<float2> hcs[2];
    std::mt19937_64 rng(seed);
    int turn = 0;
    for (int e0 = 0, take = 1; e0 < epochs; e0 += T.epochs, take = std::min(2 * take, most), turn ^= 1) {
        std::vector<int32_t> &perm = perms[turn];
        std::vector<float2> &hc = hcs[turn];
        T.epochs = std::min(std::min(take, most), epochs - e0);
        perm.resize((size_t)rows * T.epochs);
        hc.resize((size_t)nb * T.epochs);
        for (int e = 0; e < T.epochs; ++e) {   // Fisher-Yates shuffle of the row order
            int32_t *p = perm.data() + (size_t)e * rows;
            for (int64_t i = 0; i < rows; ++i) p[i] = (int32_t)i;
            for (int64_t i = rows - 1; i > 0; --i) std::swap(p[i], p[rng() % (uint64_t)(i + 1)]);
        }
        for (float2 &c : hc) {
            S.step += 1;
            c.x = (float)(1.0 - std::pow(0.9, (double)S.step));
            c.y = (float)(1.0 - std::pow(0.999, (double)S.step));
        }
        // waits for the launch before, so also for the copies out of the other
        // pair of vectors, which the next turn rewrites
        if (e0 > 0) LNE_CUDA_TRY(cudaStreamSynchronize(st));
        LNE_CUDA_TRY(cudaMemcpyAsync(idx, perm.data(), sizeof(int32_t) * perm.size(), cudaMemcpyHostToDevice, st));
        LNE_CUDA_TRY(cudaMemcpyAsync(corr, hc.data(), sizeof(float2) * hc.size(), cudaMemcpyHostToDevice, st));
        LNE_CUDA_TRY(cudaMemsetAsync(bar, 0, sizeof(uint64_t), st));
        LNE_TRACE("sur_train", st);
        const int64_t per = ceil_div(B, num_sms());
        if (per <= 2) LNE_TRY(launch_train<2>(T, st));
        else if (per <= 4) LNE_TRY(launch_train<4>(T, st));
        else LNE_TRY(launch_train<8>(T, st));
    }
    int hs[2] = {0, 0};
    LNE_CUDA_TRY(cudaMemcpyAsync(hs, status, sizeof(hs), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    if (hs[1] != 0) return fail(LNE_ERR_TIMEOUT, "a bounded grid barrier of the surrogate's training expired");
    if (final_loss) {
        float *yh = nullptr;
        double *d = nullptr;
        LNE_TRY(ws.get("sur.yall", (size_t)rows, &yh));
        LNE_TRY(ws.get("sur.loss", 1, &d));
        LNE_TRY(forward(S, X, rows, yh, st));
        sur_mse_kernel<<<1, 256, 0, st>>>(yh, t, nullptr, rows, d);
        LNE_LAUNCH_CHECK();
        LNE_CUDA_TRY(cudaMemcpyAsync(final_loss, d, sizeof(double), cudaMemcpyDeviceToHost, st));
        LNE_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return 0;
}

}  // namespace lne
