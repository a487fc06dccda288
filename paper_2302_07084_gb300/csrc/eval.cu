// Downstream objective (Sec. 6.1): one-vs-rest L2-regularised logistic
// regression on the embedding, then Micro/Macro-F1 with the top-k rule (each
// test node predicts its k highest-scoring labels, k = its number of labels).
//
// For each label l: minimise 1/2 |w|^2 + C sum_i log(1 + exp(-y_il w.x_i)),
// y in {-1, +1}, x with a constant-1 bias feature; `iters` Newton steps from
// w = 0, all labels at once, four launches a step:
//   margins   Z = X W                                  (right_multiply)
//   partials  r = C (sigma(yz) - 1) y, D = C sigma (1 - sigma); X^T r and
//             X^T diag(D) X of a block of 128 rows and one label, FP32
//   sums      G = W + sum of the X^T r blocks (FP64), H = I + sum of the
//             X^T D X blocks (three floats a sum, as good as FP64)
//   update    W_l -= H_l^-1 G_l to FP64 accuracy: FP32 Cholesky, FP64 residuals
#include <algorithm>
#include <cmath>
#include <vector>

#include "float_sum.h"
#include "runtime.h"

namespace lne {
namespace {

constexpr int kEvalRows = 128;   // rows per FP32 partial sum (and per CTA)
constexpr double kEvalBatchBytes = 256e6;   // buffers of a batch of more than one candidate

// Xa[i] = (X[idx[i]], 1, 0, ..) with rows of `pitch` floats, Ys[i][l] = +1 / -1.
// A row index outside [0, n) is not read: its row becomes zeros (label -1) and
// status bit 2 is set, which the host turns into LNE_ERR_INVALID.
__global__ void gather_rows_kernel(const float *__restrict__ X, int64_t n, int64_t ldx, int d,
                                   const uint8_t *__restrict__ lab, int L, const int32_t *__restrict__ idx, int64_t m,
                                   int pitch, float *__restrict__ Xa, float *__restrict__ Ys,
                                   int *__restrict__ status) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m * pitch;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / pitch;
        const int j = (int)(e - i * pitch);
        const int64_t r = idx[i];
        if (r < 0 || r >= n) {
            if (j == 0) atomicOr(status, 2);
            Xa[e] = 0.0f;
            continue;
        }
        Xa[e] = j < d ? X[r * ldx + j] : j == d ? 1.0f : 0.0f;
    }
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m * L; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / L;
        const int l = (int)(e - i * L);
        const int64_t r = idx[i];
        Ys[e] = (r >= 0 && r < n && lab[r * L + l]) ? 1.0f : -1.0f;
    }
}

// Number of TS x TS tiles on and above the diagonal of a da x da matrix, and
// the tile (ti, tj), ti <= tj, at position p in row order.
__host__ __device__ inline int upper_tiles(int da, int ts) {
    const int nt = (da + ts - 1) / ts;
    return nt * (nt + 1) / 2;
}
__device__ __forceinline__ void upper_tile(int p, int nt, int *ti, int *tj) {
    int i = 0;
    while (p >= nt - i) {
        p -= nt - i;
        ++i;
    }
    *ti = i;
    *tj = i + p;
}

// One block of kEvalRows rows and one label: gpart[b][l][a] = sum_r x_a R,
// hpart[b][l][e][p] = sum_r (x_a D) x_c for entry e = (a % TS) TS + c % TS of
// the upper tile p (entry-major, so that a warp's stores are contiguous), rows
// in ascending order. Bound by the FP32 FMAs (rows x labels x da (da + 1) / 2):
// a thread owns a TS x TS tile in registers, so a row costs it TS / 2 16-byte
// shared-memory loads and TS multiplications by D for TS^2 FMAs; rows are
// staged 32 at a time by asynchronous copies into two buffers, so the next
// ones arrive during the sums. TS = 8 for d >= 64, where the tiles fill the
// warps (d = 128: 153 tiles on 160 threads); below, 4 x 4 tiles keep more
// threads busy (d = 32: 45 tiles on 64 threads, with 8 x 8 15 on 32).
// Measured (5,156 rows, d = 128, 39 labels): 126 us a Newton step; the FP32 pipe
// is about half busy, at 15 warps an SM (128 registers) the rest is latency and
// the last wave. A thread per entry with two loads per FMA took 1.5 ms.
// Staged rows with TS = 8 hold the first four columns of every tile, then the
// last four, so that neighbouring tiles' 16-byte loads hit neighbouring banks.
constexpr int kEvalStage = 32;

template <int TS, bool BATCH>
__global__ void __launch_bounds__(256) hess_partial_kernel(const float *__restrict__ Xa, const float *__restrict__ Z,
                                                           const float *__restrict__ Ys, int64_t m, int da, int L,
                                                           int Ly,
                                                           float C, int ntiles, float *__restrict__ hpart,
                                                           float *__restrict__ gpart) {
    extern __shared__ __align__(16) float xs[];   // two buffers of kEvalStage rows
    __shared__ float2 s_w[kEvalRows];             // (D, R) of the rows
    const int nt = (da + TS - 1) / TS, pitch = nt * TS, quads = pitch / 4;
    const int tid = threadIdx.x;
    const int l = blockIdx.y, cand = BATCH ? l / Ly : 0;   // the candidate's rows; its labels are every candidate's
    if (BATCH) Xa += cand * m * pitch;
    const int64_t r0 = (int64_t)blockIdx.x * kEvalRows;
    const int rows = (int)imin64(kEvalRows, m - r0);
    auto stage = [&](int s0, float *to) {
        const float *src = Xa + (r0 + s0) * pitch;
        const int total = min(kEvalStage, rows - s0) * quads;
        for (int e = tid; e < total; e += blockDim.x) {
            const int r = e / quads, q = e - r * quads;
            const int at = TS == 8 ? (q & 1) * nt + (q >> 1) : q;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(to + r * pitch + 4 * at);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + 4 * e) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0, xs);
    for (int r = tid; r < rows; r += blockDim.x) {
        const float y = Ys[(r0 + r) * Ly + (l - cand * Ly)];
        const float sg = 1.0f / (1.0f + expf(-y * Z[(r0 + r) * L + l]));
        s_w[r] = make_float2(C * sg * (1.0f - sg), C * (sg - 1.0f) * y);
    }
    int ti = 0, tj = 0;
    const bool active = tid < ntiles;   // threads without a tile sum tile (0, 0) along and store nothing
    if (active) upper_tile(tid, nt, &ti, &tj);
    float2 acc[TS][TS / 2];
#pragma unroll
    for (int u = 0; u < TS; ++u)
#pragma unroll
        for (int v = 0; v < TS / 2; ++v) acc[u][v] = make_float2(0.f, 0.f);
    float g = 0.f;
    const int gc = min(tid, pitch - 1);   // column tid of a staged row: the gradient's
    const int ga = TS == 8 ? (gc & 4 ? nt * 4 : 0) + (gc >> 3) * 4 + (gc & 3) : gc;
    for (int s0 = 0, buf = 0; s0 < rows; s0 += kEvalStage, buf ^= 1) {
        const int ns = min(kEvalStage, rows - s0);
        const float *x = xs + buf * (kEvalStage * pitch);
        if (s0 + kEvalStage < rows) {
            stage(s0 + kEvalStage, xs + (buf ^ 1) * (kEvalStage * pitch));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
#pragma unroll 2
        for (int r = 0; r < ns; ++r) {
            float a[TS], b[TS];
            const float2 w = s_w[s0 + r];
#pragma unroll
            for (int h = 0; h < TS / 4; ++h) {
                const float4 p = *reinterpret_cast<const float4 *>(x + r * pitch + h * nt * 4 + ti * 4);
                const float4 q = *reinterpret_cast<const float4 *>(x + r * pitch + h * nt * 4 + tj * 4);
                a[4 * h] = p.x * w.x, a[4 * h + 1] = p.y * w.x, a[4 * h + 2] = p.z * w.x, a[4 * h + 3] = p.w * w.x;
                b[4 * h] = q.x, b[4 * h + 1] = q.y, b[4 * h + 2] = q.z, b[4 * h + 3] = q.w;
            }
            g = fmaf(x[r * pitch + ga], w.y, g);
#pragma unroll
            for (int u = 0; u < TS; ++u)
#pragma unroll
                for (int v = 0; v < TS / 2; ++v)
                    f2_add_prod(acc[u][v], make_float2(a[u], a[u]), make_float2(b[2 * v], b[2 * v + 1]));
        }
        __syncthreads();   // this buffer is refilled next
    }
    if (tid < da) gpart[((int64_t)blockIdx.x * L + l) * da + tid] = g;
    if (!active) return;
    float *out = hpart + ((int64_t)blockIdx.x * L + l) * ntiles * (TS * TS) + tid;
#pragma unroll
    for (int u = 0; u < TS; ++u)
#pragma unroll
        for (int v = 0; v < TS / 2; ++v) {
            out[(int64_t)(u * TS + 2 * v) * ntiles] = acc[u][v].x;
            out[(int64_t)(u * TS + 2 * v + 1) * ntiles] = acc[u][v].y;
        }
}

// (hi, lo) += p: hi takes the rounded sum, lo its exact rounding error.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float p) {
    const float s = __fadd_rn(hi, p), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(p, b)));
    hi = s;
}

// H_l = I + sum_b hpart[b][l] (both triangles; FP64 in H, as a float pair in
// Hp) and G = W + sum_b gpart[b] (FP64). The Hessian's sums over the row blocks are
// running sums in three floats (float_sum.h), as good as FP64 ones: FP64 additions and
// conversions run at 1/64 of the FP32 rate on this GPU and would bound this pass. A sum
// past FP32's range is taken in FP64. Measured (d = 128, 39 labels, 41 row blocks): 24.7
// us a step; sums in two floats, 46 bits, 22.3.
template <int TS>
__global__ void __launch_bounds__(256) newton_reduce_kernel(const float *__restrict__ gpart,
                                                            const float *__restrict__ hpart, int nblk, int da, int L,
                                                            int ntiles, const double *__restrict__ W,
                                                            double *__restrict__ G, double *__restrict__ H,
                                                            float2 *__restrict__ Hp) {
    const int l = blockIdx.y;
    const int64_t stride = (int64_t)L * ntiles * (TS * TS);
    const int total = ntiles * TS * TS;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < total) {
        const int q = e / ntiles, nt = (da + TS - 1) / TS;
        int ti, tj;
        upper_tile(e - q * ntiles, nt, &ti, &tj);
        const int a = ti * TS + q / TS, c = tj * TS + q % TS;
        if (a <= c && c < da) {
            const float *src = hpart + (int64_t)l * total + e;
            FloatSum sum = {a == c ? 1.f : 0.f, 0.f, 0.f};
#pragma unroll 16
            for (int b = 0; b < nblk; ++b) float_sum_add(sum, src[b * stride]);
            double h = float_sum_value(sum);
            if (!(fabs(h) <= 3.0e38)) {   // past FP32's range, or not finite
                h = a == c ? 1.0 : 0.0;
                for (int b = 0; b < nblk; ++b) h += (double)src[b * stride];
            }
            const int64_t at = (int64_t)l * da * da;
            H[at + a * da + c] = H[at + c * da + a] = h;
            const float s = __fadd_rn(sum.hi, sum.lo);
            float rest = __fsub_rn(sum.lo, __fsub_rn(s, sum.hi));   // |lo| <= |hi|: exact
            rest = __fadd_rn(rest, sum.tail);
            Hp[at + a * da + c] = Hp[at + c * da + a] = make_float2(s, rest);
        }
    } else if (e - total < da) {
        const int a = e - total;
        double s = W[a * L + l];
        for (int b = 0; b < nblk; ++b) s += gpart[((int64_t)b * L + l) * da + a];
        G[a * L + l] = s;
    }
}

// Per label (one CTA each): W[:, l] -= H_l^-1 G[:, l].
//
// H is factored in FP32 (blocked Cholesky in shared memory, 32-wide panels)
// and the solution refined with residuals G - H x, first in float-pair
// arithmetic (about 46 bits, 1 us), then in FP64 until the next correction
// would be below an FP64 ulp of x, so x is as accurate as an FP64
// factorisation's: FP64 FMAs run at 2 a cycle and SM here, which puts the FP64
// factorisation alone at 170 us for d = 128 (129^3 / 3 FMAs), against 5 us for
// an FP64 residual. Measured at d = 128: 64 us a step (the FP64 factorisation
// with one-thread triangular solves: 0.5 ms). Refinement converges when the condition number is below about
// 1e6 (H = I + X^T D X: 1 + C |X|^2 / 4 at most); where it does not, or the
// FP32 factorisation breaks down, the label takes the FP64 factorisation
// (newton_solve_fp64).
constexpr int kSolveThreads = 512;
constexpr int kNB = 32;

__host__ __device__ inline int solve_pad(int da) { return (da + kNB - 1) / kNB * kNB; }
__host__ __device__ inline int solve_smem(int da) {
    const int dp = solve_pad(da);
    const int fp32 = (dp * (dp + 4) + (dp / kNB) * kNB * (kNB + 1) + dp) * 4 + (7 * da + (da & 1)) * 8;
    const int fp64 = (da * da + da) * 8;
    return fp32 > fp64 ? fp32 : fp64;
}

// The FP64 factorisation of one label's Hessian (shared memory A: da x da,
// then the right-hand side) and its solve; status bit 1: not positive definite.
__device__ void newton_solve_fp64(const double *__restrict__ Hl, const double *__restrict__ G, int da, int L, int l,
                                  double *A, double *__restrict__ W, int *__restrict__ status) {
    double *rhs = A + da * da;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    __shared__ double s_inv;
    for (int e = tid; e < da * da; e += blockDim.x) A[e] = Hl[e];
    for (int a = tid; a < da; a += blockDim.x) rhs[a] = G[a * L + l];
    __syncthreads();
    // upper Cholesky H = R^T R, R in the upper triangle of A
    for (int k = 0; k < da; ++k) {
        if (tid == 0) {
            const double akk = A[k * da + k];
            if (!(akk > 0.0)) {
                atomicOr(status, 1);
                A[k * da + k] = 1.0;
                s_inv = 1.0;
            } else {
                const double dk = sqrt(akk);
                A[k * da + k] = dk;
                s_inv = 1.0 / dk;
            }
        }
        __syncthreads();
        const double inv = s_inv;
        for (int j = k + 1 + tid; j < da; j += blockDim.x) A[k * da + j] *= inv;
        __syncthreads();
        for (int i = k + 1 + warp; i < da; i += nw) {
            const double aki = A[k * da + i];
            for (int j = i + lane; j < da; j += 32) A[i * da + j] = fma(-aki, A[k * da + j], A[i * da + j]);
        }
        __syncthreads();
    }
    // R^T y = rhs (forward), then R delta = y (backward), one thread
    if (tid == 0) {
        for (int i = 0; i < da; ++i) {
            double s = rhs[i];
            for (int k = 0; k < i; ++k) s -= A[k * da + i] * rhs[k];
            rhs[i] = s / A[i * da + i];
        }
        for (int i = da - 1; i >= 0; --i) {
            double s = rhs[i];
            for (int k = i + 1; k < da; ++k) s -= A[i * da + k] * rhs[k];
            rhs[i] = s / A[i * da + i];
        }
    }
    __syncthreads();
    for (int a = tid; a < da; a += blockDim.x) W[a * L + l] -= rhs[a];
}

// FP32 upper Cholesky of the dp x dp matrix A (row stride ld, upper triangle;
// dp a multiple of 32) by the CTA, and the inverses of its 32 x 32 diagonal
// blocks (Dinv, row stride 33). *bad is set where a pivot is not positive and
// finite; rdiag: dp floats, the diagonal's reciprocals. Ends with a barrier.
__device__ __forceinline__ void chol32(float *A, int ld, int dp, float *Dinv, float *rdiag, int *bad) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    for (int p0 = 0; p0 < dp; p0 += kNB) {
        if (warp == 0) {   // diagonal block: lane j holds column j
            float a[kNB];
#pragma unroll
            for (int i = 0; i < kNB; ++i) a[i] = i <= lane ? A[(p0 + i) * ld + p0 + lane] : 0.f;
            bool ok = true;
#pragma unroll
            for (int k = 0; k < kNB; ++k) {
                const float piv = __shfl_sync(0xffffffffu, a[k], k);
                ok = ok && piv > 0.f && piv < 3.0e38f;
                const float inv = rsqrtf(piv);
                if (lane == k) rdiag[p0 + k] = inv;
                a[k] *= inv;
#pragma unroll
                for (int i = k + 1; i < kNB; ++i)
                    a[i] = fmaf(-__shfl_sync(0xffffffffu, a[k], i), a[k], a[i]);
            }
            if (!ok && lane == 0) *bad = 1;
#pragma unroll
            for (int i = 0; i < kNB; ++i)
                if (i <= lane) A[(p0 + i) * ld + p0 + lane] = a[i];
        }
        __syncthreads();
        const int j = p0 + kNB + tid;   // the panel's row block, a thread per column
        if (j < dp) {
            float x[kNB];
#pragma unroll
            for (int i = 0; i < kNB; ++i) x[i] = A[(p0 + i) * ld + j];
#pragma unroll
            for (int t = 0; t < kNB; ++t) {
                const float *rt = A + (p0 + t) * ld + p0;
                x[t] *= rdiag[p0 + t];
#pragma unroll
                for (int i = t + 1; i < kNB; ++i) x[i] = fmaf(-rt[i], x[t], x[i]);
            }
#pragma unroll
            for (int i = 0; i < kNB; ++i) A[(p0 + i) * ld + j] = x[i];
        }
        __syncthreads();
        const int base = p0 + kNB, nt = (dp - base) / 4, pairs = nt * (nt + 1) / 2;
        for (int q = tid; q < pairs; q += blockDim.x) {   // trailing 4 x 4 tiles
            // tile row from the pairs before it: rows i hold nt - i pairs
            int ti = (int)(((2 * nt + 1) - sqrtf((float)((2 * nt + 1) * (2 * nt + 1) - 8 * q))) * 0.5f);
            while (ti > 0 && ti * nt - ti * (ti - 1) / 2 > q) --ti;
            while ((ti + 1) * nt - (ti + 1) * ti / 2 <= q) ++ti;
            const int tj = ti + q - (ti * nt - ti * (ti - 1) / 2);
            float *ai = A + base + 4 * ti, *aj = A + base + 4 * tj;
            float c[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 v = *reinterpret_cast<const float4 *>(aj + (base + 4 * ti + u) * ld);
                c[u][0] = v.x, c[u][1] = v.y, c[u][2] = v.z, c[u][3] = v.w;
            }
#pragma unroll 8
            for (int k = 0; k < kNB; ++k) {
                const float4 x = *reinterpret_cast<const float4 *>(ai + (p0 + k) * ld);
                const float4 y = *reinterpret_cast<const float4 *>(aj + (p0 + k) * ld);
                const float xu[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) c[u][v] = fmaf(-xu[u], yv[v], c[u][v]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<float4 *>(aj + (base + 4 * ti + u) * ld) =
                    make_float4(c[u][0], c[u][1], c[u][2], c[u][3]);
        }
        __syncthreads();
    }
    // inverses of the diagonal blocks, a warp each, lane j its column j
    for (int b = warp; b < dp / kNB; b += nw) {
        const float *R = A + (b * kNB) * ld + b * kNB;
        float *D = Dinv + b * kNB * (kNB + 1);
        float x[kNB];
#pragma unroll
        for (int i = kNB - 1; i >= 0; --i) {
            float s = i == lane ? 1.f : 0.f;
#pragma unroll
            for (int t = i + 1; t < kNB; ++t) s = fmaf(-R[i * ld + t], x[t], s);
            x[i] = i <= lane ? s * rdiag[b * kNB + i] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kNB; ++i) D[i * (kNB + 1) + lane] = x[i];
    }
    __syncthreads();
}

// v <- R^-1 R^-T v (FP32, dp entries in shared memory). Ends with a barrier.
__device__ __forceinline__ void solve32(const float *A, int ld, int dp, const float *Dinv, float *v) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = dp / kNB;
    for (int p = 0; p < nb; ++p) {   // R^T y = v
        const float *D = Dinv + p * kNB * (kNB + 1);
        if (warp == 0) {
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < kNB; ++i) s = fmaf(D[i * (kNB + 1) + lane], v[p * kNB + i], s);
            __syncwarp();
            v[p * kNB + lane] = s;
        }
        __syncthreads();
        const int j = (p + 1) * kNB + tid;
        if (j < dp) {
            float s = v[j];
#pragma unroll
            for (int i = 0; i < kNB; ++i) s = fmaf(-A[(p * kNB + i) * ld + j], v[p * kNB + i], s);
            v[j] = s;
        }
        __syncthreads();
    }
    for (int p = nb - 1; p >= 0; --p) {   // R x = y
        const float *D = Dinv + p * kNB * (kNB + 1);
        if (warp == 0) {
            float s = 0.f;
#pragma unroll
            for (int t = 0; t < kNB; ++t) s = fmaf(D[lane * (kNB + 1) + t], v[p * kNB + t], s);
            __syncwarp();
            v[p * kNB + lane] = s;
        }
        __syncthreads();
        if (tid < p * kNB) {
            float s = v[tid];
#pragma unroll
            for (int t = 0; t < kNB; t += 4) {
                const float4 r = *reinterpret_cast<const float4 *>(A + tid * ld + p * kNB + t);
                s = fmaf(-r.x, v[p * kNB + t], s);
                s = fmaf(-r.y, v[p * kNB + t + 1], s);
                s = fmaf(-r.z, v[p * kNB + t + 2], s);
                s = fmaf(-r.w, v[p * kNB + t + 3], s);
            }
            v[tid] = s;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kSolveThreads) newton_solve_kernel(const double *__restrict__ H,
                                                                     const float2 *__restrict__ Hp,
                                                                     const double *__restrict__ G, int da, int L,
                                                                     double *__restrict__ W,
                                                                     int *__restrict__ status) {
    extern __shared__ __align__(16) double sm[];
    const int l = blockIdx.x, tid = threadIdx.x;
    const int dp = solve_pad(da), ld = dp + 4;
    double *x = sm, *r = x + da, *part = r + da;   // part: up to 4 da
    float2 *xp = reinterpret_cast<float2 *>(part + 4 * da);   // x as float pairs
    float *A = reinterpret_cast<float *>(xp + da + (da & 1)), *Dinv = A + dp * ld;
    float *v = Dinv + (dp / kNB) * kNB * (kNB + 1);
    __shared__ int s_bad, s_rexp;
    __shared__ unsigned s_dmax, s_xmax;
    const double *Hl = H + (int64_t)l * da * da;
    const float2 *Hpl = Hp + (int64_t)l * da * da;
    if (tid == 0) {
        s_bad = 0;
        s_rexp = 0;
    }
    for (int e = tid; e < dp * dp; e += blockDim.x) {
        const int i = e / dp, j = e - i * dp;
        A[i * ld + j] = i < da && j < da ? Hpl[i * da + j].x : i == j ? 1.f : 0.f;
    }
    for (int a = tid; a < da; a += blockDim.x) {
        x[a] = 0.0;
        r[a] = G[a * L + l];
    }
    __syncthreads();
    chol32(A, ld, dp, Dinv, v, &s_bad);   // v: scratch until the first solve
    // groups of da threads share a residual: group q sums columns q, q + ng, ..
    const int ng = min(4, (int)blockDim.x / da), grp = tid / da, ra = tid - grp * da;
    bool done = false, fp64 = false;
    float before = 3.0e38f, rate = 0.f;   // rate: the largest factor between corrections seen
    for (int it = 0; it < 16 && !done && !s_bad; ++it) {
        if (it > 0) {
            if (grp < ng && fp64) {
                double s = 0.0;
#pragma unroll 16
                for (int j = grp; j < da; j += ng) s = fma(Hl[j * da + ra], x[j], s);
                part[grp * da + ra] = s;
            } else if (grp < ng) {
                float hi = 0.f, lo = 0.f;
#pragma unroll 16
                for (int j = grp; j < da; j += ng) {
                    const float2 h = Hpl[j * da + ra], xj = xp[j];
                    const float p = __fmul_rn(h.x, xj.x);
                    lo = __fadd_rn(lo, fmaf(h.x, xj.y, fmaf(h.y, xj.x, fmaf(h.x, xj.x, -p))));
                    pair_add(hi, lo, p);
                }
                part[grp * da + ra] = (double)hi + (double)lo;
            }
            __syncthreads();
            if (tid < da) {
                double s = part[tid];
                for (int q = 1; q < ng; ++q) s += part[q * da + tid];
                r[tid] = G[tid * L + l] - s;
            }
        }
        // the residual scaled by a power of two into FP32's range
        if (tid == 0) s_dmax = s_xmax = 0u;
        if (tid < dp) {   // dp is a multiple of 32: whole warps
            const unsigned e = tid < da ? (__double2hiint(r[tid]) >> 20) & 0x7ff : 0u;
            const unsigned m = __reduce_max_sync(0xffffffffu, e);
            if ((tid & 31) == 0) atomicMax(&s_rexp, (int)m);
        }
        __syncthreads();
        const int re = s_rexp;
        if (re == 0 || re == 0x7ff) {   // zero (or below FP64's normal range): nothing left to correct
            if (re != 0 && tid == 0) s_bad = 1;
            done = re == 0;
            __syncthreads();
            break;
        }
        const double up = __hiloint2double((2046 - re) << 20, 0), down = __hiloint2double(re << 20, 0);   // 2^-+(re - 1023)
        if (tid < dp) v[tid] = tid < da ? (float)(r[tid] * up) : 0.f;
        __syncthreads();
        solve32(A, ld, dp, Dinv, v);
        if (tid < dp) {
            unsigned db = 0u, xb = 0u;
            if (tid < da) {
                const double dx = (double)v[tid] * down, xn = x[tid] + dx;
                x[tid] = xn;
                const float xh = (float)xn;
                xp[tid] = make_float2(xh, (float)(xn - (double)xh));
                db = __float_as_uint(fabsf((float)dx));
                xb = __float_as_uint(fabsf(xh));
            }
            db = __reduce_max_sync(0xffffffffu, db);
            xb = __reduce_max_sync(0xffffffffu, xb);
            if ((tid & 31) == 0) {
                atomicMax(&s_dmax, db);
                atomicMax(&s_xmax, xb);
            }
        }
        if (tid == 0) s_rexp = 0;
        __syncthreads();
        // the error left is about rate dmax: switch to FP64 residuals where
        // the pairs' own error comes near, stop when it is below an ulp of x,
        // give up when the corrections shrink by less than 4
        const float dmax = __uint_as_float(s_dmax), xmax = __uint_as_float(s_xmax);
        if (!(dmax < 3.0e38f)) {
            if (tid == 0) s_bad = 1;
        } else if (it > 0) {
            if (!fp64 && before > 0.f) rate = fmaxf(rate, fminf(dmax / before, 1.f));
            const float left = rate * dmax;
            if (!fp64) {
                fp64 = left <= 1.0e-9f * xmax;
                if (!fp64 && !(dmax <= 0.25f * before) && tid == 0) s_bad = 1;
            } else {
                done = dmax <= 1.0e-16f * xmax || left <= 1.0e-16f * xmax;
            }
        }
        before = dmax;
        __syncthreads();
    }
    if (done && !s_bad) {
        for (int a = tid; a < da; a += blockDim.x) W[a * L + l] -= x[a];
        return;
    }
    __syncthreads();
    newton_solve_fp64(Hl, G, da, L, l, sm, W, status);
}

// Top-k prediction and per-label TP / FP / FN counts.
__global__ void topk_f1_kernel(const float *__restrict__ S, const float *__restrict__ Ys, int64_t m, int L,
                               unsigned long long *__restrict__ counts) {
    S += blockIdx.y * m * L;   // the candidate's
    counts += 3 * L * blockIdx.y;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const float *si = S + i * L;
        const float *yi = Ys + i * L;
        int k = 0;
        for (int l = 0; l < L; ++l) k += yi[l] > 0.f;
        for (int l = 0; l < L; ++l) {
            int rank = 0;
            for (int j = 0; j < L; ++j) rank += (si[j] > si[l]) || (si[j] == si[l] && j < l);
            const bool pred = rank < k, truth = yi[l] > 0.f;
            if (pred && truth) atomicAdd(&counts[3 * l + 0], 1ull);
            if (pred && !truth) atomicAdd(&counts[3 * l + 1], 1ull);
            if (!pred && truth) atomicAdd(&counts[3 * l + 2], 1ull);
        }
    }
}

int egrid(int64_t work) { return (int)std::min<int64_t>(ceil_div(std::max<int64_t>(work, 1), 256), num_sms() * 16); }

}  // namespace

// Candidates are scored together: one launch a Newton step for all of them, as many
// as fit the buffer bound. A small candidate's kernels (33 features, a few labels)
// are all latency: 4 tasks of 8 candidates each took 26.3 ms one candidate at a
// time, 22.2 together (both with everything else alike).
int eval_batch_init(Workspace &ws, EvalBatch *b, int ncand, int64_t n, int d, const uint8_t *labels, int L,
                    const int32_t *train_idx, int64_t n_train, const int32_t *test_idx, int64_t n_test, double C,
                    int iters, cudaStream_t st) {
    if (d < 1 || L < 1 || n_train < 1 || n_test < 1 || iters < 0 || !(C > 0.0))
        return fail(LNE_ERR_INVALID, "bad Macro-F1 arguments");
    const int da = d + 1;
    if (da > 160) return fail(LNE_ERR_UNSUPPORTED, "Macro-F1 supports d <= 159");
    b->n = n;
    b->n_train = n_train;
    b->n_test = n_test;
    b->d = d;
    b->L = L;
    b->iters = iters;
    b->C = C;
    b->labels = labels;
    b->train_idx = train_idx;
    b->test_idx = test_idx;
    b->nblk = ceil_div(n_train, kEvalRows);
    b->ts = da > 64 ? 8 : 4;
    b->ntiles = upper_tiles(da, b->ts);
    b->pitch = (da + b->ts - 1) / b->ts * b->ts;
    const size_t hp = (size_t)b->nblk * L * b->ntiles * b->ts * b->ts;
    const double bytes = 4.0 * ((double)(n_train + n_test) * (b->pitch + L) + (double)b->nblk * da * L + (double)hp) +
                         16.0 * da * L * (da + 1);
    b->cap = (int)std::max(1.0, std::min({(double)ncand, kEvalBatchBytes / bytes, 65535.0 / L}));
    b->ids.clear();
    const size_t cap = (size_t)b->cap;
    LNE_TRY(ws.get("eval.Xa", cap * (size_t)(n_train * b->pitch), &b->Xa));
    LNE_TRY(ws.get("eval.Ys", (size_t)(n_train * L), &b->Ys));
    LNE_TRY(ws.get("eval.Z", cap * (size_t)(n_train * L), &b->Z));
    LNE_TRY(ws.get("eval.Xt", cap * (size_t)(n_test * b->pitch), &b->Xt));
    LNE_TRY(ws.get("eval.Yt", (size_t)(n_test * L), &b->Yt));
    LNE_TRY(ws.get("eval.St", cap * (size_t)(n_test * L), &b->St));
    LNE_TRY(ws.get("eval.W", cap * (size_t)da * L, &b->W));
    LNE_TRY(ws.get("eval.G", cap * (size_t)da * L, &b->G));
    LNE_TRY(ws.get("eval.H", cap * (size_t)L * da * da, &b->H));
    LNE_TRY(ws.get("eval.Hp", cap * (size_t)L * da * da, &b->Hp));
    LNE_TRY(ws.get("eval.gp", cap * (size_t)(b->nblk * da * L), &b->gp));
    LNE_TRY(ws.get("eval.hp", cap * hp, &b->hp));
    LNE_TRY(ws.get("eval.cnt", cap * (size_t)3 * L, &b->cnt));
    LNE_TRY(ws.get("eval.status", 1, &b->status));
    LNE_CUDA_TRY(cudaMemsetAsync(b->status, 0, sizeof(int), st));
    return 0;
}

// Gathers candidate id's rows of X (free to be reused on the stream afterwards);
// runs the batch first when it is full.
int eval_batch_add(EvalBatch *b, int id, const float *X, int64_t ldx, double *macro, double *micro, cudaStream_t st) {
    if ((int)b->ids.size() == b->cap) LNE_TRY(eval_batch_run(b, macro, micro, st));
    const int64_t slot = (int64_t)b->ids.size();
    b->ids.push_back(id);
    LNE_TRACE("eval_gather", st);
    gather_rows_kernel<<<egrid(b->n_train * b->pitch), 256, 0, st>>>(
        X, b->n, ldx, b->d, b->labels, b->L, b->train_idx, b->n_train, b->pitch, b->Xa + slot * b->n_train * b->pitch,
        b->Ys, b->status);
    LNE_LAUNCH_CHECK();
    gather_rows_kernel<<<egrid(b->n_test * b->pitch), 256, 0, st>>>(
        X, b->n, ldx, b->d, b->labels, b->L, b->test_idx, b->n_test, b->pitch, b->Xt + slot * b->n_test * b->pitch,
        b->Yt, b->status);
    LNE_LAUNCH_CHECK();
    return 0;
}

// Scores the gathered candidates: macro[id], micro[id]. Synchronises.
int eval_batch_run(EvalBatch *b, double *macro, double *micro, cudaStream_t st) {
    const int m = (int)b->ids.size(), L = b->L, da = b->d + 1, ntiles = b->ntiles, ts = b->ts, pitch = b->pitch;
    if (m == 0) return 0;
    LNE_CUDA_TRY(cudaMemsetAsync(b->W, 0, sizeof(double) * da * L * m, st));
    LNE_CUDA_TRY(cudaMemsetAsync(b->cnt, 0, sizeof(unsigned long long) * 3 * L * m, st));
    const int threads = (std::max(ntiles, da) + 31) / 32 * 32;   // at most 224 (da = 160: 210 tiles)
    const int hsmem = 2 * kEvalStage * pitch * 4;
    // the labels of all candidates in a row: label l of candidate j is column j L + l
    const int Lm = L * m;
    const dim3 hgrid((unsigned)b->nblk, (unsigned)Lm);
    const dim3 rgrid((unsigned)ceil_div((int64_t)ntiles * ts * ts + da, 256), (unsigned)Lm);
    LNE_TRY(allow_dynamic_smem(newton_solve_kernel));
    for (int it = 0; it < b->iters; ++it) {
        LNE_TRY(right_multiply(b->Xa, b->n_train, da, pitch, b->W, Lm, L, nullptr, b->Z, Lm, st, m,
                               b->n_train * pitch, L, L));
        {
            LNE_TRACE("newton_partials", st);
            auto *hess = m > 1 ? (ts == 8 ? hess_partial_kernel<8, true> : hess_partial_kernel<4, true>)
                               : (ts == 8 ? hess_partial_kernel<8, false> : hess_partial_kernel<4, false>);
            hess<<<hgrid, threads, hsmem, st>>>(b->Xa, b->Z, b->Ys, b->n_train, da, Lm, L, (float)b->C, ntiles, b->hp,
                                                b->gp);
            LNE_LAUNCH_CHECK();
        }
        {
            LNE_TRACE("newton_sums", st);
            if (ts == 8)
                newton_reduce_kernel<8><<<rgrid, 256, 0, st>>>(b->gp, b->hp, (int)b->nblk, da, Lm, ntiles, b->W, b->G,
                                                               b->H, b->Hp);
            else
                newton_reduce_kernel<4><<<rgrid, 256, 0, st>>>(b->gp, b->hp, (int)b->nblk, da, Lm, ntiles, b->W, b->G,
                                                               b->H, b->Hp);
            LNE_LAUNCH_CHECK();
        }
        {
            LNE_TRACE("newton_solve", st);
            newton_solve_kernel<<<Lm, kSolveThreads, solve_smem(da), st>>>(b->H, b->Hp, b->G, da, Lm, b->W, b->status);
            LNE_LAUNCH_CHECK();
        }
    }
    LNE_TRY(right_multiply(b->Xt, b->n_test, da, pitch, b->W, Lm, L, nullptr, b->St, L, st, m, b->n_test * pitch, L,
                           b->n_test * L));
    {
        LNE_TRACE("topk_f1", st);
        topk_f1_kernel<<<dim3((unsigned)egrid(b->n_test), (unsigned)m), 256, 0, st>>>(b->St, b->Yt, b->n_test, L,
                                                                                     b->cnt);
        LNE_LAUNCH_CHECK();
    }
    std::vector<unsigned long long> h((size_t)3 * L * m);
    int hs = 0;
    LNE_CUDA_TRY(cudaMemcpyAsync(h.data(), b->cnt, sizeof(unsigned long long) * h.size(), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaMemcpyAsync(&hs, b->status, sizeof(int), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    if (hs & 2) return fail(LNE_ERR_INVALID, "a train or test row index is outside [0, n)");
    if (hs) return fail(LNE_ERR_NUMERIC, "a logistic-regression Hessian was not positive definite");
    for (int j = 0; j < m; ++j) {
        const unsigned long long *hj = h.data() + (size_t)3 * L * j;
        double f1sum = 0.0, tp = 0, fp = 0, fn = 0;
        for (int l = 0; l < L; ++l) {
            const double t = (double)hj[3 * l], p = (double)hj[3 * l + 1], q = (double)hj[3 * l + 2];
            const double den = 2 * t + p + q;
            f1sum += den > 0 ? 2 * t / den : 0.0;
            tp += t;
            fp += p;
            fn += q;
        }
        macro[b->ids[j]] = f1sum / L;
        micro[b->ids[j]] = (2 * tp + fp + fn) > 0 ? 2 * tp / (2 * tp + fp + fn) : 0.0;
    }
    b->ids.clear();
    return 0;
}

int macro_f1(Workspace &ws, const float *X, int64_t n, int d, int64_t ldx, const uint8_t *labels, int L,
             const int32_t *train_idx, int64_t n_train, const int32_t *test_idx, int64_t n_test, double C, int iters,
             double *macro, double *micro, cudaStream_t st) {
    EvalBatch b;
    LNE_TRY(eval_batch_init(ws, &b, 1, n, d, labels, L, train_idx, n_train, test_idx, n_test, C, iters, st));
    LNE_TRY(eval_batch_add(&b, 0, X, ldx, macro, micro, st));
    return eval_batch_run(&b, macro, micro, st);
}

}  // namespace lne
