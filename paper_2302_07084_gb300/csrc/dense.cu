// Dense stages of the randomized SVD (Algorithm 4) on the GPU:
//
//   sketch         Omega = randn(n, c) from Philox4x32-10 words (Box-Muller).
//   gram           G = Y^T Y to FP64 accuracy: per-CTA partial Grams over row
//                  blocks in exact FP32 steps (float pairs), summed in FP64
//                  in a fixed order so the result is reproducible.
//   chol           G = R^T R (upper Cholesky) in FP64, a CTA per block column.
//   trsm_rows      Q = Y R^-1 by forward substitution per row (FP32): each
//                  row's solve is backward stable, so Y = Q R holds to FP32
//                  rounding whatever the conditioning of R.
//   right_multiply out = Y W for a small FP64 W (rounded to FP32), FP32 FMA.
//   cholqr2        Q = Y R1^-1, then again: the orthonormalisation used in
//                  place of eigSVD inside the power iteration (same range).
//   small_svd      SVD of the c x c factor R: FP32 one-sided Jacobi, then
//                  Ogita-Aishima refinement in FP64, so Y = Q R gives left
//                  singular vectors Q U_R -- the final eigSVD of Algorithm 4.
//   sign_fix_embed largest-magnitude entry of each column made positive, and
//                  X = U Sigma^{1/2} (Sec. 4.2).
#include <algorithm>
#include <cmath>
#include <mutex>

#include "jacobi_order.h"
#include "runtime.h"

namespace lne {
namespace {

// ---------------------------------------------------------------------------
// Gaussian sketch
// ---------------------------------------------------------------------------
__device__ __forceinline__ float log_unit(uint32_t w) {
    // ln((w + 0.5) / 2^32); near 1 use log1p of the exact integer distance.
    if (w >= 0x80000000u) {
        uint32_t m = 0u - w;   // 2^32 - w, in 1 .. 2^31
        return log1pf(-((float)m - 0.5f) * 2.3283064365386963e-10f);
    }
    return logf(((float)w + 0.5f) * 2.3283064365386963e-10f);
}

__global__ void sketch_kernel(int64_t n, int c, uint32_t k0, uint32_t k1, float *__restrict__ out,
                              int64_t ld) {
    const int nblk = (c + 3) / 4;
    const int64_t total = n * nblk;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx / nblk;
        const int cb = (int)(idx - i * nblk);
        u32x4 w = philox10(u32x4{(uint32_t)i, (uint32_t)cb, 0u, 0u}, k0, k1);
        float r0 = sqrtf(-2.0f * log_unit(w.x));
        float r1 = sqrtf(-2.0f * log_unit(w.z));
        float s0, c0, s1, c1;
        sincospif(2.0f * (((float)w.y + 0.5f) * 2.3283064365386963e-10f), &s0, &c0);
        sincospif(2.0f * (((float)w.w + 0.5f) * 2.3283064365386963e-10f), &s1, &c1);
        float z[4] = {r0 * c0, r0 * s0, r1 * c1, r1 * s1};
        float *row = out + i * ld + 4 * cb;
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (4 * cb + t < c) row[t] = z[t];
    }
}

// ---------------------------------------------------------------------------
// Gram with FP64 accuracy from FP32 arithmetic: thread (ti, tj, half), ti <= tj,
// owns 4 rows of an 8x8 tile of the upper half. Every product a*b is split exactly into
// p + e (p = fl(a b), e = fma(a, b, -p)); p enters a float pair (hi, lo) by
// an error-free two-sum, e and the two-sum's error go to lo. The pair carries
// ~46 significant bits over a CTA's rows; CTAs are summed in FP64. FP64
// arithmetic runs at a small fraction of the FP32 rate on this GPU, so this
// is several times faster than FP64 FMAs. The _rn operations keep the
// compiler from contracting the error-free transformations.
// Bound by the FP32 pipe (ten operations a product, issued as packed pairs); chunks
// of rows arrive by asynchronous copies during the sums of the chunk before. Measured
// (n = 1e6, c = 144): 4.5 ms with scalar operations and a barrier between load and
// sums, 3.7 now; n = 10,312: 64 -> 59 us. Sums on a fixed grid per chunk (a shift
// above the running sum: four operations, 1.65 ms) were given up: their error is
// relative to the columns' norms instead of to the sum, and the changed rounding
// moved tuning scores (each a count of decisions, some of them near ties). Picking
// the larger operand by compare and select (three operations fewer): 4.2 ms.
// ---------------------------------------------------------------------------
constexpr int kGramRows = 64;   // rows of a chunk (two buffers of them are staged)

constexpr int kGramThreads = 384;

// Paired FP32 arithmetic (f32x2, sm_100 and later): one instruction for two lanes
// of a float2, each rounded as the scalar operation.
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(reinterpret_cast<const uint64_t &>(a)), "l"(reinterpret_cast<const uint64_t &>(b)));
    return reinterpret_cast<const float2 &>(d);
}
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(reinterpret_cast<const uint64_t &>(a)), "l"(reinterpret_cast<const uint64_t &>(b)));
    return reinterpret_cast<const float2 &>(d);
}
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(reinterpret_cast<const uint64_t &>(a)), "l"(reinterpret_cast<const uint64_t &>(b)),
          "l"(reinterpret_cast<const uint64_t &>(c)));
    return reinterpret_cast<const float2 &>(d);
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(reinterpret_cast<const uint64_t &>(a)), "l"(reinterpret_cast<const uint64_t &>(b)));
    return reinterpret_cast<const float2 &>(d);
}

// VEC: rows are read by 16-byte copies (c, ld multiples of 4, Y 16-byte aligned).
template <bool VEC>
__global__ void __launch_bounds__(kGramThreads) gram_partial_kernel(const float *__restrict__ Y, int64_t n, int c,
                                                                    int64_t ld, int64_t rows_per_cta,
                                                                    double *__restrict__ partial) {
    extern __shared__ __align__(16) float ys[];   // two chunks of kGramRows x cp
    const int cp = (c + 7) & ~7;
    const int nt = cp / 8;
    const int nitems = nt * (nt + 1);   // (tile, half): rows 0-3 or 4-7 of an 8x8 tile
    const int tid = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_cta;
    const int64_t r1 = imin64(n, r0 + rows_per_cta);
    for (int e = tid; e < 2 * kGramRows * (cp - c); e += kGramThreads) {   // padding columns
        const int r = e / (cp - c);
        ys[r * cp + c + (e - r * (cp - c))] = 0.f;
    }
    auto stage = [&](int64_t base, float *to) {
        const int rows = (int)imin64(kGramRows, r1 - base);
        if (VEC) {
            const int q = c / 4;
            for (int e = tid; e < rows * q; e += kGramThreads) {
                const int r = e / q, k = e - r * q;
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(to + r * cp + 4 * k);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Y + (base + r) * ld + 4 * k)
                             : "memory");
            }
        } else {
            for (int e = tid; e < rows * c; e += kGramThreads) {
                const int r = e / c, k = e - r * c;
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(to + r * cp + k);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(Y + (base + r) * ld + k)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // items are processed in groups of kGramThreads (uniform trip count for the barriers)
    for (int g0 = 0; g0 < nitems; g0 += kGramThreads) {
        const int item = g0 + tid;
        const bool active = item < nitems;
        int ti = 0, tj = 0;
        const int half = item & 1;
        if (active) {
            int rem = item >> 1;
            while (rem >= nt - ti) {
                rem -= nt - ti;
                ++ti;
            }
            tj = ti + rem;
        }
        const int xa = ti * 8 + half * 4;
        float2 hi[4][4], lo[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) hi[x][y] = lo[x][y] = make_float2(0.f, 0.f);
        __syncthreads();   // the last group's chunks are done
        if (r0 < r1) stage(r0, ys);
        int buf = 0;
        for (int64_t base = r0; base < r1; base += kGramRows, buf ^= 1) {
            const int rows = (int)imin64(kGramRows, r1 - base);
            const float *yb = ys + buf * (kGramRows * cp);
            if (base + kGramRows < r1) {
                stage(base + kGramRows, ys + (buf ^ 1) * (kGramRows * cp));
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            if (active) {
                for (int r = 0; r < rows; ++r) {
                    const float *yr = yb + r * cp;
                    const float4 a4 = *reinterpret_cast<const float4 *>(yr + xa);
                    const float4 b0 = *reinterpret_cast<const float4 *>(yr + tj * 8);
                    const float4 b1 = *reinterpret_cast<const float4 *>(yr + tj * 8 + 4);
                    const float av[4] = {a4.x, a4.y, a4.z, a4.w};
                    const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                                          make_float2(b1.z, b1.w)};
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const float2 a2 = make_float2(av[x], av[x]), na2 = make_float2(-av[x], -av[x]);
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            const float2 p = f2_mul(a2, bv[y]);
                            const float2 ne = f2_fma(na2, bv[y], p);   // p - a b
                            const float2 h = hi[x][y], s = f2_add(h, p);
                            const float2 bb = f2_sub(s, h);
                            const float2 err = f2_add(f2_sub(h, f2_sub(s, bb)), f2_sub(p, bb));
                            hi[x][y] = s;
                            lo[x][y] = f2_add(lo[x][y], f2_sub(err, ne));
                        }
                    }
                }
            }
            __syncthreads();   // this buffer is rewritten next
        }
        if (active) {
            double *P = partial + (int64_t)blockIdx.x * cp * cp;
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    P[(xa + x) * cp + tj * 8 + 2 * y] = (double)hi[x][y].x + (double)lo[x][y].x;
                    P[(xa + x) * cp + tj * 8 + 2 * y + 1] = (double)hi[x][y].y + (double)lo[x][y].y;
                }
        }
    }
}

// G[a][b] = G[b][a] = sum over CTAs of the partials of the upper entry
// (a, b): 8 lanes per entry, lane q summing partials q, q + 8, ..., then a
// fixed shuffle tree, so the order is the same on every run. (The (a, b)
// entry lives in tile (a/8, b/8); tiles with a/8 == b/8 hold both orders,
// tiles above the diagonal only (a, b).)
constexpr int kGramRedLanes = 8;

// Also zeroes the tile counters of the Cholesky that follows.
__global__ void gram_reduce_kernel(const double *__restrict__ partial, int nblk, int c,
                                   double *__restrict__ G, unsigned *__restrict__ cnt) {
    if (blockIdx.x == 0 && threadIdx.x < 16) cnt[threadIdx.x] = 0u;
    constexpr int kPerWarp = 32 / kGramRedLanes;   // entries per warp and step
    const int cp = (c + 7) & ~7;
    const int nup = c * (c + 1) / 2;
    const int lane = threadIdx.x & 31, q = lane % kGramRedLanes;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // the warp's lanes take the same trip count (the shuffles need all of them)
    for (int64_t ub = warp * kPerWarp; ub < nup; ub += nwarps * kPerWarp) {
        const int64_t u = ub + lane / kGramRedLanes;
        const bool live = u < nup;
        int a = 0, b = 0;
        if (live) {   // u-th upper entry in row order: row a holds c - a entries
            int rem = (int)u;
            while (rem >= c - a) {
                rem -= c - a;
                ++a;
            }
            b = a + rem;
        }
        double s = 0.0;
        if (live)
            for (int k = q; k < nblk; k += kGramRedLanes) s += partial[(int64_t)k * cp * cp + a * cp + b];
#pragma unroll
        for (int off = kGramRedLanes / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (live && q == 0) {
            G[a * c + b] = s;
            G[b * c + a] = s;
        }
    }
}

// 1/sqrt(a) of a positive finite FP64 pivot by two Newton steps
// y <- y (3 - a y^2) / 2 from the FP32 estimate (which has 24 bits; two steps
// pass FP64's 53), so no FP64 square root or division runs on this GPU's
// narrow FP64 pipe. FP64 instructions take some 64 cycles each, conversions too: the
// FP32 rounding of the pivot and the estimate's FP64 form are taken on the bits
// where both are normal floats; pivots outside FP32's range take the plain route.
__device__ __forceinline__ double pivot_rsqrt(double a) {
    const uint64_t bits = (uint64_t)__double_as_longlong(a);
    const int e = (int)(bits >> 52) - 1023;
    double y;
    if (e >= -126 && e < 127) {   // rounded to nearest even: at most 2^127
        uint32_t f = (uint32_t)((bits >> 29) - ((uint64_t)896 << 23));
        const uint32_t rest = (uint32_t)bits & 0x1FFFFFFFu;
        f += rest > 0x10000000u || (rest == 0x10000000u && (f & 1u)) ? 1u : 0u;
        const uint32_t r = __float_as_uint(rsqrtf(__uint_as_float(f)));
        y = __longlong_as_double((long long)(((uint64_t)r + ((uint64_t)896 << 23)) << 29));
    } else {
        y = (double)rsqrtf((float)a);
        if (!(y > 0.0) || !isfinite(y)) return 1.0 / sqrt(a);
    }
    y = y * fma(-0.5 * a, y * y, 1.5);
    return y * fma(-0.5 * a, y * y, 1.5);
}

constexpr int kMaxSmemC = 160;   // largest c of the small SVD
constexpr int kOaSteps = 4;      // refinement steps
constexpr int kOaSync = 8;       // words: two of the grid barrier; two are lne_svd_small_noalloc's status, the others spare

// ---------------------------------------------------------------------------
// Cholesky (upper, G = R^T R) in FP64, 16 x 16 tiles, one CTA per block column.
// CTA j holds the tiles (i, j), i <= j, of its 16 columns in shared memory and
// takes the panels p = 0 .. j in order: it solves R_pp^T R_pj = A_pj, publishes
// R_pj, and subtracts R_pi^T R_pj from its tiles (i, j) as the other CTAs publish
// their R_pi; at p = j it factors its diagonal tile, which releases the panel to
// the CTAs on its right. cnt[i] counts the tiles CTA i has published, so a CTA
// waits for the one tile it needs instead of for a grid-wide barrier (nine
// panels of two barriers each took most of the factorisation's time). What is
// left is the chain of the diagonal: per panel 16 pivots (an FP64 reciprocal
// square root, a scaling and an update each), one tile solve and one tile
// update. Launched cooperatively, so every CTA that is waited for is resident;
// a wait gives up after 2 s and sets status[1]. A pivot that is not positive
// sets status[0] and is replaced by 1. Every entry takes its terms in ascending
// order of the pivots. Measured: see chol().
// ---------------------------------------------------------------------------
constexpr int kCholB = 16;
constexpr int kCholMaxTiles = 15;   // c <= 240

// Waits until *cnt >= want (thread 0 polls; ends with a barrier of the CTA).
__device__ __forceinline__ bool chol_wait(const unsigned *cnt, unsigned want, int *status) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        uint64_t t0 = 0;
        int ok = 1;
        for (unsigned spin = 1;; ++spin) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
            if (v >= want) break;
            if ((spin & 63u) == 0u) {
                uint64_t t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t0 == 0) t0 = t;
                if (t - t0 > 2000000000ull) {
                    atomicExch(status + 1, 1);
                    ok = 0;
                    break;
                }
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    const bool ok = s_ok != 0;
    __syncthreads();   // s_ok is written again by the next wait
    return ok;
}

// pub: the published tiles, (i, j) at ((size_t)i * nt + j) * 256; inv: the
// reciprocal diagonal.
__global__ void __launch_bounds__(256, 1) chol_kernel(const double *__restrict__ G, int c, double *__restrict__ R,
                                                      double *pub, double *inv, unsigned *cnt,
                                                      int *__restrict__ status) {
    __shared__ double tiles[kCholMaxTiles][kCholB][kCholB + 1];
    __shared__ double rp[kCholB][kCholB + 1];   // R_pp, then R_pi
    __shared__ double sinv[kCholB];
    const int nt = gridDim.x, j = blockIdx.x, tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
    const int col = 16 * j + tj;
#pragma unroll 4
    for (int i = 0; i <= j; ++i) {
        const int row = 16 * i + ti;
        tiles[i][ti][tj] = row < c && col < c ? __ldg(G + (size_t)row * c + col) : 0.0;
    }
    __syncthreads();
    auto publish = [&](int p, double v) {
        pub[((size_t)p * nt + j) * 256 + tid] = v;
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(cnt + j), "r"((unsigned)p + 1u) : "memory");
        }
    };
    for (int p = 0; p < j; ++p) {
        if (!chol_wait(cnt + p, p + 1, status)) return;
        rp[ti][tj] = __ldcg(pub + ((size_t)p * nt + p) * 256 + tid);
        if (tid < 16) sinv[tid] = __ldcg(inv + 16 * p + tid);
        __syncthreads();
        // R_pp^T x = A_pj: 16 lanes per column; lane li holds x_li and subtracts
        // r_t,li x_t as soon as x_t is final (panel p is full: p < j)
        {
            const int li = tj, q = ti;   // row in the tile, column in the tile
            double x = tiles[p][li][q];
            for (int t = 0; t < kCholB; ++t) {
                if (li == t) x *= sinv[t];
                const double xt = __shfl_sync(0xffffffffu, x, t, 16);
                if (li > t) x = fma(-rp[t][li], xt, x);
            }
            __syncthreads();
            tiles[p][li][q] = x;
        }
        __syncthreads();
        publish(p, tiles[p][ti][tj]);
        for (int i = p + 1; i < j; ++i) {
            if (!chol_wait(cnt + i, p + 1, status)) return;
            rp[ti][tj] = __ldcg(pub + ((size_t)p * nt + i) * 256 + tid);
            __syncthreads();
            double a = tiles[i][ti][tj];
#pragma unroll
            for (int t = 0; t < kCholB; ++t) a = fma(-rp[t][ti], tiles[p][t][tj], a);
            tiles[i][ti][tj] = a;
            __syncthreads();
        }
        if (ti <= tj) {
            double a = tiles[j][ti][tj];
#pragma unroll
            for (int t = 0; t < kCholB; ++t) a = fma(-tiles[p][t][ti], tiles[p][t][tj], a);
            tiles[j][ti][tj] = a;
        }
        __syncthreads();
    }
    // the diagonal tile, one entry per thread (in v); the owner of the next pivot
    // takes its reciprocal root in the same phase as the update that finishes it
    const int bs = min(kCholB, c - 16 * j);
    double v = tiles[j][ti][tj];
    auto pivot = [&](int t) {
        double d = 1.0, y = 1.0;
        const int hi = __double2hiint(v);
        if ((hi > 0 && hi < 0x7FF00000) || (hi == 0 && __double2loint(v) != 0)) {   // positive, finite
            y = pivot_rsqrt(v);
            d = v * y;
        } else if (*status == 0) {
            *status = 16 * j + t + 1;
        }
        v = d;
        sinv[t] = y;
    };
    if (tid == 0) pivot(0);
    __syncthreads();
    for (int t = 0; t < bs; ++t) {
        if (ti == t && tj >= t && tj < bs) {
            if (tj > t) v *= sinv[t];
            rp[0][tj] = v;
        }
        __syncthreads();
        if (ti > t && tj >= ti && tj < bs) {
            v = fma(-rp[0][ti], rp[0][tj], v);
            if (ti == tj && ti == t + 1) pivot(t + 1);
        }
        __syncthreads();
    }
    if (ti <= tj) tiles[j][ti][tj] = v;
    __syncthreads();
    if (j + 1 < nt) {
        if (tid < 16) inv[16 * j + tid] = sinv[tid];
        publish(j, tiles[j][ti][tj]);
    }
    for (int i = 0; i < nt; ++i) {
        const int row = 16 * i + ti;
        if (row < c && col < c) R[(size_t)row * c + col] = row <= col ? tiles[min(i, j)][ti][tj] : 0.0;
    }
}

// Q = Y R^-1 for upper-triangular R (FP64, rounded to FP32): forward
// substitution per row, q_l = (y_l - q_0 R_0l - .. - q_(l-1) R_(l-1)l) / R_ll with
// the terms subtracted in that order. A warp owns 32 RPT rows, a lane the rows
// lane and lane + 32, and takes their columns in blocks of 16: the terms of all
// columns before the block are a small matrix product (the rows' earlier q from
// shared memory, stored negated and by column; R's 16 entries of a row
// broadcast), then the block's own triangle is solved in registers. Blocks of Y
// and Q pass through a warp's staging rows, so that four lanes read or write a
// row's 64 bytes together; the next block's loads are in flight meanwhile.
// Per earlier column and RPT = 2: 6 shared-memory wavefronts for 32 FMAs a
// thread, so the FP32 pipe bounds it (n c^2 / 2 FMAs). Measured (n = 1e6,
// c = 144): 3.5 -> 0.73 ms; with a warp a row, a shuffle and c / 32 predicated
// FMAs per column, most issue slots went to neither. One warp a scheduler (R and
// the q of 256 rows fill shared memory), so latencies show: about half the
// FP32 rate.
constexpr int kTrsmB = 16;
constexpr int kTrsmPitch = kTrsmB + 4;   // floats a staging row: 8 lanes' 16-byte accesses hit all banks once

// floats of R's column blocks before block b: block b holds the rows 0 .. 16 b + 15
__host__ __device__ inline int trsm_block_at(int b) { return 128 * b * (b + 1); }
inline int trsm_smem(int c, int tile_rows) {
    const int nb = (c + kTrsmB - 1) / kTrsmB;
    return (trsm_block_at(nb) + nb * kTrsmB + tile_rows * kTrsmPitch + (nb - 1) * kTrsmB * tile_rows) * 4;
}

// VEC: 16-byte accesses to Y and Q (c, ldy, ldq multiples of 4, both aligned).
template <int RPT, bool VEC>
__global__ void __launch_bounds__(128) trsm_rows_kernel(const float *__restrict__ Y, int64_t n, int c, int64_t ldy,
                                                        const double *__restrict__ R, float *__restrict__ Q,
                                                        int64_t ldq) {
    // R by column blocks, reciprocal diagonal, staging rows, -q by column
    extern __shared__ __align__(16) float Rs[];
    constexpr int WR = 32 * RPT, ITS = WR / 8;   // rows of a warp; its 16-byte accesses a lane and block
    const int nb = (c + kTrsmB - 1) / kTrsmB, tile = blockDim.x * RPT, tid = threadIdx.x, lane = tid & 31;
    const int wrow = (tid >> 5) * WR;            // the warp's first row in the tile
    float *rdiag = Rs + trsm_block_at(nb), *stg = rdiag + nb * kTrsmB + wrow * kTrsmPitch;
    float *qs = rdiag + nb * kTrsmB + tile * kTrsmPitch + wrow;
    for (int b = 0; b < nb; ++b) {
        float *to = Rs + trsm_block_at(b);
        // staged 8 loads at a time per thread: independent loads in flight
#pragma unroll 8
        for (int e = tid; e < (b + 1) * (kTrsmB * kTrsmB); e += blockDim.x) {
            const int j = e / kTrsmB, l = b * kTrsmB + e % kTrsmB;
            to[e] = j < c && l < c ? (float)__ldg(R + j * c + l) : 0.f;
        }
    }
    for (int j = tid; j < nb * kTrsmB; j += blockDim.x) rdiag[j] = j < c ? (float)(1.0 / R[j * c + j]) : 0.f;
    __syncthreads();
    const int sr = lane >> 2, sc = 4 * (lane & 3);   // access it of a block: row 8 it + sr, columns sc .. sc + 3
    // columns l0 + sc .. of the warp's rows from row w0 on (zeros past the rows or the matrix)
    auto load = [&](int64_t w0, int l0, float4 (&v)[ITS]) {
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
            const int64_t i = w0 + 8 * it + sr;
            const float *src = Y + i * ldy + l0 + sc;
            const int left = i < n ? c - (l0 + sc) : 0;
            if (VEC) {
                v[it] = left > 0 ? *reinterpret_cast<const float4 *>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                v[it].x = left > 0 ? src[0] : 0.f;
                v[it].y = left > 1 ? src[1] : 0.f;
                v[it].z = left > 2 ? src[2] : 0.f;
                v[it].w = left > 3 ? src[3] : 0.f;
            }
        }
    };
    for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < n; t0 += (int64_t)gridDim.x * tile) {
        const int64_t w0 = t0 + wrow;
        if (w0 >= n) continue;   // whole warps
        float4 nxt[ITS];
        load(w0, 0, nxt);
        for (int b = 0; b < nb; ++b) {
#pragma unroll
            for (int it = 0; it < ITS; ++it)
                *reinterpret_cast<float4 *>(stg + (8 * it + sr) * kTrsmPitch + sc) = nxt[it];
            __syncwarp();
            if (b + 1 < nb) load(w0, (b + 1) * kTrsmB, nxt);   // arrives during this block's work
            float2 y[RPT][kTrsmB / 2];
#pragma unroll
            for (int p = 0; p < RPT; ++p)
#pragma unroll
                for (int q = 0; q < kTrsmB / 4; ++q) {
                    const float4 x =
                        *reinterpret_cast<const float4 *>(stg + (lane + 32 * p) * kTrsmPitch + 4 * q);
                    y[p][2 * q] = make_float2(x.x, x.y);
                    y[p][2 * q + 1] = make_float2(x.z, x.w);
                }
            const float *Rb = Rs + trsm_block_at(b);
#pragma unroll 4
            for (int j = 0; j < b * kTrsmB; ++j) {
                float nq[RPT];
#pragma unroll
                for (int p = 0; p < RPT; ++p) nq[p] = qs[j * tile + lane + 32 * p];
#pragma unroll
                for (int q = 0; q < kTrsmB / 4; ++q) {
                    const float4 r = *reinterpret_cast<const float4 *>(Rb + j * kTrsmB + 4 * q);
#pragma unroll
                    for (int p = 0; p < RPT; ++p) {
                        f2_add_prod(y[p][2 * q], make_float2(nq[p], nq[p]), make_float2(r.x, r.y));
                        f2_add_prod(y[p][2 * q + 1], make_float2(nq[p], nq[p]), make_float2(r.z, r.w));
                    }
                }
            }
            // the block's own triangle
            const float *Rd = Rb + b * (kTrsmB * kTrsmB);
            float v[RPT][kTrsmB];
#pragma unroll
            for (int p = 0; p < RPT; ++p)
#pragma unroll
                for (int q = 0; q < kTrsmB / 2; ++q) v[p][2 * q] = y[p][q].x, v[p][2 * q + 1] = y[p][q].y;
#pragma unroll
            for (int l = 0; l < kTrsmB; ++l) {
                const float rd = rdiag[b * kTrsmB + l];
#pragma unroll
                for (int p = 0; p < RPT; ++p) v[p][l] *= rd;
#pragma unroll
                for (int q = (l + 1) / 4; q < kTrsmB / 4; ++q) {
                    const float4 r4 = *reinterpret_cast<const float4 *>(Rd + l * kTrsmB + 4 * q);
                    const float r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                    for (int m = 4 * q; m < 4 * q + 4; ++m)
#pragma unroll
                        for (int p = 0; p < RPT; ++p)
                            if (m > l) v[p][m] = fmaf(-v[p][l], r[m - 4 * q], v[p][m]);
                }
            }
#pragma unroll
            for (int p = 0; p < RPT; ++p) {
                if (b + 1 < nb) {   // read back by this lane only
#pragma unroll
                    for (int l = 0; l < kTrsmB; ++l) qs[(b * kTrsmB + l) * tile + lane + 32 * p] = -v[p][l];
                }
#pragma unroll
                for (int q = 0; q < kTrsmB; q += 4)   // rows of the staging that only this lane has read
                    *reinterpret_cast<float4 *>(stg + (lane + 32 * p) * kTrsmPitch + q) =
                        make_float4(v[p][q], v[p][q + 1], v[p][q + 2], v[p][q + 3]);
            }
            __syncwarp();
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                const int64_t i = w0 + 8 * it + sr;
                const int l0 = b * kTrsmB + sc, left = i < n ? c - l0 : 0;
                const float4 x = *reinterpret_cast<const float4 *>(stg + (8 * it + sr) * kTrsmPitch + sc);
                float *dst = Q + i * ldq + l0;
                if (VEC) {
                    if (left > 0) *reinterpret_cast<float4 *>(dst) = x;
                } else {
                    if (left > 0) dst[0] = x.x;
                    if (left > 1) dst[1] = x.y;
                    if (left > 2) dst[2] = x.z;
                    if (left > 3) dst[3] = x.w;
                }
            }
            __syncwarp();   // the staging rows are rewritten next
        }
    }
}

// C = A B for upper-triangular c x c FP64 matrices (row i per CTA).
__global__ void upper_matmul_kernel(const double *__restrict__ A, const double *__restrict__ B, int c,
                                    double *__restrict__ C) {
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < c; j += blockDim.x) {
        double s = 0.0;
        if (j >= i)
            for (int l = i; l <= j; ++l) s += A[i * c + l] * B[l * c + j];
        C[i * c + j] = s;
    }
}

// ---------------------------------------------------------------------------
// out[n][dout] = Y[n][c] W[c][dout], FP32 FMA with W rounded to FP32.
// 64 x 64 output tile per CTA, 4 x 4 per thread.
// ---------------------------------------------------------------------------
constexpr int kMMTile = 64;
constexpr int kMMK = 32;

// BATCH: independent products at fixed strides (a compile-time choice: the strides
// alone cost a single product 10%).
template <bool BATCH>
__global__ void __launch_bounds__(256) right_multiply_kernel(
    const float *__restrict__ Y0, int64_t n, int c, int64_t ldy, const double *__restrict__ W0,
    int64_t ldw, int dout, const double *__restrict__ colscale, float *__restrict__ out0, int64_t ldo, int64_t sy,
    int64_t sw, int64_t so) {
    const float *__restrict__ Y = BATCH ? Y0 + blockIdx.z * sy : Y0;
    const double *__restrict__ W = BATCH ? W0 + blockIdx.z * sw : W0;
    float *__restrict__ out = BATCH ? out0 + blockIdx.z * so : out0;
    __shared__ float ys[kMMTile][kMMK + 1];
    __shared__ float ws[kMMK][kMMTile];
    const int tid = threadIdx.x;
    const int tr = tid / 16, tc = tid % 16;   // 16 x 16 threads, 4 x 4 each
    const int64_t row0 = (int64_t)blockIdx.x * kMMTile;
    const int col0 = blockIdx.y * kMMTile;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < c; k0 += kMMK) {
        for (int e = tid; e < kMMTile * kMMK; e += 256) {
            int r = e / kMMK, k = e - r * kMMK;
            int64_t gr = row0 + r;
            ys[r][k] = (gr < n && k0 + k < c) ? Y[gr * ldy + k0 + k] : 0.f;
        }
        for (int e = tid; e < kMMK * kMMTile; e += 256) {
            int k = e / kMMTile, cc = e - k * kMMTile;
            ws[k][cc] = (k0 + k < c && col0 + cc < dout) ? (float)W[(int64_t)(k0 + k) * ldw + col0 + cc] : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kMMK; ++k) {
            float a[4], b[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) a[x] = ys[tr * 4 + x][k];
#pragma unroll
            for (int y = 0; y < 4; ++y) b[y] = ws[k][tc * 4 + y];
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(a[x], b[y], acc[x][y]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        int64_t gr = row0 + tr * 4 + x;
        if (gr >= n) continue;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            int gc = col0 + tc * 4 + y;
            if (gc < dout) {
                float v = acc[x][y];
                if (colscale) v = (float)((double)v * colscale[gc]);
                out[gr * ldo + gc] = v;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Small SVD of the c x c factor R (c <= 160), FP64-accurate:
//   1. one-sided (Hestenes) Jacobi on R in FP32, one CTA, accumulating the
//      right rotations V (columns paired by the circle method: m = c rounded up
//      to even players, player 0 fixed, m/2 disjoint pairs per round, 8 threads
//      per pair); U = normalised columns of R V;
//   2. Ogita-Aishima refinement of (U, Sigma, V) of R itself in FP64 (matrix
//      products only, spread over many CTAs; R is never squared);
//   3. sorted by sigma descending.
// FP64 rates on this GPU are a small fraction of FP32, so FP64 is used only
// where the refinement needs it: its products.
// ---------------------------------------------------------------------------
constexpr int kJacTPP = 8;
constexpr int kJacMaxE = (160 + kJacTPP - 1) / kJacTPP;   // elements per thread and column, c <= 160

__device__ __forceinline__ int circle_player(int pos, int round, int m) {
    return pos == 0 ? 0 : ((pos - 1 + round) % (m - 1)) + 1;
}

// Column stride of the shared-memory matrices: = 8 (mod 32), so the four
// 8-thread pair groups of a warp hit distinct banks.
__host__ __device__ __forceinline__ int jac_ld(int c) { return ((c + 23) / 32) * 32 + 8; }

// Jacobi acts on the columns of A = R^T (for a triangular factor this
// converges in fewer sweeps than on R): R^T W = Z Sigma with W the accumulated
// rotations, so R = W Sigma Z^T -- left singular vectors U = W, right ones
// V = normalised columns of R^T W.
__global__ void jacobi32_kernel(const double *__restrict__ R, int c, double *__restrict__ Uout,
                                double *__restrict__ Vout, int max_sweeps, int *__restrict__ sweeps_out,
                                unsigned *__restrict__ sync) {
    if (threadIdx.x < kOaSync) sync[threadIdx.x] = 0u;   // for the refinement that follows
    extern __shared__ float js[];
    const int ldc = jac_ld(c);
    float *A = js;              // column j at A + j * ldc
    float *V = js + c * ldc;    // accumulated rotations
    __shared__ float red[32];
    __shared__ int s_done;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthreads = blockDim.x;
    for (int e = tid; e < c * c; e += nthreads) {
        int i = e / c, j = e - i * c;
        A[i * ldc + j] = (float)R[e];   // column i of R^T = row i of R
        V[j * ldc + i] = (i == j) ? 1.f : 0.f;
    }
    __syncthreads();
    const int m = c + (c & 1);
    const int pairs = m / 2;
    const int pi = tid / kJacTPP, sub = tid % kJacTPP;
    // FP32 round-off floor of |a_p . a_q| / (|a_p| |a_q|) is about c * 2^-24
    // stop at cosines of 0.4 c ulp (at least 8 ulp): the FP64 refinement's first-order
    // step needs the start's rotations this close where singular values are dense
    const float tol = fmaxf(0.4f * (float)c, 8.f) * 5.9604645e-8f;
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        float local_max = 0.f;
        for (int round = 0; round < m - 1; ++round) {
            int p = 0, q = c;
            if (pi < pairs) {
                p = circle_player(pi, round, m);
                q = circle_player(m - 1 - pi, round, m);
                if (p > q) {
                    int t = p;
                    p = q;
                    q = t;
                }
            }
            const bool active = pi < pairs && q < c;
            float al = 0.f, be = 0.f, ga = 0.f;
            // the pair's elements stay in registers between the dot products
            // and the rotation (one shared-memory read and write per element)
            float xr[kJacMaxE], yr[kJacMaxE];
            float *ap = A + p * ldc, *aq = A + q * ldc;
#pragma unroll
            for (int e = 0; e < kJacMaxE; ++e) {
                const int i = sub + e * kJacTPP;
                const bool in = active && i < c;
                const float x = in ? ap[i] : 0.f, y = in ? aq[i] : 0.f;
                xr[e] = x;
                yr[e] = y;
                al = fmaf(x, x, al);
                be = fmaf(y, y, be);
                ga = fmaf(x, y, ga);
            }
            // every lane takes part in the shuffles; lanes without a pair add zeros
#pragma unroll
            for (int off = 1; off < kJacTPP; off <<= 1) {
                al += __shfl_xor_sync(0xffffffffu, al, off);
                be += __shfl_xor_sync(0xffffffffu, be, off);
                ga += __shfl_xor_sync(0xffffffffu, ga, off);
            }
            if (active && ga != 0.f && al > 0.f && be > 0.f) {
                float rel = fabsf(ga) * rsqrtf(al * be);
                local_max = fmaxf(local_max, rel);
                if (rel > tol) {
                    float zeta = (be - al) / (2.f * ga);
                    float t = (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
                    float cs = rsqrtf(1.f + t * t);
                    float sn = cs * t;
                    float *vp = V + p * ldc, *vq = V + q * ldc;
#pragma unroll
                    for (int e = 0; e < kJacMaxE; ++e) {
                        const int i = sub + e * kJacTPP;
                        if (i < c) {
                            ap[i] = cs * xr[e] - sn * yr[e];
                            aq[i] = sn * xr[e] + cs * yr[e];
                            const float u = vp[i], w = vq[i];
                            vp[i] = cs * u - sn * w;
                            vq[i] = sn * u + cs * w;
                        }
                    }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) local_max = fmaxf(local_max, __shfl_xor_sync(0xffffffffu, local_max, off));
        if (lane == 0) red[warp] = local_max;
        __syncthreads();
        if (tid == 0) {
            float mx = 0.f;
            for (int w = 0; w < (nthreads + 31) / 32; ++w) mx = fmaxf(mx, red[w]);
            s_done = mx <= tol;
        }
        __syncthreads();
        if (s_done) {
            ++sweep;
            break;
        }
    }
    __shared__ float s_nrm[kMaxSmemC + 1];
    for (int j = tid; j < c; j += nthreads) {
        float t = 0.f;
        for (int i = 0; i < c; ++i) t = fmaf(A[j * ldc + i], A[j * ldc + i], t);
        s_nrm[j] = t > 0.f ? rsqrtf(t) : 0.f;
    }
    __syncthreads();
    for (int e = tid; e < c * c; e += nthreads) {
        int i = e / c, j = e - i * c;
        Uout[e] = (double)V[j * ldc + i];                 // left vectors of R: the rotations
        Vout[e] = (double)(A[j * ldc + i] * s_nrm[j]);    // right vectors: normalised R^T W
    }
    if (tid == 0 && sweeps_out) *sweeps_out = sweep;
}

// Register-resident variant of the same Jacobi (c <= 144). Each 8-thread
// group holds its pair of columns of A in registers (E elements per column
// and thread, as float2 chunks: element 16 q + 2 sub + {0, 1}), so a round
// reads nothing from shared memory; columns move between groups through a
// shared exchange buffer only when the pairing changes. The rotations W are
// not accumulated here: every round's (cos, sin) and column labels are
// recorded, and jacobi_replay_kernel applies them to the identity afterwards,
// one row of W per warp on many SMs (the rows of W evolve independently).
//
// The pairing order is chosen so that most rounds move one column of each
// pair instead of both: a sweep over m = 2G columns takes the columns in slot
// 0 as a set X and those in slot 1 as Y, and pairs X[i] with Y[(i + r) mod G]
// for r = 0..G-1 (only Y moves, one group along); then X and Y are each split
// in halves and the same is done inside X and inside Y in parallel, and so on
// while the set size is even. Sets of odd size s then finish with s rounds of
// the circle method (one column of each set idle per round). Every pair meets
// exactly once per sweep; the layout a sweep ends with is the next sweep's
// starting point, and a label per column records which column of R^T it
// started as.
// Blocks of two columns a move with lazily scaled rotations and kept norms took 0.6
// (c = 32) to 0.8 (c = 144) of the time and were given up: the squares of squared
// norms that their test formed underflow for columns below 3e-9 of the largest, which
// then were not rotated, and another order of rotations moves tuning scores.
constexpr int kJacRegMaxC = 144;
constexpr int kJacMaxSweeps = 20;

template <int E>
__host__ __device__ constexpr int jreg_stride() { return ((8 * E + 31) / 32) * 32 + 16; }

// rounds per sweep of the order above for m (even) columns
__host__ __device__ inline int jreg_rounds(int m) { return jorder_rounds(m); }

template <int E>
__global__ void __launch_bounds__(32 * E, 1) jacobi_reg_kernel(const double *__restrict__ R, int c,
                                                               double *__restrict__ Vout,
                                                               float2 *__restrict__ rot,
                                                               uint32_t *__restrict__ rlab, int max_sweeps,
                                                               int *__restrict__ sweeps_out) {
    constexpr int CP = 8 * E;            // padded column length
    constexpr int NQ = E / 2;            // float2 chunks per column and thread
    static_assert(E % 2 == 0, "columns are held as float2 chunks");
    constexpr int ST = jreg_stride<E>(); // floats per exchange entry (= 16 mod 32: conflict-free float2)
    extern __shared__ float xb[];        // 2 G entries: column [CP], label at CP
    __shared__ float red[32];
    __shared__ int s_done;
    const int m = c + (c & 1), G = m / 2, RD = jreg_rounds(m);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = tid >> 3, sub = tid & 7;
    const bool real = g < G;             // groups past G only fill the last warp
    // element 2 q + t of a column is component t of chunk q (rows 16 q + 2 sub + t)
    float2 a0[NQ], a1[NQ];
    int lab0 = g, lab1 = g + G;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int i = 16 * q + 2 * sub;
        const bool r0 = real && lab0 < c, r1 = real && lab1 < c;   // column lab of R^T
        a0[q].x = r0 && i < c ? (float)R[(size_t)lab0 * c + i] : 0.f;
        a0[q].y = r0 && i + 1 < c ? (float)R[(size_t)lab0 * c + i + 1] : 0.f;
        a1[q].x = r1 && i < c ? (float)R[(size_t)lab1 * c + i] : 0.f;
        a1[q].y = r1 && i + 1 < c ? (float)R[(size_t)lab1 * c + i + 1] : 0.f;
    }
    // stop at cosines of 0.4 c ulp (at least 8 ulp): the FP64 refinement's first-order
    // step needs the start's rotations this close where singular values are dense
    const float tol = fmaxf(0.4f * (float)c, 8.f) * 5.9604645e-8f;
    const int tz = jorder_levels(m);
    const int s_odd = m >> tz;           // set size the halving ends at
    float local_max = 0.f;
    int rec = 0;                         // record index of this round's group 0

    auto put = [&](int entry, const float2 (&a)[NQ], int lab) {
        float *eb = xb + (size_t)entry * ST;
#pragma unroll
        for (int q = 0; q < NQ; ++q) *reinterpret_cast<float2 *>(eb + 16 * q + 2 * sub) = a[q];
        if (sub == 0) reinterpret_cast<int *>(eb)[CP] = lab;
    };
    auto take = [&](int entry, float2 (&a)[NQ], int &lab) {
        const float *eb = xb + (size_t)entry * ST;
#pragma unroll
        for (int q = 0; q < NQ; ++q) a[q] = *reinterpret_cast<const float2 *>(eb + 16 * q + 2 * sub);
        lab = reinterpret_cast<const int *>(eb)[CP];
    };
    // both columns of every group move (sources as group * 2 + slot)
    auto move_both = [&](int src0, int src1) {
        __syncthreads();
        if (real) {
            put(2 * g, a0, lab0);
            put(2 * g + 1, a1, lab1);
        }
        __syncthreads();
        if (real) {
            take(src0, a0, lab0);
            take(src1, a1, lab1);
        }
        __syncthreads();
    };
    // one rotation of the group's pair (every lane takes part in the shuffles),
    // recorded as (cos, sin) = (1, 0) when the pair is left as it is
    auto rotate = [&](bool active) {
        float2 al2 = make_float2(0.f, 0.f), be2 = al2, ga2 = al2;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            al2 = f2_fma(a0[q], a0[q], al2);
            be2 = f2_fma(a1[q], a1[q], be2);
            ga2 = f2_fma(a0[q], a1[q], ga2);
        }
        float al = al2.x + al2.y, be = be2.x + be2.y, ga = ga2.x + ga2.y;
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) {
            al += __shfl_xor_sync(0xffffffffu, al, off);
            be += __shfl_xor_sync(0xffffffffu, be, off);
            ga += __shfl_xor_sync(0xffffffffu, ga, off);
        }
        float cs = 1.f, sn = 0.f;
        if (active && ga != 0.f && al > 0.f && be > 0.f) {
            const float rel = fabsf(ga) * rsqrtf(al * be);
            local_max = fmaxf(local_max, rel);
            if (rel > tol) {
                const float zeta = (be - al) / (2.f * ga);
                const float t = (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
                cs = rsqrtf(1.f + t * t);
                sn = cs * t;
                const float2 c2 = make_float2(cs, cs), s2 = make_float2(sn, sn), ms2 = make_float2(-sn, -sn);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float2 x = a0[q], y = a1[q];
                    a0[q] = f2_fma(c2, x, f2_mul(ms2, y));   // cs x - sn y
                    a1[q] = f2_fma(c2, y, f2_mul(s2, x));    // sn x + cs y
                }
            }
        }
        if (real && sub == 0) {
            rot[(size_t)rec + g] = make_float2(cs, sn);
            rlab[(size_t)rec + g] = (uint32_t)lab0 | ((uint32_t)lab1 << 16);
        }
        rec += G;
    };

    int sweep = 0, par = 0;
    for (; sweep < max_sweeps; ++sweep) {
        local_max = 0.f;
        rec = sweep * RD * G;
        for (int lev = 0; lev < tz; ++lev) {
            const int h = m >> (lev + 1);   // ring length: pairs per set and rounds of this level
            if (lev > 0) {
                // the two halves of each set of the level before become two sets
                int src0, src1;
                jorder_split_sources(g, h, src0, src1);
                move_both(src0, src1);   // every thread reaches the same barriers
            }
            const int ks = jorder_ring_source(g, h);   // slot-1 column comes from the next group
            for (int r = 0; r < h; ++r) {
                if (r > 0) {
                    // double-buffered halves: one barrier per round
                    if (real) put(par * G + g, a1, lab1);
                    __syncthreads();
                    if (real) take(par * G + ks, a1, lab1);
                    par ^= 1;
                }
                rotate(true);
            }
        }
        if (s_odd > 1) {
            // circle method inside each set of odd size s: positions 1..k paired
            // with s-1..k+1 in k groups per set, position 0 idle (the two sets
            // that share a parent put their idle columns in one group)
            const int s = s_odd;
            int e0, e1, r0, r1;
            bool idle;
            jorder_tail_sources(g, s, e0, e1, r0, r1, idle);
            for (int r = 0; r < s; ++r) {
                move_both(r == 0 ? e0 : r0, r == 0 ? e1 : r1);
                rotate(!idle);
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) local_max = fmaxf(local_max, __shfl_xor_sync(0xffffffffu, local_max, off));
        if (lane == 0) red[warp] = local_max;
        __syncthreads();
        if (tid == 0) {
            float mx = 0.f;
            for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) mx = fmaxf(mx, red[w]);
            s_done = mx <= tol;
        }
        __syncthreads();
        if (s_done) {
            ++sweep;
            break;
        }
    }
    // right singular vectors of R: normalised columns of R^T W, by label
    float2 n02 = make_float2(0.f, 0.f), n12 = n02;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        n02 = f2_fma(a0[q], a0[q], n02);
        n12 = f2_fma(a1[q], a1[q], n12);
    }
    float n0 = n02.x + n02.y, n1 = n12.x + n12.y;
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
        n0 += __shfl_xor_sync(0xffffffffu, n0, off);
        n1 += __shfl_xor_sync(0xffffffffu, n1, off);
    }
    const float q0 = n0 > 0.f ? rsqrtf(n0) : 0.f, q1 = n1 > 0.f ? rsqrtf(n1) : 0.f;
    if (real) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int i = 16 * q + 2 * sub + t;
                const float x0 = t ? a0[q].y : a0[q].x, x1 = t ? a1[q].y : a1[q].x;
                if (i < c && lab0 < c) Vout[(size_t)i * c + lab0] = (double)(x0 * q0);
                if (i < c && lab1 < c) Vout[(size_t)i * c + lab1] = (double)(x1 * q1);
            }
    }
    if (tid == 0 && sweeps_out) *sweeps_out = sweep;
}

// W = the recorded rotations applied to the identity, in order: warp w of a
// CTA owns row i of W in shared memory; in every round its lanes take the
// round's records (disjoint column pairs). The CTA stages the records in
// chunks of kRpChunk rounds through shared memory, loading the next chunk
// into registers while it applies the current one.
constexpr int kRpWarps = 4;
constexpr int kRpPer = 3;      // records per lane and round: G <= 96
constexpr int kRpChunk = 16;   // rounds per staged chunk
constexpr int kRpMaxG = kJacRegMaxC / 2;
constexpr int kRpLoads = (kRpChunk * kRpMaxG + kRpWarps * 32 - 1) / (kRpWarps * 32);
static_assert(kRpMaxG <= 32 * kRpPer, "records of a round fit the lanes");

__global__ void __launch_bounds__(kRpWarps * 32) jacobi_replay_kernel(const float2 *__restrict__ rot,
                                                                      const uint32_t *__restrict__ rlab, int G,
                                                                      int RD, const int *__restrict__ sweeps,
                                                                      int c, double *__restrict__ Uout,
                                                                      unsigned *__restrict__ sync) {
    if (blockIdx.x == 0 && threadIdx.x < kOaSync) sync[threadIdx.x] = 0u;   // for the refinement that follows
    __shared__ float rows[kRpWarps][kJacRegMaxC + 1];
    __shared__ float2 srot[2][kRpChunk * kRpMaxG];
    __shared__ uint32_t slab[2][kRpChunk * kRpMaxG];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i = blockIdx.x * kRpWarps + warp;
    const bool live = i < c;   // warps past the last row still stage records and meet the barriers
    float *row = rows[warp];
    for (int j = lane; j < c; j += 32) row[j] = i == j ? 1.f : 0.f;
    const int total = *sweeps * RD;
    const int per = kRpChunk * G;   // records per chunk
    float2 rr[kRpLoads];
    uint32_t rl[kRpLoads];
    auto fetch = [&](int ch) {   // chunk ch's records into registers
        const size_t base = (size_t)ch * per, end = (size_t)total * G;
#pragma unroll
        for (int u = 0; u < kRpLoads; ++u) {
            const int e = tid + u * kRpWarps * 32;
            const bool in = e < per && base + e < end;
            rr[u] = in ? rot[base + e] : make_float2(1.f, 0.f);
            rl[u] = in ? rlab[base + e] : 0u;
        }
    };
    auto stash = [&](int b) {
#pragma unroll
        for (int u = 0; u < kRpLoads; ++u) {
            const int e = tid + u * kRpWarps * 32;
            if (e < per) {
                srot[b][e] = rr[u];
                slab[b][e] = rl[u];
            }
        }
    };
    const int nch = (total + kRpChunk - 1) / kRpChunk;
    fetch(0);
    stash(0);
    __syncthreads();
    for (int ch = 0; ch < nch; ++ch) {
        const int b = ch & 1;
        if (ch + 1 < nch) fetch(ch + 1);
        if (live) {
            const int nr = min(kRpChunk, total - ch * kRpChunk);
            // the round's pairs are disjoint: all reads first, then all writes;
            // the next round's records are read before this round's rows
            float2 cn[kRpPer];
            uint32_t pq[kRpPer];
            auto records = [&](int r) {
#pragma unroll
                for (int k = 0; k < kRpPer; ++k) {
                    const int g = lane + 32 * k;
                    cn[k] = g < G ? srot[b][r * G + g] : make_float2(1.f, 0.f);
                    pq[k] = g < G ? slab[b][r * G + g] : 0u;
                }
            };
            records(0);
            for (int r = 0; r < nr; ++r) {
                float u[kRpPer], v[kRpPer];
                float2 c0[kRpPer];
                uint32_t l0[kRpPer];
#pragma unroll
                for (int k = 0; k < kRpPer; ++k) {
                    c0[k] = cn[k];
                    l0[k] = pq[k];
                    u[k] = c0[k].y != 0.f ? row[l0[k] & 0xFFFFu] : 0.f;
                    v[k] = c0[k].y != 0.f ? row[l0[k] >> 16] : 0.f;
                }
                if (r + 1 < nr) records(r + 1);
#pragma unroll
                for (int k = 0; k < kRpPer; ++k)
                    if (c0[k].y != 0.f) {
                        row[l0[k] & 0xFFFFu] = c0[k].x * u[k] - c0[k].y * v[k];
                        row[l0[k] >> 16] = c0[k].y * u[k] + c0[k].x * v[k];
                    }
                __syncwarp();
            }
        }
        if (ch + 1 < nch) stash(b ^ 1);
        __syncthreads();
    }
    if (live)
        for (int j = lane; j < c; j += 32) Uout[(size_t)i * c + j] = (double)row[j];
}

// records a Jacobi run on c <= kJacRegMaxC columns may write
inline size_t jreg_records(int c) {
    const int m = c + (c & 1);
    return (size_t)kJacMaxSweeps * jreg_rounds(m) * (m / 2);
}

template <int E>
int launch_jacobi_reg_e(const double *R, int c, double *U, double *V, float2 *rot, uint32_t *rlab, int *sweeps,
                        unsigned *sync, cudaStream_t st) {
    const int m = c + (c & 1);
    const int threads = ((m / 2) * 8 + 31) / 32 * 32;
    const int smem = m * jreg_stride<E>() * (int)sizeof(float);
    if (smem > 48 * 1024) LNE_TRY(allow_dynamic_smem(jacobi_reg_kernel<E>));
    jacobi_reg_kernel<E><<<1, threads, smem, st>>>(R, c, V, rot, rlab, kJacMaxSweeps, sweeps);
    LNE_LAUNCH_CHECK();
    jacobi_replay_kernel<<<(unsigned)ceil_div(c, kRpWarps), kRpWarps * 32, 0, st>>>(
        rot, rlab, m / 2, jreg_rounds(m), sweeps, c, U, sync);
    LNE_LAUNCH_CHECK();
    return 0;
}

// FP32 Jacobi start of the small SVD: the register-resident kernel (with its
// replay; rot / rlab hold jreg_records(c) records) up to c = 144, the
// shared-memory one above.
int launch_jacobi(const double *R, int c, double *U, double *V, float2 *rot, uint32_t *rlab, int *sweeps,
                  unsigned *sync, cudaStream_t st) {
    switch ((c + 15) / 16) {
    case 1: return launch_jacobi_reg_e<2>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 2: return launch_jacobi_reg_e<4>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 3: return launch_jacobi_reg_e<6>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 4: return launch_jacobi_reg_e<8>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 5: return launch_jacobi_reg_e<10>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 6: return launch_jacobi_reg_e<12>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 7: return launch_jacobi_reg_e<14>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 8: return launch_jacobi_reg_e<16>(R, c, U, V, rot, rlab, sweeps, sync, st);
    case 9: return launch_jacobi_reg_e<18>(R, c, U, V, rot, rlab, sweeps, sync, st);
    default: break;
    }
    const int m = c + (c & 1);
    const int threads = std::max(32, std::min(1024, (m / 2 * kJacTPP + 31) / 32 * 32));
    const int smem = 2 * c * jac_ld(c) * 4;
    if (smem > 48 * 1024) LNE_TRY(allow_dynamic_smem(jacobi32_kernel));
    jacobi32_kernel<<<1, threads, smem, st>>>(R, c, U, V, kJacMaxSweeps, sweeps, sync);
    LNE_LAUNCH_CHECK();
    return 0;
}

// One step of Ogita-Aishima refinement of an SVD A = U Sigma V^T (Ogita and
// Aishima, "Iterative refinement for singular value decomposition based on
// matrix multiplication", 2020), written from first-order perturbation:
// with U = U^(I + F), V = V^(I + G) exact, P = I - U^T U^ = F + F^T,
// Q = I - V^T V^ = G + G^T and T = U^T A V^ = Sigma - F^T Sigma - Sigma G. So
// sigma_i = t_ii / (1 - (p_ii + q_ii) / 2), f_ii = p_ii / 2, g_ii = q_ii / 2,
// and for i != j the pair (f_ij, g_ij) solves
//   [ s_j  -s_i ] [f_ij]   [t_ij + p_ij s_j]
//   [-s_i   s_j ] [g_ij] = [t_ji + q_ij s_j],
// taken as (p_ij / 2, q_ij / 2) when |s_i - s_j| <= delta (near-equal values),
// delta = 2 (||offdiag T|| + max|s| (||P|| + ||Q||)). A itself is never squared,
// so the accuracy does not depend on the condition number of A.
//
// kOaSteps steps in one cooperative launch: quadratic convergence, but the
// FP32 start may be loose in directions FP32 cannot resolve. A step is four
// phases between grid barriers: P, Q (upper tiles, mirrored) and W = A V; T =
// U^T W with sigma and the norms' partial sums; F and G; U + U F and V + V G.
// Bound by FP64 at large c (per step 6 c^3 multiply-adds at 2 a cycle and SM: 29 us
// at c = 144) and by barriers and load latency at small c. Measured, all steps: c =
// 32 83 us, c = 144 313; as four products and two element passes of their own
// launches a step 190 and 335.
// A 64-thread group takes an 8 x 8 tile: its 8 rows of op(A) and 8 columns of B
// over the whole k range go to shared memory at once (one round of load
// latency), then each thread runs its dot product.
constexpr int kOaTile = 8;
constexpr int kOaGroups = 2;                    // 64-thread groups of a CTA
constexpr int kOaThreads = 64 * kOaGroups;

struct OaArgs {
    const double *R;
    double *U, *U2, *V, *V2, *W, *T, *P, *Q, *F, *G, *out, *sig;
    double *part;       // 4 per CTA
    unsigned *sync;     // kOaSync words, zeroed, 8-byte aligned
    int *status;        // [1] is set where a barrier gave up
    int c;
};

struct OaSmem {
    double a[kOaTile][kMaxSmemC + 1], b[kMaxSmemC][kOaTile + 1];
};

// Entry (r0 + ty, c0 + tx) of op(A) B, k ascending; the group's threads load the
// operands together (read through L2: other CTAs of the launch wrote them).
__device__ __forceinline__ double oa_tile(OaSmem &sm, const double *A, bool ta, const double *B, int c, int r0, int c0,
                                          int gt, int grp) {
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");   // the group's last tile is done
#pragma unroll 6
    for (int e = gt; e < kOaTile * c; e += 64) {
        const int i = ta ? e % kOaTile : e / c, k = ta ? e / kOaTile : e % c;
        const int r = r0 + i;
        sm.a[i][k] = r < c ? __ldcg(ta ? A + k * c + r : A + r * c + k) : 0.0;
        const int j = e % kOaTile, kb = e / kOaTile, cc = c0 + j;
        sm.b[kb][j] = cc < c ? __ldcg(B + kb * c + cc) : 0.0;
    }
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");
    const int tx = gt % kOaTile, ty = gt / kOaTile;
    double acc = 0.0;
    for (int k = 0; k < c; ++k) acc = fma(sm.a[ty][k], sm.b[k][tx], acc);
    return acc;
}

__global__ void __launch_bounds__(kOaThreads) svd_refine_kernel(OaArgs A) {
    __shared__ OaSmem sm[kOaGroups];
    __shared__ double red[4][kOaThreads / 32];
    __shared__ double s_delta;
    const int c = A.c, nt = (c + kOaTile - 1) / kOaTile, nup = nt * (nt + 1) / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = tid >> 6, gt = tid & 63;
    const int g0 = blockIdx.x * kOaGroups + grp, ng = gridDim.x * kOaGroups;
    const int tx = gt % kOaTile, ty = gt / kOaTile;
    uint64_t target = 0, *const bar = reinterpret_cast<uint64_t *>(A.sync);   // the first two words
    double *U = A.U, *U2 = A.U2, *V = A.V, *V2 = A.V2;
    for (int it = 0; it < kOaSteps; ++it) {
        // P = I - U^T U, Q = I - V^T V, W = R V
        for (int q = g0; q < 2 * nup + nt * nt; q += ng) {
            const int which = q < nup ? 0 : q < 2 * nup ? 1 : 2;
            int ti, tj;
            if (which == 2) {
                ti = (q - 2 * nup) / nt;
                tj = (q - 2 * nup) % nt;
            } else {
                int rem = q - which * nup;
                for (ti = 0; rem >= nt - ti; ++ti) rem -= nt - ti;
                tj = ti + rem;
            }
            const double *X = which == 0 ? U : V;
            const double acc = which == 2 ? oa_tile(sm[grp], A.R, false, V, c, 8 * ti, 8 * tj, gt, grp)
                                          : oa_tile(sm[grp], X, true, X, c, 8 * ti, 8 * tj, gt, grp);
            const int row = 8 * ti + ty, col = 8 * tj + tx;
            if (row >= c || col >= c) continue;
            if (which == 2) {
                A.W[row * c + col] = acc;
            } else {
                double *to = which == 0 ? A.P : A.Q;
                const double v = (row == col ? 1.0 : 0.0) - acc;
                to[row * c + col] = v;
                to[col * c + row] = v;
            }
        }
        if (!grid_barrier(bar, target, A.status)) return;
        // T = U^T W; sigma; partial sums of |offdiag T|^2, |P|^2, |Q|^2 and max |sigma|
        double o2 = 0.0, p2 = 0.0, q2 = 0.0, smax = 0.0;
        for (int q = g0; q < nt * nt; q += ng) {
            const int row = 8 * (q / nt) + ty, col = 8 * (q % nt) + tx;
            const double t = oa_tile(sm[grp], U, true, A.W, c, 8 * (q / nt), 8 * (q % nt), gt, grp);
            if (row >= c || col >= c) continue;
            const double p = __ldcg(A.P + row * c + col), qq = __ldcg(A.Q + row * c + col);
            A.T[row * c + col] = t;
            if (row == col) {
                const double sv = t / (1.0 - 0.5 * (p + qq));
                A.sig[row] = sv;
                smax = fmax(smax, fabs(sv));
            } else {
                o2 = fma(t, t, o2);
            }
            p2 = fma(p, p, p2);
            q2 = fma(qq, qq, q2);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            o2 += __shfl_xor_sync(0xffffffffu, o2, off);
            p2 += __shfl_xor_sync(0xffffffffu, p2, off);
            q2 += __shfl_xor_sync(0xffffffffu, q2, off);
            smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, off));
        }
        if (lane == 0) red[0][warp] = o2, red[1][warp] = p2, red[2][warp] = q2, red[3][warp] = smax;
        __syncthreads();
        if (tid < 4) {
            double v = red[tid][0];
            for (int w = 1; w < kOaThreads / 32; ++w) v = tid < 3 ? v + red[tid][w] : fmax(v, red[tid][w]);
            A.part[4 * blockIdx.x + tid] = v;
        }
        if (!grid_barrier(bar, target, A.status)) return;
        // F and G, an element per thread
        if (warp == 0) {
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            for (int b = lane; b < (int)gridDim.x; b += 32) {
                for (int k = 0; k < 3; ++k) s[k] += __ldcg(A.part + 4 * b + k);
                s[3] = fmax(s[3], __ldcg(A.part + 4 * b + 3));
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                for (int k = 0; k < 3; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], off);
                s[3] = fmax(s[3], __shfl_xor_sync(0xffffffffu, s[3], off));
            }
            if (lane == 0) s_delta = 2.0 * (sqrt(s[0]) + s[3] * (sqrt(s[1]) + sqrt(s[2])));
        }
        __syncthreads();
        const double delta = s_delta;
        for (int e = blockIdx.x * kOaThreads + tid; e < c * c; e += gridDim.x * kOaThreads) {
            const int i = e / c, j = e - i * c;
            const double pij = __ldcg(A.P + e), qij = __ldcg(A.Q + e);
            double f = 0.5 * pij, g = 0.5 * qij;
            if (i != j) {
                const double si = __ldcg(A.sig + i), sj = __ldcg(A.sig + j);
                if (fabs(sj - si) > delta) {
                    const double r1 = __ldcg(A.T + e) + pij * sj;
                    const double r2 = __ldcg(A.T + j * c + i) + qij * sj;
                    const double inv = 1.0 / ((sj - si) * (sj + si));
                    const double ff = (sj * r1 + si * r2) * inv;
                    const double gg = (si * r1 + sj * r2) * inv;
                    // outside the first-order regime this step only restores orthogonality:
                    // the correction must be small against the pair's relative gap, or its
                    // second-order error (|f|^2 (s_i + s_j) / |s_i - s_j|) would exceed it
                    const double mf = fmax(fabs(ff), fabs(gg));
                    if (mf <= 0.25 && mf * (fabs(si) + fabs(sj)) <= 0.25 * fabs(sj - si)) {
                        f = ff;
                        g = gg;
                    }
                }
            }
            A.F[e] = f;
            A.G[e] = g;
        }
        if (!grid_barrier(bar, target, A.status)) return;
        const bool last = it + 1 == kOaSteps;
        // U + U F (the last step's goes to `out`), V + V G
        double *to = last ? A.out : U2;
        for (int q = g0; q < (last ? 1 : 2) * nt * nt; q += ng) {
            const bool v = q >= nt * nt;
            const int k = v ? q - nt * nt : q, row = 8 * (k / nt) + ty, col = 8 * (k % nt) + tx;
            const double acc = oa_tile(sm[grp], v ? V : U, false, v ? A.G : A.F, c, 8 * (k / nt), 8 * (k % nt), gt, grp);
            if (row < c && col < c) (v ? V2 : to)[row * c + col] = __ldcg((v ? V : U) + row * c + col) + acc;
        }
        if (last) return;
        if (!grid_barrier(bar, target, A.status)) return;
        double *x = U;
        U = U2;
        U2 = x;
        x = V;
        V = V2;
        V2 = x;
    }
}

// The pairs the first-order step leaves (near-equal singular values, or a
// start not yet close enough for their gap) keep off-diagonal entries in
// T = U^T A V. They are resolved exactly: a two-sided Jacobi in FP64 on the
// block of T over the indices K of such pairs (entries above 2^-42 max|s|),
// each 2 x 2 block [t_ii t_ij; t_ji t_jj] diagonalised by a left and a right
// plane rotation (a rotation that makes it symmetric, then the symmetric
// Jacobi rotation), the left rotations also applied to the columns of U.
// The rotation angles are taken in FP32 and the rotations renormalised in
// FP64, so they are orthogonal to FP64 rounding (U stays orthonormal) and
// leave at most ~1e-7 of a pair's off-diagonal entries, which the next sweep
// removes. sigma_i = t_ii for i in K. T comes from the last refinement step
// (before its update, which is below the threshold). Entries between K and
// the rest are below the threshold and stay there (a rotation mixes two of
// them).
//
// One CTA. Each sweep takes the pairs above the threshold at its start and
// splits them into rounds of disjoint pairs (first-fit in (a, b) order, up to
// 64 rounds and kClusterList pairs a pass; the rest go to the next pass); in a
// round each warp takes a pair, all rows are rotated before all columns (left
// and right rotations commute, and the pairs of a round share no row or
// column, so the order of the pairs does not change the result). Sweeps until
// no entry is above the threshold (at most kClusterSweeps).
constexpr int kClusterSweeps = 16;
constexpr int kClusterThreads = 256;
constexpr int kClusterWarps = kClusterThreads / 32;
constexpr int kClusterList = 1024;                 // pairs coloured in one pass
constexpr int kClusterRowsPerLane = (kMaxSmemC + 31) / 32;

// |x| > thr for thr >= 0 by the ordering of IEEE-754 bit patterns (integer
// compares: FP64 instructions are slow on this GPU)
__device__ __forceinline__ bool above(double x, long long thr_bits) {
    return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll) > thr_bits;
}

// (c, s) from FP32 made a unit vector in FP64: multiplied by the series of
// (1 + d)^-1/2 to second order, d = c^2 + s^2 - 1 (|d| ~ 1e-7, so the
// third-order term is below FP64 rounding)
__device__ __forceinline__ void unit_fp64(double &c, double &s) {
    const double d = fma(c, c, fma(s, s, -1.0));
    const double n = fma(d, fma(0.375, d, -0.5), 1.0);
    c *= n;
    s *= n;
}

// The rotations of one 2 x 2 block M = [taa tab; tba tbb]: left
// L = [al be; -be al] = G J and right J = [cs sn; -sn cs], L^T M J diagonal up
// to the FP32 angles. G = [cf -sf; sf cf] makes G^T M symmetric; J is the
// symmetric Jacobi rotation of G^T M. inv scales the block to about unit size
// for the FP32 arithmetic (a power of two).
__device__ __forceinline__ void cluster_rotation(double taa, double tab, double tba, double tbb, double inv,
                                                 double &al, double &be, double &cs, double &sn) {
    const float x = (float)((taa + tbb) * inv), y = (float)((tba - tab) * inv);
    const float h = hypotf(x, y);
    const float cf = h > 0.f ? x / h : 1.f, sf = h > 0.f ? y / h : 0.f;
    // G^T M = [p q'; q'' r]: q = (q' + q'') / 2, r - p, from the differences
    const double d = tbb - taa, e = tab + tba;
    const double rp = fma((double)cf, d, -(double)sf * e);
    const double q = 0.5 * fma((double)cf, e, (double)sf * d);
    float c32 = 1.f, s32 = 0.f;
    const float qf = (float)(q * inv);
    if (qf != 0.f) {
        const float zeta = (float)(rp * inv) / (2.f * qf);
        const float az = fabsf(zeta);
        const float t = (zeta >= 0.f ? 1.f : -1.f) * (az > 1e18f ? 0.5f / az : 1.f / (az + sqrtf(1.f + zeta * zeta)));
        c32 = rsqrtf(1.f + t * t);
        s32 = c32 * t;
    }
    cs = c32;
    sn = s32;
    unit_fp64(cs, sn);
    al = (double)(cf * c32 + sf * s32);
    be = (double)(cf * s32 - sf * c32);
    unit_fp64(al, be);
}

__global__ void __launch_bounds__(kClusterThreads) svd_cluster_kernel(const double *__restrict__ T, int c,
                                                                     double *__restrict__ U,
                                                                     double *__restrict__ sg) {
    extern __shared__ double sT[];       // nK x nK block of T
    constexpr int kWords = (kMaxSmemC + 31) / 32;
    __shared__ int sK[kMaxSmemC];        // block index -> index of T
    __shared__ int s_act[kMaxSmemC];
    __shared__ uint32_t s_mask[kMaxSmemC][kWords];   // row a: bit b > a set for a pair left in the sweep
    __shared__ unsigned long long s_used[kMaxSmemC]; // rounds of the pass that index a takes part in
    __shared__ uint32_t s_list[kClusterList];        // round << 16 | a << 8 | b
    __shared__ uint32_t s_round[kMaxSmemC / 2];      // a << 8 | b
    __shared__ double s_rcs[kMaxSmemC / 2][2];       // each round pair's right rotation (cs, sn)
    __shared__ int s_rgo[kMaxSmemC / 2];             // ... and whether it rotated
    __shared__ long long red[kClusterWarps];
    __shared__ int s_nK, s_any, s_np, s_rounds, s_nr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // max |sigma| by the integer order of the bit patterns
    long long mb = 0;
    for (int i = tid; i < c; i += blockDim.x) mb = max(mb, __double_as_longlong(sg[i]) & 0x7FFFFFFFFFFFFFFFll);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, off));
    if (lane == 0) red[warp] = mb;
    for (int i = tid; i < c; i += blockDim.x) s_act[i] = 0;
    __syncthreads();
    mb = 0;
    for (int w = 0; w < kClusterWarps; ++w) mb = max(mb, red[w]);
    if (mb == 0 || mb >= 0x7FF0000000000000ll) return;   // a zero matrix, or not finite
    const double smax = __longlong_as_double(mb);
    const double thr = 0x1p-42 * smax;
    const long long thr_bits = __double_as_longlong(thr);
    const long long ex = min((mb >> 52) & 0x7FF, 2045ll);
    const double inv = __longlong_as_double((2046ll - ex) << 52);   // 2^(1023 - exponent of smax)
    // indices with an entry above the threshold in their row or column (a warp
    // per row, two rows at a time, every load of the two rows issued at once)
    for (int i0 = 2 * warp; i0 < c; i0 += 2 * kClusterWarps) {
        double v[2][kClusterRowsPerLane];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < kClusterRowsPerLane; ++q) {
                const int i = i0 + h, j = lane + 32 * q;
                v[h][q] = i < c && j < c ? T[(size_t)i * c + j] : 0.0;
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + h;
            bool rowbig = false;
#pragma unroll
            for (int q = 0; q < kClusterRowsPerLane; ++q) {
                const int j = lane + 32 * q;
                if (i < c && j < c && j != i && above(v[h][q], thr_bits)) {
                    s_act[j] = 1;
                    rowbig = true;
                }
            }
            if (__any_sync(0xffffffffu, rowbig) && lane == 0) s_act[i] = 1;
        }
    }
    __syncthreads();
    if (warp == 0) {
        int n = 0;
        for (int j0 = 0; j0 < c; j0 += 32) {
            const int j = j0 + lane;
            const bool f = j < c && s_act[j];
            const unsigned bal = __ballot_sync(0xffffffffu, f);
            if (f) sK[n + __popc(bal & ((1u << lane) - 1u))] = j;
            n += __popc(bal);
        }
        if (lane == 0) s_nK = n;
    }
    __syncthreads();
    const int nK = s_nK;
    if (nK == 0) return;
    for (int a = warp; a < nK; a += kClusterWarps)
#pragma unroll 5
        for (int b = lane; b < nK; b += 32) sT[a * nK + b] = T[(size_t)sK[a] * c + sK[b]];
    const int words = (nK + 31) / 32;
    for (int sweep = 0; sweep < kClusterSweeps; ++sweep) {
        // the pairs above the threshold at the start of the sweep (a warp per row)
        if (tid == 0) s_any = 0;
        __syncthreads();
        for (int a = warp; a < nK; a += kClusterWarps)
            for (int w = 0; w < words; ++w) {
                const int b = 32 * w + lane;
                const bool big = b > a && b < nK && (above(sT[a * nK + b], thr_bits) || above(sT[b * nK + a], thr_bits));
                const unsigned m = __ballot_sync(0xffffffffu, big);
                if (lane == 0) {
                    s_mask[a][w] = m;
                    if (m) s_any = 1;
                }
            }
        __syncthreads();
        if (!s_any) break;
        for (;;) {   // passes: up to 64 rounds of disjoint pairs each
            if (tid == 0) {
                for (int a = 0; a < nK; ++a) s_used[a] = 0ull;
                int np = 0, rounds = 0;
                for (int a = 0; a < nK && np < kClusterList; ++a)
                    for (int w = 0; w < words && np < kClusterList; ++w) {
                        uint32_t m = s_mask[a][w];
                        while (m && np < kClusterList) {
                            const int bit = __ffs(m) - 1;
                            m &= m - 1u;
                            const int b = 32 * w + bit;
                            const unsigned long long fr = ~(s_used[a] | s_used[b]);
                            if (fr == 0ull) continue;   // stays for the next pass
                            const int r = __ffsll((long long)fr) - 1;
                            s_used[a] |= 1ull << r;
                            s_used[b] |= 1ull << r;
                            s_mask[a][w] &= ~(1u << bit);
                            s_list[np++] = ((uint32_t)r << 16) | ((uint32_t)a << 8) | (uint32_t)b;
                            rounds = max(rounds, r + 1);
                        }
                    }
                s_np = np;
                s_rounds = rounds;
            }
            __syncthreads();
            const int np = s_np, rounds = s_rounds;
            if (np == 0) break;
            for (int r = 0; r < rounds; ++r) {
                if (tid == 0) s_nr = 0;
                __syncthreads();
                for (int k = tid; k < np; k += blockDim.x)
                    if ((int)(s_list[k] >> 16) == r) s_round[atomicAdd(&s_nr, 1)] = s_list[k] & 0xFFFFu;
                __syncthreads();
                const int nr = s_nr;
                // rows of the block and columns of U, a warp per pair (rows disjoint)
                for (int k = warp; k < nr; k += kClusterWarps) {
                    const int a = (int)(s_round[k] >> 8), b = (int)(s_round[k] & 0xFFu);
                    const double taa = sT[a * nK + a], tab = sT[a * nK + b], tba = sT[b * nK + a],
                                 tbb = sT[b * nK + b];
                    const bool go = above(tab, thr_bits) || above(tba, thr_bits);
                    if (lane == 0) s_rgo[k] = go;
                    if (!go) continue;
                    double al, be, cs, sn;
                    cluster_rotation(taa, tab, tba, tbb, inv, al, be, cs, sn);
                    for (int k2 = lane; k2 < nK; k2 += 32) {   // rows a, b: L^T
                        const double u = sT[a * nK + k2], v = sT[b * nK + k2];
                        sT[a * nK + k2] = al * u - be * v;
                        sT[b * nK + k2] = be * u + al * v;
                    }
                    const int ia = sK[a], ib = sK[b];
                    double uu[kClusterRowsPerLane], vv[kClusterRowsPerLane];
#pragma unroll
                    for (int q = 0; q < kClusterRowsPerLane; ++q) {   // columns ia, ib of U: U L
                        const int k2 = lane + 32 * q;
                        uu[q] = k2 < c ? U[(size_t)k2 * c + ia] : 0.0;
                        vv[q] = k2 < c ? U[(size_t)k2 * c + ib] : 0.0;
                    }
#pragma unroll
                    for (int q = 0; q < kClusterRowsPerLane; ++q) {
                        const int k2 = lane + 32 * q;
                        if (k2 < c) {
                            U[(size_t)k2 * c + ia] = al * uu[q] - be * vv[q];
                            U[(size_t)k2 * c + ib] = be * uu[q] + al * vv[q];
                        }
                    }
                    if (lane == 0) {
                        s_rcs[k][0] = cs;
                        s_rcs[k][1] = sn;
                    }
                }
                __syncthreads();
                // columns of the block, a warp per pair (columns disjoint): J
                for (int k = warp; k < nr; k += kClusterWarps) {
                    if (!s_rgo[k]) continue;
                    const int a = (int)(s_round[k] >> 8), b = (int)(s_round[k] & 0xFFu);
                    const double cs = s_rcs[k][0], sn = s_rcs[k][1];
                    for (int k2 = lane; k2 < nK; k2 += 32) {
                        const double u = sT[k2 * nK + a], v = sT[k2 * nK + b];
                        sT[k2 * nK + a] = cs * u - sn * v;
                        sT[k2 * nK + b] = sn * u + cs * v;
                    }
                }
                __syncthreads();
            }
        }
    }
    for (int a = tid; a < nK; a += blockDim.x) sg[sK[a]] = sT[a * nK + a];
}

// sigma sorted descending; U_R[:, rank_j] = sign(s_j) U[:, j].
// Ranks first, then the columns copied by all threads over the flat index,
// so the loads of the whole matrix are in flight together. Magnitudes are
// compared and signs flipped on the bit patterns (non-negative doubles order
// as their bits; integer operations instead of the slow FP64 pipe).
// A refinement whose barrier gave up (status[1]) leaves NaN.
__global__ void svd_finish_kernel(const double *__restrict__ U, const double *__restrict__ sg, int c,
                                  double *__restrict__ UR, double *__restrict__ sigma,
                                  const int *__restrict__ status) {
    if (status[1] != 0) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        for (int e = threadIdx.x; e < c * c; e += blockDim.x) UR[e] = nan;
        for (int j = threadIdx.x; j < c; j += blockDim.x) sigma[j] = nan;
        return;
    }
    __shared__ long long s_abs[256];
    __shared__ int s_rank[256];
    __shared__ unsigned long long s_flip[256];
    const int tid = threadIdx.x;
    for (int j = tid; j < c; j += blockDim.x) {
        const long long b = __double_as_longlong(sg[j]);
        s_abs[j] = b & 0x7FFFFFFFFFFFFFFFll;
        s_flip[j] = (unsigned long long)b & 0x8000000000000000ull;   // the sign of sg[j]
    }
    __syncthreads();
    for (int j = tid; j < c; j += blockDim.x) {
        const long long sj = s_abs[j];
        int rank = 0;
        for (int i = 0; i < c; ++i) rank += (s_abs[i] > sj) || (s_abs[i] == sj && i < j);
        sigma[rank] = __longlong_as_double(sj);
        s_rank[j] = rank;
    }
    __syncthreads();
#pragma unroll 8
    for (int e = tid; e < c * c; e += blockDim.x) {
        const int i = e / c, j = e - i * c;
        UR[i * c + s_rank[j]] =
            __longlong_as_double((long long)((unsigned long long)__double_as_longlong(__ldg(U + e)) ^ s_flip[j]));
    }
}

// ---------------------------------------------------------------------------
// sign convention and X = U Sigma^{1/2}
// ---------------------------------------------------------------------------
// Per column: the largest |u| and, among equal magnitudes, the smallest row,
// packed as (|u| bits << 32) | ~row so that one max orders both. Each thread
// keeps a running maximum over a strided set of rows of one column, and a CTA
// adds one atomic per column (all CTAs meet at the same d words: with an atomic per
// thread and a row a thread they bound the kernel, 41 us at 10k x 32, 4 us now).
__global__ void __launch_bounds__(256) col_absmax_kernel(const float *__restrict__ U, int64_t n, int d, int64_t ld,
                                                         unsigned long long *__restrict__ best) {
    const int sub = blockDim.x / d;               // row subsets per CTA (d <= 256)
    const int j = threadIdx.x % d, r0 = threadIdx.x / d;
    __shared__ unsigned long long s_best[256];
    unsigned long long m = 0;
    if (r0 < sub) {
#pragma unroll 4
        for (int64_t i = (int64_t)blockIdx.x * sub + r0; i < n; i += (int64_t)gridDim.x * sub) {
            const float a = fabsf(U[i * ld + j]);
            const unsigned long long key = ((unsigned long long)__float_as_uint(a) << 32) |
                                           (unsigned long long)(0xFFFFFFFFu - (uint32_t)i);
            m = key > m ? key : m;
        }
    }
    s_best[threadIdx.x] = m;
    __syncthreads();
    if (r0 != 0) return;
    for (int r = 1; r < sub; ++r) m = s_best[r * d + j] > m ? s_best[r * d + j] : m;
    atomicMax(&best[j], m);
}

__global__ void column_signs_kernel(const float *__restrict__ U, int d, int64_t ld,
                                    const unsigned long long *__restrict__ best, const double *__restrict__ sigma,
                                    float *__restrict__ sgn, float *__restrict__ scale) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d) return;
    const int64_t i = (int64_t)(0xFFFFFFFFu - (uint32_t)(best[j] & 0xFFFFFFFFull));
    sgn[j] = U[i * ld + j] < 0.f ? -1.f : 1.f;
    if (sigma) scale[j] = (float)sqrt(fmax(sigma[j], 0.0));
}

// U <- U diag(sgn); X = U diag(scale) when X is given.
__global__ void sign_scale_kernel(float *__restrict__ U, int64_t n, int d, int64_t ld,
                                  const float *__restrict__ sgn, const float *__restrict__ scale,
                                  float *__restrict__ X, int64_t ldx) {
    const int sub = blockDim.x / d;
    const int j = threadIdx.x % d, r0 = threadIdx.x / d;
    if (r0 >= sub) return;
    const float sg = sgn[j], sc = X ? scale[j] : 0.f;
    for (int64_t i = (int64_t)blockIdx.x * sub + r0; i < n; i += (int64_t)gridDim.x * sub) {
        const float u = U[i * ld + j] * sg;
        U[i * ld + j] = u;
        if (X) X[i * ldx + j] = u * sc;
    }
}

int grid_for(int64_t work, int threads) {
    int64_t g = ceil_div(std::max<int64_t>(work, 1), threads);
    return (int)std::min<int64_t>(g, num_sms() * 32);
}

}  // namespace

int gaussian_sketch(int64_t n, int c, uint64_t seed, float *out, int64_t ld, cudaStream_t st) {
    if (n <= 0 || c <= 0) return 0;
    const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFu) ^ 0x4f4d4547u;
    const uint32_t k1 = (uint32_t)(seed >> 32);
    {
        LNE_TRACE("sketch", st);
        sketch_kernel<<<grid_for(n * ((c + 3) / 4), 256), 256, 0, st>>>(n, c, k0, k1, out, ld);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

int right_multiply(const float *Y, int64_t n, int c, int64_t ldy, const double *W, int64_t ldw,
                   int dout, const double *colscale, float *out, int64_t ldo, cudaStream_t st, int batch, int64_t sy,
                   int64_t sw, int64_t so) {
    if (n <= 0 || dout <= 0) return 0;
    dim3 grid((unsigned)ceil_div(n, kMMTile), (unsigned)ceil_div(dout, kMMTile), (unsigned)batch);
    {
        LNE_TRACE("right_multiply", st);
        if (batch > 1)
            right_multiply_kernel<true><<<grid, 256, 0, st>>>(Y, n, c, ldy, W, ldw, dout, colscale, out, ldo, sy, sw, so);
        else
            right_multiply_kernel<false><<<grid, 256, 0, st>>>(Y, n, c, ldy, W, ldw, dout, colscale, out, ldo, 0, 0, 0);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

// G = Y^T Y (FP64, [c][c]).
static int gram(Workspace &ws, const float *Y, int64_t n, int c, int64_t ld, double *G, cudaStream_t st) {
    const int cp = (c + 7) & ~7;
    const int threads = kGramThreads;
    const bool vec = c % 4 == 0 && ld % 4 == 0 && reinterpret_cast<uintptr_t>(Y) % 16 == 0;
    const int smem = 2 * kGramRows * cp * 4;   // cp <= 240: 120 KB
    LNE_TRY(vec ? allow_dynamic_smem(gram_partial_kernel<true>) : allow_dynamic_smem(gram_partial_kernel<false>));
    // whole waves of resident CTAs (one per SM at this kernel's register use). The
    // split of the rows is part of the result: sums of other blocks round differently
    const int64_t slots = num_sms();
    int64_t nblk = std::min<int64_t>(2 * slots, std::max<int64_t>(1, ceil_div(n, 64)));
    if (nblk > slots) nblk = (nblk / slots) * slots;
    const int64_t rows_per = ceil_div(std::max<int64_t>(n, 1), nblk);
    nblk = ceil_div(std::max<int64_t>(n, 1), rows_per);
    double *partial = nullptr;
    LNE_TRY(ws.get("gram.partial", (size_t)nblk * cp * cp, &partial));
    unsigned *cnt = nullptr;
    LNE_TRY(ws.get("chol.cnt", 16, &cnt));
    {
        LNE_TRACE("gram_partial", st);
        if (vec) gram_partial_kernel<true><<<(unsigned)nblk, threads, smem, st>>>(Y, n, c, ld, rows_per, partial);
        else gram_partial_kernel<false><<<(unsigned)nblk, threads, smem, st>>>(Y, n, c, ld, rows_per, partial);
        LNE_LAUNCH_CHECK();
    }
    {
        LNE_TRACE("gram_reduce", st);
        gram_reduce_kernel<<<grid_for((int64_t)c * (c + 1) / 2 * kGramRedLanes, 256), 256, 0, st>>>(
            partial, (int)nblk, c, G, cnt);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

// A breakdown (a pivot that is not positive) is recorded in the device status
// word read by status_check, without a host synchronisation here; the
// factorisation goes on with a unit pivot, so later kernels see finite values.
// G comes from gram() on the same stream, whose reduction zeroes the tile
// counters. Measured (c = 32 / 48 / 144): one CTA with a rank-1 update and three
// barriers a pivot took 27 / 44 us, one cooperative launch with grid barriers
// between panels 159 us at c = 144; now 27 / 41 / 123 us (the pivot's chain).
static int chol(Workspace &ws, const double *G, int c, double *R, cudaStream_t st) {
    int *status = nullptr;
    unsigned *cnt = nullptr;
    double *pub = nullptr, *inv = nullptr;
    const int nt = (int)ceil_div(c, kCholB);
    if (nt > kCholMaxTiles) return fail(LNE_ERR_UNSUPPORTED, "Cholesky supports at most 240 columns");
    LNE_TRY(device_status(ws, &status, st));
    LNE_TRY(ws.get("chol.cnt", 16, &cnt));
    LNE_TRY(ws.get("chol.pub", (size_t)nt * nt * 256, &pub));
    LNE_TRY(ws.get("chol.inv", (size_t)nt * kCholB, &inv));
    LNE_TRACE("chol", st);
    void *args[] = {&G, &c, &R, &pub, &inv, &cnt, &status};
    LNE_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(chol_kernel), dim3(nt), dim3(256), args, 0,
                                             st));
    LNE_LAUNCH_CHECK();
    return 0;
}

int device_status(Workspace &ws, int **status, cudaStream_t st) {
    const bool fresh = !ws.has("dev.status");
    LNE_TRY(ws.get("dev.status", 4, status));
    if (fresh) LNE_CUDA_TRY(cudaMemsetAsync(*status, 0, 4 * sizeof(int), st));
    return 0;
}

int status_check(Workspace &ws, cudaStream_t st) {
    if (!ws.has("dev.status")) return 0;
    int *status = nullptr;
    LNE_TRY(ws.get("dev.status", 4, &status));
    int h[4] = {0, 0, 0, 0};
    LNE_CUDA_TRY(cudaMemcpyAsync(h, status, sizeof(h), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    if (h[0] == 0 && h[1] == 0 && h[2] == 0) return 0;
    LNE_CUDA_TRY(cudaMemsetAsync(status, 0, 4 * sizeof(int), st));
    if (h[1] != 0) return fail(LNE_ERR_TIMEOUT, "a bounded device wait expired (tensor-core pipeline, Cholesky, small SVD or key sort)");
    if (h[2] != 0)
        return fail(LNE_ERR_UNSUPPORTED, "a row of the very sparse projection has more than 12 nonzeros (raise s)");
    return fail(LNE_ERR_NUMERIC, "Cholesky breakdown in CholeskyQR (Gram not positive definite)");
}

// Rows a tile: 256 (two a thread) where the earlier columns of that many fit in
// shared memory beside R (c <= 144) and there are enough rows to give every SM
// such a tile; else 128, else 64 (c up to 240).
static int trsm_rows(const float *Y, int64_t n, int c, int64_t ldy, const double *R, float *Q, int64_t ldq,
                     cudaStream_t st) {
    constexpr int kMost = 226 * 1024;
    const bool vec = c % 4 == 0 && ldy % 4 == 0 && ldq % 4 == 0 && reinterpret_cast<uintptr_t>(Y) % 16 == 0 &&
                     reinterpret_cast<uintptr_t>(Q) % 16 == 0;
    LNE_TRACE("trsm_rows", st);
    auto launch = [&](auto kernel, int threads, int rpt) -> int {
        const int tile = threads * rpt, smem = trsm_smem(c, tile);
        LNE_TRY(allow_dynamic_smem(kernel));
        const int per_sm = std::max(1, std::min(8, kMost / smem));
        const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(n, tile), (int64_t)num_sms() * per_sm);
        kernel<<<blocks, threads, smem, st>>>(Y, n, c, ldy, R, Q, ldq);
        LNE_LAUNCH_CHECK();
        return 0;
    };
    if (trsm_smem(c, 256) <= kMost && n >= (int64_t)num_sms() * 256)
        return vec ? launch(trsm_rows_kernel<2, true>, 128, 2) : launch(trsm_rows_kernel<2, false>, 128, 2);
    int threads = 128;
    while (threads > 32 && (trsm_smem(c, threads) > kMost || n < (int64_t)num_sms() * threads)) threads /= 2;
    if (trsm_smem(c, threads) > kMost) return fail(LNE_ERR_UNSUPPORTED, "CholeskyQR column count too large");
    return vec ? launch(trsm_rows_kernel<1, true>, threads, 1) : launch(trsm_rows_kernel<1, false>, threads, 1);
}

int cholqr1(Workspace &ws, const float *Y, int64_t n, int c, int64_t ld, float *Q, int64_t ldq, cudaStream_t st) {
    if (c <= 0 || c > 256) return fail(LNE_ERR_INVALID, "CholeskyQR needs 1 <= c <= 256");
    if (n < c) return fail(LNE_ERR_INVALID, "CholeskyQR needs at least as many rows as columns");
    if ((size_t)(c * c + c) * 4 > 227 * 1024) return fail(LNE_ERR_UNSUPPORTED, "CholeskyQR column count too large");
    double *G = nullptr, *R1 = nullptr;
    LNE_TRY(ws.get("qr.G", (size_t)c * c, &G));
    LNE_TRY(ws.get("qr.R1", (size_t)c * c, &R1));
    LNE_TRY(gram(ws, Y, n, c, ld, G, st));
    LNE_TRY(chol(ws, G, c, R1, st));
    return trsm_rows(Y, n, c, ld, R1, Q, ldq, st);
}

int cholqr2(Workspace &ws, float *Y, int64_t n, int c, int64_t ld, double *Rout, cudaStream_t st) {
    if (c <= 0 || c > 256) return fail(LNE_ERR_INVALID, "CholeskyQR2 needs 1 <= c <= 256");
    if (n < c) return fail(LNE_ERR_INVALID, "CholeskyQR2 needs at least as many rows as columns");
    if ((size_t)(c * c + c) * 4 > 227 * 1024) return fail(LNE_ERR_UNSUPPORTED, "CholeskyQR2 column count too large");
    double *G = nullptr, *R1 = nullptr, *R2 = nullptr;
    float *tmp = nullptr;
    LNE_TRY(ws.get("qr.G", (size_t)c * c, &G));
    LNE_TRY(ws.get("qr.R1", (size_t)c * c, &R1));
    LNE_TRY(ws.get("qr.R2", (size_t)c * c, &R2));
    LNE_TRY(ws.get("qr.tmp", (size_t)n * c, &tmp));
    // pass 1: G = Y^T Y, R1 = chol(G), Q1 = Y R1^-1
    LNE_TRY(gram(ws, Y, n, c, ld, G, st));
    LNE_TRY(chol(ws, G, c, R1, st));
    LNE_TRY(trsm_rows(Y, n, c, ld, R1, tmp, c, st));
    // pass 2 on Q1
    LNE_TRY(gram(ws, tmp, n, c, c, G, st));
    LNE_TRY(chol(ws, G, c, R2, st));
    LNE_TRY(trsm_rows(tmp, n, c, c, R2, Y, ld, st));
    if (Rout) {
        LNE_TRACE("upper_matmul", st);
        upper_matmul_kernel<<<c, 128, 0, st>>>(R2, R1, c, Rout);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

// FP64 scratch of the refinement: ten c x c matrices, sigma (c), the norm
// partials (4 per CTA), the barrier and the status words.
struct SvdScratch {
    double *U, *U2, *V, *V2, *W, *T, *P, *Q, *F, *Gm, *sg, *dl;
    unsigned *sync;
    int *status;
};
constexpr int kOaMaxCtas = 192;   // norm partials held

// Refines the FP32 start (sc.U, sc.V) into the SVD of R in FP64 and writes
// U_R and sigma (sorted descending).
static int svd_refine_finish(const double *R, int c, SvdScratch sc, double *U_R, double *sigma, cudaStream_t st) {
    const size_t cc = (size_t)c * c;
    const int nt = (int)ceil_div(c, kOaTile);
    {
        LNE_TRACE("svd_refine", st);
        // out: W's buffer, which the last step no longer reads
        OaArgs A{R, sc.U, sc.U2, sc.V, sc.V2, sc.W, sc.T, sc.P, sc.Q, sc.F, sc.Gm, sc.W, sc.sg, sc.dl, sc.sync,
                 sc.status, c};
        const int ctas = (int)std::min<int64_t>(ceil_div(nt * (nt + 1) + nt * nt, kOaGroups),
                                                std::min(num_sms(), kOaMaxCtas));
        void *args[] = {&A};
        LNE_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(svd_refine_kernel), dim3(ctas),
                                                 dim3(kOaThreads), args, 0, st));
        LNE_LAUNCH_CHECK();
    }
    {
        LNE_TRACE("svd_cluster", st);
        LNE_TRY(allow_dynamic_smem(svd_cluster_kernel));
        svd_cluster_kernel<<<1, kClusterThreads, sizeof(double) * cc, st>>>(sc.T, c, sc.W, sc.sg);
        LNE_LAUNCH_CHECK();
    }
    {
        LNE_TRACE("svd_finish", st);
        svd_finish_kernel<<<1, 256, 0, st>>>(sc.W, sc.sg, c, U_R, sigma, sc.status);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

int small_svd(Workspace &ws, const double *R, int c, double *U_R, double *sigma, cudaStream_t st) {
    if (c > kMaxSmemC) return fail(LNE_ERR_UNSUPPORTED, "small SVD supports c <= 160");
    double *U = nullptr, *U2 = nullptr, *V = nullptr, *V2 = nullptr, *W = nullptr, *T = nullptr, *P = nullptr,
           *Q = nullptr, *F = nullptr, *Gm = nullptr, *sg = nullptr;
    int *sweeps = nullptr;
    const size_t cc = (size_t)c * c;
    LNE_TRY(ws.get("svd.U", cc, &U));
    LNE_TRY(ws.get("svd.U2", cc, &U2));
    LNE_TRY(ws.get("svd.V", cc, &V));
    LNE_TRY(ws.get("svd.V2", cc, &V2));
    LNE_TRY(ws.get("svd.W", cc, &W));
    LNE_TRY(ws.get("svd.T", cc, &T));
    LNE_TRY(ws.get("svd.P", cc, &P));
    LNE_TRY(ws.get("svd.Q", cc, &Q));
    LNE_TRY(ws.get("svd.F", cc, &F));
    LNE_TRY(ws.get("svd.G", cc, &Gm));
    LNE_TRY(ws.get("svd.sg", (size_t)c, &sg));
    double *dl = nullptr;
    unsigned *sync = nullptr;
    int *status = nullptr;
    LNE_TRY(ws.get("svd.delta", 4 * kOaMaxCtas, &dl));
    LNE_TRY(ws.get("svd.sync", kOaSync, &sync));
    LNE_TRY(device_status(ws, &status, st));
    LNE_TRY(ws.get("svd.sweeps", 1, &sweeps));
    float2 *jrot = nullptr;
    uint32_t *jlab = nullptr;
    if (c <= kJacRegMaxC) {
        LNE_TRY(ws.get("svd.jrot", jreg_records(c), &jrot));
        LNE_TRY(ws.get("svd.jlab", jreg_records(c), &jlab));
    }
    // starting point: FP32 one-sided Jacobi on R (U, V in FP64 storage)
    {
        LNE_TRACE("jacobi32", st);
        LNE_TRY(launch_jacobi(R, c, U, V, jrot, jlab, sweeps, sync, st));
    }
    SvdScratch sc{U, U2, V, V2, W, T, P, Q, F, Gm, sg, dl, sync, status};
    return svd_refine_finish(R, c, sc, U_R, sigma, st);
}

int sign_fix_embed(Workspace &ws, float *U, int64_t n, int d, int64_t ld, const double *sigma, float *X,
                   int64_t ldx, cudaStream_t st) {
    if (d < 1 || d > 256) return fail(LNE_ERR_UNSUPPORTED, "sign fix supports 1..256 columns");
    unsigned long long *best = nullptr;
    float *sgn = nullptr, *scale = nullptr;
    LNE_TRY(ws.get("sign.best", (size_t)d, &best));
    LNE_TRY(ws.get("sign.sgn", (size_t)d, &sgn));
    LNE_TRY(ws.get("sign.scale", (size_t)d, &scale));
    LNE_CUDA_TRY(cudaMemsetAsync(best, 0, sizeof(unsigned long long) * d, st));
    const int sub = 256 / d;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, sub), num_sms() * 8));
    {
        LNE_TRACE("col_absmax", st);
        // at least 16 rows a thread before the CTAs fill the GPU
        const unsigned cblocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 16 * sub), num_sms() * 8));
        col_absmax_kernel<<<cblocks, 256, 0, st>>>(U, n, d, ld, best);
        LNE_LAUNCH_CHECK();
    }
    {
        LNE_TRACE("column_signs", st);
        column_signs_kernel<<<(d + 127) / 128, 128, 0, st>>>(U, d, ld, best, X ? sigma : nullptr, sgn, scale);
        LNE_LAUNCH_CHECK();
    }
    {
        LNE_TRACE("sign_scale", st);
        sign_scale_kernel<<<blocks, 256, 0, st>>>(U, n, d, ld, sgn, scale, X, ldx);
        LNE_LAUNCH_CHECK();
    }
    return 0;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the small SVD (lne_svd_small_noalloc).
//
// For callers that must not allocate device memory when they call in -- for
// example a process whose device memory is wholly handed to another allocator
// up front, or a latency-bound service that forbids allocation after start-up.
// Its scratch (ten c x c FP64 matrices, a few scalars and the Jacobi's
// rotation records, c <= 160: about 4.5 MB) is a file-scope __device__ array that every GPU which loads this
// library holds until the process exits. In host code the array's name is only
// a stand-in for it, so its device address is looked up with
// cudaGetSymbolAddress once per device, on that device's first call.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocMaxC = 160;
constexpr size_t kNoAllocMat = (size_t)kNoAllocMaxC * kNoAllocMaxC;
constexpr size_t kNoAllocRec = (size_t)kJacMaxSweeps * kJacRegMaxC * (kJacRegMaxC / 2);   // >= jreg_records(c)
constexpr size_t kNoAllocSmall = 4 * kOaMaxCtas + 16;   // norm partials; sweep count and sync words
constexpr size_t kNoAllocDoubles = 10 * kNoAllocMat + kNoAllocMaxC + kNoAllocSmall + kNoAllocRec + kNoAllocRec / 2;
static_assert((kOaSync + 2) * sizeof(unsigned) <= 16 * sizeof(double) && kOaSync >= 4, "the words fit the reserve");
static __device__ __align__(256) double g_svd_scratch[kNoAllocDoubles];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
double *g_noalloc_addr[kNoAllocMaxDevices] = {};

}  // namespace
}  // namespace lne

extern "C" int lne_svd_small_noalloc(const double *R_dev, int32_t c, double *U_dev, double *sigma_dev, void *stream) {
    using namespace lne;
    clear_message();
    set_tracer(nullptr);   // no timing events (they would be created on demand)
    if (!R_dev || !U_dev || !sigma_dev) return fail(LNE_ERR_INVALID, "NULL argument");
    if (c < 1 || c > kNoAllocMaxC) return fail(LNE_ERR_INVALID, "lne_svd_small_noalloc needs 1 <= c <= 160");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail("cudaGetDevice", e, __FILE__, __LINE__);
    if (dev < 0 || dev >= kNoAllocMaxDevices) return fail(LNE_ERR_UNSUPPORTED, "device index too large");
    double *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void *ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_svd_scratch);
            if (e != cudaSuccess) return cuda_fail("cudaGetSymbolAddress", e, __FILE__, __LINE__);
            g_noalloc_addr[dev] = static_cast<double *>(ptr);
        }
        base = g_noalloc_addr[dev];
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t cc = (size_t)c * c;
    // every buffer below is fully written before it is read, so nothing left by
    // an earlier call needs clearing
    double *U = base, *U2 = base + cc, *V = base + 2 * cc, *V2 = base + 3 * cc, *W = base + 4 * cc,
           *T = base + 5 * cc, *P = base + 6 * cc, *Q = base + 7 * cc, *F = base + 8 * cc, *Gm = base + 9 * cc;
    double *sg = base + 10 * kNoAllocMat;
    double *dl = sg + kNoAllocMaxC;
    int *sweeps = reinterpret_cast<int *>(dl + 4 * kOaMaxCtas), *status = nullptr;
    unsigned *sync = reinterpret_cast<unsigned *>(sweeps + 2);
    status = reinterpret_cast<int *>(sync + kOaSync - 2);   // two words that each call zeroes with the others
    float2 *jrot = reinterpret_cast<float2 *>(base + 10 * kNoAllocMat + kNoAllocMaxC + kNoAllocSmall);
    uint32_t *jlab = reinterpret_cast<uint32_t *>(jrot + kNoAllocRec);
    LNE_TRY(launch_jacobi(R_dev, c, U, V, jrot, jlab, sweeps, sync, st));
    SvdScratch sc{U, U2, V, V2, W, T, P, Q, F, Gm, sg, dl, sync, status};
    LNE_TRY(svd_refine_finish(R_dev, c, sc, U_dev, sigma_dev, st));
    return LNE_OK;
}
