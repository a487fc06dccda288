// Sorting and run-length counting of 64-bit pair keys, for graphs whose pair
// space does not fit a dense count table (the hash aggregation of Sec. 5.2
// done as sort + run-length instead: exact counts, deterministic order).
//
// radix_sort_u64: stable LSD radix sort, 8 bits per pass over bits [lo, hi),
// optional 32-bit payload. One kernel counts the digits of every pass; then a
// pass is one launch that reads and writes the keys once: a tile of 4096 keys
// ranks its keys by digit (each warp alone on 512 consecutive keys, by
// groups of equal digits and its own row of counters), stages them in shared
// memory in digit order, learns how many keys of each digit precede the tile from
// the tiles before it (decoupled lookback: a tile publishes its counts, then its
// prefix), and writes each digit's run contiguously. Bound by HBM: 16 bytes a key
// (24 with a payload) and pass.
// run_length: unique keys of a sorted array and their multiplicities (run starts
// counted per chunk of 1024 keys, one scan over the chunks, then a warp per chunk
// writes its runs); run_length_weighted sums a per-arc 64-bit weight over each run
// instead (edge downsampling).
#include "common.cuh"
#include "runtime.h"

namespace lne {
namespace {

constexpr int kRleThreads = 256;
constexpr int kRleChunk = 1024;   // keys a warp

// Exclusive scan of the 256 values v (one per thread) over the block.
__device__ __forceinline__ int64_t block_scan256(int64_t v, int64_t *s_warp) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int64_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    __syncthreads();
    return before + x - v;
}

// 256 threads with 16 keys each. Measured over 2e8 keys (five passes and the
// count): 5.4 ms without a payload at four CTAs an SM (three 5.7, 384 threads 5.8,
// 12 or 24 keys a thread 6.2 and 5.7), 6.8 ms with one at three (four spill: 7.2).
constexpr int kPassThreads = 256;
static_assert(kPassThreads == 256, "a thread per digit");
constexpr int kPassWarps = kPassThreads / 32;
constexpr int kPassItems = 16;
constexpr int kPassTile = kPassThreads * kPassItems;   // 4096 keys per tile
constexpr int kMaxPasses = 8;   // lo + 8 passes <= 64

// hist[p][d] = keys whose digit of pass p is d (zeroed before).
__global__ void __launch_bounds__(512) radix_count_kernel(const uint64_t *__restrict__ keys, int64_t n, int lo,
                                                          int passes, unsigned long long *__restrict__ hist) {
    __shared__ uint32_t h[kMaxPasses][256];
    for (int e = threadIdx.x; e < passes * 256; e += blockDim.x) h[e >> 8][e & 255] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
        uint64_t k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) k[u] = i + u * stride < n ? __ldcs(keys + i + u * stride) : 0ull;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i + u * stride >= n) break;
            for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(uint32_t)(k[u] >> (lo + 8 * p)) & 255u], 1u);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < passes * 256; e += blockDim.x) {
        const uint32_t c = h[e >> 8][e & 255];
        if (c) atomicAdd(hist + e, (unsigned long long)c);
    }
}

// hist[p][.] -> exclusive prefix sums over the digits, one CTA of 256 per pass.
__global__ void __launch_bounds__(256) radix_base_kernel(unsigned long long *__restrict__ hist) {
    __shared__ int64_t s_warp[8];
    unsigned long long *row = hist + 256 * blockIdx.x;
    const int64_t v = (int64_t)row[threadIdx.x];
    row[threadIdx.x] = (unsigned long long)block_scan256(v, s_warp);
}

// A tile's published word for a digit: the upper 8 bits say of which pass and
// what (2 pass + 1: the tile's own count, 2 pass + 2: the count up to and with
// the tile), the rest is the value. A pass does not see the words of the passes
// before it (smaller tags), so the array is zeroed once per sort.
__device__ __forceinline__ uint64_t tile_word(int tag, uint64_t v) { return ((uint64_t)tag << 56) | v; }
__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Which lanes of the warp hold the same digit: __match_any_sync for every fourth
// group of keys, eight ballots for the others. Match alone keeps its pipe busy 63%
// of the pass (7.3 ms for the five passes instead of 5.8, 384 threads), ballots
// alone the issue slots (6.0).
constexpr int kMatchEvery = 4;
// The lanes whose digit d is this lane's.
__device__ __forceinline__ unsigned same_digit(uint32_t d) {
    unsigned peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned one = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        peers &= ~(one ^ (unsigned)((int)(d << (31 - b)) >> 31));
    }
    return peers;
}

// One pass. Tiles are taken in order from a counter, so the tiles a tile waits
// for are running or done. A wait gives up after 2 s, sets status[1] and the CTA
// ends without writing its keys, as do CTAs that find it set while they wait. A CTA
// that finds it set when it starts does nothing: after a pass that gave up its
// output holds stale words, whose digits were never counted and would be placed
// past the buffers' ends.
template <bool VALS>
__global__ void __launch_bounds__(kPassThreads, VALS ? 3 : 4) radix_pass_kernel(
    const uint64_t *__restrict__ kin, const uint32_t *__restrict__ vin, int64_t n, int shift, int pass,
    const unsigned long long *__restrict__ base, uint64_t *__restrict__ words, unsigned *__restrict__ next_tile,
    uint64_t *__restrict__ kout, uint32_t *__restrict__ vout, int *status) {
    extern __shared__ uint64_t sk[];                                   // kPassTile staged keys
    uint32_t *sv = reinterpret_cast<uint32_t *>(sk + kPassTile);      // kPassTile staged payloads
    __shared__ uint16_t s_wc[kPassWarps][256];   // per warp and digit: count, then where its keys go in the tile
    __shared__ int64_t s_delta[256];             // output position minus tile position of the digit's keys
    __shared__ int64_t s_warp[8];
    __shared__ uint32_t s_tile;
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_tile = atomicAdd(next_tile, 1u);
        s_fail = *reinterpret_cast<volatile int *>(status + 1);
    }
    for (int e = tid; e < kPassWarps * 256; e += kPassThreads) s_wc[e >> 8][e & 255] = 0;
    __syncthreads();
    if (s_fail) return;
    const int64_t tile = s_tile, i0 = tile * kPassTile;
    const int nt = (int)imin64(kPassTile, n - i0);
    // the warp's 512 consecutive keys, all requested up front
    const int w0 = warp * (32 * kPassItems);
    uint64_t k[kPassItems];
#pragma unroll
    for (int i = 0; i < kPassItems; ++i) {
        const int li = w0 + 32 * i + lane;
        k[i] = li < nt ? __ldcs(kin + i0 + li) : ~0ull;   // past the end: the largest digit, ranked last
    }
    uint32_t rank[kPassItems / 2];   // among the warp's keys of the same digit, two to a register
#pragma unroll
    for (int i = 0; i < kPassItems; ++i) {
        const uint32_t d = (uint32_t)(k[i] >> shift) & 255u;
        const unsigned peers = i % kMatchEvery == 0 ? __match_any_sync(0xffffffffu, d) : same_digit(d);
        const uint32_t before = s_wc[warp][d];
        const uint32_t lr = (uint32_t)__popc(peers & ((1u << lane) - 1u));
        if (i & 1) rank[i / 2] |= (before + lr) << 16;
        else rank[i / 2] = before + lr;
        __syncwarp();
        if (lr == 0) s_wc[warp][d] = (uint16_t)(before + (uint32_t)__popc(peers));
        __syncwarp();
    }
    __syncthreads();
    uint64_t *mine = words + tile * 256 + tid;   // thread = digit from here on
    int64_t count = 0;
    uint32_t lbase = 0;   // start of the digit in the tile
    {   // warps' counts -> their starting ranks; the tile's count is published
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < kPassWarps; ++w) {
            const uint32_t x = s_wc[w][tid];
            s_wc[w][tid] = (uint16_t)c;
            c += x;
        }
        count = c - (tid == 255 ? (uint32_t)(kPassTile - nt) : 0u);
        st_relaxed(mine, tile_word(2 * pass + (tile == 0 ? 2 : 1), (uint64_t)count));
        lbase = (uint32_t)block_scan256(count, s_warp);
#pragma unroll
        for (int w = 0; w < kPassWarps; ++w) s_wc[w][tid] += (uint16_t)lbase;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPassItems; ++i) {
        const int li = w0 + 32 * i + lane;
        const uint32_t d = (uint32_t)(k[i] >> shift) & 255u;
        const uint32_t pos = s_wc[warp][d] + ((i & 1) ? rank[i / 2] >> 16 : rank[i / 2] & 0xffffu);
        sk[pos] = k[i];
        if (VALS && li < nt) sv[pos] = __ldcs(vin + i0 + li);
    }
    {   // keys of digit tid in the tiles before: four words at a time
        int64_t sum = 0;
        bool done = tile == 0;
        uint64_t t0 = 0;
        for (int64_t q = tile - 1; !done;) {
            uint64_t x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = q - u >= 0 ? ld_relaxed(words + (q - u) * 256 + tid) : 0ull;
            bool moved = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int tag = (int)(x[u] >> 56);
                if (done || tag < 2 * pass + 1) break;   // not published yet: read it again
                sum += (int64_t)(x[u] & 0x00FFFFFFFFFFFFFFull);
                done = tag == 2 * pass + 2;
                --q;
                moved = true;
            }
            if (!done && !moved) {
                uint64_t t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t0 == 0) t0 = t;
                if (t - t0 > 2000000000ull || *reinterpret_cast<volatile int *>(status + 1) != 0) {
                    atomicExch(status + 1, 1);
                    s_fail = 1;
                    break;
                }
            }
        }
        if (tile > 0 && done) st_relaxed(mine, tile_word(2 * pass + 2, (uint64_t)(sum + count)));
        s_delta[tid] = (int64_t)base[tid] + sum - (int64_t)lbase;
    }
    __syncthreads();
    if (s_fail) return;
    for (int li = tid; li < nt; li += kPassThreads) {
        const uint64_t x = sk[li];
        const int64_t g = s_delta[(uint32_t)(x >> shift) & 255u] + li;
        kout[g] = x;
        if (VALS) vout[g] = sv[li];
    }
}

// Run starts of a sorted array, counted per chunk of kRleChunk keys (a warp each).
__global__ void __launch_bounds__(kRleThreads) rle_count_kernel(const uint64_t *__restrict__ keys, int64_t n,
                                                                uint32_t *__restrict__ chunk_cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t chunk = ((int64_t)blockIdx.x * kRleThreads + threadIdx.x) >> 5;
    const int64_t i0 = chunk * kRleChunk;
    if (i0 >= n) return;
    const int64_t iend = imin64(n, i0 + kRleChunk);
    uint32_t c = 0;
#pragma unroll 8
    for (int64_t g = i0 + lane; g < iend; g += 32) c += (g == 0 || keys[g] != keys[g - 1]) ? 1u : 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) chunk_cnt[chunk] = c;
}

// Unique keys and their run lengths, a warp per chunk: 32 consecutive keys at a
// time, the run starts among them by ballot, so reads and writes are coalesced
// (a thread per 32 consecutive keys read 32 sectors a load and took 2.4 of
// run_length's 2.9 ms at 2e8 keys). A run that starts and ends in the chunk is
// stored; the pieces of one that crosses a chunk's edge are added atomically
// (integer sums, so the result does not depend on the order), which keeps a run
// of any length parallel. The outputs are zeroed beforehand. WEIGHTED: instead of
// the length, the 64-bit sum of w[arc] over the run's payloads.
template <bool WEIGHTED>
__global__ void __launch_bounds__(kRleThreads) rle_write_kernel(const uint64_t *__restrict__ keys, int64_t n,
                                                                const int64_t *__restrict__ chunk_off,
                                                                uint64_t *__restrict__ ukeys,
                                                                uint32_t *__restrict__ counts,
                                                                const uint32_t *__restrict__ arcs,
                                                                const uint64_t *__restrict__ w,
                                                                uint64_t *__restrict__ wsum) {
    constexpr int kAhead = 8;   // loads in flight a lane
    const int lane = threadIdx.x & 31;
    const int64_t chunk = ((int64_t)blockIdx.x * kRleThreads + threadIdx.x) >> 5;
    const int64_t i0 = chunk * kRleChunk;
    if (i0 >= n) return;   // whole warps
    const int64_t iend = imin64(n, i0 + kRleChunk);
    auto store = [&](int64_t run, uint64_t v) {
        if (WEIGHTED) wsum[run] = v;
        else counts[run] = (uint32_t)v;
    };
    auto add = [&](int64_t run, uint64_t v) {
        if (WEIGHTED) atomicAdd(reinterpret_cast<unsigned long long *>(wsum) + run, (unsigned long long)v);
        else atomicAdd(counts + run, (uint32_t)v);
    };
    int64_t run = chunk_off[chunk] - 1;   // the run that is open
    uint64_t acc = 0;                     // its sum so far in this chunk
    bool here = false;                    // whether it started in this chunk
    uint64_t before = i0 > 0 ? keys[i0 - 1] : 0ull;
    for (int64_t g0 = i0; g0 < iend; g0 += 32 * kAhead) {
        uint64_t k[kAhead];
        uint64_t x[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int64_t g = g0 + 32 * u + lane;
            k[u] = g < iend ? keys[g] : 0ull;
            x[u] = WEIGHTED ? (g < iend ? __ldg(w + arcs[g]) : 0ull) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int64_t g = g0 + 32 * u + lane;
            const int nv = (int)imin64(32, iend - (g0 + 32 * u));   // keys of this step
            if (nv <= 0) break;
            uint64_t prev = __shfl_up_sync(0xffffffffu, k[u], 1);
            if (lane == 0) prev = before;
            before = __shfl_sync(0xffffffffu, k[u], nv - 1);
            const bool head = lane < nv && (g == 0 || k[u] != prev);
            const unsigned heads = __ballot_sync(0xffffffffu, head);
            uint64_t upto = (uint64_t)lane + 1;   // sum over the lanes up to and with this one
            if (WEIGHTED) {
                upto = x[u];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint64_t y = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += y;
                }
            }
            const uint64_t all = WEIGHTED ? __shfl_sync(0xffffffffu, upto, 31) : (uint64_t)nv;
            if (heads == 0) {
                acc += all;
                continue;
            }
            const int first = __ffs(heads) - 1, last = 31 - __clz(heads);
            const unsigned above = lane < 31 ? heads & ~((2u << lane) - 1u) : 0u;   // starts after this lane
            const int next = above ? __ffs(above) - 1 : 32;
            uint64_t below = __shfl_up_sync(0xffffffffu, upto, 1);
            if (lane == 0) below = 0;
            const uint64_t at_next = __shfl_sync(0xffffffffu, upto, (next - 1) & 31);
            acc += __shfl_sync(0xffffffffu, below, first);
            if (lane == 0) {   // the open run ends here
                if (here) store(run, acc);
                else if (acc) add(run, acc);
            }
            if (head) {
                const int64_t r = run + 1 + __popc(heads & ((1u << lane) - 1u));
                ukeys[r] = k[u];
                if (next < 32) store(r, at_next - below);
            }
            run += __popc(heads);
            acc = all - __shfl_sync(0xffffffffu, below, last);
            here = true;
        }
    }
    if (lane == 0) {
        if (here && (iend >= n || keys[iend] != before)) store(run, acc);
        else if (acc) add(run, acc);
    }
}

// Number of keys below `key` in a sorted array (one thread, binary search).
__global__ void lower_bound_kernel(const uint64_t *__restrict__ keys, int64_t n, uint64_t key,
                                   int64_t *__restrict__ out) {
    int64_t lo = 0, hi = n;   // keys[0, lo) < key <= keys[hi, n)
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (keys[mid] < key) lo = mid + 1; else hi = mid;
    }
    *out = lo;
}

}  // namespace

int count_below(Workspace &ws, const uint64_t *keys, int64_t n, uint64_t key, int64_t *count, cudaStream_t st) {
    int64_t *d = nullptr;
    LNE_TRY(ws.temp("sort.bound", 1, &d));
    lower_bound_kernel<<<1, 1, 0, st>>>(keys, n, key, d);
    LNE_LAUNCH_CHECK();
    LNE_CUDA_TRY(cudaMemcpyAsync(count, d, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    return 0;
}

// Measured over 2e8 keys of 38 bits (five passes) and 1.1e8 mirrored ones with a
// payload (five passes before, three over the row bits now): 14.3 ms with a
// histogram, a scan and a scatter launch a pass (the scatter with four CTA
// barriers per 256 keys), 7.5 ms now with the one count of all digits (0.58 ms).
int radix_sort_u64(Workspace &ws, uint64_t *keys, uint64_t *keys_alt, uint32_t *vals, uint32_t *vals_alt,
                   int64_t n, int lo, int hi, bool *in_alt, cudaStream_t st) {
    *in_alt = false;
    if (n <= 1 || hi <= lo) return 0;
    const int passes = (hi - lo + 7) / 8;
    // the last digit is whole: the padding of a last tile has to be the largest one
    if (lo < 0 || hi > 64 || lo + 8 * passes > 64) return fail(LNE_ERR_INVALID, "radix sort bits out of range");
    const int64_t ntiles = ceil_div(n, (int64_t)kPassTile);
    uint64_t *words = nullptr;
    unsigned long long *hist = nullptr;
    unsigned *next = nullptr;
    int *status = nullptr;
    LNE_TRY(ws.temp("sort.words", (size_t)256 * ntiles, &words));
    LNE_TRY(ws.get("sort.hist", (size_t)256 * kMaxPasses, &hist));
    LNE_TRY(ws.get("sort.next", kMaxPasses, &next));
    LNE_TRY(device_status(ws, &status, st));
    const int smem = kPassTile * (8 + (vals ? 4 : 0));
    LNE_TRY(allow_dynamic_smem(radix_pass_kernel<true>));
    LNE_TRY(allow_dynamic_smem(radix_pass_kernel<false>));
    {
        LNE_TRACE("radix_count", st);
        LNE_CUDA_TRY(cudaMemsetAsync(words, 0, sizeof(uint64_t) * 256 * (size_t)ntiles, st));
        LNE_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * 256 * kMaxPasses, st));
        LNE_CUDA_TRY(cudaMemsetAsync(next, 0, sizeof(unsigned) * kMaxPasses, st));
        radix_count_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n, 2048), num_sms() * 4), 512, 0, st>>>(
            keys, n, lo, passes, hist);
        LNE_LAUNCH_CHECK();
        radix_base_kernel<<<passes, 256, 0, st>>>(hist);
        LNE_LAUNCH_CHECK();
    }
    uint64_t *ka = keys, *kb = keys_alt;
    uint32_t *va = vals, *vb = vals_alt;
    for (int p = 0; p < passes; ++p) {
        LNE_TRACE("radix_pass", st);
        if (vals)
            radix_pass_kernel<true><<<(unsigned)ntiles, kPassThreads, smem, st>>>(
                ka, va, n, lo + 8 * p, p, hist + 256 * p, words, next + p, kb, vb, status);
        else
            radix_pass_kernel<false><<<(unsigned)ntiles, kPassThreads, smem, st>>>(
                ka, nullptr, n, lo + 8 * p, p, hist + 256 * p, words, next + p, kb, nullptr, status);
        LNE_LAUNCH_CHECK();
        std::swap(ka, kb);
        std::swap(va, vb);
        *in_alt = !*in_alt;
    }
    return status_check(ws, st);   // an expired wait leaves keys unwritten: nothing may use them
}

namespace {

int run_length_impl(Workspace &ws, const uint64_t *keys, int64_t n, uint64_t *ukeys, uint32_t *counts,
                    const uint32_t *arcs, const uint64_t *w, uint64_t *wsum, int64_t *nunique, cudaStream_t st) {
    *nunique = 0;
    if (n <= 0) return 0;
    const int64_t nchunks = ceil_div(n, (int64_t)kRleChunk);
    const unsigned grid = (unsigned)ceil_div(n, (int64_t)kRleChunk * (kRleThreads / 32));
    uint32_t *cc = nullptr;
    int64_t *coff = nullptr;
    LNE_TRY(ws.get("rle.cnt", (size_t)nchunks, &cc));
    LNE_TRY(ws.get("rle.off", (size_t)nchunks + 1, &coff));
    LNE_TRACE("run_length", st);
    rle_count_kernel<<<grid, kRleThreads, 0, st>>>(keys, n, cc);
    LNE_LAUNCH_CHECK();
    LNE_TRY(scan_exclusive_u32_to_i64(cc, coff, nchunks, st));
    int64_t u = 0;
    LNE_CUDA_TRY(cudaMemcpyAsync(&u, coff + nchunks, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    if (wsum) LNE_CUDA_TRY(cudaMemsetAsync(wsum, 0, sizeof(uint64_t) * (size_t)u, st));
    else LNE_CUDA_TRY(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * (size_t)u, st));
    if (wsum)
        rle_write_kernel<true><<<grid, kRleThreads, 0, st>>>(keys, n, coff, ukeys, nullptr, arcs, w, wsum);
    else
        rle_write_kernel<false><<<grid, kRleThreads, 0, st>>>(keys, n, coff, ukeys, counts, nullptr, nullptr, nullptr);
    LNE_LAUNCH_CHECK();
    LNE_CUDA_TRY(cudaStreamSynchronize(st));
    *nunique = u;
    return 0;
}

}  // namespace

int run_length(Workspace &ws, const uint64_t *keys, int64_t n, uint64_t *ukeys, uint32_t *counts,
               int64_t *nunique, cudaStream_t st) {
    return run_length_impl(ws, keys, n, ukeys, counts, nullptr, nullptr, nullptr, nunique, st);
}

int run_length_weighted(Workspace &ws, const uint64_t *keys, const uint32_t *arcs, const uint64_t *w, int64_t n,
                        uint64_t *ukeys, uint64_t *wsum, int64_t *nunique, cudaStream_t st) {
    return run_length_impl(ws, keys, n, ukeys, nullptr, arcs, w, wsum, nunique, st);
}

}  // namespace lne
