// The key sort and the run lengths at the edges of their tiles (4096 keys) and chunks
// (1024 keys), against std::stable_sort and a loop: full last tiles, last tiles of one
// and two keys, bit ranges that start and end inside a byte, all-ones keys (which look
// like the padding of the last tile), with and without a payload. Prints "ok".
#include <algorithm>
#include <cstdio>
#include <numeric>
#include <random>
#include <vector>

#include "lne.h"
#include "runtime.h"

template <typename T>
static std::vector<T> down(const T *d, size_t n) {
    std::vector<T> h(n);
    cudaMemcpy(h.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost);
    return h;
}

static int fails(const char *what, int64_t n, int lo, int hi, int kind) {
    std::printf("%s: n %lld bits [%d, %d) kind %d\n", what, (long long)n, lo, hi, kind);
    return 1;
}

int main() {
    lne::Workspace ws;
    std::mt19937_64 rng(3);
    const int64_t sizes[] = {1, 2, 31, 33, 1023, 1024, 1025, 4094, 4095, 4096, 4097, 4098, 8191, 8192, 8193, 12288, 12289};
    const int ranges[][2] = {{0, 8}, {0, 22}, {0, 38}, {0, 40}, {0, 64}, {11, 22}, {17, 34}, {31, 62}, {5, 14}};
    for (int64_t n : sizes)
        for (const auto &r : ranges)
            for (int kind = 0; kind < 3; ++kind) {   // random, few values, half of them all ones in the range
                const int lo = r[0], hi = r[1];
                const int width = hi - lo, top = lo + 8 * ((width + 7) / 8);
                // bits from hi to the last compared byte's end have to order alike: zero, but
                // for whole keys of ones
                const uint64_t in = hi == 64 ? ~0ull : (1ull << hi) - 1ull;
                std::vector<uint64_t> k(n);
                std::vector<uint32_t> v(n);
                std::iota(v.begin(), v.end(), 0u);
                for (auto &x : k) {
                    x = rng() & in;
                    if (kind == 1) x = (rng() % 3) << lo;
                    if (kind == 2 && (rng() & 1)) x = ~0ull;
                }
                const uint64_t mask = (top >= 64 ? ~0ull : (1ull << top) - 1ull) & ~((1ull << lo) - 1ull);
                std::vector<uint32_t> order(v);
                std::stable_sort(order.begin(), order.end(), [&](uint32_t a, uint32_t b) { return (k[a] & mask) < (k[b] & mask); });
                for (int vals = 0; vals < 2; ++vals) {
                    uint64_t *a, *b;
                    uint32_t *va, *vb;
                    if (ws.get("a", (size_t)n, &a) || ws.get("b", (size_t)n, &b) || ws.get("va", (size_t)n, &va) ||
                        ws.get("vb", (size_t)n, &vb))
                        return fails("no memory", n, lo, hi, kind);
                    cudaMemcpy(a, k.data(), 8 * n, cudaMemcpyHostToDevice);
                    cudaMemcpy(va, v.data(), 4 * n, cudaMemcpyHostToDevice);
                    bool alt = false;
                    if (lne::radix_sort_u64(ws, a, b, vals ? va : nullptr, vals ? vb : nullptr, n, lo, hi, &alt, nullptr))
                        return fails("sort failed", n, lo, hi, kind);
                    const auto sk = down(alt ? b : a, n);
                    const auto sv = down(alt ? vb : va, n);
                    for (int64_t i = 0; i < n; ++i)
                        if (sk[i] != k[order[i]] || (vals && sv[i] != order[i])) return fails("order", n, lo, hi, kind);
                }
                if (lo != 0) continue;
                // run lengths of the sorted keys, and sums of a 64-bit weight over the runs
                std::vector<uint64_t> s(n), w(n), uk, sum;
                std::vector<uint32_t> arcs(n), cnt;
                for (int64_t i = 0; i < n; ++i) {
                    s[i] = k[order[i]];
                    arcs[i] = (uint32_t)(rng() % n);
                    w[i] = rng() >> 20;
                }
                std::sort(s.begin(), s.end());
                for (int64_t i = 0; i < n; ++i) {
                    if (i == 0 || s[i] != s[i - 1]) uk.push_back(s[i]), cnt.push_back(0), sum.push_back(0);
                    ++cnt.back();
                    sum.back() += w[arcs[i]];
                }
                uint64_t *ds, *du, *dw, *dsum;
                uint32_t *dc, *da;
                if (ws.get("s", (size_t)n, &ds) || ws.get("u", (size_t)n, &du) || ws.get("w", (size_t)n, &dw) ||
                    ws.get("sum", (size_t)n, &dsum) || ws.get("c", (size_t)n, &dc) || ws.get("arcs", (size_t)n, &da))
                    return fails("no memory", n, lo, hi, kind);
                cudaMemcpy(ds, s.data(), 8 * n, cudaMemcpyHostToDevice);
                cudaMemcpy(dw, w.data(), 8 * n, cudaMemcpyHostToDevice);
                cudaMemcpy(da, arcs.data(), 4 * n, cudaMemcpyHostToDevice);
                int64_t u = 0;
                if (lne::run_length(ws, ds, n, du, dc, &u, nullptr) || u != (int64_t)uk.size() || down(du, u) != uk ||
                    down(dc, u) != cnt)
                    return fails("run lengths", n, lo, hi, kind);
                if (lne::run_length_weighted(ws, ds, da, dw, n, du, dsum, &u, nullptr) || u != (int64_t)uk.size() ||
                    down(du, u) != uk || down(dsum, u) != sum)
                    return fails("run sums", n, lo, hi, kind);
            }
    {   // a last digit that reaches past bit 63 is refused
        uint64_t *a, *b;
        bool alt = false;
        if (ws.get("a", (size_t)64, &a) || ws.get("b", (size_t)64, &b)) return fails("no memory", 64, 1, 64, 0);
        if (lne::radix_sort_u64(ws, a, b, nullptr, nullptr, 64, 1, 64, &alt, nullptr) != LNE_ERR_INVALID)
            return fails("not refused", 64, 1, 64, 0);
    }
    const cudaError_t e = cudaDeviceSynchronize();
    std::printf(e == cudaSuccess ? "ok\n" : "%s\n", cudaGetErrorString(e));
    return e != cudaSuccess;
}
