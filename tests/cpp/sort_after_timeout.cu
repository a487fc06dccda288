// A key sort that starts with the context's status word 1 (an expired wait) set must
// write nothing and report the time-out, and the next one must sort. The keys are
// whole, so nothing here can be placed out of range either way. The buffers have
// guard words behind them. Prints "ok".
#include <cstdio>
#include <algorithm>
#include <vector>

#include "lne.h"
#include "runtime.h"

int main() {
    lne::Workspace ws;
    const int64_t n = 3 * 4096 + 17, guard = 4096;
    std::vector<uint64_t> k(n + guard), back(n + guard);
    std::vector<uint32_t> v(n + guard);
    uint64_t x = 88172645463325252ull;
    for (int64_t i = 0; i < n + guard; ++i) {
        x ^= x << 13, x ^= x >> 7, x ^= x << 17;
        k[i] = x & 0xFFFFFFFFFFull;
        v[i] = (uint32_t)i;
    }
    uint64_t *a = nullptr, *b = nullptr;
    uint32_t *va = nullptr, *vb = nullptr;
    const size_t kb = sizeof(uint64_t) * (n + guard), vbytes = sizeof(uint32_t) * (n + guard);
    if (ws.get("a", (size_t)(n + guard), &a) || ws.get("b", (size_t)(n + guard), &b) ||
        ws.get("va", (size_t)(n + guard), &va) || ws.get("vb", (size_t)(n + guard), &vb))
        return std::printf("no memory\n"), 1;
    int *status = nullptr, set = 1;
    if (lne::device_status(ws, &status, nullptr)) return std::printf("no status\n"), 1;
    for (int vals = 0; vals < 2; ++vals) {
        bool in_alt = false;
        cudaMemcpy(a, k.data(), kb, cudaMemcpyHostToDevice);
        cudaMemcpy(va, v.data(), vbytes, cudaMemcpyHostToDevice);
        cudaMemset(b, 0xA5, kb);
        cudaMemset(vb, 0xA5, vbytes);
        cudaMemcpy(status + 1, &set, sizeof(int), cudaMemcpyHostToDevice);
        int rc = lne::radix_sort_u64(ws, a, b, vals ? va : nullptr, vals ? vb : nullptr, n, 0, 40, &in_alt, nullptr);
        if (rc != LNE_ERR_TIMEOUT) return std::printf("expected a time-out, got %d\n", rc), 1;
        cudaMemcpy(back.data(), a, kb, cudaMemcpyDeviceToHost);
        if (back != k) return std::printf("the keys changed\n"), 1;
        cudaMemcpy(back.data(), b, kb, cudaMemcpyDeviceToHost);
        for (uint64_t w : back)
            if (w != 0xA5A5A5A5A5A5A5A5ull) return std::printf("the other buffer was written\n"), 1;
        rc = lne::radix_sort_u64(ws, a, b, vals ? va : nullptr, vals ? vb : nullptr, n, 0, 40, &in_alt, nullptr);
        if (rc) return std::printf("the next sort failed: %d\n", rc), 1;
        cudaMemcpy(back.data(), in_alt ? b : a, kb, cudaMemcpyDeviceToHost);
        std::vector<uint64_t> ref(k.begin(), k.begin() + n);
        std::sort(ref.begin(), ref.end());
        if (!std::equal(ref.begin(), ref.end(), back.begin())) return std::printf("not sorted\n"), 1;
        cudaMemcpy(back.data(), a, kb, cudaMemcpyDeviceToHost);
        if (!std::equal(k.begin() + n, k.end(), back.begin() + n)) return std::printf("guard words written\n"), 1;
    }
    cudaError_t e = cudaDeviceSynchronize();
    std::printf(e == cudaSuccess ? "ok\n" : "%s\n", cudaGetErrorString(e));
    return e != cudaSuccess;
}
