// relearn_morton_order_noalloc over scratch that holds anything: the static array is filled
// with a byte pattern before each call, on both sides of the one-cluster form (40,960
// positions). The positions lie on a grid of exact quotients, so the codes are formed here
// in the same float operations. Exit status: 0, or 1 with the first call that differs.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <vector>

#include "octree.cu"

void rl::note_launch() {}

static uint32_t spread(uint32_t v)
{
    uint32_t r = 0;
    for (int b = 0; b < 10; ++b) r |= ((v >> b) & 1u) << (3 * b);
    return r;
}

static bool check(int64_t n, int fill)
{
    std::vector<float> p[3];
    std::vector<uint32_t> code(n, 0u);
    uint32_t seed = 12345u + (uint32_t)n;
    for (int a = 0; a < 3; ++a) {
        p[a].resize(n);
        for (int64_t i = 0; i < n; ++i) {
            seed = seed * 1664525u + 1013904223u;
            // the box is [0, 1024], so a coordinate's cell is its integer part (at most 1023)
            const uint32_t q = i == 0 ? 0u : i == 1 ? 1024u : (seed >> 12) % 1024u;
            p[a][i] = (float)q;
            code[i] |= spread(std::min(q, 1023u)) << a;
        }
    }
    std::vector<int32_t> want(n);
    std::iota(want.begin(), want.end(), 0);
    std::stable_sort(want.begin(), want.end(),
                     [&](int32_t a, int32_t b) { return code[a] < code[b]; });
    float *x[3];
    for (int a = 0; a < 3; ++a) {
        if (cudaMalloc(&x[a], n * 4) != cudaSuccess) return false;
        cudaMemcpy(x[a], p[a].data(), n * 4, cudaMemcpyHostToDevice);
    }
    uint32_t *codes;
    int32_t *perm;
    cudaMalloc(&codes, n * 4);
    cudaMalloc(&perm, n * 4);
    if (fill >= 0) {
        void *scratch = nullptr;
        cudaGetSymbolAddress(&scratch, rl::g_noalloc_scratch);
        cudaMemset(scratch, fill, rl::kNoAllocBytes);
    }
    const relearn_status s = relearn_morton_order_noalloc(n, x[0], x[1], x[2], nullptr, nullptr,
                                                          codes, perm, nullptr);
    std::vector<int32_t> got(n, -1);
    std::vector<uint32_t> got_codes(n, 0u);
    const cudaError_t e = cudaDeviceSynchronize();
    cudaMemcpy(got.data(), perm, n * 4, cudaMemcpyDeviceToHost);
    cudaMemcpy(got_codes.data(), codes, n * 4, cudaMemcpyDeviceToHost);
    bool ok = s == RELEARN_OK && e == cudaSuccess && got == want;
    for (int64_t k = 0; ok && k < n; ++k) ok = got_codes[k] == code[want[k]];
    if (!ok) printf("n %lld, fill %d: status %d, %s\n", (long long)n, fill, (int)s,
                    cudaGetErrorString(e));
    for (int a = 0; a < 3; ++a) cudaFree(x[a]);
    cudaFree(codes);
    cudaFree(perm);
    return ok;
}

int main()
{
    for (int64_t n : {700, 40960, 40961, 300000})
        for (int fill : {-1, 0, 1, 0xFF, 0x5A})
            if (!check(n, fill)) return 1;
    // a context made anew after a reset of the device (with nothing in flight) is served too
    if (cudaDeviceReset() != cudaSuccess) return 1;
    for (int64_t n : {700, 40961})
        if (!check(n, -1)) return 1;
    return 0;
}
