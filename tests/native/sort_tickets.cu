// A pass of the radix sort whose ticket counter starts high, as it can when another sort
// draws from the same counter: tiles past the grid touch nothing. The tile states lie
// between guard words that have to stay as they are. Exit status: 0, or 1 with the first
// guard word that changed.
#include <cstdio>
#include <vector>

#include "sort.cu"

void rl::note_launch() {}

int main()
{
    using namespace rl;
    constexpr int64_t n = 3 * kTile + 5, tiles = 4, words = tiles * kRadix;
    constexpr int64_t guard = 2 * tiles * kRadix; // farther than any ticket below reaches
    const uint32_t mark = 0xA5A5A5A5u;
    for (uint32_t first : {0u, 1u, 3u, 4u, 7u}) {
        uint32_t *keys[2], *hist, *state[2];
        int32_t *vals[2];
        for (int k = 0; k < 2; ++k) {
            cudaMalloc(&keys[k], n * 4);
            cudaMalloc(&vals[k], n * 4);
            cudaMemset(keys[k], 0, n * 4);
            cudaMemset(vals[k], 0, n * 4);
            cudaMalloc(&state[k], (words + 2 * guard) * 4);
            cudaMemset(state[k], 0xA5, (words + 2 * guard) * 4);
            // the tiles before the first ticket have published that they hold nothing
            std::vector<uint32_t> s(words, 0u);
            if (k == 0)
                for (int64_t i = 0; i < words && i < (int64_t)first * kRadix; ++i)
                    s[i] = state_of_prefix(0u);
            cudaMemcpy(state[k] + guard, s.data(), words * 4, cudaMemcpyHostToDevice);
        }
        cudaMalloc(&hist, kHead * 4);
        cudaMemset(hist, 0, kHead * 4);
        uint32_t *ticket = hist + kMaxPasses * kRadix;
        cudaMemcpy(ticket, &first, 4, cudaMemcpyHostToDevice);
        pass_kernel<uint32_t><<<(unsigned)tiles, kThreads>>>(
            keys[0], vals[0], keys[1], vals[1], n, nullptr, 0, hist, ticket, ticket + kMaxPasses,
            state[0] + guard, state[1] + guard, nullptr);
        if (cudaDeviceSynchronize() != cudaSuccess) return 1;
        for (int k = 0; k < 2; ++k) {
            std::vector<uint32_t> s(words + 2 * guard);
            cudaMemcpy(s.data(), state[k], s.size() * 4, cudaMemcpyDeviceToHost);
            for (int64_t i = 0; i < (int64_t)s.size(); ++i)
                if ((i < guard || i >= guard + words) && s[i] != mark) {
                    printf("first ticket %u: state set %d, word %lld past the start\n", first, k,
                           (long long)(i - guard));
                    return 1;
                }
        }
        for (int k = 0; k < 2; ++k) {
            cudaFree(keys[k]);
            cudaFree(vals[k]);
            cudaFree(state[k]);
        }
        cudaFree(hist);
    }
    return 0;
}
