// Stable LSD radix sort of (key, int32 value) pairs with 8-bit digits, one pass over the
// data per digit (the published one-sweep scheme of Adinets and Merrill 2022, on the
// decoupled look-back of Merrill and Garland 2016): a first kernel counts the digits of every position at once; each pass
// then takes its tiles by ticket, ranks a tile's keys (each warp with eight votes per key, the
// warps ordered by a per-digit prefix), publishes the tile's digit counts and adds up those of
// the tiles before it (decoupled look-back, one thread per digit), and scatters.
// The element count may live on the device (grids are sized by capacity and tiles past
// the count do nothing), so the sort needs no host round trip.
//
// A tile only waits for tiles with smaller tickets, which are held by blocks already
// running that publish their counts before they wait themselves, so every wait ends; each
// is still bounded (kSortSpin reads, then RELEARN_ERR_TIMEOUT in the status word, no tile
// waits any more, and the sort's result is void).
//
// Against a count, a device-wide scan of the tiles' counts and a scatter per digit (three
// kernels that each read or write everything), with match.any for the ranks (600 cycles
// for 32 different digits, eight votes 130) and scattered writes: the Morton order of
// 700,001 positions 143 -> 75 us, a pass 26 -> 9 us. Bound by latency: one tile's loads,
// ranks, look-back (a few L2 round trips) and writes, 2 to 3 tiles per SM. Blocks of 512
// threads, 4 keys each: 300,000 / 700,001 / 2^20 positions 54 / 76 / 98 us; 8 keys 60 /
// 80 / 93; 256 threads of 8 keys 59 / 79 / 102, of 16 keys 75 / 108 / 125.
#include "internal.h"
#include "tile_state.h"

namespace rl {

namespace {
#ifndef RELEARN_SORT_THREADS
#define RELEARN_SORT_THREADS 512
#endif
#ifndef RELEARN_SORT_ITEMS
#define RELEARN_SORT_ITEMS 4
#endif
constexpr int kThreads = RELEARN_SORT_THREADS;
constexpr int kWarps = kThreads / 32;
constexpr int kRadix = 256;
constexpr int kMaxPasses = 8;
constexpr int kItems = RELEARN_SORT_ITEMS;   // keys per thread
constexpr int kTile = kThreads * kItems;      // keys per block
constexpr int kSortSpin = 1 << 18;

__device__ __forceinline__ int64_t bounded_count(int64_t max_n, const int32_t *d_count)
{
    if (!d_count) return max_n;
    int64_t c = *d_count;
    if (c < 0) c = 0;
    return c < max_n ? c : max_n;
}

// Digit counts of every pass: hist[pass][digit] (zeroed before).
template <typename K>
__global__ void __launch_bounds__(kThreads)
    hist_kernel(const K *__restrict__ keys, int64_t max_n, const int32_t *d_count, int passes,
                uint32_t *__restrict__ hist)
{
    __shared__ uint32_t h[kMaxPasses * kRadix];
    for (int i = threadIdx.x; i < passes * kRadix; i += kThreads) h[i] = 0;
    __syncthreads();
    const int64_t n = bounded_count(max_n, d_count);
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * kThreads) {
        const K k = keys[i];
        for (int p = 0; p < passes; ++p)
            atomicAdd(&h[p * kRadix + ((uint32_t)(k >> (8 * p)) & 0xFFu)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kThreads)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// One pass. hist: this pass's digit counts; ticket, abort: zeroed before; state: this
// pass's tile states, zeroed before; next_state: the next pass's, zeroed here.
template <typename K>
__global__ void __launch_bounds__(kThreads)
    pass_kernel(const K *__restrict__ keys_in, const int32_t *__restrict__ vals_in,
                K *__restrict__ keys_out, int32_t *__restrict__ vals_out, int64_t max_n,
                const int32_t *d_count, int shift, const uint32_t *__restrict__ hist,
                uint32_t *ticket, uint32_t *abort_, uint32_t *state, uint32_t *next_state,
                int32_t *status)
{
    __shared__ uint32_t wcnt[kWarps][kRadix];
    __shared__ uint32_t s_base[kRadix], s_sum[kWarps], s_loc[kWarps];
    __shared__ uint32_t s_tile;
    __shared__ K s_key[kTile];
    __shared__ int32_t s_val[kTile];
    const int64_t n = bounded_count(max_n, d_count);
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    for (int i = threadIdx.x; i < kWarps * kRadix; i += kThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const int64_t tile = s_tile;
    // Sorts that share scratch and overlap (relearn_morton_order_noalloc states that such
    // calls race) draw from one ticket counter: their results are void, but no tile past
    // this grid's has a state to write.
    if (tile >= gridDim.x) return;
    if (threadIdx.x < kRadix) next_state[tile * kRadix + threadIdx.x] = 0;
    const int64_t tile0 = tile * kTile;
    if (tile0 >= n) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = tile0 + (int64_t)warp * (32 * kItems);
    const uint32_t lt = lanemask_lt();
    K k[kItems];
    int32_t v[kItems];
    uint32_t rank[kItems];
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        const int64_t i = base + s * 32 + lane;
        const bool ok = i < n;
        k[s] = ok ? keys_in[i] : ~K(0);
        v[s] = ok ? vals_in[i] : 0;
    }
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        // keys past the end rank after every other key of their digit (they are the tile's
        // last) and are not counted
        const uint32_t dig = (uint32_t)(k[s] >> shift) & 0xFFu;
        uint32_t peers = 0xffffffffu; // lanes with this digit
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (dig >> b) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
        }
        const uint32_t live = __ballot_sync(0xffffffffu, base + s * 32 + lane < n);
        const uint32_t before = wcnt[warp][dig];
        __syncwarp();
        if ((peers & lt) == 0u) wcnt[warp][dig] = before + __popc(peers & live);
        __syncwarp();
        rank[s] = before + __popc(peers & lt);
    }
    __syncthreads();
    { // thread d < 256: digit d of the tile
        const int d = threadIdx.x;
        const bool on = d < kRadix;
        volatile uint32_t *st = state;
        uint32_t cnt = 0, total = 0;
        if (on) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t c = wcnt[w][d];
                wcnt[w][d] = cnt;
                cnt += c;
            }
            st[tile * kRadix + d] = tile == 0 ? state_of_prefix(cnt) : state_of_count(cnt);
            total = hist[d];
        }
        // where digit d starts among all keys, and in the tile
        uint32_t inc = total, loc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            const uint32_t u = __shfl_up_sync(0xffffffffu, loc, o);
            if (lane >= o) {
                inc += t;
                loc += u;
            }
        }
        if (lane == 31) {
            s_sum[warp] = inc;
            s_loc[warp] = loc;
        }
        __syncthreads();
        if (on) {
            uint32_t start = inc - total;
            loc -= cnt;
            for (int w = 0; w < warp; ++w) {
                start += s_sum[w];
                loc += s_loc[w];
            }
#pragma unroll
            for (int w = 0; w < kWarps; ++w) wcnt[w][d] += loc;
            // the counts of the tiles before this one, the nearest eight at a time: the words
            // themselves are added up, and what marks them is taken off at the end
            uint32_t words = 0;
            int spin = 0;
            int64_t t = tile - 1;
            while (t >= 0) {
                uint32_t f[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    f[q] = t - q >= 0 ? (uint32_t)st[(t - q) * kRadix + d] : state_of_prefix(0u);
                bool done = false;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (done || !state_published(f[q])) break; // read again
                    words += f[q];
                    done = state_is_prefix(f[q]);
                    --t;
                }
                if (done) break;
                if (!state_published(f[0]) &&
                    (++spin >= kSortSpin || *(volatile uint32_t *)abort_ != 0u)) {
                    if (status) set_status(status, RELEARN_ERR_TIMEOUT);
                    *(volatile uint32_t *)abort_ = 1u;
                    break;
                }
            }
            const uint32_t prefix =
                tile > 0 ? state_sum(words, (uint32_t)(tile - 1 - t)) : 0u;
            if (tile > 0) st[tile * kRadix + d] = state_of_prefix(prefix + cnt);
            s_base[d] = start + prefix - loc;
        }
    }
    __syncthreads();
    // through shared memory in digit order, so that consecutive threads write consecutive
    // places of a digit's run (direct scattered writes take a sector per key and per value:
    // a pass over 700,001 pairs 23 us against 17.7)
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        const uint32_t dig = (uint32_t)(k[s] >> shift) & 0xFFu;
        const uint32_t at = wcnt[warp][dig] + rank[s];
        if (base + s * 32 + lane < n) {
            s_key[at] = k[s];
            s_val[at] = v[s];
        }
    }
    __syncthreads();
    const int m = (int)min((int64_t)kTile, n - tile0);
#pragma unroll 4
    for (int j = threadIdx.x; j < m; j += kThreads) {
        const K key = s_key[j];
        const uint32_t pos = s_base[(uint32_t)(key >> shift) & 0xFFu] + j;
        if (pos < n) { // unless a wait ran out
            keys_out[pos] = key;
            vals_out[pos] = s_val[j];
        }
    }
}

// Scratch: the passes' digit counts, tickets, the abort flag and the word of
// sort_zero_word, then two sets of tile states, used in turn (each pass clears the next
// one's).
constexpr int64_t kHead = kMaxPasses * kRadix + kMaxPasses + 8;

template <typename K>
cudaError_t radix_sort(K *keys, K *keys_alt, int32_t *vals, int32_t *vals_alt, int64_t max_n,
                       const int32_t *d_count, int end_bit, SortScratch &s, cudaStream_t st,
                       int *which, bool counted)
{
    *which = 0;
    if (max_n <= 0 || end_bit <= 0) return cudaSuccess;
    const int passes = (end_bit + 7) / 8;
    const int64_t nb = (max_n + kTile - 1) / kTile;
    if (sort_blocks_needed(max_n) > s.max_blocks || nb > 0x7fffffff || passes > kMaxPasses)
        return cudaErrorInvalidValue;
    uint32_t *hist = reinterpret_cast<uint32_t *>(s.hist);
    uint32_t *ticket = hist + kMaxPasses * kRadix, *abort_ = ticket + kMaxPasses;
    uint32_t *state[2] = {hist + kHead, hist + kHead + nb * kRadix};
    if (!counted) {
        const cudaError_t e = cudaMemsetAsync(
            hist, 0, (kHead + nb * kRadix) * sizeof(uint32_t), st);
        if (e) return e;
        const int64_t hb = std::min<int64_t>((max_n + 1023) / 1024, 8 * s.num_sms);
        hist_kernel<K><<<(unsigned)hb, kThreads, 0, st>>>(keys, max_n, d_count, passes, hist);
        note_launch();
    }
    K *kin = keys, *kout = keys_alt;
    int32_t *vin = vals, *vout = vals_alt;
    for (int p = 0; p < passes; ++p) {
        pass_kernel<K><<<(unsigned)nb, kThreads, 0, st>>>(
            kin, vin, kout, vout, max_n, d_count, 8 * p, hist + p * kRadix, ticket + p, abort_,
            state[p & 1], state[(p + 1) & 1], s.scan.status);
        note_launch();
        std::swap(kin, kout);
        std::swap(vin, vout);
        *which ^= 1;
    }
    return cudaGetLastError();
}
} // namespace

int64_t sort_blocks_needed(int64_t max_n) { return (max_n + kTile - 1) / kTile; }
int64_t sort_scratch_words(int64_t blocks) { return kHead + 2 * kRadix * blocks; }

uint32_t *sort_counts(SortScratch &s) { return reinterpret_cast<uint32_t *>(s.hist); }
uint32_t *sort_zero_word(SortScratch &s)
{
    return sort_counts(s) + kMaxPasses * kRadix + kMaxPasses + 1;
}

cudaError_t sort_clear_u32(int64_t n, SortScratch &s, cudaStream_t st)
{
    const int64_t nb = (n + kTile - 1) / kTile;
    if (sort_blocks_needed(n) > s.max_blocks) return cudaErrorInvalidValue;
    return cudaMemsetAsync(s.hist, 0, (kHead + nb * kRadix) * sizeof(uint32_t), st);
}

cudaError_t radix_sort_u32(uint32_t *keys, uint32_t *keys_alt, int32_t *vals, int32_t *vals_alt,
                           int64_t max_n, const int32_t *d_count, int end_bit, SortScratch &s,
                           cudaStream_t st, int *which, bool counted)
{
    return radix_sort<uint32_t>(keys, keys_alt, vals, vals_alt, max_n, d_count, end_bit, s, st,
                                which, counted);
}

cudaError_t radix_sort_u64(uint64_t *keys, uint64_t *keys_alt, int32_t *vals, int32_t *vals_alt,
                           int64_t max_n, const int32_t *d_count, int end_bit, SortScratch &s,
                           cudaStream_t st, int *which)
{
    return radix_sort<uint64_t>(keys, keys_alt, vals, vals_alt, max_n, d_count, end_bit, s, st,
                                which, false);
}

} // namespace rl
