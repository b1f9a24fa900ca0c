// Acceptance, apply, synapse store, deletion and spike delivery
// (Sec. III-A "Update of synapses" and "Update of electrical activity").
//
// Acceptance groups requests by target with a counting pass (histogram, scan,
// scatter). A target with no more requests than vacant dendritic elements
// accepts them all; an over-requested target accepts a request iff fewer than
// vac_de other requests to it have a smaller (priority, source, element) key,
// which is the same set as sorting by that key and taking the first vac_de.
// Requests are numbered in (source id, element) order, so that key orders exactly
// like the 64-bit (priority << 32 | request number), which the scatter stores in the
// target's bucket: ranking a request reads its bucket once, in order.
//
// The store is the synapse multiset. Updates append their new synapses; the
// canonical order (source, then target) with an out-row pointer array and an
// in-view (rows by target, each ordered by source) is restored only when deletion
// or an export needs it. Spike delivery reads the store in any order: each
// synapse of a spiking source adds its sign to its target with an integer atomic
// (exact, so the order does not matter).
#include "cluster.cuh"
#include "internal.h"

namespace rl {

namespace {

#define GRID_STRIDE(i, n)                                                                         \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n);                     \
         i += (int64_t)gridDim.x * blockDim.x)

int id_bits(int64_t n)
{
    int b = 1;
    while (b < 31 && ((int64_t)1 << b) < n) ++b;
    return b;
}

// ---------------------------------------------------------------- acceptance
__global__ void accept_count_kernel(const int32_t *d_Q, const int32_t *__restrict__ req_src,
                                    const int32_t *__restrict__ req_elem,
                                    const int32_t *__restrict__ req_tgt,
                                    uint32_t *__restrict__ prio, int32_t *__restrict__ tcnt,
                                    uint64_t seed, uint32_t step)
{
    const int64_t Q = *d_Q;
    GRID_STRIDE(r, Q)
    {
        int32_t t = req_tgt[r];
        if (t < 0) continue;
        atomicAdd(&tcnt[t], 1);
        prio[r] = philox_x((uint32_t)req_src[r], step, ((uint32_t)req_elem[r] << 8) | 0xFFu, 1u,
                           seed);
    }
}

__device__ __forceinline__ uint64_t request_key(uint32_t prio, int64_t r)
{
    return ((uint64_t)prio << 32) | (uint64_t)(uint32_t)r;
}

// Each request takes a slot of its target's bucket by counting the target's count
// down (the bucket's order does not matter: the decision ranks keys).
__global__ void accept_scatter_kernel(const int32_t *d_Q, const int32_t *__restrict__ req_tgt,
                                      const uint32_t *__restrict__ prio,
                                      const int32_t *__restrict__ toff,
                                      int32_t *__restrict__ tcnt, uint64_t *__restrict__ bucket)
{
    const int64_t Q = *d_Q;
    GRID_STRIDE(r, Q)
    {
        int32_t t = req_tgt[r];
        if (t < 0) continue;
        bucket[toff[t] + atomicSub(&tcnt[t], 1) - 1] = request_key(prio[r], r);
    }
}

// Whether request r to target t is accepted. A target's request count is the difference
// of neighbouring bucket offsets (one read of two adjacent words).
__device__ __forceinline__ bool accepted(int64_t r, int32_t t, const uint32_t *prio,
                                         const int32_t *toff, const uint64_t *bucket,
                                         const int32_t *vac_de)
{
    const int32_t v = max(vac_de[t], 0);
    const int32_t o = toff[t], rt = toff[t + 1] - o;
    if (rt <= v) return true;
    if (v == 0) return false;
    const uint64_t kr = request_key(prio[r], r); // keys are distinct
    const uint64_t *bk = bucket + o;
    int32_t below = 0;
    for (int32_t k = 0; k < rt && below < v; ++k) below += bk[k] < kr ? 1 : 0;
    return below < v;
}

__global__ void accept_decide_kernel(const int32_t *d_Q, const int32_t *__restrict__ req_tgt,
                                     const uint32_t *__restrict__ prio,
                                     const int32_t *__restrict__ toff,
                                     const uint64_t *__restrict__ bucket,
                                     const int32_t *__restrict__ vac_de,
                                     uint8_t *__restrict__ acc, int32_t *__restrict__ flag,
                                     int64_t *declined)
{
    const int64_t Q = *d_Q;
    int64_t dec = 0;
    GRID_STRIDE(r, Q)
    {
        const int32_t t = req_tgt[r];
        uint8_t a = 0;
        if (t >= 0) {
            a = accepted(r, t, prio, toff, bucket, vac_de) ? 1 : 0;
            dec += a ? 0 : 1;
        }
        acc[r] = a;
        flag[r] = a; // scanned by the apply step into the new synapses' positions
    }
    for (int off = 16; off; off >>= 1) dec += __shfl_xor_sync(0xffffffffu, dec, off);
    if ((threadIdx.x & 31) == 0 && dec)
        atomicAdd(reinterpret_cast<unsigned long long *>(declined), (unsigned long long)dec);
}

// ---------------------------------------------------------------- apply
// New store size check: formed = *d_formed; nothing is applied on overflow. The
// store grows here: the apply kernel writes the new synapses from *d_base (the old
// size) on.
__global__ void apply_check_kernel(const int64_t *d_formed, int32_t *d_nsyn, int32_t *d_new,
                                   int32_t *d_base, int64_t *d_nsyn64, int64_t max_synapses,
                                   int32_t *status, int64_t *d_formed_out)
{
    int64_t f = *d_formed;
    const int32_t base = *d_nsyn;
    const bool failed = *(volatile int32_t *)status != 0; // an earlier kernel reported an error
    *d_base = base;
    if (failed || (int64_t)base + f > max_synapses) {
        if (!failed) set_status(status, RELEARN_ERR_CAPACITY);
        *d_new = -1;
        *d_formed_out = 0;
    } else {
        *d_new = (int32_t)f;
        *d_formed_out = f;
        *d_nsyn = base + (int32_t)f;
    }
    *d_nsyn64 = *d_nsyn;
}

__global__ void apply_kernel(const int32_t *d_Q, const int32_t *d_new, const int32_t *d_base,
                             const int32_t *__restrict__ req_src,
                             const int32_t *__restrict__ req_tgt, const uint8_t *__restrict__ acc,
                             const int32_t *__restrict__ newpos, const uint8_t *__restrict__ type,
                             int32_t *vac_ax, int32_t *vac_de, int32_t *__restrict__ syn_src,
                             int32_t *__restrict__ syn_tgt, int8_t *__restrict__ syn_sign)
{
    if (*d_new < 0) return;
    const int64_t Q = *d_Q;
    const int32_t base = *d_base;
    GRID_STRIDE(r, Q)
    {
        if (!acc[r]) continue;
        const int32_t s = req_src[r], t = req_tgt[r];
        atomicSub(&vac_ax[s], 1);
        atomicSub(&vac_de[t], 1);
        const int32_t k = base + newpos[r];
        syn_src[k] = s;
        syn_tgt[k] = t;
        syn_sign[k] = type[s] ? (int8_t)-1 : (int8_t)1;
    }
}

// ---------------------------------------------------------------- store
__global__ void unpack_keys_kernel(const int32_t *d_nsyn, const uint64_t *__restrict__ key,
                                   const int32_t *__restrict__ val, int bits,
                                   int32_t *__restrict__ src, int32_t *__restrict__ tgt,
                                   int8_t *__restrict__ sign)
{
    const int64_t m = *d_nsyn;
    const uint64_t mask = ((uint64_t)1 << bits) - 1;
    GRID_STRIDE(k, m)
    {
        uint64_t kk = key[k];
        src[k] = (int32_t)(kk >> bits);
        tgt[k] = (int32_t)(kk & mask);
        sign[k] = (int8_t)val[k];
    }
}

__global__ void degree_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                              const int32_t *__restrict__ tgt, int32_t *__restrict__ out_cnt,
                              int32_t *__restrict__ in_cnt)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        atomicAdd(&out_cnt[src[k]], 1);
        atomicAdd(&in_cnt[tgt[k]], 1);
    }
}

// The canonical order without a global sort: each synapse goes to its source's row
// (any order within the row), then takes its rank in the row by (target, place in
// the row). Rows are short (a neuron's bound elements), so ranking by counting is
// cheaper than sorting the whole store; equal (source, target) records are
// identical (the sign follows the source), so their order does not matter.
__global__ void row_scatter_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                                   const int32_t *__restrict__ tgt, const int8_t *__restrict__ sign,
                                   const int32_t *__restrict__ out_ptr, int32_t *__restrict__ left,
                                   int32_t *__restrict__ row_src, int32_t *__restrict__ row_tgt,
                                   int32_t *__restrict__ row_sign)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        const int32_t s = src[k];
        const int32_t r = out_ptr[s] + atomicSub(&left[s], 1) - 1;
        row_src[r] = s;
        row_tgt[r] = tgt[k];
        row_sign[r] = sign[k];
    }
}

// Where record r of a row belongs: its rank in the row by (target, place in the row).
__device__ __forceinline__ int32_t row_place(int64_t r, const int32_t *row_src,
                                             const int32_t *row_tgt, const int32_t *out_ptr)
{
    const int32_t s = row_src[r], t = row_tgt[r];
    const int32_t b = out_ptr[s], e = out_ptr[s + 1];
    int32_t rank = 0;
    for (int32_t j = b; j < e; ++j) {
        const int32_t tj = row_tgt[j];
        rank += (tj < t || (tj == t && j < r)) ? 1 : 0;
    }
    return b + rank;
}

__global__ void row_rank_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ row_src,
                                const int32_t *__restrict__ row_tgt,
                                const int32_t *__restrict__ row_sign,
                                const int32_t *__restrict__ out_ptr, int32_t *__restrict__ src,
                                int32_t *__restrict__ tgt, int8_t *__restrict__ sign)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(r, m)
    {
        const int32_t w = row_place(r, row_src, row_tgt, out_ptr);
        src[w] = row_src[r];
        tgt[w] = row_tgt[r];
        sign[w] = (int8_t)row_sign[r];
    }
}

// In-view: synapse numbers k (canonical order) grouped by target, each row ordered by
// k (i.e. by source), by the same scatter-then-rank.
__global__ void in_scatter_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ tgt,
                                  const int32_t *__restrict__ in_ptr, int32_t *__restrict__ left,
                                  int32_t *__restrict__ row_k)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        const int32_t t = tgt[k];
        row_k[in_ptr[t] + atomicSub(&left[t], 1) - 1] = (int32_t)k;
    }
}

__device__ __forceinline__ int32_t in_place(int64_t r, const int32_t *row_k, const int32_t *tgt,
                                            const int32_t *in_ptr)
{
    const int32_t k = row_k[r], t = tgt[k];
    const int32_t b = in_ptr[t], e = in_ptr[t + 1];
    int32_t rank = 0;
    for (int32_t j = b; j < e; ++j) rank += row_k[j] < k ? 1 : 0;
    return b + rank;
}

__global__ void in_rank_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ tgt,
                               const int32_t *__restrict__ in_ptr,
                               const int32_t *__restrict__ row_k, int32_t *__restrict__ in_syn)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(r, m)
    {
        in_syn[in_place(r, row_k, tgt, in_ptr)] = row_k[r];
    }
}

// ---------------------------------------------------------------- deletion
// Neuron i retracts vacant elements first; what is left breaks bound ones.
__device__ __forceinline__ int32_t retract(int64_t i, const int32_t *retract_, int32_t *vac,
                                           int32_t degree)
{
    const int32_t r = max(retract_[i], 0), v = vac[i];
    const int32_t t = r < v ? r : max(v, 0);
    vac[i] = v - t;
    return min(r - t, degree);
}

__global__ void delete_needs_kernel(int64_t n, const int32_t *__restrict__ retract_ax,
                                    const int32_t *__restrict__ retract_de, int32_t *vac_ax,
                                    int32_t *vac_de, const int32_t *__restrict__ out_ptr,
                                    const int32_t *__restrict__ in_ptr,
                                    int32_t *__restrict__ need_ax, int32_t *__restrict__ need_de)
{
    GRID_STRIDE(i, n)
    {
        need_ax[i] = retract(i, retract_ax, vac_ax, out_ptr[i + 1] - out_ptr[i]);
        need_de[i] = retract(i, retract_de, vac_de, in_ptr[i + 1] - in_ptr[i]);
    }
}

// The priority of slot k of its out-row and of its in-row, where the row breaks some of
// its slots but not all (select_row reads no others).
__device__ __forceinline__ void slot_priorities(int64_t k, const int32_t *src, const int32_t *tgt,
                                                const int32_t *in_syn, const int32_t *out_ptr,
                                                const int32_t *in_ptr, const int32_t *need_ax,
                                                const int32_t *need_de, uint32_t *prio_ax,
                                                uint32_t *prio_de, uint64_t seed, uint32_t step)
{
    const int32_t i = src[k], wi = need_ax[i], bi = out_ptr[i];
    if (wi > 0 && wi < out_ptr[i + 1] - bi)
        prio_ax[k] = philox_x((uint32_t)i, step, (uint32_t)(k - bi), 2u, seed);
    const int32_t j = tgt[in_syn[k]], wj = need_de[j], bj = in_ptr[j];
    if (wj > 0 && wj < in_ptr[j + 1] - bj)
        prio_de[k] = philox_x((uint32_t)j, step, (uint32_t)(k - bj), 3u, seed);
}

__global__ void delete_prio_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                                   const int32_t *__restrict__ in_syn,
                                   const int32_t *__restrict__ tgt,
                                   const int32_t *__restrict__ out_ptr,
                                   const int32_t *__restrict__ in_ptr,
                                   const int32_t *__restrict__ need_ax,
                                   const int32_t *__restrict__ need_de,
                                   uint32_t *__restrict__ prio_ax, uint32_t *__restrict__ prio_de,
                                   uint8_t *__restrict__ sel_ax, uint8_t *__restrict__ sel_de,
                                   uint64_t seed, uint32_t step)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        slot_priorities(k, src, tgt, in_syn, out_ptr, in_ptr, need_ax, need_de, prio_ax, prio_de,
                        seed, step);
        sel_ax[k] = 0;
        sel_de[k] = 0;
    }
}

// Row i picks its `want` slots with the smallest (priority, slot).
__device__ __forceinline__ void select_row(int32_t b, int32_t deg, int32_t want,
                                           const uint32_t *prio, const int32_t *map, uint8_t *sel)
{
    if (want <= 0) return;
    for (int32_t k = 0; k < deg; ++k) {
        bool take = want >= deg; // all of them
        if (!take) {
            const uint32_t pk = prio[b + k];
            int32_t below = 0;
            for (int32_t o = 0; o < deg && below < want; ++o) {
                const uint32_t po = prio[b + o];
                if (po < pk || (po == pk && o < k)) ++below;
            }
            take = below < want;
        }
        if (take) sel[map ? map[b + k] : b + k] = 1;
    }
}

__global__ void delete_select_kernel(int64_t n, const int32_t *__restrict__ ptr,
                                     const int32_t *__restrict__ need,
                                     const uint32_t *__restrict__ prio,
                                     const int32_t *__restrict__ map, uint8_t *__restrict__ sel)
{
    GRID_STRIDE(i, n)
    {
        const int32_t b = ptr[i];
        select_row(b, ptr[i + 1] - b, need[i], prio, map, sel);
    }
}

__global__ void delete_apply_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                                    const int32_t *__restrict__ tgt,
                                    const uint8_t *__restrict__ sel_ax,
                                    const uint8_t *__restrict__ sel_de, int32_t *vac_ax,
                                    int32_t *vac_de, int32_t *__restrict__ keep)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        const bool a = sel_ax[k], d = sel_de[k];
        if (a && !d) atomicAdd(&vac_de[tgt[k]], 1);
        if (d && !a) atomicAdd(&vac_ax[src[k]], 1);
        keep[k] = (a || d) ? 0 : 1;
    }
}

__global__ void compact_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                               const int32_t *__restrict__ tgt, const int8_t *__restrict__ sign,
                               const uint8_t *__restrict__ sel_ax,
                               const uint8_t *__restrict__ sel_de,
                               const int32_t *__restrict__ pos, int bits,
                               uint64_t *__restrict__ key, int32_t *__restrict__ val)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(k, m)
    {
        if (sel_ax[k] || sel_de[k]) continue;
        int32_t w = pos[k];
        key[w] = ((uint64_t)(uint32_t)src[k] << bits) | (uint32_t)tgt[k];
        val[w] = sign[k];
    }
}

__global__ void shrink_store_kernel(int32_t *d_nsyn, const int64_t *d_kept, int64_t *d_broken,
                                    int64_t *d_nsyn64)
{
    int64_t kept = *d_kept;
    *d_broken = (int64_t)*d_nsyn - kept;
    *d_nsyn = (int32_t)kept;
    *d_nsyn64 = kept;
}

// ---------------------------------------------------------------- spikes
// input[t] += sign for every synapse s -> t of a spiking source (input zeroed first).
// A thread takes W neighbouring synapses: each synapse is a chain of dependent reads
// (source, its spike or rate, target, atomic), and four chains in flight per thread wait
// for them together (1.8 million synapses, 5 % firing, with the zeroing of the inputs:
// 12.4 -> 10.9 us a call, of which about 9 are the two launches). A store that the
// resident threads cover with one synapse each takes W = 1 (see deliver_width).
template <int W>
struct Some {
    int32_t v[W];
};

// Entries W q .. W q + W - 1 of a store array (16-byte aligned), `fill` past its end m.
template <int W>
__device__ __forceinline__ Some<W> some_of(const int32_t *__restrict__ a, int64_t q, int64_t m,
                                           int32_t fill)
{
    Some<W> f;
    if (W == 4 && 4 * q + 4 <= m) {
        const int4 w = __ldg(reinterpret_cast<const int4 *>(a) + q);
        f.v[0] = w.x;
        f.v[1 % W] = w.y;
        f.v[2 % W] = w.z;
        f.v[3 % W] = w.w;
    } else {
#pragma unroll
        for (int k = 0; k < W; ++k) f.v[k] = W * q + k < m ? a[W * q + k] : fill;
    }
    return f;
}

template <int W>
__device__ __forceinline__ void some_spikes(int64_t q, int64_t m, const int32_t *src,
                                            const int32_t *tgt, const int8_t *sign,
                                            const uint8_t *spiked, int32_t *input)
{
    const Some<W> s = some_of<W>(src, q, m, -1);
    uint8_t on[W];
#pragma unroll
    for (int k = 0; k < W; ++k) on[k] = s.v[k] >= 0 ? spiked[s.v[k]] : 0;
#pragma unroll
    for (int k = 0; k < W; ++k)
        if (on[k]) atomicAdd(&input[tgt[W * q + k]], (int32_t)sign[W * q + k]);
}

template <int W>
__global__ void spikes_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                              const int32_t *__restrict__ tgt, const int8_t *__restrict__ sign,
                              const uint8_t *__restrict__ spiked, int32_t *__restrict__ input)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(q, (m + W - 1) / W) some_spikes<W>(q, m, src, tgt, sign, spiked, input);
}

// Firing-rate delivery (Sec. IV-B): the receiver t decides once per step and per
// source s whether s spiked, spiked iff philox({s, t, step, 4}).x < rate[s] * 2^32;
// duplicates of (s, t) share that decision (each copy computes the same word).
// The comparison is exact: the product is (a power of two), and a whole word lies below
// it exactly if it lies below the product rounded up to a whole number. No FP64: two
// conversions, a product and a comparison of it per synapse cost more than the generator.
__device__ __forceinline__ bool rate_fires(int32_t s, int32_t t, float rate, uint64_t seed,
                                           uint32_t step)
{
    const uint32_t w = philox_x((uint32_t)s, (uint32_t)t, step, 4u, seed);
    if (rate >= 1.0f) return true;
    return rate > 0.0f && w < __float2uint_ru(__fmul_rn(rate, 4294967296.0f)); // NaN: never
}

template <int W>
__device__ __forceinline__ void some_rates(int64_t q, int64_t m, const int32_t *src,
                                           const int32_t *tgt, const int8_t *sign,
                                           const float *rate, uint64_t seed, uint32_t step,
                                           int32_t *input)
{
    const Some<W> s = some_of<W>(src, q, m, -1), t = some_of<W>(tgt, q, m, 0);
    float r[W];
#pragma unroll
    for (int k = 0; k < W; ++k) r[k] = s.v[k] >= 0 ? rate[s.v[k]] : 0.0f;
#pragma unroll
    for (int k = 0; k < W; ++k)
        if (rate_fires(s.v[k], t.v[k], r[k], seed, step))
            atomicAdd(&input[t.v[k]], (int32_t)sign[W * q + k]);
}

// As spikes_kernel (1.8 million synapses 19.7 -> 14.4 us a call, 3.4 million 31.0 -> 18.6;
// one, two or four synapses per thread are the same here: the generator bounds it).
template <int W>
__global__ void rates_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                             const int32_t *__restrict__ tgt, const int8_t *__restrict__ sign,
                             const float *__restrict__ rate, uint64_t seed, uint32_t step,
                             int32_t *__restrict__ input)
{
    const int64_t m = *d_nsyn;
    GRID_STRIDE(q, (m + W - 1) / W) some_rates<W>(q, m, src, tgt, sign, rate, seed, step, input);
}

// ---------------------------------------------------------------- small networks
// The steps above for a small network, one launch per call (see cluster.cuh): the same
// arithmetic and, where an order matters, the same order. Pointers without __restrict__:
// one step reads what another wrote in the same launch.
#define CLUSTER_STRIDE(i, n)                                                                      \
    for (int64_t i = cluster_form::first(); i < (n); i += cluster_form::kStride)

// Rows longer than kLongRow (a hub's requests or synapses) are not ranked by counting:
// that takes the square of the length, which 16 SMs take several times as long over as the
// general kernels' 152. Instead each run of kRun entries is sorted (one block per run, in
// shared memory), and an entry's place is its place in its own run plus a binary search in
// each other one. One target taking every request of 20,000 / 40,000 neurons, 1,000 /
// 2,000 vacancies: update 4.07 / 15.6 ms by counting, 0.30 / 0.95 here, 1.9 / 3.7 by the
// general kernels; canonical order with an in-degree of 20,000: 840 us, 197, 443. The flag
// any_long (set by the scans of the row lengths) keeps the passes out of networks without
// such rows.
constexpr int32_t kLongRow = 256, kRun = cluster_form::kThreads;

// Sorts every run of kRun entries of the rows ptr[i] .. ptr[i + 1] longer than kLongRow (at
// most kSmallItems entries in all), by keys of type K below the largest of K: load(i) is
// entry i's key, store(i, key) puts it back. Called by the whole cluster; a barrier has to
// follow.
template <class K, class Load, class Store>
__device__ __forceinline__ void sort_runs(const int32_t *ptr, int64_t n, K largest, Load load,
                                          Store store)
{
    namespace cf = cluster_form;
    __shared__ K s_key[kRun];
    __shared__ int32_t s_row[kSmallItems / kLongRow];
    __shared__ int32_t s_rows;
    const int t = threadIdx.x, rank = (int)cooperative_groups::this_cluster().block_rank();
    if (t == 0) s_rows = 0;
    __syncthreads();
    for (int64_t i = t; i < n; i += cf::kThreads) // every block lists every long row
        if (ptr[i + 1] - ptr[i] > kLongRow) s_row[atomicAdd(&s_rows, 1)] = (int32_t)i;
    __syncthreads();
    for (int q = 0; q < s_rows; ++q) {
        const int32_t b = ptr[s_row[q]], e = ptr[s_row[q] + 1];
        for (int32_t s = b; s < e; s += kRun) {
            if ((s / kRun) % cf::kBlocks != rank) continue; // the same block for every list order
            s_key[t] = s + t < e ? load(s + t) : largest;
            __syncthreads();
            for (int k = 2; k <= kRun; k <<= 1) // bitonic sort
                for (int j = k >> 1; j; j >>= 1) {
                    const int p = t ^ j;
                    if (p > t) {
                        const K x = s_key[t], y = s_key[p];
                        if ((x > y) == ((t & k) == 0)) {
                            s_key[t] = y;
                            s_key[p] = x;
                        }
                    }
                    __syncthreads();
                }
            if (s + t < e) store(s + t, s_key[t]);
            __syncthreads();
        }
    }
}

// How many entries of the row b .. e (its runs sorted by keys) come before entry r, whose
// key is given: smaller keys, and of equal ones those at smaller places. r = -1: how many
// keys are smaller.
template <class K>
__device__ __forceinline__ int32_t place_in_runs(const K *keys, int32_t b, int32_t e, K key,
                                                 int64_t r)
{
    int32_t place = 0;
    for (int32_t s = b; s < e; s += kRun) {
        const int32_t end = min(s + kRun, e);
        int32_t lo = s, hi = end;
        if (r >= s && r < end) {
            place += (int32_t)r - s;
            continue;
        }
        const bool ties = end <= r;
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (keys[mid] < key || (ties && keys[mid] == key))
                lo = mid + 1;
            else
                hi = mid;
        }
        place += lo - s;
    }
    return place;
}

struct StoreArgs {
    int64_t n, max_synapses;
    int32_t *d_nsyn;
    int64_t *d_nsyn64;
    int32_t *src, *tgt;
    int8_t *sign;
    uint64_t seed;
    uint32_t step;
};

StoreArgs store_args(relearn_ctx *c, uint64_t seed, uint32_t step)
{
    return StoreArgs{c->n,         c->max_synapses, c->d_i32 + I32_NSYN, c->d_i64 + I64_NSYN,
                     c->d_syn_src, c->d_syn_tgt,    c->d_syn_sign,       seed,
                     step};
}

struct AcceptArgs {
    const int32_t *d_Q;
    int32_t *status;
    const int32_t *req_src, *req_elem, *req_tgt;
    uint32_t *prio;
    int32_t *tcnt, *toff;
    uint64_t *bucket;
    int32_t *any_long;
    uint8_t *acc;
    int64_t *declined, *formed;
    int32_t *vac_ax, *vac_de;
    const uint8_t *type;
};

// As accepted, for a request of a long row (runs sorted).
__device__ __forceinline__ bool accepted_long(int64_t r, int32_t t, const AcceptArgs &a)
{
    const int32_t v = max(a.vac_de[t], 0), b = a.toff[t], e = a.toff[t + 1];
    if (e - b <= v) return true;
    return v > 0 && place_in_runs(a.bucket, b, e, request_key(a.prio[r], r), -1) < v;
}

// Acceptance and apply of an update.
__global__ void __cluster_dims__(cluster_form::kBlocks, 1, 1)
    __launch_bounds__(cluster_form::kThreads) accept_apply_small_kernel(AcceptArgs a, StoreArgs st)
{
    namespace cf = cluster_form;
    const int64_t Q = *a.d_Q;
    const int64_t base = *st.d_nsyn;
    const bool failed = *(volatile int32_t *)a.status != 0; // an earlier kernel's error
    CLUSTER_STRIDE(i, st.n + 1) a.tcnt[i] = 0;
    if (cf::first() == 0) {
        *a.declined = 0;
        *a.any_long = 0;
    }
    cf::sync();
    CLUSTER_STRIDE(r, Q)
    {
        const int32_t t = a.req_tgt[r];
        if (t < 0) continue;
        atomicAdd(&a.tcnt[t], 1);
        a.prio[r] = philox_x((uint32_t)a.req_src[r], st.step,
                             ((uint32_t)a.req_elem[r] << 8) | 0xFFu, 1u, st.seed);
    }
    cf::sync();
    auto count = [&](int64_t i) { return cf::I32{a.tcnt[i]}; };
    cf::scan<cf::I32>(st.n + 1, count, count,
                      [&](int64_t i, cf::I32 prefix, cf::I32 requests, cf::I32) {
                          a.toff[i] = prefix.v;
                          if (requests.v > kLongRow) *a.any_long = 1;
                      });
    cf::sync();
    const bool any_long = *(volatile int32_t *)a.any_long != 0;
    CLUSTER_STRIDE(r, Q)
    {
        const int32_t t = a.req_tgt[r];
        if (t >= 0)
            a.bucket[a.toff[t] + atomicSub(&a.tcnt[t], 1) - 1] = request_key(a.prio[r], r);
    }
    cf::sync();
    if (any_long) {
        sort_runs(a.toff, st.n, ~uint64_t(0), [&](int64_t i) { return a.bucket[i]; },
                  [&](int64_t i, uint64_t key) { a.bucket[i] = key; });
        cf::sync();
    }
    int64_t dec = 0;
    // every decision is made before the first vacancy changes (the scan's barrier)
    const cf::I32 formed = cf::scan<cf::I32>(
        Q,
        [&](int64_t r) {
            const int32_t t = a.req_tgt[r];
            const bool ok =
                t >= 0 && (any_long && a.toff[t + 1] - a.toff[t] > kLongRow
                               ? accepted_long(r, t, a)
                               : accepted(r, t, a.prio, a.toff, a.bucket, a.vac_de));
            dec += t >= 0 && !ok ? 1 : 0;
            a.acc[r] = ok ? 1 : 0;
            return cf::I32{ok ? 1 : 0};
        },
        [&](int64_t r) { return cf::I32{a.acc[r]}; },
        [&](int64_t r, cf::I32 prefix, cf::I32 ok, cf::I32 total) {
            // nothing is applied on overflow
            if (!ok.v || failed || base + total.v > st.max_synapses) return;
            const int32_t s = a.req_src[r], t = a.req_tgt[r];
            atomicSub(&a.vac_ax[s], 1);
            atomicSub(&a.vac_de[t], 1);
            const int64_t k = base + prefix.v;
            st.src[k] = s;
            st.tgt[k] = t;
            st.sign[k] = a.type[s] ? (int8_t)-1 : (int8_t)1;
        });
    for (int off = 16; off; off >>= 1) dec += __shfl_xor_sync(0xffffffffu, dec, off);
    if ((threadIdx.x & 31) == 0 && dec)
        atomicAdd(reinterpret_cast<unsigned long long *>(a.declined), (unsigned long long)dec);
    if (cf::first() == 0) {
        const bool fits = base + formed.v <= st.max_synapses;
        if (!failed && !fits) set_status(a.status, RELEARN_ERR_CAPACITY);
        const int64_t f = failed || !fits ? 0 : formed.v;
        *a.formed = f;
        *st.d_nsyn = (int32_t)(base + f);
        *st.d_nsyn64 = base + f;
    }
    cf::sync();
}

struct DeleteArgs {
    bool canonical; // the views below are those of the store
    int32_t *out_cnt, *in_cnt, *out_ptr, *in_ptr;
    int32_t *row_src, *row_tgt, *row_sign, *row_k, *in_syn, *any_long;
    const int32_t *retract_ax, *retract_de;
    int32_t *vac_ax, *vac_de, *need_ax, *need_de;
    uint32_t *prio_ax, *prio_de;
    uint8_t *sel_ax, *sel_de;
    int64_t *broken;
};

// The canonical order and its views, then the deletion pass (see canonicalise_store and
// delete_synapses).
__global__ void __cluster_dims__(cluster_form::kBlocks, 1, 1)
    __launch_bounds__(cluster_form::kThreads) delete_small_kernel(DeleteArgs a, StoreArgs st)
{
    namespace cf = cluster_form;
    const int64_t n = st.n, m = *st.d_nsyn;
    if (!a.canonical) {
        CLUSTER_STRIDE(i, n + 1) a.out_cnt[i] = a.in_cnt[i] = 0;
        if (cf::first() == 0) *a.any_long = 0;
        cf::sync();
        CLUSTER_STRIDE(k, m)
        {
            atomicAdd(&a.out_cnt[st.src[k]], 1);
            atomicAdd(&a.in_cnt[st.tgt[k]], 1);
        }
        cf::sync();
        auto counts = [&](int64_t i) { return cf::I64x2{a.out_cnt[i], a.in_cnt[i]}; };
        cf::scan<cf::I64x2>(n + 1, counts, counts,
                            [&](int64_t i, cf::I64x2 prefix, cf::I64x2 degree, cf::I64x2) {
                                a.out_ptr[i] = (int32_t)prefix.a;
                                a.in_ptr[i] = (int32_t)prefix.b;
                                if (degree.a > kLongRow || degree.b > kLongRow) *a.any_long = 1;
                            });
        cf::sync();
        const bool any_long = *(volatile int32_t *)a.any_long != 0;
        CLUSTER_STRIDE(k, m)
        {
            const int32_t s = st.src[k];
            const int32_t r = a.out_ptr[s] + atomicSub(&a.out_cnt[s], 1) - 1;
            a.row_src[r] = s;
            a.row_tgt[r] = st.tgt[k];
            a.row_sign[r] = st.sign[k];
        }
        cf::sync();
        if (any_long) { // by (target, sign): the sign moves with its record
            sort_runs(a.out_ptr, n, 0x7fffffff,
                      [&](int64_t i) { return 2 * a.row_tgt[i] + (a.row_sign[i] > 0 ? 1 : 0); },
                      [&](int64_t i, int32_t key) {
                          a.row_tgt[i] = key >> 1;
                          a.row_sign[i] = key & 1 ? 1 : -1;
                      });
            cf::sync();
        }
        CLUSTER_STRIDE(r, m)
        {
            const int32_t s = a.row_src[r], b = a.out_ptr[s], e = a.out_ptr[s + 1];
            const int32_t w = any_long && e - b > kLongRow
                                  ? b + place_in_runs(a.row_tgt, b, e, a.row_tgt[r], r)
                                  : row_place(r, a.row_src, a.row_tgt, a.out_ptr);
            st.src[w] = a.row_src[r];
            st.tgt[w] = a.row_tgt[r];
            st.sign[w] = (int8_t)a.row_sign[r];
        }
        cf::sync();
        CLUSTER_STRIDE(k, m)
        {
            const int32_t t = st.tgt[k];
            a.row_k[a.in_ptr[t] + atomicSub(&a.in_cnt[t], 1) - 1] = (int32_t)k;
        }
        cf::sync();
        if (any_long) {
            sort_runs(a.in_ptr, n, 0x7fffffff, [&](int64_t i) { return a.row_k[i]; },
                      [&](int64_t i, int32_t k) { a.row_k[i] = k; });
            cf::sync();
        }
        CLUSTER_STRIDE(r, m)
        {
            const int32_t k = a.row_k[r], t = st.tgt[k], b = a.in_ptr[t], e = a.in_ptr[t + 1];
            a.in_syn[any_long && e - b > kLongRow
                         ? b + place_in_runs(a.row_k, b, e, k, r)
                         : in_place(r, a.row_k, st.tgt, a.in_ptr)] = k;
        }
        cf::sync();
    }
    CLUSTER_STRIDE(i, n)
    {
        a.need_ax[i] = retract(i, a.retract_ax, a.vac_ax, a.out_ptr[i + 1] - a.out_ptr[i]);
        a.need_de[i] = retract(i, a.retract_de, a.vac_de, a.in_ptr[i + 1] - a.in_ptr[i]);
    }
    cf::sync();
    CLUSTER_STRIDE(k, m)
    {
        a.sel_ax[k] = 0;
        a.sel_de[k] = 0;
        slot_priorities(k, st.src, st.tgt, a.in_syn, a.out_ptr, a.in_ptr, a.need_ax, a.need_de,
                        a.prio_ax, a.prio_de, st.seed, st.step);
    }
    cf::sync();
    CLUSTER_STRIDE(i, n)
    {
        const int32_t b = a.out_ptr[i], d = a.in_ptr[i];
        select_row(b, a.out_ptr[i + 1] - b, a.need_ax[i], a.prio_ax, nullptr, a.sel_ax);
        select_row(d, a.in_ptr[i + 1] - d, a.need_de[i], a.prio_de, a.in_syn, a.sel_de);
    }
    cf::sync();
    const cf::I32 kept = cf::scan<cf::I32>(
        m,
        [&](int64_t k) {
            const bool x = a.sel_ax[k], d = a.sel_de[k];
            if (x && !d) atomicAdd(&a.vac_de[st.tgt[k]], 1);
            if (d && !x) atomicAdd(&a.vac_ax[st.src[k]], 1);
            return cf::I32{x || d ? 0 : 1};
        },
        [&](int64_t k) { return cf::I32{a.sel_ax[k] || a.sel_de[k] ? 0 : 1}; },
        [&](int64_t k, cf::I32 prefix, cf::I32 keep, cf::I32) {
            if (!keep.v) return;
            a.row_src[prefix.v] = st.src[k];
            a.row_tgt[prefix.v] = st.tgt[k];
            a.row_sign[prefix.v] = st.sign[k];
        });
    cf::sync();
    CLUSTER_STRIDE(w, kept.v)
    {
        st.src[w] = a.row_src[w];
        st.tgt[w] = a.row_tgt[w];
        st.sign[w] = (int8_t)a.row_sign[w];
    }
    if (cf::first() == 0) {
        *a.broken = m - kept.v;
        *st.d_nsyn = kept.v;
        *st.d_nsyn64 = kept.v;
    }
}

// input = 0, then as spikes_kernel (spiked given) or rates_kernel: one launch instead of a
// memset and a kernel (called directly, 4,000 to 40,000 neurons: spikes 10.2 -> 8.3 us,
// rates 10.4 -> 8.6; for graphs see deliver_small).
__global__ void __cluster_dims__(cluster_form::kBlocks, 1, 1)
    __launch_bounds__(cluster_form::kThreads)
    deliver_small_kernel(const int32_t *d_nsyn, const int32_t *__restrict__ src,
                         const int32_t *__restrict__ tgt, const int8_t *__restrict__ sign,
                         const uint8_t *__restrict__ spiked, const float *__restrict__ rate,
                         uint64_t seed, uint32_t step, int64_t n, int32_t *input)
{
    namespace cf = cluster_form;
    const int64_t m = *d_nsyn;
    CLUSTER_STRIDE(i, n) input[i] = 0;
    cf::sync();
    CLUSTER_STRIDE(q, (m + 3) / 4)
    {
        if (spiked)
            some_spikes<4>(q, m, src, tgt, sign, spiked, input);
        else
            some_rates<4>(q, m, src, tgt, sign, rate, seed, step, input);
    }
}

} // namespace

namespace {

// Synapses per thread of the general delivery kernels, by the store's capacity: up to one
// and a half per resident thread, four to a thread leave the chip idle (in a graph of 40
// calls, us a call, spikes / rates, one -> four per thread: 32,904 3.2 / 3.2 -> 3.6 / 4.1,
// 400,946 3.5 / 3.7 -> 3.7 / 4.4, 800,072 4.4 / 4.5 -> 3.8 / 4.7, 1,601,212 5.9 / 6.3 ->
// 4.1 / 5.8, 4,186,726 8.3 / 9.9 -> 5.8 / 9.2).
int deliver_width(const relearn_ctx *c)
{
    return c->max_synapses <= 3072 * (int64_t)c->num_sms ? 1 : 4;
}

// Whether a delivery runs as one cluster kernel (see deliver_small_kernel): called
// directly, it saves a launch. Replayed from a graph it saves none, and the general form
// spreads over the whole GPU; only where the inputs take at most 4 KB is the general form's
// zeroing node slow (a graph of 40 calls, us a call, spikes / rates, cluster and general:
// 1,000 neurons 2.9 / 3.7 and 6.2 / 6.2, 2,000 3.0 / 3.6 and 3.1 / 3.1, 16,000 3.2 / 4.0 and
// 3.2 / 3.2, 40,000 4.4 / 5.7 and 3.3 / 3.2).
bool deliver_small(const relearn_ctx *c, cudaStream_t st)
{
    if (!small_network(c)) return false;
    if (c->n <= 1024) return true;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError(); // the launch reports what is wrong with the stream
        return true;
    }
    return cs == cudaStreamCaptureStatusNone;
}

} // namespace

cudaError_t deliver_rates(relearn_ctx *c, const float *rate, uint64_t seed, uint32_t step,
                          int32_t *input, cudaStream_t st)
{
    if (deliver_small(c, st)) {
        deliver_small_kernel<<<cluster_form::kBlocks, cluster_form::kThreads, 0, st>>>(
            c->d_i32 + I32_NSYN, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign, nullptr, rate, seed, step, c->n,
            input);
        note_launch();
        return cudaGetLastError();
    }
    cudaError_t e;
    if ((e = cudaMemsetAsync(input, 0, c->n * sizeof(int32_t), st))) return e;
    const int w = deliver_width(c);
    (w == 1 ? rates_kernel<1> : rates_kernel<4>)
        <<<grid_for((c->max_synapses + w - 1) / w, 256, c->num_sms), 256, 0, st>>>(
            c->d_i32 + I32_NSYN, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign, rate, seed, step,
            input);
    note_launch();
    return cudaGetLastError();
}

cudaError_t accept_requests(relearn_ctx *c, const relearn_params &p, const int32_t *vac_de,
                            cudaStream_t st)
{
    cudaError_t e;
    const int64_t n = c->n;
    const int32_t *dQ = c->d_i32 + I32_Q;
    const unsigned gq = grid_for(c->max_searches, 256, c->num_sms);
    if ((e = cudaMemsetAsync(c->d_tcnt, 0, (n + 1) * sizeof(int32_t), st))) return e;
    if ((e = cudaMemsetAsync(c->d_i64 + I64_DECLINED, 0, sizeof(int64_t), st))) return e;
    accept_count_kernel<<<gq, 256, 0, st>>>(dQ, c->d_req_src, c->d_req_elem, c->d_req_tgt,
                                            c->d_req_prio, c->d_tcnt, p.seed, (uint32_t)p.step);
    note_launch();
    if ((e = scan_exclusive(c->d_tcnt, c->d_toff, n + 1, nullptr, nullptr, c->scan, st))) return e;
    accept_scatter_kernel<<<gq, 256, 0, st>>>(dQ, c->d_req_tgt, c->d_req_prio, c->d_toff,
                                              c->d_tcnt, c->d_bucket);
    note_launch();
    accept_decide_kernel<<<gq, 256, 0, st>>>(dQ, c->d_req_tgt, c->d_req_prio, c->d_toff,
                                             c->d_bucket,
                                             vac_de, c->d_req_acc, c->d_newpos,
                                             c->d_i64 + I64_DECLINED);
    note_launch();
    return cudaGetLastError();
}

// The store in canonical order (source, then target) with its views: out-row
// pointers, in-row pointers and the in-view. Counting pass, two scans, then one
// scatter and one in-row ranking per side (see row_scatter_kernel).
cudaError_t canonicalise_store(relearn_ctx *c, cudaStream_t st)
{
    cudaError_t e;
    const int64_t n = c->n;
    const int32_t *dm = c->d_i32 + I32_NSYN;
    const unsigned gs = grid_for(c->max_synapses, 256, c->num_sms);
    int32_t *out_cnt = c->d_cnt, *in_cnt = c->d_tcnt;
    int32_t *row_src = c->d_val, *row_sign = c->d_val_alt;
    int32_t *row_tgt = reinterpret_cast<int32_t *>(c->d_key32);
    int32_t *row_k = reinterpret_cast<int32_t *>(c->d_key32_alt);
    if ((e = cudaMemsetAsync(out_cnt, 0, (n + 1) * sizeof(int32_t), st))) return e;
    if ((e = cudaMemsetAsync(in_cnt, 0, (n + 1) * sizeof(int32_t), st))) return e;
    degree_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_src, c->d_syn_tgt, out_cnt, in_cnt);
    note_launch();
    if ((e = scan_exclusive(out_cnt, c->d_out_ptr, n + 1, nullptr, nullptr, c->scan, st)))
        return e;
    if ((e = scan_exclusive(in_cnt, c->d_in_ptr, n + 1, nullptr, nullptr, c->scan, st))) return e;
    row_scatter_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign,
                                           c->d_out_ptr, out_cnt, row_src, row_tgt, row_sign);
    note_launch();
    row_rank_kernel<<<gs, 256, 0, st>>>(dm, row_src, row_tgt, row_sign, c->d_out_ptr,
                                        c->d_syn_src, c->d_syn_tgt, c->d_syn_sign);
    note_launch();
    in_scatter_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_tgt, c->d_in_ptr, in_cnt, row_k);
    note_launch();
    in_rank_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_tgt, c->d_in_ptr, row_k, c->d_in_syn);
    note_launch();
    c->canonical = true;
    return cudaGetLastError();
}

bool synapses_clusters()
{
    return cluster_form::placeable(accept_apply_small_kernel) &&
           cluster_form::placeable(delete_small_kernel) &&
           cluster_form::placeable(deliver_small_kernel);
}

cudaError_t accept_apply_small(relearn_ctx *c, const relearn_params &p, int32_t *vac_ax,
                               int32_t *vac_de, const uint8_t *type, cudaStream_t st)
{
    AcceptArgs a;
    a.d_Q = c->d_i32 + I32_Q;
    a.status = c->d_status;
    a.req_src = c->d_req_src;
    a.req_elem = c->d_req_elem;
    a.req_tgt = c->d_req_tgt;
    a.prio = c->d_req_prio;
    a.tcnt = c->d_tcnt;
    a.toff = c->d_toff;
    a.bucket = c->d_bucket;
    a.any_long = c->d_i32 + I32_LONG;
    a.acc = c->d_req_acc;
    a.declined = c->d_i64 + I64_DECLINED;
    a.formed = c->d_i64 + I64_FORMED;
    a.vac_ax = vac_ax;
    a.vac_de = vac_de;
    a.type = type;
    accept_apply_small_kernel<<<cluster_form::kBlocks, cluster_form::kThreads, 0, st>>>(
        a, store_args(c, p.seed, (uint32_t)p.step));
    note_launch();
    c->canonical = false; // as in apply_requests
    return cudaGetLastError();
}

cudaError_t apply_requests(relearn_ctx *c, int32_t *vac_ax, int32_t *vac_de, const uint8_t *type,
                           cudaStream_t st)
{
    cudaError_t e;
    const int32_t *dQ = c->d_i32 + I32_Q;
    const unsigned gq = grid_for(c->max_searches, 256, c->num_sms);
    // d_newpos holds the acceptance flags (written by the acceptance step)
    if ((e = scan_exclusive(c->d_newpos, c->d_newpos, c->max_searches, dQ,
                            c->d_i64 + I64_SCAN_TOTAL, c->scan, st)))
        return e;
    apply_check_kernel<<<1, 1, 0, st>>>(c->d_i64 + I64_SCAN_TOTAL, c->d_i32 + I32_NSYN,
                                        c->d_i32 + I32_NEW, c->d_i32 + I32_BASE,
                                        c->d_i64 + I64_NSYN, c->max_synapses, c->d_status,
                                        c->d_i64 + I64_FORMED);
    note_launch();
    apply_kernel<<<gq, 256, 0, st>>>(dQ, c->d_i32 + I32_NEW, c->d_i32 + I32_BASE, c->d_req_src,
                                     c->d_req_tgt, c->d_req_acc, c->d_newpos, type, vac_ax,
                                     vac_de, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign);
    note_launch();
    // new synapses sit unsorted at the end of the store until an operation needs the
    // canonical order (deletion, export); spike delivery reads the store in any order
    c->canonical = false;
    return cudaGetLastError();
}

cudaError_t delete_synapses(relearn_ctx *c, const relearn_params &p, const int32_t *retract_ax,
                            const int32_t *retract_de, int32_t *vac_ax, int32_t *vac_de,
                            cudaStream_t st)
{
    cudaError_t e;
    const int64_t n = c->n;
    const int bits = id_bits(c->max_neurons);
    const int32_t *dm = c->d_i32 + I32_NSYN;
    const unsigned gs = grid_for(c->max_synapses, 256, c->num_sms);
    const unsigned gn = grid_for(n, 256, c->num_sms);
    if (small_network(c)) {
        DeleteArgs a;
        a.canonical = c->canonical;
        a.out_cnt = c->d_cnt;
        a.in_cnt = c->d_tcnt;
        a.out_ptr = c->d_out_ptr;
        a.in_ptr = c->d_in_ptr;
        a.row_src = c->d_val;
        a.row_sign = c->d_val_alt;
        a.row_tgt = reinterpret_cast<int32_t *>(c->d_key32);
        a.row_k = reinterpret_cast<int32_t *>(c->d_key32_alt);
        a.in_syn = c->d_in_syn;
        a.any_long = c->d_i32 + I32_LONG;
        a.retract_ax = retract_ax;
        a.retract_de = retract_de;
        a.vac_ax = vac_ax;
        a.vac_de = vac_de;
        a.need_ax = c->d_need_ax;
        a.need_de = c->d_need_de;
        a.prio_ax = c->d_prio_ax;
        a.prio_de = c->d_prio_de;
        a.sel_ax = c->d_sel_ax;
        a.sel_de = c->d_sel_de;
        a.broken = c->d_i64 + I64_BROKEN;
        delete_small_kernel<<<cluster_form::kBlocks, cluster_form::kThreads, 0, st>>>(
            a, store_args(c, p.seed, (uint32_t)p.step));
        note_launch();
        c->canonical = false; // as below
        return cudaGetLastError();
    }
    if (!c->canonical && (e = canonicalise_store(c, st))) return e;
    delete_needs_kernel<<<gn, 256, 0, st>>>(n, retract_ax, retract_de, vac_ax, vac_de,
                                            c->d_out_ptr, c->d_in_ptr, c->d_need_ax,
                                            c->d_need_de);
    note_launch();
    delete_prio_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_src, c->d_in_syn, c->d_syn_tgt,
                                           c->d_out_ptr, c->d_in_ptr, c->d_need_ax,
                                           c->d_need_de, c->d_prio_ax, c->d_prio_de,
                                           c->d_sel_ax, c->d_sel_de, p.seed, (uint32_t)p.step);
    note_launch();
    delete_select_kernel<<<gn, 256, 0, st>>>(n, c->d_out_ptr, c->d_need_ax, c->d_prio_ax, nullptr,
                                             c->d_sel_ax);
    note_launch();
    delete_select_kernel<<<gn, 256, 0, st>>>(n, c->d_in_ptr, c->d_need_de, c->d_prio_de,
                                             c->d_in_syn, c->d_sel_de);
    note_launch();
    delete_apply_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_src, c->d_syn_tgt, c->d_sel_ax,
                                            c->d_sel_de, vac_ax, vac_de, c->d_keep);
    note_launch();
    if ((e = scan_exclusive(c->d_keep, c->d_keep, c->max_synapses, dm, c->d_i64 + I64_SCAN_TOTAL,
                            c->scan, st)))
        return e;
    compact_kernel<<<gs, 256, 0, st>>>(dm, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign, c->d_sel_ax,
                                       c->d_sel_de, c->d_keep, bits, c->d_key, c->d_val);
    note_launch();
    shrink_store_kernel<<<1, 1, 0, st>>>(c->d_i32 + I32_NSYN, c->d_i64 + I64_SCAN_TOTAL,
                                         c->d_i64 + I64_BROKEN, c->d_i64 + I64_NSYN);
    note_launch();
    unpack_keys_kernel<<<gs, 256, 0, st>>>(dm, c->d_key, c->d_val, bits, c->d_syn_src,
                                           c->d_syn_tgt, c->d_syn_sign);
    note_launch();
    // the kept synapses are in canonical order; their views are rebuilt when an
    // operation next needs them (the next update appends anyway)
    c->canonical = false;
    return cudaGetLastError();
}

namespace {

// Typed dendrite pools: the axons of one type, and writing them back.
__global__ void select_type_kernel(const int32_t *__restrict__ vac_ax,
                                   const uint8_t *__restrict__ type, int kind, int64_t n,
                                   int32_t *__restrict__ out)
{
    GRID_STRIDE(i, n) out[i] = type[i] == kind ? vac_ax[i] : 0;
}

__global__ void merge_type_kernel(const int32_t *__restrict__ part,
                                  const uint8_t *__restrict__ type, int kind, int64_t n,
                                  int32_t *__restrict__ vac_ax)
{
    GRID_STRIDE(i, n)
    {
        if (type[i] == kind) vac_ax[i] = part[i];
    }
}

} // namespace

cudaError_t select_type(relearn_ctx *c, const int32_t *vac_ax, const uint8_t *type, int kind,
                        int32_t *out, cudaStream_t st)
{
    select_type_kernel<<<grid_for(c->n, 256, c->num_sms), 256, 0, st>>>(vac_ax, type, kind, c->n,
                                                                        out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t merge_type(relearn_ctx *c, const int32_t *part, const uint8_t *type, int kind,
                       int32_t *vac_ax, cudaStream_t st)
{
    merge_type_kernel<<<grid_for(c->n, 256, c->num_sms), 256, 0, st>>>(part, type, kind, c->n,
                                                                       vac_ax);
    note_launch();
    return cudaGetLastError();
}

cudaError_t deliver_spikes(relearn_ctx *c, const uint8_t *spiked, int32_t *input,
                           cudaStream_t st)
{
    if (deliver_small(c, st)) {
        deliver_small_kernel<<<cluster_form::kBlocks, cluster_form::kThreads, 0, st>>>(
            c->d_i32 + I32_NSYN, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign, spiked, nullptr, 0, 0, c->n,
            input);
        note_launch();
        return cudaGetLastError();
    }
    cudaError_t e;
    if ((e = cudaMemsetAsync(input, 0, c->n * sizeof(int32_t), st))) return e;
    const int w = deliver_width(c);
    (w == 1 ? spikes_kernel<1> : spikes_kernel<4>)
        <<<grid_for((c->max_synapses + w - 1) / w, 256, c->num_sms), 256, 0, st>>>(
            c->d_i32 + I32_NSYN, c->d_syn_src, c->d_syn_tgt, c->d_syn_sign, spiked, input);
    note_launch();
    return cudaGetLastError();
}

} // namespace rl
