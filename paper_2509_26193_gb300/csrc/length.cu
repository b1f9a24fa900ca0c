// Differentiable form (not in the paper): the expected synapse length over each
// source's root frontier and its adjoint.
//
// For a source i with m_i = vac_ax[i] > 0, its root frontier F_i is the set of
// candidates of its first draw (Sec. III-B search from the root, criterion of
// Sec. II), its own leaf excluded. With D_ik = |x_i - c_k|^2, d_ik = sqrt(D_ik),
// a_ik = N_k exp(-D_ik / sigma^2), S_i = sum_k a_ik and q_ik = a_ik / S_i:
//   l_i = sum_k q_ik d_ik,   L = sum_i m_i l_i / M,   M = sum of m_i with S_i > 0.
// Adjoint (criterion and topology constant):
//   dl_i/dsigma = (2 / sigma^3) sum_k q_ik (d_ik - l_i) (D_ik - Dbar_i),
//   dl_i/dc_k   = q_ik r_ik (2 (d_ik - l_i) / sigma^2 - 1 / d_ik),  r = x_i - c_k,
//   dl_i/dx_i   = -sum_k dl_i/dc_k,   dc_k/dx_j = w_j / N_k  (w = vac_de).
//
// Forward: one walk of the root frontiers of 32 sources at a time (group walks, below),
// FP32 attractions with Kahan-compensated sums; S, l and Dbar formed in FP64 and kept
// per source with the exponent shift. Backward: the same walk again, recomputing every
// attraction (nothing per candidate is stored), accumulating the centroid adjoints
// G_k = sum_i (m_i / M) dl_i/dc_k per node in FP64 and each source's direct term in
// registers (Kahan-compensated FP32: it is a sum of terms of both signs that nearly
// cancel); then every neuron j adds w_j * sum over its cells k of G_k / N_k (its leaf's
// parent chain, in FP64).
//
// Node adjoints: the warp sums its lanes' (x, y, z) contributions to eight nodes at a
// time (a transpose reduction that leaves each component's total on one lane) and adds
// the totals to the nodes with FP64 atomics. One FP32 vector atomic per lane and
// candidate (an earlier design) was L2-atomic-bound and its order-dependent FP32 sums
// left element-wise gradient errors up to 6e-3 of the cancellation-aware scale at 2^18
// neurons; FP64 sums of warp partials bring every element within the FP32 arithmetic of
// its terms.
//
// Measured (GB300, uniform cube, theta 0.3, the forward and backward calls with their
// small kernels, one-node-per-step union walks -> group walks): 2^18 neurons forward
// 1.77 -> 1.55 ms, backward 5.75 -> 2.66 ms; 5,003 neurons, forward + backward
// 5.5 -> 0.18 ms. Bound by instruction issue (70 to 73 % active at 2^18: per entry and
// group about 16 instructions of forward sums, 40 of backward ones, and 16 of walking).
#include "cluster.cuh"
#include "internal.h"

namespace rl {

namespace {

constexpr float kTinyL = 8.673617e-19f; // 2^-60: below this S is redone with a shift

struct LenArgs {
    const Node *__restrict__ nodes;
    const FamNode *__restrict__ fam;
    const float4 *__restrict__ pos;
    const int32_t *__restrict__ perm;
    const int32_t *__restrict__ act_src;
    const int32_t *__restrict__ leaf_of;
    const int32_t *__restrict__ vac_ax;
    int64_t n;              // neurons
    const Geom *geom;       // the network's
    const int64_t *d_total; // active sources
    int32_t *redo;          // groups left to redo_kernel: their number, its work counter,
                            // its blocks done
    int32_t *redo_list;     // [n] which
    int64_t *evals_total;   // candidates visited (both passes)
    const SearchConst *sc;
    float4 *state;  // [n] per Morton position
    double *lsum;   // [4]
    double *mean;   // forward: the caller's, or NULL
    int32_t *work;
    // backward
    double *G;           // [4 * nodes] centroid adjoints (x, y, z, unused) in FP64
    float *gx, *gy, *gz; // id order
    const double *gout;  // upstream gradient of the mean (NULL = 1)
    double *gsigma;
};

__device__ __forceinline__ float att(float cnt, float D, float k2, float k2sh)
{
    return __fmul_rn(cnt, ex2_approx(__fmaf_rn(-k2, D, k2sh)));
}

__device__ __forceinline__ void kahan(float &sum, float &c, float a)
{
    const float y = __fsub_rn(a, c);
    const float t = __fadd_rn(sum, y);
    c = __fsub_rn(__fsub_rn(t, sum), y);
    sum = t;
}

struct Fwd {
    float s = 0.f, sc = 0.f, a = 0.f, ac = 0.f, b = 0.f, bc = 0.f;
    float dmin2 = __builtin_huge_valf();
};

struct Bwd {
    float cov = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
    float cx = 0.f, cy = 0.f, cz = 0.f; // Kahan compensation of the direct term
};

struct Src {
    float3 x;
    int32_t self;
    float l, Db, invS, k2sh, w; // backward: state and (m_i gout / M)
};

// One candidate (accepted, count > 0, not the source's own leaf).
__device__ __forceinline__ void fwd_visit(Fwd &f, float cnt, float D, float k2, float k2sh)
{
    const float at = att(cnt, D, k2, k2sh);
    const float d = sqrt_approx(D);
    kahan(f.s, f.sc, at);
    kahan(f.a, f.ac, __fmul_rn(at, d));
    kahan(f.b, f.bc, __fmul_rn(at, D));
    f.dmin2 = fminf(f.dmin2, D);
}

// Returns the node's adjoint contribution (m_i / M) dl_i/dc_k in (ox, oy, oz).
__device__ __forceinline__ void bwd_visit(Bwd &b, const Src &s, float cnt, float rx, float ry,
                                          float rz, float D, float k2, float two_s2, float &ox,
                                          float &oy, float &oz)
{
    const float q = __fmul_rn(att(cnt, D, k2, s.k2sh), s.invS);
    const float d = sqrt_approx(D);
    const float dl = __fsub_rn(d, s.l);
    b.cov = __fmaf_rn(__fmul_rn(q, dl), __fsub_rn(D, s.Db), b.cov);
    const float inv_d = d > 0.0f ? rcp_approx(d) : 0.0f;
    const float kap = __fmul_rn(__fmul_rn(q, __fmaf_rn(two_s2, dl, -inv_d)), s.w);
    ox = __fmul_rn(kap, rx);
    oy = __fmul_rn(kap, ry);
    oz = __fmul_rn(kap, rz);
    kahan(b.gx, b.cx, -ox);
    kahan(b.gy, b.cy, -oy);
    kahan(b.gz, b.cz, -oz);
}

// One lane's own contribution straight to the node (lane-by-lane walks, rare).
__device__ __forceinline__ void add_node(double *G, int32_t p, float ox, float oy, float oz)
{
    atomicAdd(&G[4 * (int64_t)p + 0], (double)ox);
    atomicAdd(&G[4 * (int64_t)p + 1], (double)oy);
    atomicAdd(&G[4 * (int64_t)p + 2], (double)oz);
}

// A lane's own walk of its root frontier (stackless: expand = p + 1, accept or
// empty = escape).
template <bool kBack>
__device__ int32_t lane_walk(const LenArgs &a, const Src &s, int32_t p, int32_t end,
                             uint32_t thr0, float k2, float k2sh, float two_s2, Fwd &f, Bwd &b)
{
    int32_t visited = 0;
    while (p < end) {
        const float4 g = __ldg(reinterpret_cast<const float4 *>(&a.nodes[p].g));
        const int2 t = __ldg(reinterpret_cast<const int2 *>(&a.nodes[p].t));
        const float rx = __fsub_rn(s.x.x, g.x), ry = __fsub_rn(s.x.y, g.y),
                    rz = __fsub_rn(s.x.z, g.z);
        const float D = __fmaf_rn(rx, rx, __fmaf_rn(ry, ry, __fmul_rn(rz, rz)));
        const bool has = g.w > 0.0f;
        const bool pass = __float_as_uint(D) + (uint32_t)t.y > thr0;
        if (has && pass && p != s.self) {
            ++visited;
            if constexpr (!kBack) {
                fwd_visit(f, g.w, D, k2, k2sh);
            } else {
                float ox, oy, oz;
                bwd_visit(b, s, g.w, rx, ry, rz, D, k2, two_s2, ox, oy, oz);
                add_node(a.G, p, ox, oy, oz);
            }
        }
        p = (has && !pass) ? p + 1 : max(t.x, p + 1);
    }
    return visited;
}

// ---- group walks --------------------------------------------------------------
// Both passes visit, for each group of 32 sources (adjacent in Morton order), every
// node that at least one of them accepts, once, with the set of sources that take it.
// The order is free here (unlike the search's draw), which makes the walk cheap: the
// lanes of a warp hold nodes, eight families of up to eight children at a time, and put
// each node to the criterion for the whole group at once; the accepted ones are then
// evaluated in chunks of 32, lanes holding sources, the nodes read from shared memory
// (a 16-byte broadcast from there costs 2.3 cycles of the SM, the 32-byte broadcast from
// L1 of a one-node-per-step walk 8.2, which bounded that walk together with its 31
// instructions per step).
//
// The group's test is conservative: D = fma(rx, rx, fma(ry, ry, rz * rz)) with
// rx = fl(x - cx) is non-decreasing in |rx|, |ry| and |rz| (rounding is monotone), so the
// same expression on the smallest and largest |x - cx| over the group's bounding box
// bounds every source's D exactly. A node whose lower bound passes is taken by every
// source that reaches it, one whose upper bound fails is expanded for all of them, and
// the few in between are tested source by source when their chunk is evaluated (their
// subtree goes on with the sources that rejected it).
//
// A pending node carries its set of sources as a mask. With fewer than one group to two
// resident warps, 2, 4 or 8 warps of a block share a group: each keeps every second,
// fourth or eighth of the first pending nodes, and their sums are added through shared
// memory (5,000 neurons: 135 groups for 3,648 warps). The line, groups x warps per group
// at most twice the resident warps (forward + backward): 60,000 neurons 1.19 ms, at
// most once 1.29, four times 1.24; 2^18 4.39, 4.41, 4.82 ms.

constexpr int kGroupWarps = 8;      // warps per block
constexpr int kPend = 256;          // pending nodes per warp
constexpr int kEntries = 128;       // accepted nodes per warp waiting for evaluation
constexpr int kLenChunk = 32;       // entries evaluated at a time
constexpr uint32_t kTestFlag = 0x80000000u;
constexpr uint32_t kLastSibling = 1u; // in FamNode::shift

struct __align__(16) GroupShared {
    float4 xy[kLenChunk / 2]; // entries 2k, 2k + 1: x, x, y, y
    float4 zc[kLenChunk / 2]; // z, z, count, count
    uint32_t mask[kLenChunk]; // sources that reach the entry
    int32_t pre[kLenChunk];
    uint32_t shift[kLenChunk];
    uint2 pend[kPend];        // first child, mask
    uint2 out[kEntries];      // node (| kTestFlag), mask
    int32_t self[32];         // the sources' own leaves (ascending; idle lanes: the largest int)
};

using Pair = unsigned long long; // two packed floats
__device__ __forceinline__ Pair pack2(float a, float b)
{
    Pair r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(Pair v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ Pair sub2(Pair a, Pair b)
{
    Pair r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b)
{
    Pair r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ Pair add2(Pair a, Pair b)
{
    Pair r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c)
{
    Pair r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ void kahan2(Pair &sum, Pair &c, Pair a)
{
    const Pair y = sub2(a, c);
    const Pair t = add2(sum, y);
    c = sub2(sub2(t, sum), y);
    sum = t;
}

// Two compensated sums side by side, one over the even entries, one over the odd ones.
struct Sum2 {
    Pair s = 0ull, c = 0ull;
    __device__ __forceinline__ void add(Pair a) { kahan2(s, c, a); }
    __device__ __forceinline__ void add_one(float a) // into the even one
    {
        float s0, s1, c0, c1;
        unpack2(s, s0, s1);
        unpack2(c, c0, c1);
        kahan(s0, c0, a);
        s = pack2(s0, s1);
        c = pack2(c0, c1);
    }
    __device__ __forceinline__ double total() const
    {
        float s0, s1, c0, c1;
        unpack2(s, s0, s1);
        unpack2(c, c0, c1);
        return ((double)s0 - (double)c0) + ((double)s1 - (double)c1);
    }
};

struct FwdSums {
    Sum2 s, a, b; // attraction, attraction x d, attraction x D
};
struct BwdSums {
    Sum2 cov;
    Sum2 gx, gy, gz; // the direct term, negated
};

__device__ __forceinline__ void load_fam(const FamNode *n, float4 &g, int4 &t)
{
    float v[8];
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
          "=f"(v[7])
        : "l"(n));
    g = make_float4(v[0], v[1], v[2], v[3]);
    t = make_int4(__float_as_int(v[4]), __float_as_int(v[5]), __float_as_int(v[6]),
                  __float_as_int(v[7]));
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float dist2_of(float rx, float ry, float rz)
{
    return __fmaf_rn(rx, rx, __fmaf_rn(ry, ry, __fmul_rn(rz, rz)));
}

// A pending subtree without room to expand it: its sources walk it one by one. Called
// only while the pending list is nearly full.
template <bool kBack>
__device__ __noinline__ void walk_pending(const LenArgs &a, const Src &s, uint2 item,
                                          uint32_t thr0, float k2, float two_s2, float sums[4],
                                          int64_t &evals)
{
    const int lane = threadIdx.x & 31;
    const FamNode *kid = a.fam + item.x;
    const int32_t p0 = kid->pre;
    const int32_t end = a.nodes[kid->up].t.escape;
    Fwd f;
    Bwd b;
    if ((item.y >> lane) & 1u)
        evals += lane_walk<kBack>(a, s, p0, end, thr0, k2, s.k2sh, two_s2, f, b);
    if constexpr (kBack) {
        sums[0] = b.cov;
        sums[1] = __fsub_rn(b.cx, b.gx);
        sums[2] = __fsub_rn(b.cy, b.gy);
        sums[3] = __fsub_rn(b.cz, b.gz);
    } else {
        sums[0] = __fsub_rn(f.s, f.sc);
        sums[1] = __fsub_rn(f.a, f.ac);
        sums[2] = __fsub_rn(f.b, f.bc);
        sums[3] = f.dmin2;
    }
    __syncwarp();
}

// The walk of one group by one warp (all lanes converged).
struct GroupWalk {
    const FamNode *__restrict__ fam;
    GroupShared *s;
    uint32_t thr0;
    float lx, hx, ly, hy, lz, hz; // bounding box of the sources
    int32_t self_lo, self_hi;     // range of the sources' own leaves (pre-order)
    int32_t base, top;            // pending nodes: pend[base .. top)
    int32_t outc;                 // entries: out[0 .. outc)

    // members: the lanes that are sources, at least one
    __device__ __forceinline__ void start(uint32_t members, float3 x, int32_t self)
    {
        const int lane = threadIdx.x & 31;
        const float inf = __int_as_float(0x7f800000);
        const bool in = (members >> lane) & 1u;
        lx = warp_min(in ? x.x : inf);
        hx = -warp_min(in ? -x.x : inf);
        ly = warp_min(in ? x.y : inf);
        hy = -warp_min(in ? -x.y : inf);
        lz = warp_min(in ? x.z : inf);
        hz = -warp_min(in ? -x.z : inf);
        self_lo = __shfl_sync(0xffffffffu, self, __ffs(members) - 1);
        self_hi = __shfl_sync(0xffffffffu, self, 31 - __clz(members));
        s->self[lane] = self;
        if (lane == 0) s->pend[0] = make_uint2((uint32_t)__ldg(&fam[0].kids), members);
        base = 0;
        top = 1;
        outc = 0;
        __syncwarp();
    }

    // Expands up to eight pending nodes, the last ones (or the first ones, so that the
    // list grows evenly over the tree): at most 64 more pending nodes and entries.
    template <bool kFront>
    __device__ __forceinline__ void expand()
    {
        const int lane = threadIdx.x & 31;
        const uint32_t lt = lanemask_lt();
        const int ns = min(8, top - base);
        const int c = lane & 7;
        uint2 it[2];
        bool slot_on[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int slot = (lane >> 3) + 4 * h;
            slot_on[h] = slot < ns;
            it[h] = slot < ns ? s->pend[kFront ? base + slot : top - 1 - slot]
                              : make_uint2(0u, 0u); // family 0 holds the root alone
        }
        if (kFront)
            base += ns;
        else
            top -= ns;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && ns <= 4) break;
            const uint32_t k = it[h].x + c;
            float4 g;
            int4 t;
            load_fam(&fam[k], g, t);
            const uint32_t shift = (uint32_t)t.w & ~kLastSibling;
            // the family ends at its last sibling; one of more than eight (a bucket's
            // leaves) goes on as another pending node
            const uint32_t ends = __ballot_sync(0xffffffffu, ((uint32_t)t.w & kLastSibling) != 0u);
            const uint32_t fam_ends = (ends >> (lane & 24)) & 0xffu;
            const bool act = slot_on[h] && (fam_ends & ((1u << c) - 1u)) == 0u;
            bool near_ok = true, far_ok = true; // the criterion at the bounds of D
            if (!node_is_leaf(shift)) {
                const float ax = __fsub_rn(lx, g.x), bx = __fsub_rn(hx, g.x);
                const float ay = __fsub_rn(ly, g.y), by = __fsub_rn(hy, g.y);
                const float az = __fsub_rn(lz, g.z), bz = __fsub_rn(hz, g.z);
                const float D0 = dist2_of(fmaxf(fmaxf(ax, -bx), 0.0f), fmaxf(fmaxf(ay, -by), 0.0f),
                                          fmaxf(fmaxf(az, -bz), 0.0f));
                const float D1 = dist2_of(fmaxf(fabsf(ax), fabsf(bx)), fmaxf(fabsf(ay), fabsf(by)),
                                          fmaxf(fabsf(az), fabsf(bz)));
                // (a centroid that is not a number is accepted, as by each source alone)
                near_ok = __float_as_uint(D0) + shift > thr0 || D1 != D1;
                far_ok = __float_as_uint(D1) + shift > thr0;
            }
            const bool has = act && g.w > 0.0f;
            const uint32_t entry = __ballot_sync(0xffffffffu, has && far_ok);
            const uint32_t open = __ballot_sync(0xffffffffu, has && !far_ok);
            if (has && far_ok)
                s->out[outc + __popc(entry & lt)] =
                    make_uint2(near_ok ? k : k | kTestFlag, it[h].y);
            if (has && !far_ok)
                s->pend[top + __popc(open & lt)] = make_uint2((uint32_t)t.z, it[h].y);
            top += __popc(open);
            outc += __popc(entry);
            // (a zero byte in ends: none of its eight nodes is a last sibling)
            if ((ends - 0x01010101u) & ~ends & 0x80808080u) {
                const bool more = act && c == 7 && fam_ends == 0u;
                const uint32_t rest = __ballot_sync(0xffffffffu, more);
                if (more) s->pend[top + __popc(rest & lt)] = make_uint2(k + 1u, it[h].y);
                top += __popc(rest);
            }
        }
        __syncwarp();
    }

    // Of the pending nodes and entries keep every wpg-th, from the sub-th on.
    __device__ __forceinline__ void take_share(int sub, int wpg)
    {
        const int lane = threadIdx.x & 31;
        auto thin = [&](uint2 *v, int from, int to) {
            int kept = 0;
            for (int i0 = 0; from + sub + wpg * i0 < to; i0 += 32) {
                const int q = from + sub + wpg * (i0 + lane);
                const bool ok = q < to;
                const uint2 w = ok ? v[q] : make_uint2(0u, 0u);
                __syncwarp();
                if (ok) v[i0 + lane] = w; // never past the place it was read from
                __syncwarp();
                kept += __popc(__ballot_sync(0xffffffffu, ok));
            }
            return kept;
        };
        top = thin(s->pend, base, top);
        base = 0;
        outc = thin(s->out, 0, outc);
    }

    // The next chunk: the last n <= 32 entries into xy, zc, mask, pre and shift, filled up
    // with entries that no source takes. Returns the entries that have to be tested
    // source by source; kids = the first child of this lane's entry.
    __device__ __forceinline__ uint32_t gather(int n, uint32_t &kids, int64_t &evals)
    {
        const int lane = threadIdx.x & 31;
        outc -= n;
        kids = 0u;
        bool tst = false;
        if (lane < n) {
            const uint2 w = s->out[outc + lane];
            float4 g;
            int4 t;
            load_fam(&fam[w.x & ~kTestFlag], g, t);
            tst = (w.x & kTestFlag) != 0u;
            uint32_t m = w.y;
            const uint32_t shift = (uint32_t)t.w & ~kLastSibling;
            if (node_is_leaf(shift) && t.x >= self_lo && t.x <= self_hi) {
                int lo = 0; // a source does not take its own leaf
#pragma unroll
                for (int o = 16; o; o >>= 1)
                    if (s->self[lo + o] <= t.x) lo += o;
                if (s->self[lo] == t.x) m &= ~(1u << lo);
            }
            // a position that is not a number makes the sums of the sources that take it
            // not a number, and no other's
            if (g.x != g.x || g.y != g.y || g.z != g.z)
                g = make_float4(lx, ly, lz, __int_as_float(0x7fc00000));
            float *xy = reinterpret_cast<float *>(s->xy) + (lane >> 1) * 4 + (lane & 1);
            float *zc = reinterpret_cast<float *>(s->zc) + (lane >> 1) * 4 + (lane & 1);
            xy[0] = g.x;
            xy[2] = g.y;
            zc[0] = g.z;
            zc[2] = g.w;
            s->mask[lane] = m;
            s->pre[lane] = t.x;
            s->shift[lane] = shift;
            kids = (uint32_t)t.z;
            evals += __popc(m);
        } else { // padding
            float *xy = reinterpret_cast<float *>(s->xy) + (lane >> 1) * 4 + (lane & 1);
            float *zc = reinterpret_cast<float *>(s->zc) + (lane >> 1) * 4 + (lane & 1);
            xy[0] = lx;
            xy[2] = ly;
            zc[0] = lz;
            zc[2] = 0.0f;
            s->mask[lane] = 0u;
        }
        const uint32_t tests = __ballot_sync(0xffffffffu, tst);
        __syncwarp();
        return tests;
    }

    // Puts the marked entries of the chunk to the criterion, source by source (x: this
    // lane's): their masks keep the sources that take them, and below them the sources
    // that do not go on. Apart from the sums, so that those run without a branch (tests
    // inside their loop kept its chains of dependent operations from overlapping: 2^18
    // neurons, forward 1.71 against 1.55 ms).
    __device__ __forceinline__ void resolve(uint32_t tests, uint32_t kids, float3 x,
                                            int64_t &evals)
    {
        const int lane = threadIdx.x & 31;
        const uint32_t bit = 1u << lane;
        uint32_t rej = 0u; // of entry `lane`
        const float *xy = reinterpret_cast<const float *>(s->xy);
        const float *zc = reinterpret_cast<const float *>(s->zc);
        while (tests) { // two at a time (an odd last one twice)
            const int j0 = __ffs(tests) - 1;
            tests &= tests - 1;
            const int j1 = tests ? __ffs(tests) - 1 : j0;
            tests &= tests - 1;
            const int k0 = (j0 >> 1) * 4 + (j0 & 1), k1 = (j1 >> 1) * 4 + (j1 & 1);
            const float D0 = dist2_of(__fsub_rn(x.x, xy[k0]), __fsub_rn(x.y, xy[k0 + 2]),
                                      __fsub_rn(x.z, zc[k0]));
            const float D1 = dist2_of(__fsub_rn(x.x, xy[k1]), __fsub_rn(x.y, xy[k1 + 2]),
                                      __fsub_rn(x.z, zc[k1]));
            const bool f0 = !(__float_as_uint(D0) + s->shift[j0] > thr0);
            const bool f1 = !(__float_as_uint(D1) + s->shift[j1] > thr0);
            const uint32_t r0 = __ballot_sync(0xffffffffu, f0 && (s->mask[j0] & bit));
            const uint32_t r1 = __ballot_sync(0xffffffffu, f1 && (s->mask[j1] & bit));
            if (lane == j0) rej = r0;
            if (lane == j1) rej = r1;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, rej != 0u);
        if (rej) {
            s->mask[lane] &= ~rej;
            s->pend[top + __popc(m & lanemask_lt())] = make_uint2(kids, rej);
        }
        top += __popc(m);
        evals -= __popc(rej);
        __syncwarp();
    }
};

// The chunk's sums of this lane's source (kNear: and its nearest D).
template <bool kNear>
__device__ __forceinline__ void fwd_chunk(const GroupShared *g, int n, const Src &src, float k2,
                                          FwdSums &f, float &nearest)
{
    const uint32_t bit = 1u << (threadIdx.x & 31);
    const Pair xx = pack2(src.x.x, src.x.x), yy = pack2(src.x.y, src.x.y),
               zz = pack2(src.x.z, src.x.z), nk2 = pack2(-k2, -k2),
               sh = pack2(src.k2sh, src.k2sh);
#pragma unroll 4
    for (int j = 0; j < n; j += 2) {
        const ulonglong2 xy = *reinterpret_cast<const ulonglong2 *>(&g->xy[j >> 1]);
        const ulonglong2 zc = *reinterpret_cast<const ulonglong2 *>(&g->zc[j >> 1]);
        const uint2 m = *reinterpret_cast<const uint2 *>(&g->mask[j]);
        const Pair rx = sub2(xx, xy.x), ry = sub2(yy, xy.y), rz = sub2(zz, zc.x);
        const Pair D = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
        const bool on0 = (m.x & bit) != 0u, on1 = (m.y & bit) != 0u;
        float D0, D1, e0, e1;
        unpack2(D, D0, D1);
        unpack2(fma2(nk2, D, sh), e0, e1);
        float a0, a1;
        unpack2(mul2(zc.y, pack2(ex2_approx(e0), ex2_approx(e1))), a0, a1);
        const Pair at = pack2(on0 ? a0 : 0.0f, on1 ? a1 : 0.0f);
        f.s.add(at);
        f.a.add(mul2(at, pack2(sqrt_approx(D0), sqrt_approx(D1))));
        f.b.add(mul2(at, D));
        if constexpr (kNear) {
            if (on0) nearest = fminf(nearest, D0);
            if (on1) nearest = fminf(nearest, D1);
        }
    }
}

// Sums over the 32 lanes of v[e][c] (8 entries, x, y, z), as a transpose reduction: at
// each level a lane keeps half of its values and sends the other half, so that after
// five levels lane 4 e + c holds the total of entry e, component c (31 adds and 24
// shuffles for 24 totals).
__device__ __forceinline__ float warp_sum_8x3(float v[8][3], int lane)
{
#pragma unroll
    for (int lev = 0; lev < 3; ++lev) {
        const int o = 16 >> lev, half = 4 >> lev;
        const bool hi = lane & o;
#pragma unroll
        for (int e = 0; e < half; ++e)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float keep = hi ? v[e + half][c] : v[e][c];
                const float send = hi ? v[e][c] : v[e + half][c];
                v[e][c] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
            }
    }
    const bool c1 = lane & 2, c0 = lane & 1;
    float k0 = c1 ? v[0][2] : v[0][0], k1 = c1 ? 0.0f : v[0][1];
    k0 = __fadd_rn(k0, __shfl_xor_sync(0xffffffffu, c1 ? v[0][0] : v[0][2], 2));
    k1 = __fadd_rn(k1, __shfl_xor_sync(0xffffffffu, c1 ? v[0][1] : 0.0f, 2));
    return __fadd_rn(c0 ? k1 : k0, __shfl_xor_sync(0xffffffffu, c0 ? k0 : k1, 1));
}

// The chunk's terms of this lane's source: its covariance and direct term, and the
// warp's contributions to the entries' adjoints, eight entries at a time: summed over
// the warp in FP32, then one FP64 atomic per entry and component.
__device__ __forceinline__ void bwd_chunk(const GroupShared *g, int n, const Src &src, float k2,
                                          float two_s2, double *G, BwdSums &b)
{
    const int lane = threadIdx.x & 31;
    const uint32_t bit = 1u << lane;
    const Pair xx = pack2(src.x.x, src.x.x), yy = pack2(src.x.y, src.x.y),
               zz = pack2(src.x.z, src.x.z), nk2 = pack2(-k2, -k2),
               sh = pack2(src.k2sh, src.k2sh), inv_s = pack2(src.invS, src.invS),
               ll = pack2(src.l, src.l), db = pack2(src.Db, src.Db),
               ww = pack2(src.w, src.w), ts = pack2(two_s2, two_s2);
    for (int j0 = 0; j0 < n; j0 += 8) {
        float v[8][3];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const int j = j0 + u;
            const ulonglong2 xy = *reinterpret_cast<const ulonglong2 *>(&g->xy[j >> 1]);
            const ulonglong2 zc = *reinterpret_cast<const ulonglong2 *>(&g->zc[j >> 1]);
            const uint2 m = *reinterpret_cast<const uint2 *>(&g->mask[j]);
            const Pair rx = sub2(xx, xy.x), ry = sub2(yy, xy.y), rz = sub2(zz, zc.x);
            const Pair D = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
            const bool on0 = (m.x & bit) != 0u, on1 = (m.y & bit) != 0u;
            float D0, D1, e0, e1, a0, a1;
            unpack2(D, D0, D1);
            unpack2(fma2(nk2, D, sh), e0, e1);
            unpack2(mul2(zc.y, pack2(ex2_approx(e0), ex2_approx(e1))), a0, a1);
            const Pair q = mul2(pack2(on0 ? a0 : 0.0f, on1 ? a1 : 0.0f), inv_s);
            const float d0 = sqrt_approx(D0), d1 = sqrt_approx(D1);
            const Pair dl = sub2(pack2(d0, d1), ll);
            b.cov.add(mul2(mul2(q, dl), sub2(D, db)));
            const Pair ninv = pack2(d0 > 0.0f ? -rcp_approx(d0) : 0.0f,
                                    d1 > 0.0f ? -rcp_approx(d1) : 0.0f);
            const Pair kap = mul2(mul2(q, fma2(ts, dl, ninv)), ww);
            const Pair ox = mul2(kap, rx), oy = mul2(kap, ry), oz = mul2(kap, rz);
            b.gx.add(ox);
            b.gy.add(oy);
            b.gz.add(oz);
            unpack2(ox, v[u][0], v[u + 1][0]);
            unpack2(oy, v[u][1], v[u + 1][1]);
            unpack2(oz, v[u][2], v[u + 1][2]);
        }
        const float t = warp_sum_8x3(v, lane);
        const int e = j0 + (lane >> 2);
        if ((lane & 3) < 3 && e < n && t != 0.0f)
            atomicAdd(&G[4 * (int64_t)g->pre[e] + (lane & 3)], (double)t);
    }
}

// One walk of a group by this warp, the sub-th of wpg that share it, with what each pass
// adds up of the entries: the forward sums, these and the nearest D, or the adjoint.
// members: the lanes whose sources take part, at least one.
enum Pass { kSums, kNearSums, kAdjoint };
template <Pass kPass>
__device__ __forceinline__ void group_pass(const LenArgs &a, GroupWalk &w, const Src &s,
                                           uint32_t members, int sub, int wpg, float k2,
                                           float two_s2, FwdSums &f, BwdSums &b, float &nearest,
                                           int64_t &evals)
{
    w.start(members, s.x, s.self);
    if (wpg > 1) { // a pending list long enough to share out (at most 140 nodes)
        while (w.top - w.base > 0 && w.top - w.base < 8 * wpg && w.top <= 72 &&
               w.outc < kEntries - 64)
            w.expand<true>();
        w.take_share(sub, wpg);
    }
    for (;;) {
        while (w.outc < kLenChunk && w.top > 0) {
            // no room to expand: many sources at a small theta, or few far apart (uniform
            // cubes, subtrees of a forward call: 2^18 neurons at theta 0.3 88, 0.25 3,298, 0.2
            // 45,117; theta 0 none to 33,001 neurons, 5,277 at 65,001)
            if (w.top > kPend - 64 - kLenChunk) {
                const uint2 it = w.s->pend[--w.top];
                float part[4];
                walk_pending<kPass == kAdjoint>(a, s, it, w.thr0, k2, two_s2, part, evals);
                if constexpr (kPass == kAdjoint) {
                    b.cov.add_one(part[0]);
                    b.gx.add_one(part[1]);
                    b.gy.add_one(part[2]);
                    b.gz.add_one(part[3]);
                } else {
                    f.s.add_one(part[0]);
                    f.a.add_one(part[1]);
                    f.b.add_one(part[2]);
                    if constexpr (kPass == kNearSums) nearest = fminf(nearest, part[3]);
                }
            } else {
                w.expand<false>();
            }
        }
        const int n = min(w.outc, kLenChunk);
        if (n == 0) break;
        uint32_t kids;
        const uint32_t tests = w.gather(n, kids, evals);
        if (tests) w.resolve(tests, kids, s.x, evals);
        if constexpr (kPass == kAdjoint)
            bwd_chunk(w.s, n, s, k2, two_s2, a.G, b);
        else
            fwd_chunk<kPass == kNearSums>(w.s, n, s, k2, f, nearest);
        __syncwarp(); // the chunk is overwritten next
    }
}

using BlockSums = double[kGroupWarps][3][32];

// Warps that share a group (see above for the line).
__device__ __forceinline__ int warps_per_group(int32_t groups)
{
    int wpg = kGroupWarps;
    while (wpg > 1 && (int64_t)groups * wpg > 2 * (int64_t)gridDim.x * kGroupWarps) wpg >>= 1;
    return wpg;
}

// Takes the next of `count` groups for this warp (or, shared by wpg warps each, the next
// kGroupWarps / wpg groups for the block, the last of them possibly past the count). False:
// none left.
__device__ __forceinline__ bool next_group(int32_t *work, int32_t count, int wpg, int32_t &s_next,
                                           int32_t &at)
{
    if (wpg == 1) {
        if ((threadIdx.x & 31) == 0) at = atomicAdd(work, 1);
        at = __shfl_sync(0xffffffffu, at, 0);
        return at < count;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_next = atomicAdd(work, kGroupWarps / wpg);
    __syncthreads();
    at = s_next + (int32_t)(threadIdx.x >> 5) / wpg;
    return s_next < count;
}

// Lanes that take no part (on: this one does) follow a lane that does.
__device__ __forceinline__ void follow(uint32_t members, bool on, float3 &x)
{
    const int f = __ffs(members) - 1;
    const float mx = __shfl_sync(0xffffffffu, x.x, f), my = __shfl_sync(0xffffffffu, x.y, f),
                mz = __shfl_sync(0xffffffffu, x.z, f);
    if (!on) x = make_float3(mx, my, mz);
}

// A source without a finite position has no finite distance and is left out.
__device__ __forceinline__ bool finite_at(float4 p)
{
    return fabsf(p.x) + fabsf(p.y) + fabsf(p.z) < __int_as_float(0x7f800000);
}

// A source's state from its sums, and its share of the mean's numerator and denominator.
__device__ __forceinline__ void finish_source(const LenArgs &a, int32_t sp, int32_t i, double S,
                                              double sa, double sb, float k2sh, double &my0,
                                              double &my1)
{
    float4 st = make_float4(0.f, 0.f, 0.f, k2sh);
    if (S > 0.0) {
        const double l = sa / S;
        st.x = (float)l;
        st.y = (float)(sb / S);
        st.z = (float)(1.0 / S);
        const double m = (double)a.vac_ax[i];
        my0 += m * l;
        my1 += m;
    }
    a.state[sp] = st;
}

__device__ __forceinline__ void add_totals(const LenArgs &a, double my0, double my1,
                                           int64_t my_evals)
{
    for (int o = 16; o; o >>= 1) {
        my0 += __shfl_xor_sync(0xffffffffu, my0, o);
        my1 += __shfl_xor_sync(0xffffffffu, my1, o);
        my_evals += __shfl_xor_sync(0xffffffffu, my_evals, o);
    }
    if ((threadIdx.x & 31) != 0) return;
    if (my_evals)
        atomicAdd(reinterpret_cast<unsigned long long *>(a.evals_total),
                  (unsigned long long)my_evals);
    if (my1 > 0.0) {
        atomicAdd(&a.lsum[0], my0);
        atomicAdd(&a.lsum[1], my1);
    }
}

// Sources whose every attraction underflows need their sums again, with the exponents
// shifted by their nearest D (an exact common factor). The forward pass leaves their groups
// to redo_kernel, the sources marked by a shift of -1 in their state: those whose sums came
// out too small, and, without a walk, whole groups with an isolated source. redo_kernel
// walks a group for the sums and the nearest D at once, and again, shifted, for the
// sources that need it. It also forms the mean, which is all it does where nothing
// underflows. A kernel of its own: as a part of the forward kernel, called from it, the
// same made that one 6 us slower for 1,000 neurons. A forward call in which a tenth / a
// third / nearly all of the sources underflow (a cube of 62 um spacing, sigma 8 / 6 / 1.5
// um), us, each such lane walking its own frontier twice -> here: 5,003 neurons 606 / 634 /
// 655 -> 130 / 135 / 138; 60,000 2,480 / 2,640 / 2,760 -> 747 / 812 / 840; 2^18 4,550 / 4,900 /
// 7,140 -> 2,775 / 3,060 / 3,155. Where nothing underflows (sigma 800 um, replayed from a
// graph): 86 -> 84, 419 -> 407, 1,560 -> 1,510; called directly 91 -> 96 (5,003 neurons).
constexpr float kMarked = -1.0f;

// Whether one of the group's sources (on: this lane's is one, at Morton position sp) has
// none of the four positions on either side of its own in Morton order within the distance
// at which an attraction still counts (2^-50): a guess that its sums will underflow.
__device__ __forceinline__ bool isolated(const LenArgs &a, bool on, int64_t sp, float3 x, float k2)
{
    bool near = !on;
    for (int k = 1; k <= 4 && __any_sync(0xffffffffu, !near); ++k)
        for (int64_t q : {sp - k, sp + k})
            if (!near && q >= 0 && q < a.n) {
                const float4 p = a.pos[q];
                near = __fmul_rn(k2, dist2_of(__fsub_rn(x.x, p.x), __fsub_rn(x.y, p.y),
                                              __fsub_rn(x.z, p.z))) < 50.0f;
            }
    return __any_sync(0xffffffffu, !near);
}

// 3 blocks per SM (80 registers): 2^18 neurons, forward + backward 4.21 ms; 4 blocks
// (64 registers, spills) 4.49, 2 blocks 4.25 (60,000 neurons: 1.13, 1.22, 1.29 ms).
#ifndef RELEARN_LEN_MIN_BLOCKS
#define RELEARN_LEN_MIN_BLOCKS 3
#endif
template <bool kBack>
__global__ void __launch_bounds__(32 * kGroupWarps, RELEARN_LEN_MIN_BLOCKS)
    length_kernel(LenArgs a)
{
    __shared__ GroupShared s_group[kGroupWarps];
    __shared__ BlockSums s_sum;
    __shared__ int32_t s_next;
    const int32_t A = (int32_t)*a.d_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float k2 = __ldg(&a.sc->k2);
    const float sigma = __ldg(&a.sc->sigma);
    const float two_s2 = (float)(2.0 / ((double)sigma * (double)sigma));
    double wscale = 0.0;
    if constexpr (kBack) {
        const double M = a.lsum[1];
        wscale = M > 0.0 ? (a.gout ? *a.gout : 1.0) / M : 0.0;
    }
    const int32_t groups = (A + 31) / 32;
    const int wpg = warps_per_group(groups), sub = warp & (wpg - 1);
    double my0 = 0.0, my1 = 0.0;
    int64_t my_evals = 0;
    GroupWalk w;
    w.fam = a.fam;
    w.s = &s_group[warp];
    w.thr0 = __ldg(&a.sc->thr0);
    // in a domain whose diagonal is within an attraction's reach no source is isolated
    const float ext = kBack ? 0.0f : (float)a.geom->ext;
    const bool wide = 3.0f * k2 * ext * ext > 50.0f;
    int32_t gr = 0;
    while (next_group(a.work, groups, wpg, s_next, gr)) {
        const int64_t slot = (int64_t)gr * 32 + lane;
        const bool live = slot < A;
        const int32_t sp = live ? a.act_src[slot] : -1;
        Src s;
        const float4 xp = live ? a.pos[sp] : make_float4(0.f, 0.f, 0.f, 0.f);
        s.x = make_float3(xp.x, xp.y, xp.z);
        s.self = live ? a.leaf_of[sp] : 0x7fffffff;
        const int32_t i = live ? a.perm[sp] : 0;
        s.l = s.Db = s.invS = s.k2sh = s.w = 0.0f;
        bool on_src = live && finite_at(xp);
        if constexpr (kBack) {
            if (live) {
                const float4 st = a.state[sp];
                s.l = st.x;
                s.Db = st.y;
                s.invS = st.z;
                s.k2sh = st.w;
            }
            on_src = on_src && s.invS > 0.0f;
            s.w = on_src ? (float)((double)a.vac_ax[i] * wscale) : 0.0f;
        }
        FwdSums f;
        BwdSums b;
        const uint32_t members = __ballot_sync(0xffffffffu, on_src);
        bool left = false; // the whole group is left to redo_kernel
        if constexpr (!kBack)
            if (wide) left = isolated(a, on_src, sp, s.x, k2);
        if (members && !left) {
            follow(members, on_src, s.x);
            float unused;
            group_pass<kBack ? kAdjoint : kSums>(a, w, s, members, sub, wpg, k2, two_s2, f, b,
                                                 unused, my_evals);
        }
        double t0, t1, t2;
        if constexpr (kBack) {
            t0 = b.gx.total();
            t1 = b.gy.total();
            t2 = b.gz.total();
            if (on_src) my0 += (double)s.w * b.cov.total(); // * 2 / sigma^3 below
        } else {
            t0 = f.s.total();
            t1 = f.a.total();
            t2 = f.b.total();
        }
        if (wpg > 1) {
            s_sum[warp][0][lane] = t0;
            s_sum[warp][1][lane] = t1;
            s_sum[warp][2][lane] = t2;
            __syncthreads();
            if (sub != 0) continue;
            for (int k = 1; k < wpg; ++k) {
                t0 += s_sum[warp + k][0][lane];
                t1 += s_sum[warp + k][1][lane];
                t2 += s_sum[warp + k][2][lane];
            }
        }
        if constexpr (!kBack) {
            const bool again = on_src && (left || t0 < (double)kTinyL);
            if (__any_sync(0xffffffffu, again) && lane == 0)
                a.redo_list[atomicAdd(a.redo, 1)] = gr;
            if (again)
                a.state[sp] = make_float4(0.f, 0.f, 0.f, kMarked);
            else if (live)
                finish_source(a, sp, i, t0, t1, t2, 0.0f, my0, my1);
        } else if (on_src) { // the sums hold the negated direct term
            a.gx[i] = (float)-t0;
            a.gy[i] = (float)-t1;
            a.gz[i] = (float)-t2;
        }
        __syncwarp();
    }
    if constexpr (!kBack) {
        add_totals(a, my0, my1, my_evals);
    } else {
        for (int o = 16; o; o >>= 1) {
            my0 += __shfl_xor_sync(0xffffffffu, my0, o);
            my_evals += __shfl_xor_sync(0xffffffffu, my_evals, o);
        }
        if (lane == 0 && my_evals)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.evals_total),
                      (unsigned long long)my_evals);
        if (lane == 0 && a.gsigma && my0 != 0.0) {
            const double sd = (double)sigma;
            atomicAdd(a.gsigma, my0 * 2.0 / (sd * sd * sd));
        }
    }
}

// Each lane's sums and nearest D over the warps that share its group, in their order.
// Every warp of the block calls it and gets its group's.
__device__ __forceinline__ void group_totals(BlockSums &sums, int sub, int wpg, double t[3],
                                             float &nearest)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < 3; ++k) sums[warp][k][lane] = t[k];
    __syncthreads();
    for (int k = 0; k < 3; ++k) {
        t[k] = sums[warp - sub][k][lane];
        for (int q = 1; q < wpg; ++q) t[k] += sums[warp - sub + q][k][lane];
    }
    __syncthreads();
    sums[warp][0][lane] = (double)nearest;
    __syncthreads();
    for (int q = 0; q < wpg; ++q) nearest = fminf(nearest, (float)sums[warp - sub + q][0][lane]);
    __syncthreads();
}

// mean = sum m l / M (NaN when M = 0).
__device__ __forceinline__ void publish_mean(const LenArgs &a)
{
    const volatile double *sum = a.lsum;
    const double M = sum[1];
    const double m = M > 0.0 ? sum[0] / M : __longlong_as_double(0x7ff8000000000000LL);
    a.lsum[2] = m;
    if (a.mean) *a.mean = m;
}

__global__ void __launch_bounds__(32 * kGroupWarps, RELEARN_LEN_MIN_BLOCKS) redo_kernel(LenArgs a)
{
    __shared__ GroupShared s_group[kGroupWarps];
    __shared__ BlockSums s_sum;
    __shared__ int32_t s_next;
    const int32_t groups = a.redo[0];
    if (groups == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) publish_mean(a);
        return;
    }
    const int32_t A = (int32_t)*a.d_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float k2 = __ldg(&a.sc->k2), inf = __int_as_float(0x7f800000);
    const int wpg = warps_per_group(groups), sub = warp & (wpg - 1);
    double my0 = 0.0, my1 = 0.0;
    int64_t my_evals = 0;
    GroupWalk w;
    w.fam = a.fam;
    w.s = &s_group[warp];
    w.thr0 = __ldg(&a.sc->thr0);
    int32_t at = 0;
    while (next_group(a.redo + 1, groups, wpg, s_next, at)) {
        const int64_t slot = at < groups ? (int64_t)a.redo_list[at] * 32 + lane : A;
        const int32_t sp = slot < A ? a.act_src[slot] : -1;
        // (the states of marked sources alone are written, by the warp with sub 0, after the
        // last barrier that follows these reads)
        const bool marked = sp >= 0 && a.state[sp].w == kMarked;
        Src s{};
        const float4 xp = marked ? a.pos[sp] : make_float4(0.f, 0.f, 0.f, 0.f);
        s.x = make_float3(xp.x, xp.y, xp.z);
        s.self = sp >= 0 ? a.leaf_of[sp] : 0x7fffffff;
        uint32_t members = __ballot_sync(0xffffffffu, marked);
        double t[3] = {0.0, 0.0, 0.0};
        float nearest = inf;
        BwdSums unused;
        if (members) {
            FwdSums f;
            follow(members, marked, s.x);
            group_pass<kNearSums>(a, w, s, members, sub, wpg, k2, 0.0f, f, unused, nearest,
                                  my_evals);
            t[0] = f.s.total();
            t[1] = f.a.total();
            t[2] = f.b.total();
        }
        if (wpg > 1) group_totals(s_sum, sub, wpg, t, nearest);
        const bool shifted = marked && t[0] < (double)kTinyL && nearest < inf;
        if (shifted) s.k2sh = __fmul_rn(k2, nearest);
        members = __ballot_sync(0xffffffffu, shifted);
        if (wpg > 1 ? __syncthreads_or(members != 0u) : members != 0u) {
            FwdSums f;
            if (members)
                group_pass<kSums>(a, w, s, members, sub, wpg, k2, 0.0f, f, unused, nearest,
                                  my_evals);
            double u[3] = {f.s.total(), f.a.total(), f.b.total()};
            if (wpg > 1) group_totals(s_sum, sub, wpg, u, nearest);
            if (shifted)
                for (int k = 0; k < 3; ++k) t[k] = u[k];
        }
        if (sub == 0 && marked)
            finish_source(a, sp, a.perm[sp], t[0], t[1], t[2], s.k2sh, my0, my1);
        __syncwarp();
    }
    add_totals(a, my0, my1, my_evals);
    __threadfence(); // the totals, before the block counts as done
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(a.redo + 2, 1) == (int32_t)gridDim.x - 1) {
        __threadfence();
        publish_mean(a);
    }
}

// ---- family order ---------------------------------------------------------------
// Slot 0 holds the root, and the children of node v are the slots 1 + k0[v] .. in Morton
// order, k0 the exclusive prefix over pre-order of the nodes' child counts. Rank of node
// v among its siblings (children of u):
__device__ __forceinline__ int32_t sibling_rank(const Node *__restrict__ nodes, int32_t u,
                                                int32_t v)
{
    if (nodes[u].t.shift == (uint32_t)kMaxDepth << 24) return v - u - 1; // a bucket's leaves
    int32_t r = 0;
    for (int32_t q = u + 1; q < v; q = nodes[q].t.escape) ++r; // at most seven before it
    return r;
}

// Child counts: a node's last child (same escape) knows its own rank. Leaves have none.
__device__ __forceinline__ void family_count(const Node *__restrict__ nodes,
                                             const int32_t *__restrict__ parent, int32_t v,
                                             int32_t *count)
{
    const NodeTopo t = nodes[v].t;
    if (node_is_leaf(t.shift)) count[v] = 0;
    const int32_t u = parent[v];
    if (u >= 0 && nodes[u].t.escape == t.escape) count[u] = sibling_rank(nodes, u, v) + 1;
}

__device__ __forceinline__ void family_emit(const Node *__restrict__ nodes,
                                            const int32_t *__restrict__ parent, int32_t v,
                                            const int32_t *k0, FamNode *fam)
{
    const Node nd = nodes[v];
    const int32_t u = parent[v];
    const bool last = u < 0 || nodes[u].t.escape == nd.t.escape;
    FamNode f;
    f.cx = nd.g.cx;
    f.cy = nd.g.cy;
    f.cz = nd.g.cz;
    f.cnt = nd.g.cnt;
    f.pre = v;
    f.up = u;
    f.kids = node_is_leaf(nd.t.shift) ? 0u : (uint32_t)(1 + k0[v]);
    f.shift = nd.t.shift | (last ? kLastSibling : 0u);
    fam[u < 0 ? 0 : 1 + k0[u] + sibling_rank(nodes, u, v)] = f;
}

// What a forward pass sets up: the active sources (vac_ax > 0) in Morton order, the tree
// in family order with the geometry the bottom-up update just formed, its sums and its
// work counter zeroed: the steps before and after the two prefix sums (over flag and k0),
// or, for networks of at most kSmallLen neurons, all of it as one cluster kernel. Whole
// forward call on the device, us, with a launch for each step -> with two kernels and two
// prefix sums -> with the cluster kernel: 1,000 neurons 71 -> 62 -> 52, 5,003 105 -> 97 ->
// 86, 16,000 151 -> 142 -> 138, 24,000 206 -> 200 -> 199, 40,000 320 -> 311 -> 317.
struct PrepArgs {
    const int32_t *vac_ax, *perm;
    int64_t n;
    int32_t *flag, *off, *act_src;
    int64_t *active;
    const Node *nodes;
    const int32_t *parent;
    const int64_t *d_num_nodes;
    int32_t *k0;
    FamNode *fam;
    double *lsum;
    int32_t *work, *redo;
};
constexpr int64_t kSmallLen = 16384;

#define GRID_STRIDE(i, n)                                                                         \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n);                     \
         i += (int64_t)gridDim.x * blockDim.x)
#define CLUSTER_STRIDE(i, n)                                                                      \
    for (int64_t i = cluster_form::first(); i < (n); i += cluster_form::kStride)

__device__ __forceinline__ int32_t active_flag(const PrepArgs &a, int64_t s)
{
    return a.vac_ax[a.perm[s]] > 0 ? 1 : 0;
}

__device__ __forceinline__ void clear_sums(const PrepArgs &a)
{
    for (int k = 0; k < 4; ++k) a.lsum[k] = 0.0;
    *a.work = 0;
    a.redo[0] = a.redo[1] = a.redo[2] = 0;
}

__global__ void len_count_kernel(PrepArgs a)
{
    const int64_t m = *a.d_num_nodes;
    if (blockIdx.x == 0 && threadIdx.x == 0) clear_sums(a);
    GRID_STRIDE(s, a.n + 1) a.flag[s] = s < a.n ? active_flag(a, s) : 0;
    GRID_STRIDE(v, m) family_count(a.nodes, a.parent, (int32_t)v, a.k0);
}

__global__ void len_emit_kernel(PrepArgs a)
{
    const int64_t m = *a.d_num_nodes;
    GRID_STRIDE(s, a.n)
    {
        if (a.flag[s]) a.act_src[a.off[s]] = (int32_t)s;
    }
    GRID_STRIDE(v, m) family_emit(a.nodes, a.parent, (int32_t)v, a.k0, a.fam);
}

__global__ void __cluster_dims__(cluster_form::kBlocks, 1, 1)
    __launch_bounds__(cluster_form::kThreads) len_prepare_small_kernel(PrepArgs a)
{
    namespace cf = cluster_form;
    const int64_t m = *a.d_num_nodes;
    CLUSTER_STRIDE(v, m) family_count(a.nodes, a.parent, (int32_t)v, a.k0);
    const cf::I32 total = cf::scan<cf::I32>(
        a.n, [&](int64_t s) { return cf::I32{a.flag[s] = active_flag(a, s)}; },
        [&](int64_t s) { return cf::I32{a.flag[s]}; },
        [&](int64_t s, cf::I32 prefix, cf::I32 on, cf::I32) {
            if (on.v) a.act_src[prefix.v] = (int32_t)s;
        });
    if (cf::first() == 0) {
        clear_sums(a);
        *a.active = total.v;
    }
    cf::sync(); // the child counts and the scan's shared words
    cf::scan<cf::I32>(
        m, [&](int64_t v) { return cf::I32{a.k0[v]}; },
        [&](int64_t v) { return cf::I32{a.k0[v]}; },
        [&](int64_t v, cf::I32 prefix, cf::I32, cf::I32) { a.k0[v] = prefix.v; });
    cf::sync();
    CLUSTER_STRIDE(v, m) family_emit(a.nodes, a.parent, (int32_t)v, a.k0, a.fam);
}

// ell[id] = l (NaN for excluded neurons).
__global__ void len_finish_kernel(const float4 *__restrict__ state,
                                  const int32_t *__restrict__ flag,
                                  const int32_t *__restrict__ perm, int64_t n, float *ell)
{
    GRID_STRIDE(s, n)
    {
        const float4 st = state[s];
        ell[perm[s]] = flag[s] && st.z > 0.0f ? st.x : __int_as_float(0x7fc00000);
    }
}

// What a backward pass adds into, zeroed in one launch.
__global__ void len_zero_kernel(double4 *G, const int64_t *d_num_nodes, int64_t n, float *gx,
                                float *gy, float *gz, double *gsigma, int32_t *work)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *work = 0;
        if (gsigma) *gsigma = 0.0;
    }
    const int64_t m = *d_num_nodes;
    GRID_STRIDE(k, m) G[k] = make_double4(0.0, 0.0, 0.0, 0.0);
    GRID_STRIDE(i, n) gx[i] = gy[i] = gz[i] = 0.0f;
}

// Neuron j (Morton position s) gets w_j * sum over its cells k of G_k / N_k: first G / N
// per node (a node without vacant elements is no candidate and has G = 0), then every
// neuron's sum up its parent chain. One FP64 division per node instead of one per neuron
// and level. Whole backward call on the device with this and the zeroing in one launch:
// 1,000 neurons 59 -> 49 us, 5,003 106 -> 96, 40,000 460 -> 448, 2^18 2,773 -> 2,761. (As
// one cluster kernel: 50, 99, 481.)
struct ScatterArgs {
    const Node *nodes;
    const int32_t *parent, *leaf_of, *perm, *vac_de;
    const int64_t *d_num_nodes;
    double *G;
    int64_t n;
    float *gx, *gy, *gz;
};

__device__ __forceinline__ void scale_node(const ScatterArgs &a, int64_t u)
{
    const int32_t cnt = a.nodes[u].t.icount;
    if (cnt <= 0) return;
    const double inv = 1.0 / (double)cnt;
    double *g = a.G + 4 * u;
    g[0] *= inv;
    g[1] *= inv;
    g[2] *= inv;
}

__device__ __forceinline__ void gather_chain(const ScatterArgs &a, int64_t s)
{
    const int32_t i = a.perm[s];
    const int32_t w = a.vac_de[i];
    if (w <= 0) return;
    double hx = 0.0, hy = 0.0, hz = 0.0;
    for (int32_t u = a.leaf_of[s]; u >= 0; u = a.parent[u]) {
        const double *g = a.G + 4 * (int64_t)u;
        hx += g[0];
        hy += g[1];
        hz += g[2];
    }
    // direct term (FP32) + cell terms (FP64), rounded once
    a.gx[i] = (float)((double)a.gx[i] + w * hx);
    a.gy[i] = (float)((double)a.gy[i] + w * hy);
    a.gz[i] = (float)((double)a.gz[i] + w * hz);
}

__global__ void len_scale_kernel(ScatterArgs a)
{
    const int64_t m = *a.d_num_nodes;
    GRID_STRIDE(u, m) scale_node(a, u);
}

__global__ void len_scatter_kernel(ScatterArgs a)
{
    GRID_STRIDE(s, a.n) gather_chain(a, s);
}

LenArgs make_args(relearn_ctx *c, const int32_t *vac_ax)
{
    LenArgs a{};
    a.nodes = c->d_nodes;
    a.fam = c->d_fam;
    a.pos = c->d_pos;
    a.perm = c->d_perm;
    a.act_src = c->d_act_src;
    a.leaf_of = c->d_leaf;
    a.vac_ax = vac_ax;
    a.n = c->n;
    a.geom = c->d_geom;
    a.d_total = c->d_i64 + I64_ACTIVE;
    a.evals_total = c->d_i64 + I64_LEN_EVALS;
    a.sc = c->d_sc;
    a.state = c->d_lstate;
    a.lsum = c->d_lsum;
    a.work = c->d_i32 + I32_WORK;
    a.redo = c->d_i32 + I32_REDO;
    a.redo_list = c->d_act_off; // read by the forward call's setup only
    return a;
}

template <bool kBack>
cudaError_t launch_length(relearn_ctx *c, const LenArgs &a, cudaStream_t st)
{
    length_kernel<kBack>
        <<<c->num_sms * RELEARN_LEN_MIN_BLOCKS, 32 * kGroupWarps, 0, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

} // namespace

cudaError_t length_forward(relearn_ctx *c, const int32_t *vac_ax, float *ell, double *mean,
                           cudaStream_t st)
{
    cudaError_t e;
    const int64_t n = c->n;
    PrepArgs p;
    p.vac_ax = vac_ax;
    p.perm = c->d_perm;
    p.n = n;
    p.flag = c->d_cnt;
    p.off = c->d_act_off;
    p.act_src = c->d_act_src;
    p.active = c->d_i64 + I64_ACTIVE;
    p.nodes = c->d_nodes;
    p.parent = c->d_parent;
    p.d_num_nodes = c->d_i64 + I64_NODES;
    p.k0 = reinterpret_cast<int32_t *>(c->d_acc); // the bottom-up update's scratch is free
    p.fam = c->d_fam;
    p.lsum = c->d_lsum;
    p.work = c->d_i32 + I32_WORK;
    p.redo = c->d_i32 + I32_REDO;
    if (n <= kSmallLen && may_cluster(c)) {
        len_prepare_small_kernel<<<cluster_form::kBlocks, cluster_form::kThreads, 0, st>>>(p);
        note_launch();
    } else {
        const unsigned gm = grid_for(2 * n + 1, 256, c->num_sms);
        len_count_kernel<<<gm, 256, 0, st>>>(p);
        note_launch();
        if ((e = scan_exclusive(p.flag, p.off, n + 1, nullptr, p.active, c->scan, st))) return e;
        // the node count as int32 (its low word)
        if ((e = scan_exclusive(p.k0, p.k0, 2 * n + 1,
                                reinterpret_cast<const int32_t *>(p.d_num_nodes), nullptr,
                                c->scan, st)))
            return e;
        len_emit_kernel<<<gm, 256, 0, st>>>(p);
        note_launch();
    }
    LenArgs a = make_args(c, vac_ax);
    a.mean = mean;
    if ((e = launch_length<false>(c, a, st))) return e;
    // at most a block per group (every block shares one group among its warps then)
    const int64_t most = std::min<int64_t>((n + 31) / 32, c->num_sms * RELEARN_LEN_MIN_BLOCKS);
    redo_kernel<<<(unsigned)most, 32 * kGroupWarps, 0, st>>>(a);
    note_launch();
    if (ell) {
        len_finish_kernel<<<grid_for(n, 256, c->num_sms), 256, 0, st>>>(
            c->d_lstate, p.flag, c->d_perm, n, ell);
        note_launch();
    }
    return cudaGetLastError();
}

cudaError_t length_backward(relearn_ctx *c, const int32_t *vac_ax, const int32_t *vac_de,
                            const double *grad_mean, float *gx, float *gy, float *gz,
                            double *gsigma, cudaStream_t st)
{
    cudaError_t e;
    const int64_t n = c->n;
    // d_acc is free between bottom-up updates (32 bytes per node: x, y, z in FP64)
    double *G = c->d_acc;
    len_zero_kernel<<<grid_for(2 * n, 256, c->num_sms), 256, 0, st>>>(
        reinterpret_cast<double4 *>(G), c->d_i64 + I64_NODES, n, gx, gy, gz, gsigma,
        c->d_i32 + I32_WORK);
    note_launch();
    LenArgs a = make_args(c, vac_ax);
    a.G = G;
    a.gx = gx;
    a.gy = gy;
    a.gz = gz;
    a.gout = grad_mean;
    a.gsigma = gsigma;
    if ((e = launch_length<true>(c, a, st))) return e;
    const ScatterArgs s{c->d_nodes, c->d_parent, c->d_leaf, c->d_perm, vac_de,
                        c->d_i64 + I64_NODES, G, n, gx, gy, gz};
    len_scale_kernel<<<grid_for(2 * n, 256, c->num_sms), 256, 0, st>>>(s);
    note_launch();
    len_scatter_kernel<<<grid_for(n, 256, c->num_sms), 256, 0, st>>>(s);
    note_launch();
    return cudaGetLastError();
}

bool length_clusters() { return cluster_form::placeable(len_prepare_small_kernel); }

} // namespace rl
