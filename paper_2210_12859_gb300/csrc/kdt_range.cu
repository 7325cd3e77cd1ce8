// Range queries and payload reductions.
//
// Ball: every point within a fixed radius of a query point; box: every point
// inside an axis-aligned box.  Sec. 3 notes that other query primitives only
// change the in-range test and what processNode does, and that a non-ordered
// traversal is a simplification of the ordered one; both queries use the
// unordered machine's order (a node, its left subtree, its right subtree) with a
// fixed range instead of a shrinking one.  Two kernels:
//   box_range_kernel   walks the box tree (kdt_box.cuh) and finds the same hits
//                      in the same order as the machine; templated over the
//                      processNode action:
//     ACT_COUNT   count the hits;
//     ACT_FILL    write the hits to the query's slice [offsets[q], offsets[q+1])
//                 in traversal order (count and fill walk the same nodes in
//                 the same order, so no atomics are needed); hits wait in a
//                 ring in shared memory, and from the slice's first 16-byte
//                 boundary on are written four at a time as 16-byte stores, the
//                 slice's unaligned head and its last partial group one word
//                 at a time;
//     ACT_REDUCE  sum a per-point payload over the hits in traversal order
//                 (the point types with payload, e.g. photon power, that Sec. 3
//                 names; the fixed-radius photon-map density estimate on top);
//   range_visits_kernel  the machine itself, for the count of the nodes that it
//                 processes (KDT_RANGE_VISITS).
// A payload is attached to the tree in node order; kNN reductions gather it
// through the inverse permutation after an ordinary kNN query.
#include <string.h>

#include "kdt_box.cuh"
#include "kdt_learned.cuh"
#include "kdt_query.cuh"

namespace kdt {
namespace {

constexpr int RANGE_THREADS = 128;
// traversal steps between two claim rounds of a warp (as for kNN, 64 beats 16)
constexpr int RANGE_CLAIM_STEPS = 64;
enum : int { ACT_COUNT = 0, ACT_FILL = 1, ACT_REDUCE = 2 };
// binary32 rounding of pi
constexpr float PI_F = 3.14159265358979323846f;

struct RangeArgs {
    const float4 *nodes;
    const int32_t *ids;
    int N, D;
    const float *a;  // ball: centres; box: lower corners   [Q][D]
    const float *b;  // box: upper corners                  [Q][D]
    int64_t Q;
    const uint32_t *perm;  // traversal order -> query index, or NULL
    float r2;
    int32_t *counts;
    const int64_t *offsets;
    int32_t *out_ids;
    float *out_d2;
    const float *payload;  // [N][C] in node order (ACT_REDUCE)
    int C;
    int mode;              // KDT_REDUCE_*
    float *out;            // [Q][C] (ACT_REDUCE)
    bool vec_fill;         // ACT_FILL: outputs 16-byte aligned, groups of four hits stored at once
    int *err;
    unsigned long long *counter;
};

template <int LAYOUT>
__device__ __forceinline__ uint32_t node_id(const NodeVal<LAYOUT> &nd, const int32_t *__restrict__ ids, int n)
{
    if constexpr (LAYOUT == 0)
        return nd.id;
    else if constexpr (LAYOUT == 3)
        return nd.id & NODE_ID_MASK;
    else
        return (uint32_t)__ldg(ids + n);
}

// Final value of a reduction: no hit -> 0; mean: / count; density: / fl(pi * R2).
__device__ __forceinline__ float finish_reduce(float s, int64_t n, int mode, float R2)
{
    if (n == 0)
        return 0.f;
    if (mode == KDT_REDUCE_MEAN)
        return __fdiv_rn(s, (float)n);
    if (mode == KDT_REDUCE_DENSITY)
        return __fdiv_rn(s, __fmul_rn(PI_F, R2));
    return s;
}

// One lane's range query: the query box / ball and the processNode action's
// state.
// The fill's hits wait in a ring of FILL_RING entries a thread in shared
// memory (entry: the hit's place in the output, modulo the ring; a column a
// thread, so that any mix of entries is free of bank conflicts) until a group
// of four on a 16-byte boundary is complete.  Staging a hit is two predicated
// stores, against a branch, a shift of eight registers and selects in a loop
// over the hits of the warp's busiest lane: the search of 10^6 balls, r = 0.002,
// takes 2.63 ms instead of 2.82.
constexpr int FILL_RING = 16;
template <bool FILL>
struct FillStage {
};
template <>
struct FillStage<true> {
    int64_t base;
    int32_t limit;
    int32_t done;   // hits written
    int32_t *s_id;  // this thread's column of the rings
    float *s_d2;
    int stride;
};

template <int LAYOUT, int KIND, int ACT>
struct RangeLane : FillStage<ACT == ACT_FILL> {
    static constexpr int NC = LayoutTraits<LAYOUT>::NC;
    float lo[NC], hi[KIND == 1 ? NC : 1];
    float acc[ACT == ACT_REDUCE ? KDT_PAYLOAD_MAX_C : 1];
    int32_t count;  // hits of one query are below N < 2^30

    // false: no point is in range of a query that is not a number
    __device__ __forceinline__ bool start(const RangeArgs &a, int64_t qi)
    {
        load_query<LAYOUT>(a.a, qi, a.D, lo);
        bool nan = false;
#pragma unroll
        for (int j = 0; j < NC; ++j)
            nan = nan || lo[j] != lo[j];
        if constexpr (KIND == 1) {
            load_query<LAYOUT>(a.b, qi, a.D, hi);
#pragma unroll
            for (int j = 0; j < NC; ++j)
                nan = nan || hi[j] != hi[j];
        }
        count = 0;
        if constexpr (ACT == ACT_FILL) {
            this->base = a.offsets[qi];
            // saturated: a slice longer than any hit count, or negative, still
            // ends with count != limit and the range error
            const int64_t len = a.offsets[qi + 1] - this->base;
            this->limit = (int32_t)(len < 0 ? -1 : (len > INT32_MAX ? INT32_MAX : len));
            this->done = 0;
        }
        if constexpr (ACT == ACT_REDUCE) {
#pragma unroll
            for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
                acc[c] = 0.f;
        }
        return !nan;
    }

    __device__ __forceinline__ bool test(const RangeArgs &a, const NodeVal<LAYOUT> &nd, float &d2) const
    {
        if constexpr (KIND == 0) {
            d2 = dist2<NC>(nd.c, lo);
            return d2 <= a.r2;
        } else {
            bool hit = true;
#pragma unroll
            for (int j = 0; j < NC; ++j)
                hit = hit && lo[j] <= nd.c[j] && nd.c[j] <= hi[j];
            return hit;
        }
    }

    // fill: a hit into the ring
    __device__ __forceinline__ void stage(uint32_t id, float d2)
    {
        const int e = (int)(((uint32_t)this->base + (uint32_t)count) & (FILL_RING - 1)) * this->stride;
        this->s_id[e] = (int32_t)id;
        if (KIND == 0)
            this->s_d2[e] = d2;
        ++count;
    }
    __device__ __forceinline__ void write_one(const RangeArgs &a)
    {
        const int64_t pos = this->base + this->done;
        const int e = (int)((uint32_t)pos & (FILL_RING - 1)) * this->stride;
        if (this->done < this->limit) {
            a.out_ids[pos] = this->s_id[e];
            if (KIND == 0 && a.out_d2)
                a.out_d2[pos] = this->s_d2[e];
        }
        ++this->done;
    }
    // fill: the ring's complete groups of four to the output, single words up
    // to the slice's first 16-byte boundary (or throughout, for unaligned
    // outputs) and past a limit that the count does not keep
    __device__ __forceinline__ void flush(const RangeArgs &a)
    {
        while (count > this->done) {
            const int64_t pos = this->base + this->done;
            if (!a.vec_fill || (pos & 3) != 0 || this->done + 4 > this->limit) {
                if (a.vec_fill && (pos & 3) == 0 && count - this->done < 4)
                    break;
                write_one(a);
                continue;
            }
            if (count - this->done < 4)
                break;
            const int e = (int)((uint32_t)pos & (FILL_RING - 1)) * this->stride, st = this->stride;  // a group does not wrap
            *reinterpret_cast<int4 *>(a.out_ids + pos) =
                make_int4(this->s_id[e], this->s_id[e + st], this->s_id[e + 2 * st], this->s_id[e + 3 * st]);
            if (KIND == 0 && a.out_d2)
                *reinterpret_cast<float4 *>(a.out_d2 + pos) =
                    make_float4(this->s_d2[e], this->s_d2[e + st], this->s_d2[e + 2 * st], this->s_d2[e + 3 * st]);
            this->done += 4;
        }
    }

    // processNode of a hit: node n, the point id
    __device__ __forceinline__ void hit(const RangeArgs &a, int n, uint32_t id, float d2)
    {
        if constexpr (ACT == ACT_FILL) {
            stage(id, d2);
            if (count - this->done > FILL_RING - 9)
                flush(a);
        } else {
            if constexpr (ACT == ACT_REDUCE) {
                const float *p = a.payload + (int64_t)n * a.C;
#pragma unroll
                for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
                    if (c < a.C)
                        acc[c] = __fadd_rn(acc[c], __ldg(p + c));
            }
            ++count;
        }
    }

    // boxes of a record that can hold a point in range, a bit each
    __device__ __forceinline__ uint32_t boxes(const RangeArgs &a, const float4 *__restrict__ rec, f32x2 one) const
    {
        uint32_t in = 0;
        if constexpr (KIND == 0) {
            float d[4];
            box_dist4<NC>(rec, lo, one, d);
#pragma unroll
            for (int c = 0; c < 4; ++c)
                in |= d[c] <= a.r2 ? 1u << c : 0u;
        } else {
            in = 15u;
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const Float8 b = load8(rec + 2 * j);  // lo[4], hi[4]
                uint32_t m = 0;
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    m |= b.v[c] <= hi[j] && lo[j] <= b.v[4 + c] ? 1u << c : 0u;
                in &= m;
            }
        }
        return in;
    }

    // points of a group in range, a bit each
    __device__ __forceinline__ uint32_t points(const RangeArgs &a, const float4 *__restrict__ g, f32x2 one,
                                               float (&d)[8]) const
    {
        uint32_t in = 0;
        if constexpr (KIND == 0) {
            group_dist8<NC>(g, lo, one, d);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                in |= d[c] <= a.r2 ? 1u << c : 0u;
        } else {
            in = 255u;
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const Float8 x = load8(g + 2 * j);
                uint32_t m = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    m |= lo[j] <= x.v[c] && x.v[c] <= hi[j] ? 1u << c : 0u;
                in &= m;
            }
        }
        return in;
    }

    // the query's end: the last partial group of the fill, the count or the
    // reduction written out
    __device__ __forceinline__ void finish(const RangeArgs &a, int64_t qi)
    {
        if constexpr (ACT == ACT_FILL) {
            while (this->done < count)
                write_one(a);
            if (count != this->limit)
                atomicOr(a.err, ERR_RANGE);
        } else {
            if (a.counts)
                a.counts[qi] = count;
            if constexpr (ACT == ACT_REDUCE) {
#pragma unroll
                for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
                    if (c < a.C)
                        a.out[qi * a.C + c] = finish_reduce(acc[c], count, a.mode, a.r2);
            }
        }
    }
};

// One lane's place in the box tree for a fixed range, in the machine's order:
// node, left subtree, right subtree.  A record's node is binary node v, its
// boxes are v's grandchildren, and v's point and its children's points come
// from the level-order nodes.  What is left to do below v are five bits in
// order: the left child's two subtrees, the right child's point, its two
// subtrees (v's and the left child's points are dealt with on entry).  The
// range is fixed, so the bits set on entry stay true and no record is read
// twice.  The records above keep theirs in `trail`, five bits each, the root's
// in root_bits: 12 records below the root for N < 2^30.
struct RangeWalk {
    uint32_t v, bits, root_bits;
    unsigned long long trail;
    __device__ __forceinline__ void start(uint32_t root)
    {
        v = root;
        bits = 0;
        root_bits = 0;
        trail = 0;
    }
    __device__ __forceinline__ void descend(uint32_t root, uint32_t c)
    {
        if (v == root)
            root_bits = bits;
        else
            trail = trail << 5 | bits;
        v = 4 * v + c;
        bits = 0;
    }
    // to the nearest record with something left; false: none
    __device__ __forceinline__ bool pop(uint32_t root)
    {
        if (trail) {
            const int up = (__ffsll((long long)trail) - 1) / 5;
            v >>= 2 * (up + 1);
            trail >>= 5 * up;
            bits = (uint32_t)trail & 31u;
            trail >>= 5;
            return true;
        }
        v = root;
        bits = root_bits;
        root_bits = 0;
        return bits != 0;
    }
};

// KIND 0: ball of squared radius r2 around a[q]; KIND 1: box [a[q], b[q]].
// Persistent lanes, and the warp's turns between records and buckets, as in
// box_knn_kernel.  The bucket's point from above is some other node's: it is
// met there.
//
// Bound: L1 wavefronts of the records that incoherent lanes read (count, 88 %),
// issue slots of the hits' staging (fill, 74 %).  Against the state machine's
// kernels (one plane a test; its bottom nodes walked with their leaves): 10^6
// balls of 35 hits count 1.43 -> 0.92 ms, fill 1.90 -> 1.35; photon density of
// 2^18 93 -> 62 us.  Lanes on records 0 / 2 / 4 / 8 / 16 and free 8 / 16 / 24 before
// the warp turns: 4 and 16 are best, the others up to 16 % slower.
constexpr int RANGE_RECORD_LANES = 4, RANGE_FREE_LANES = 16;

template <int LAYOUT, int KIND, int ACT>
__global__ void __launch_bounds__(RANGE_THREADS) box_range_kernel(const RangeArgs a, const BoxArgs b)
{
    constexpr int NC = LayoutTraits<LAYOUT>::NC;
    const BoxRef tree = b.tree;
    const f32x2 one = pair(b.one, b.one);
    const bool odd = (tree.leaf & 0xaaaaaaaau) != 0;
    const uint32_t root = odd ? 0u : 1u;
    RangeLane<LAYOUT, KIND, ACT> L;
    if constexpr (ACT == ACT_FILL) {
        extern __shared__ int32_t s_ring[];
        L.stride = blockDim.x;
        L.s_id = s_ring + threadIdx.x;
        L.s_d2 = reinterpret_cast<float *>(s_ring + FILL_RING * blockDim.x) + threadIdx.x;
    }
    RangeWalk w;
    w.start(root);
    int64_t qi = -1;
    bool busy = false, first = true, exhausted = false;
    const int64_t lanes = (int64_t)gridDim.x * blockDim.x;
    // a node's point: hit or not
    auto at_node = [&](uint32_t u) {
        const NodeVal<LAYOUT> nd = fetch<LAYOUT, false>(a.nodes, nullptr, 0, (int)u - 1);
        float d2 = 0.f;
        if (L.test(a, nd, d2))
            L.hit(a, (int)u - 1, node_id<LAYOUT>(nd, a.ids, (int)u - 1), d2);
    };
    // the next thing to do at v or above: leaves v at a node to enter
    auto advance = [&]() {
        for (;;) {
            if (w.bits == 0 && !w.pop(root))
                return false;
            const uint32_t c = __ffs(w.bits) - 1;
            w.bits &= w.bits - 1;
            if (c == 2) {
                at_node(2 * w.v + 1);
            } else {
                w.descend(root, c < 2 ? c : c - 1);
                return true;
            }
        }
    };
    for (;;) {
        const unsigned free_lanes = __ballot_sync(0xffffffffu, !busy && !exhausted);
        const unsigned busy_lanes = __ballot_sync(0xffffffffu, busy);
        if (!busy_lanes || __popc(free_lanes) >= RANGE_FREE_LANES) {
            if (!busy && qi >= 0) {
                L.finish(a, qi);
                qi = -1;
            }
            const bool need = !busy && !exhausted;
            int64_t slot;
            if (first)
                slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
            else if (lanes >= a.Q)
                slot = a.Q;
            else
                slot = claim_slot(need, a.counter);
            if (need) {
                if (!first && slot < a.Q)
                    slot += lanes;
                if (slot < a.Q) {
                    qi = a.perm ? (int64_t)a.perm[slot] : slot;
                    busy = L.start(a, qi);
                    w.start(root);
                    // with an odd LB the root's point is no record's node
                    if (busy && odd)
                        at_node(1);
                } else {
                    exhausted = true;
                }
            }
            first = false;
            if (__all_sync(0xffffffffu, !busy && exhausted && qi < 0))
                break;
        }
        for (;;) {
            if (busy && w.v < tree.leaf) {
                uint32_t in = L.boxes(a, tree.rec + (size_t)w.v * BoxFormat<NC>::REC, one);
                uint32_t right = 0;
                if (w.v == 0) {
                    in &= 12u;
                } else {
                    at_node(w.v);
                    const NodeVal<LAYOUT> l = fetch<LAYOUT, false>(a.nodes, nullptr, 0, 2 * (int)w.v - 1);
                    const NodeVal<LAYOUT> r = fetch<LAYOUT, false>(a.nodes, nullptr, 0, 2 * (int)w.v);
                    float d2 = 0.f, dr = 0.f;
                    if (L.test(a, l, d2))
                        L.hit(a, 2 * (int)w.v - 1, node_id<LAYOUT>(l, a.ids, 2 * (int)w.v - 1), d2);
                    right = L.test(a, r, dr);
                }
                w.bits = (in & 3u) | right << 2 | (in & 12u) << 1;
                busy = advance();
            }
            if (__popc(__ballot_sync(0xffffffffu, busy && w.v < tree.leaf)) <= RANGE_RECORD_LANES)
                break;
        }
        if (busy && w.v >= tree.leaf) {
            const uint32_t i = w.v - tree.leaf;
            const float4 *g = tree.grp + (size_t)(i + min(i, tree.big)) * BoxFormat<NC>::GRP;
            const bool two = i < tree.big;
            float d[2][8];
            uint32_t in0 = L.points(a, g, one, d[0]) & 127u, in1 = 0;
            if (two)
                in1 = L.points(a, g + BoxFormat<NC>::GRP, one, d[1]);
            // place p of the two groups is the bucket's node h = p + 1 (first
            // group) or p, counted from its root 1; the order of hits is node,
            // left subtree, right subtree: rank of h = 1 .. 15 there, and back
            constexpr int RANK[16] = {0, 0, 1, 8, 2, 5, 9, 12, 3, 4, 6, 7, 10, 11, 13, 14};
            constexpr unsigned long long NODE_AT = 0xFE7DC63BA598421ull;  // h of rank 0, 1, ... from the low nibble
            if constexpr (ACT == ACT_COUNT) {
                L.count += __popc(in0) + __popc(in1);
            } else if constexpr (ACT == ACT_FILL) {
                // the ring holds at most FILL_RING - 9 hits here: room for eight more
                const Float8 id0 = load8(g + 2 * NC);
                Float8 id1 = id0;
                if (two)
                    id1 = load8(g + BoxFormat<NC>::GRP + 2 * NC);
#pragma unroll
                for (int rank = 0; rank < 15; ++rank) {
                    const int h = (int)(NODE_AT >> (4 * rank)) & 15;
                    if (h < 8 ? in0 >> (h - 1) & 1u : in1 >> (h - 8) & 1u)
                        L.stage(__float_as_uint(h < 8 ? id0.v[(h - 1) & 7] : id1.v[h & 7]),
                                h < 8 ? d[0][(h - 1) & 7] : d[1][h & 7]);
                    if (rank == 7)
                        L.flush(a);
                }
                L.flush(a);
            } else {
                uint32_t order = 0;
#pragma unroll
                for (int h = 1; h < 16; ++h)
                    order |= (h < 8 ? in0 >> (h - 1) & 1u : in1 >> (h - 8) & 1u) << RANK[h];
                while (order) {
                    const int rank = __ffs(order) - 1;
                    order &= order - 1;
                    const int h = (int)(NODE_AT >> (4 * rank)) & 15;
                    const int up = 31 - __clz(h);
                    L.hit(a, (int)((w.v << up) + (uint32_t)(h - (1 << up))) - 1, 0u, 0.f);
                }
            }
            busy = advance();
        }
    }
}

// The unordered machine of Sec. 3.2 with a fixed range: processed nodes of
// every query.  The step bound 3N + 3 is checked once a round.
template <int LAYOUT, int KIND>
__global__ void __launch_bounds__(RANGE_THREADS) range_visits_kernel(const RangeArgs a)
{
    constexpr int NC = LayoutTraits<LAYOUT>::NC;
    float lo[NC], hi[NC];
    int64_t qi = -1;
    bool exhausted = false;
    int curr = 0, prev = -1, dim = 0, visits = 0;
    uint32_t steps = 0;
    const uint32_t cap = 3u * (uint32_t)a.N + 3u;
    const int bottom = a.N >> 2;  // from here on a node's children have no children
    for (;;) {
        const bool need = qi < 0 && !exhausted;
        const int64_t slot = claim_slot(need, a.counter);
        if (need) {
            if (slot < a.Q) {
                qi = a.perm ? (int64_t)a.perm[slot] : slot;
                load_query<LAYOUT>(a.a, qi, a.D, lo);
                if (KIND == 1)
                    load_query<LAYOUT>(a.b, qi, a.D, hi);
                curr = 0;
                prev = -1;
                dim = 0;
                visits = 0;
                steps = 0;
            } else {
                exhausted = true;
            }
        }
        if (__all_sync(0xffffffffu, qi < 0))
            break;
        if (qi < 0)
            continue;
        bool done = false;
        if (steps > cap) {
            atomicOr(a.err, ERR_TRAVERSAL);
            done = true;
        }
        for (int s = 0; s < RANGE_CLAIM_STEPS && !done; ++s) {
            ++steps;
            const NodeVal<LAYOUT> nd = fetch<LAYOUT, false>(a.nodes, nullptr, 0, curr);
            const bool from_parent = prev < curr;
            const int lc = 2 * curr + 1, rc = lc + 1;
            const int parent = (curr - 1) >> 1;
            visits += from_parent;
            const int sdim = split_dim_of<LAYOUT>(nd, dim);
            const float split_at = select_dim<NC>(nd.c, sdim);
            bool left_ok, right_ok;
            if constexpr (KIND == 0) {
                const float sd = __fsub_rn(select_dim<NC>(lo, sdim), split_at);
                const float sd2 = __fmul_rn(sd, sd);
                left_ok = sd <= 0.f || sd2 <= a.r2;
                right_ok = sd > 0.f || sd2 <= a.r2;
            } else {
                // left subtree coordinates are <= split, right ones >= split
                left_ok = select_dim<NC>(lo, sdim) <= split_at;
                right_ok = select_dim<NC>(hi, sdim) >= split_at;
            }
            left_ok = left_ok && lc < a.N;
            right_ok = right_ok && rc < a.N;
            int next;
            if (from_parent && curr >= bottom) {
                // the children are leaves: entered and left again
                visits += left_ok + right_ok;
                next = parent;
            } else if (from_parent)
                next = left_ok ? lc : (right_ok ? rc : parent);
            else if (prev == lc)
                next = right_ok ? rc : parent;
            else
                next = parent;
            if (next < 0) {
                done = true;
                break;
            }
            if (next == parent)
                dim = dim == 0 ? a.D - 1 : dim - 1;
            else
                dim = dim + 1 == a.D ? 0 : dim + 1;
            prev = curr;
            curr = next;
        }
        if (!done)
            continue;
        a.counts[qi] = visits;
        qi = -1;
    }
}

template <int LAYOUT, int KIND, int ACT>
int launch_one(const RangeArgs &a, const BoxArgs &b, cudaStream_t s)
{
    const void *fn = (const void *)box_range_kernel<LAYOUT, KIND, ACT>;
    // few queries: small blocks, so that they spread over the SMs
    int threads = RANGE_THREADS;
    while (threads > 32 && a.Q < (int64_t)num_sms() * threads)
        threads >>= 1;
    const size_t smem = ACT == ACT_FILL ? (size_t)threads * FILL_RING * 4 * (KIND == 0 ? 2 : 1) : 0;
    const int64_t grid = std::min<int64_t>(grid_for_kernel(fn, threads, smem), (a.Q + threads - 1) / threads);
    if (grid * threads < a.Q)
        KDT_CUDA(cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s));
    KDT_LAUNCH box_range_kernel<LAYOUT, KIND, ACT><<<(unsigned)grid, threads, smem, s>>>(a, b);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

template <int LAYOUT, int KIND>
int launch_visits(const RangeArgs &a, cudaStream_t s)
{
    KDT_CUDA(cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s));
    const int grid = grid_for_kernel((const void *)range_visits_kernel<LAYOUT, KIND>, RANGE_THREADS, 0);
    KDT_LAUNCH range_visits_kernel<LAYOUT, KIND><<<grid, RANGE_THREADS, 0, s>>>(a);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

template <int LAYOUT>
int launch_range_layout(int kind, int act, bool visits, const RangeArgs &a, const BoxArgs &b, cudaStream_t s)
{
    if (visits)
        return kind == 0 ? launch_visits<LAYOUT, 0>(a, s) : launch_visits<LAYOUT, 1>(a, s);
    if (kind == 0) {
        if (act == ACT_COUNT)
            return launch_one<LAYOUT, 0, ACT_COUNT>(a, b, s);
        if (act == ACT_FILL)
            return launch_one<LAYOUT, 0, ACT_FILL>(a, b, s);
        return launch_one<LAYOUT, 0, ACT_REDUCE>(a, b, s);
    }
    if (act == ACT_COUNT)
        return launch_one<LAYOUT, 1, ACT_COUNT>(a, b, s);
    return launch_one<LAYOUT, 1, ACT_FILL>(a, b, s);
}

int run_range(const kdt_tree *t, int kind, int act, int flags, RangeArgs a, cudaStream_t s)
{
    pool_setup_once();
    const bool morton = flags & KDT_MORTON;
    Scratch sc(s);
    KDT_TRY(sc.alloc(carve_size({64}) + (morton ? morton_scratch_bytes(a.Q) : 0)));
    Carve c{(char *)sc.p};
    a.counter = c.take<unsigned long long>(8);
    a.nodes = t->nodes;
    a.ids = t->ids;
    a.N = (int)t->N;
    a.D = t->D;
    a.err = t->err;
    a.perm = nullptr;
    if (morton)
        KDT_TRY(query_order(t, a.a, a.Q, false, c.base + c.off, const_cast<uint32_t **>(&a.perm), s));
    BoxArgs b;
    b.tree = box_ref(t->N, t->box_rec, t->box_grp);
    const bool visits = flags & KDT_RANGE_VISITS;
    switch (t->layout) {
    case 0: return launch_range_layout<0>(kind, act, visits, a, b, s);
    case 1: return launch_range_layout<1>(kind, act, visits, a, b, s);
    case 3: return launch_range_layout<3>(kind, act, visits, a, b, s);
    default: return launch_range_layout<2>(kind, act, visits, a, b, s);
    }
}

__global__ void counts_to_u64_kernel(const int32_t *__restrict__ counts, int64_t Q, unsigned long long *__restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= Q; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = i < Q ? (unsigned long long)(counts[i] > 0 ? counts[i] : 0) : 0ull;
}

// payload[id][C] (input order) -> node order; node_of[id] = node
template <int LAYOUT>
__global__ void payload_permute_kernel(const float4 *__restrict__ nodes, const int32_t *__restrict__ ids, int64_t N,
                                       const float *__restrict__ in, int C, float *__restrict__ out,
                                       int32_t *__restrict__ node_of)
{
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
        const NodeVal<LAYOUT> nd = fetch<LAYOUT, false>(nodes, nullptr, 0, (int)n);
        const int64_t id = node_id<LAYOUT>(nd, ids, (int)n);
        for (int c = 0; c < C; ++c)
            out[n * C + c] = in[id * C + c];
        node_of[id] = (int32_t)n;
    }
}

// Sum of the payload over each query's kNN list in list order (ascending
// (d2, id)); density radius R2 = the farthest found neighbour's d2.
__global__ void knn_reduce_kernel(const int32_t *__restrict__ ids, const float *__restrict__ d2, int64_t Q, int k,
                                  const int32_t *__restrict__ node_of, const float *__restrict__ payload, int C,
                                  int mode, float *__restrict__ out)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q; q += (int64_t)gridDim.x * blockDim.x) {
        const int32_t *row = ids + q * k;
        int n = 0;
        while (n < k && row[n] >= 0)
            ++n;
        const float R2 = n ? d2[q * k + n - 1] : 0.f;
        float acc[KDT_PAYLOAD_MAX_C];
#pragma unroll
        for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
            acc[c] = 0.f;
        for (int i = 0; i < n; ++i) {
            const float *p = payload + (int64_t)node_of[row[i]] * C;
#pragma unroll
            for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
                if (c < C)
                    acc[c] = __fadd_rn(acc[c], __ldg(p + c));
        }
#pragma unroll
        for (int c = 0; c < KDT_PAYLOAD_MAX_C; ++c)
            if (c < C)
                out[q * C + c] = finish_reduce(acc[c], n, mode, R2);
    }
}

unsigned grid_for(int64_t n)
{
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 16));
}

int check_range(const kdt_tree *t, int64_t Q, const void *a, const void *b, bool need_b, int flags)
{
    if (!t)
        return set_error(KDT_EINVAL, "tree is NULL");
    if (Q < 0 || Q >= ((int64_t)1 << 32))
        return set_error(KDT_EINVAL, "Q must be in [0, 2^32)");
    if (Q > 0 && (!a || (need_b && !b)))
        return set_error(KDT_EINVAL, "NULL query pointer");
    if (flags & ~(KDT_MORTON | KDT_RANGE_VISITS))
        return set_error(KDT_EINVAL, "range queries take no flag but KDT_MORTON and KDT_RANGE_VISITS (got %#x)",
                         flags);
    return KDT_OK;
}

int check_radius(float radius)
{
    if (!(radius >= 0.f))
        return set_error(KDT_EINVAL, "radius must be >= 0 (got %g)", (double)radius);
    return KDT_OK;
}

RangeArgs blank_args()
{
    RangeArgs a;
    memset(&a, 0, sizeof(a));
    return a;
}

// 16-byte stores of the fill pass only into 16-byte aligned outputs
bool fill_vectorizable(const int32_t *ids, const float *d2)
{
    return ((uintptr_t)ids & 15u) == 0 && ((uintptr_t)d2 & 15u) == 0;
}

}  // namespace
}  // namespace kdt

using namespace kdt;

extern "C" {

int kdt_radius_count(const kdt_tree *t, const float *d_q, int64_t Q, float radius, int flags, int32_t *d_counts,
                     void *stream)
{
    KDT_TRY(check_range(t, Q, d_q, nullptr, false, flags));
    KDT_TRY(check_radius(radius));
    if (Q > 0 && !d_counts)
        return set_error(KDT_EINVAL, "NULL counts");
    if (Q == 0)
        return KDT_OK;
    RangeArgs a = blank_args();
    a.a = d_q;
    a.Q = Q;
    a.r2 = radius * radius;
    a.counts = d_counts;
    return run_range(t, 0, ACT_COUNT, flags, a, (cudaStream_t)stream);
}

int kdt_radius_fill(const kdt_tree *t, const float *d_q, int64_t Q, float radius, int flags, const int64_t *d_offsets,
                    int32_t *d_ids, float *d_d2, void *stream)
{
    KDT_TRY(check_range(t, Q, d_q, nullptr, false, flags));
    if (flags & KDT_RANGE_VISITS)
        return set_error(KDT_EINVAL, "KDT_RANGE_VISITS applies to the count calls only");
    KDT_TRY(check_radius(radius));
    if (Q > 0 && (!d_offsets || !d_ids))
        return set_error(KDT_EINVAL, "NULL offsets / ids");
    if (Q == 0)
        return KDT_OK;
    RangeArgs a = blank_args();
    a.a = d_q;
    a.Q = Q;
    a.r2 = radius * radius;
    a.offsets = d_offsets;
    a.out_ids = d_ids;
    a.out_d2 = d_d2;
    a.vec_fill = fill_vectorizable(d_ids, d_d2);
    return run_range(t, 0, ACT_FILL, flags, a, (cudaStream_t)stream);
}

int kdt_box_count(const kdt_tree *t, const float *d_lo, const float *d_hi, int64_t Q, int flags, int32_t *d_counts,
                  void *stream)
{
    KDT_TRY(check_range(t, Q, d_lo, d_hi, true, flags));
    if (Q > 0 && !d_counts)
        return set_error(KDT_EINVAL, "NULL counts");
    if (Q == 0)
        return KDT_OK;
    RangeArgs a = blank_args();
    a.a = d_lo;
    a.b = d_hi;
    a.Q = Q;
    a.counts = d_counts;
    return run_range(t, 1, ACT_COUNT, flags, a, (cudaStream_t)stream);
}

int kdt_box_fill(const kdt_tree *t, const float *d_lo, const float *d_hi, int64_t Q, int flags,
                 const int64_t *d_offsets, int32_t *d_ids, void *stream)
{
    KDT_TRY(check_range(t, Q, d_lo, d_hi, true, flags));
    if (flags & KDT_RANGE_VISITS)
        return set_error(KDT_EINVAL, "KDT_RANGE_VISITS applies to the count calls only");
    if (Q > 0 && (!d_offsets || !d_ids))
        return set_error(KDT_EINVAL, "NULL offsets / ids");
    if (Q == 0)
        return KDT_OK;
    RangeArgs a = blank_args();
    a.a = d_lo;
    a.b = d_hi;
    a.Q = Q;
    a.offsets = d_offsets;
    a.out_ids = d_ids;
    a.vec_fill = fill_vectorizable(d_ids, nullptr);
    return run_range(t, 1, ACT_FILL, flags, a, (cudaStream_t)stream);
}

int kdt_offsets(const int32_t *d_counts, int64_t Q, int64_t *d_offsets, int64_t *h_total, void *stream)
{
    if (Q < 0 || !d_offsets || (Q > 0 && !d_counts))
        return set_error(KDT_EINVAL, "bad offsets arguments");
    cudaStream_t s = (cudaStream_t)stream;
    pool_setup_once();
    unsigned long long *out = (unsigned long long *)d_offsets;
    const int64_t n = Q + 1;
    Scratch sc(s);
    KDT_TRY(sc.alloc((scan_scratch_elems(n) + 1) * sizeof(unsigned long long)));
    KDT_LAUNCH counts_to_u64_kernel<<<grid_for(n), 256, 0, s>>>(d_counts, Q, out);
    KDT_TRY(exclusive_scan_u64(out, n, (unsigned long long *)sc.p, s));
    if (h_total) {
        KDT_CUDA(cudaMemcpyAsync(h_total, d_offsets + Q, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        KDT_CUDA(cudaStreamSynchronize(s));
    }
    return KDT_OK;
}

int kdt_tree_set_payload(kdt_tree *t, const float *d_payload, int C, void *stream)
{
    if (!t)
        return set_error(KDT_EINVAL, "tree is NULL");
    if (C < 1 || C > KDT_PAYLOAD_MAX_C || (t->N > 0 && !d_payload))
        return set_error(KDT_EINVAL, "payload: C must be in [1, %d] and the pointer non-NULL", KDT_PAYLOAD_MAX_C);
    cudaStream_t s = (cudaStream_t)stream;
    KDT_CUDA(cudaStreamSynchronize(s));
    cudaFree(t->payload);
    cudaFree(t->node_of);
    t->payload = nullptr;
    t->node_of = nullptr;
    t->payload_c = 0;
    const int64_t N = std::max<int64_t>(t->N, 1);
    KDT_CUDA(cudaMalloc(&t->payload, (size_t)N * C * sizeof(float)));
    KDT_CUDA(cudaMalloc(&t->node_of, (size_t)N * sizeof(int32_t)));
    if (t->N > 0) {
        const unsigned g = grid_for(t->N);
        switch (t->layout) {
        case 0: KDT_LAUNCH payload_permute_kernel<0><<<g, 256, 0, s>>>(t->nodes, t->ids, t->N, d_payload, C,
                                                                     t->payload, t->node_of); break;
        case 1: KDT_LAUNCH payload_permute_kernel<1><<<g, 256, 0, s>>>(t->nodes, t->ids, t->N, d_payload, C,
                                                                     t->payload, t->node_of); break;
        case 3: KDT_LAUNCH payload_permute_kernel<3><<<g, 256, 0, s>>>(t->nodes, t->ids, t->N, d_payload, C,
                                                                     t->payload, t->node_of); break;
        default: KDT_LAUNCH payload_permute_kernel<2><<<g, 256, 0, s>>>(t->nodes, t->ids, t->N, d_payload, C,
                                                                      t->payload, t->node_of); break;
        }
        KDT_CUDA(cudaGetLastError());
    }
    t->payload_c = C;
    return KDT_OK;
}

int kdt_radius_reduce(const kdt_tree *t, const float *d_q, int64_t Q, float radius, int flags, int mode, float *d_out,
                      int32_t *d_counts, void *stream)
{
    KDT_TRY(check_range(t, Q, d_q, nullptr, false, flags));
    if (flags & KDT_RANGE_VISITS)
        return set_error(KDT_EINVAL, "KDT_RANGE_VISITS applies to the count calls only");
    KDT_TRY(check_radius(radius));
    if (mode < KDT_REDUCE_SUM || mode > KDT_REDUCE_DENSITY)
        return set_error(KDT_EINVAL, "unknown reduction mode %d", mode);
    if (t->payload_c == 0)
        return set_error(KDT_EINVAL, "the tree has no payload (kdt_tree_set_payload)");
    if (Q > 0 && !d_out)
        return set_error(KDT_EINVAL, "NULL output");
    if (Q == 0)
        return KDT_OK;
    RangeArgs a = blank_args();
    a.a = d_q;
    a.Q = Q;
    a.r2 = radius * radius;
    a.counts = d_counts;
    a.payload = t->payload;
    a.C = t->payload_c;
    a.mode = mode;
    a.out = d_out;
    return run_range(t, 0, ACT_REDUCE, flags, a, (cudaStream_t)stream);
}

int kdt_knn_reduce(const kdt_tree *t, const float *d_q, int64_t Q, int k, float max_radius, int flags, int mode,
                   float *d_out, void *stream)
{
    if (!t)
        return set_error(KDT_EINVAL, "tree is NULL");
    if (mode < KDT_REDUCE_SUM || mode > KDT_REDUCE_DENSITY)
        return set_error(KDT_EINVAL, "unknown reduction mode %d", mode);
    if (t->payload_c == 0)
        return set_error(KDT_EINVAL, "the tree has no payload (kdt_tree_set_payload)");
    if (k < 1 || k > 64)
        return set_error(KDT_EINVAL, "k must be in [1, 64] (got %d)", k);
    if (Q < 0 || (Q > 0 && (!d_q || !d_out)))
        return set_error(KDT_EINVAL, "bad query count or NULL pointer");
    if (Q == 0)
        return KDT_OK;
    cudaStream_t s = (cudaStream_t)stream;
    pool_setup_once();
    Scratch sc(s);
    KDT_TRY(sc.alloc(carve_size({(size_t)Q * k * 4, (size_t)Q * k * 4})));
    Carve c{(char *)sc.p};
    int32_t *ids = c.take<int32_t>((size_t)Q * k);
    float *d2 = c.take<float>((size_t)Q * k);
    KDT_TRY(kdt_knn(t, d_q, Q, k, max_radius, flags, ids, d2, stream));
    KDT_LAUNCH knn_reduce_kernel<<<grid_for(Q), 256, 0, s>>>(ids, d2, Q, k, t->node_of, t->payload, t->payload_c, mode,
                                                             d_out);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

}  // extern "C"
