// The box tree: a second, read-only form of a k-d tree for queries that need
// only the result.
//
// The state machine of Sec. 3.2 tests one coordinate per node: a subtree is
// skipped when its splitting plane is farther than the cull radius.  A query
// between dense clusters lies near many planes of clusters that are far from
// it in the other coordinates, so it walks them.  With the bounding box of
// every subtree at hand the test is the distance to the box, in all
// coordinates, and most of those subtrees are skipped at once.
//
// Exactness.  For a query q and a box [lo, hi] that holds point p, in every
// coordinate t_j = max(fl(lo_j - q_j), fl(q_j - hi_j), 0) <= |fl(p_j - q_j)|
// because rounding is monotone; squares, and sums taken in the same order,
// keep the inequality.  So the box's distance, computed with the arithmetic of
// the points' distances, is never above the FP32 distance of a point in it:
// a skipped box (distance > cull radius) holds no point that the list would
// take.  Ties enter the box (<=), so equal distances are ordered by id as ever.
//
// Layout.  With H the last level, the subtrees rooted on level
// LB = max(H - 3, 0) are the buckets: 7 to 15 nodes of the tree, and one of the
// 2^LB - 1 nodes above.  Each of these is handed down to a bucket beside its
// splitting plane such that no bucket gets two: a node that receives one from
// above passes it to the child on its side of the plane and its own point to
// the other child; a node that receives none passes its own to the left.
// Either child touches the plane that the point lies on, so the buckets' boxes
// hardly grow, and the nodes above the buckets hold boxes alone.
//   bucket i: one group of 8 points (7 nodes + 1), or two (15 + 1) for the
//     first `big` buckets (those with nodes on the last level); group
//     i + min(i, big).  A group is [coordinate][8] floats, then [8] ids; places
//     without a point hold NaN, which no distance test takes.
//   record v: the boxes of the 4 grandchildren of binary node v, as
//     [coordinate][lo | hi][4] floats.  v counts nodes from 1 with the root 1
//     and the children 2v, 2v + 1, so the bucket i is v = 2^LB + i, and the
//     four children of v are 4v .. 4v + 3.  Only every second level has
//     records; with LB odd the root record is v = 0, whose children 2 and 3
//     are the root's two.
#pragma once

#include <type_traits>

#include "kdt_query.cuh"

namespace kdt {

constexpr int BOX_GROUP = 8;  // points per group
constexpr int BOX_LAUNCHES = 4;  // launches of a box tree's build: three for LB <= 26, one for small trees (kdt_box.cu)

template <int NC>
struct BoxFormat {
    static constexpr int REC = 2 * NC;        // float4 per record
    static constexpr int GRP = 2 * (NC + 1);  // float4 per group
};

__host__ __device__ __forceinline__ int box_coords(int D) { return D <= 3 ? 3 : (D == 4 ? 4 : 8); }

struct BoxShape {
    int LB;           // level of the bucket roots
    int64_t buckets;  // 2^LB
    int64_t big;      // buckets of two groups
    __host__ __device__ __forceinline__ explicit BoxShape(int64_t n)
    {
        const Topo tp(n);
        LB = tp.H > 3 ? tp.H - 3 : 0;
        buckets = (int64_t)1 << LB;
        big = tp.H >= 3 ? (tp.M + 7) / 8 : 0;
    }
    __host__ __device__ __forceinline__ int64_t records() const { return LB ? buckets / 2 : 0; }
    __host__ __device__ __forceinline__ int64_t groups() const { return buckets + big; }
    // first group of bucket i, and how many it has
    __host__ __device__ __forceinline__ int64_t group(int64_t i) const { return i + (i < big ? i : big); }
    __host__ __device__ __forceinline__ int count(int64_t i) const { return i < big ? 2 : 1; }
};

// Node at place m of a bucket's group k, root: the bucket's (m = 7 of the first
// group holds the point from above instead).  First group: the seven nodes of the
// bucket's first three levels; second: the eight of its fourth.
__host__ __device__ __forceinline__ int bucket_node(int root, int k, int m)
{
    const int up = k ? 3 : (m < 1 ? 0 : (m < 3 ? 1 : 2));
    return ((root + 1) << up) - 1 + (k ? m : m + 1 - (1 << up));
}

// Two FP32 values in one 64-bit register: sm_103a adds and multiplies such
// pairs in one instruction, each half rounded like the single operation.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pair(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 split(f32x2 p)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}
// a + b as a * 1 + b, one rounding.  The sum of two packed products written
// with add.rn.f32x2 came back a unit in the last place off: contracted to a
// fused multiply-add in spite of the rounding modifiers.  `one` is 1.0 twice,
// from the kernel's arguments, so that no compiler can know it and see a sum.
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b, f32x2 one)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(one), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// 32 bytes in one load (records and groups are multiples of 32 bytes on
// 32-byte boundaries): half the L1 wavefronts of two 16-byte loads, which bound
// the walks of incoherent lanes.
struct Float8 {
    float v[8];
};
__device__ __forceinline__ Float8 load8(const void *p)
{
    Float8 r;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
        : "l"(p));
    return r;
}

// t_j squared and summed in the order of dist2
template <int NC>
__device__ __forceinline__ void box_dist4(const float4 *__restrict__ rec, const float (&q)[NC], f32x2 one, float (&d)[4])
{
    f32x2 s[2];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const Float8 b = load8(rec + 2 * j);  // lo[4], hi[4]
        const f32x2 l[2] = {pair(b.v[0], b.v[1]), pair(b.v[2], b.v[3])};
        const f32x2 h[2] = {pair(b.v[4], b.v[5]), pair(b.v[6], b.v[7])};
        const f32x2 qq = pair(q[j], q[j]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float2 u = split(sub2(l[c], qq)), w = split(sub2(qq, h[c]));
            const f32x2 t = pair(fmaxf(fmaxf(u.x, w.x), 0.f), fmaxf(fmaxf(u.y, w.y), 0.f));
            const f32x2 tt = mul2(t, t);
            s[c] = j == 0 ? tt : add2(s[c], tt, one);
        }
    }
    const float2 u = split(s[0]), v = split(s[1]);
    d[0] = u.x;
    d[1] = u.y;
    d[2] = v.x;
    d[3] = v.y;
}

template <int NC>
__device__ __forceinline__ void group_dist8(const float4 *__restrict__ g, const float (&q)[NC], f32x2 one, float (&d)[8])
{
    f32x2 s[4];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const Float8 b = load8(g + 2 * j);
        const f32x2 x[4] = {pair(b.v[0], b.v[1]), pair(b.v[2], b.v[3]), pair(b.v[4], b.v[5]), pair(b.v[6], b.v[7])};
        const f32x2 qq = pair(q[j], q[j]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const f32x2 t = sub2(x[c], qq);
            const f32x2 tt = mul2(t, t);
            s[c] = j == 0 ? tt : add2(s[c], tt, one);
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float2 u = split(s[c]);
        d[2 * c] = u.x;
        d[2 * c + 1] = u.y;
    }
}

// One lane's place in the box tree, without a stack of nodes: the node v and,
// for every record above it, the four bits of children still to be looked at,
// the nearest record's in the low bits (14 records at most for N < 2^30).
// far[] holds, per record above, the distance of the nearest of these
// children: on the way up a record whose children are all out of range by now
// is passed without loading it again (of 26 record visits a query on surface
// points, k = 16, 9 were such).  It lies in shared memory, a column a thread.
struct BoxWalk {
    static constexpr int MAX_RECORDS = 14;
    uint32_t v;
    uint32_t mask;  // children of v to look at, while v has a record
    unsigned long long trail;
    float *far;     // of the next record down; `stride` floats to the next
    __device__ __forceinline__ void start(uint32_t leaf, float *far_)
    {
        // leaf = 2^LB: an odd LB has the root record 0 with children 2 and 3
        const bool odd = (leaf & 0xaaaaaaaau) != 0;
        v = odd ? 0u : 1u;
        mask = odd ? 12u : 15u;
        trail = 0;
        far = far_;
    }
    // back to the nearest record with a child left in range; false: none
    __device__ __forceinline__ bool pop(float cull, int stride)
    {
        while (trail) {
            const int up = (__ffsll((long long)trail) - 1) >> 2;
            v >>= 2 * (up + 1);
            trail >>= 4 * up;
            mask = (uint32_t)trail & 15u;
            trail >>= 4;
            far -= (up + 1) * stride;
            if (*far <= cull)
                return true;
        }
        return false;
    }
    // the nearest child of v in range, or back up; false: the walk is over
    template <int NC>
    __device__ __forceinline__ bool step(const float4 *__restrict__ rec, const float (&q)[NC], f32x2 one, float cull,
                                         int stride)
    {
        float d[4];
        box_dist4<NC>(rec + (size_t)v * BoxFormat<NC>::REC, q, one, d);
        // distances are >= 0, so their bits order them; the child's number
        // takes the two low bits (the order of near-equal boxes is free)
        uint32_t key[4], in = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const bool ok = (mask >> c & 1u) && d[c] <= cull;
            key[c] = ok ? (__float_as_uint(d[c]) & ~3u) | c : 0xffffffffu;
            in |= ok ? 1u << c : 0u;
        }
        if (in == 0)
            return pop(cull, stride);
        // the two smallest
        const uint32_t a = min(key[0], key[1]), b = max(key[0], key[1]);
        const uint32_t e = min(key[2], key[3]), f = max(key[2], key[3]);
        const uint32_t c = min(a, e) & 3u;
        const uint32_t next = min(max(a, e), min(b, f));
        *far = __uint_as_float(next & ~3u);
        far += stride;
        trail = trail << 4 | (in ^ (1u << c));
        v = 4 * v + c;
        mask = 15u;
        return true;
    }
};

// A box tree in memory.
struct BoxRef {
    const float4 *rec, *grp;
    uint32_t leaf;  // 2^LB
    uint32_t big;
};

struct BoxArgs {
    BoxRef tree = {nullptr, nullptr, 1, 0};
    const BoxRef *trees = nullptr;  // forests: one a tree (leaf = 0: no points)
    float one = 1.f;                // of the packed sums (add2)
};

inline BoxRef box_ref(int64_t n, const float4 *rec, const float4 *grp)
{
    const BoxShape sh(n);
    return {rec, grp, (uint32_t)sh.buckets, (uint32_t)sh.big};
}

__device__ __forceinline__ void order_keys(unsigned long long &a, unsigned long long &b)
{
    const bool sw = b < a;
    const unsigned long long t = sw ? b : a;
    b = sw ? a : b;
    a = t;
}

// Eight keys into the sorted list at once: Batcher's 19-exchange sort of the
// eight, then the half-cleaner and merge of a bitonic sequence, which keeps
// the K smallest of both.
template <int K>
__device__ __forceinline__ void merge8(unsigned long long (&L)[K], unsigned long long (&c)[8])
{
    constexpr int A[19] = {0, 2, 4, 6, 0, 1, 4, 5, 1, 5, 0, 1, 2, 3, 2, 3, 1, 3, 5};
    constexpr int B[19] = {1, 3, 5, 7, 2, 3, 6, 7, 2, 6, 4, 5, 6, 7, 4, 5, 2, 4, 6};
#pragma unroll
    for (int i = 0; i < 19; ++i)
        order_keys(c[A[i]], c[B[i]]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        unsigned long long &l = L[K - 8 + i];
        const unsigned long long x = c[7 - i];
        l = x < l ? x : l;
    }
#pragma unroll
    for (int h = K / 2; h > 0; h >>= 1)
#pragma unroll
        for (int i = 0; i < K; ++i)
            if ((i & h) == 0)
                order_keys(L[i], L[i + h]);
}

// Takers of the warp's busiest lane from which a group is merged whole
// (K = 8, 16): an insertion of one key is 6 K selects and compares, the merge
// of eight about 190 (K = 8) or 340 (K = 16), once for all lanes.  Measured
// with 1, 2, 3, 4, 5 and never: surface k = 16 2.97 / 2.92 / 2.87 / 2.87 / 2.90 /
// 3.87 ms, clustered 2^24 k = 8 19.4 / 19.0 / 18.7 / 18.5 / 18.5 / 20.0 ms.
constexpr int BOX_MERGE_FROM = 4;

// Points of the bucket that the list takes.  The test marks them for all
// points first; the marked ones are then inserted lane by lane, so that a
// warp runs the insertion as often as its busiest lane needs it and not once
// for every place in which any lane has a taker.
template <int NC, int K, class List>
__device__ __forceinline__ void box_bucket(const BoxRef &b, uint32_t i, const float (&q)[NC], f32x2 one, List &list)
{
    const float4 *g = b.grp + (size_t)(i + min(i, b.big)) * BoxFormat<NC>::GRP;
    const int groups = i < b.big ? 2 : 1;
    for (int k = 0; k < groups; ++k, g += BoxFormat<NC>::GRP) {
        float d[8];
        group_dist8<NC>(g, q, one, d);
        const float worst = list.cull();
        uint32_t take = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            take |= d[c] <= worst ? 1u << c : 0u;
        const uint32_t *ids = reinterpret_cast<const uint32_t *>(g + 2 * NC);
        if constexpr (K == 8 || K == 16) {
            const int most = __reduce_max_sync(__activemask(), __popc(take));
            if (most >= BOX_MERGE_FROM) {
                const Float8 id = load8(ids);
                unsigned long long key[8];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    key[c] = take >> c & 1u ? pack_key(d[c], __float_as_uint(id.v[c])) : ~0ull;
                merge8<K>(list.L, key);
                continue;
            }
        }
        while (take) {
            const int c = __ffs(take) - 1;
            take &= take - 1;
            const uint32_t id = __ldg(ids + c);
            float dc = d[0];
#pragma unroll
            for (int j = 1; j < 8; ++j)
                dc = c == j ? d[j] : dc;
            const unsigned long long key = pack_key(dc, id);
            if (key < list.worst())
                list.insert(key);
        }
    }
}

// The tree's box arrays (box_tree_bytes bytes at a 128-byte boundary), and their
// contents from its level-order nodes; the same for all trees of a forest.
size_t box_tree_bytes(int64_t n, int D);
void box_tree_place(kdt_tree *t, void *p);
int build_box_tree(const kdt_tree *t, cudaStream_t s);
int build_box_forest(kdt_forest *f, cudaStream_t s);
// Calls that the box tree serves: ordered queries for results, the learned
// radius among them.  Counts of processed nodes are counts of the state
// machine; the unordered machine, the ablations and lists spread over groups
// of lanes are forms that a caller asks for by name.
inline bool box_query_serves(const QueryArgs &a, int flags, int mode)
{
    return (mode == MODE_RESULTS || (mode == MODE_BOUNDED && !a.visits)) && a.out_ids && a.group == 1 &&
           !(flags & (KDT_UNORDERED | KDT_PLAIN_STEP | KDT_CLOSE_FIRST | KDT_STACK));
}
// kNN of one tree, and of a forest's queries (a.T, a.node_off and a.q_off set)
int launch_box_query(int layout, const BoxRef &tree, const QueryArgs &a, int mode, cudaStream_t s);
inline int launch_box_query(const kdt_tree *t, const QueryArgs &a, int mode, cudaStream_t s)
{
    return launch_box_query(t->layout, box_ref(t->N, t->box_rec, t->box_grp), a, mode, s);
}
int launch_box_forest(const kdt_forest *f, const QueryArgs &a, cudaStream_t s);

}  // namespace kdt
