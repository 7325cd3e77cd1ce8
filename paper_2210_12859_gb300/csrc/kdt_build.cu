// GPU builder of left-balanced, complete, level-order k-d trees.
//
// The tree is the one a serial median builder produces (Sec. 4 states that a
// parallel builder emits exactly that tree): for a subtree of n points at
// level l the points are ordered by (coordinate l mod D, input index), the
// element of rank L(n) (left-subtree size of a complete tree of n nodes)
// becomes the node, the lower ranks form the left subtree and the higher ranks
// the right subtree.
//
// Design.  For every dimension e the builder keeps a list of point indices
// sorted by (coordinate e, input index) (one stable radix sort per dimension).
// Positions of every list are laid out in IN-ORDER: the points of the subtree
// of node t always occupy the in-order range of t's subtree.  Then, at level l
// with split dimension d:
//   * the list of d needs no work: within a segment the element at in-order
//     position p goes left iff p lies in the left subtree's in-order range,
//     becomes the node iff p is t's own in-order position, else goes right.
//     That is purely topological (closed-form in-order <-> node maps), so one
//     pass over the list writes each point's side and emits the level's nodes;
//   * every other list still needed later is stably partitioned inside each
//     segment into [left | node | right] with a segmented scan of the side
//     flags, which keeps each part sorted by its own key.
// These passes run over arrays of N elements only for the levels whose subtrees
// are larger than SUB_N points; then one block a subtree builds all the levels
// that are left in shared memory (sub_kernel).  With them the build of 2^24
// points is 12 passes over the lists instead of 24, and that of 20 k points 23
// launches instead of 160.  T > 1 trees are built in the same passes: lists are
// first sorted by (tree, coordinate, index) and every position knows its tree.
#include <algorithm>

#include "kdt_internal.cuh"

namespace kdt {
namespace {

constexpr int BT = 256;          // threads per block, builder kernels
constexpr int PITEMS = 4;        // items per thread, partition scan
constexpr int PTILE = BT * PITEMS;

enum : uint8_t { SIDE_LEFT = 0, SIDE_NODE = 1, SIDE_RIGHT = 2 };

// Largest subtree that one block builds in shared memory.  Large builds take
// the largest that leaves two blocks on an SM, since every level above costs a
// pass over all lists (2^24 points: 0.31 ms a level); small ones, which fill few
// SMs either way and whose blocks are bound by instruction issue, a smaller one.
constexpr int SUB_LOG2_LARGE = 12, SUB_LOG2_SMALL = 10;
constexpr int64_t SUB_SMALL_TOTAL = (int64_t)1 << 18;
inline int sub_log2_of(int64_t total) { return total <= SUB_SMALL_TOTAL ? SUB_LOG2_SMALL : SUB_LOG2_LARGE; }

// A forest's small trees are built whole by blocks of their size, in a launch
// for each class of sizes: up to 2^7 points (a warp), up to 2^10, and the rest,
// a block of 2^sub_log2 points a subtree.  A block of 4096 points costs its
// threads and barriers whatever it holds: 100 000 clouds of 10 points are built
// in 1.8 ms instead of 9.5 (of 40: 2.8 instead of 15.1), 50 000 of 20 beside one
// of 3 M in 4.4 instead of 9.2.
constexpr int SUB_LOG2_TINY = 7;
inline int sub_class_of(int64_t n, int sub_log2)
{
    if (n <= (int64_t)1 << SUB_LOG2_TINY)
        return 0;
    return n <= (int64_t)1 << SUB_LOG2_SMALL && sub_log2 > SUB_LOG2_SMALL ? 1 : 2;
}

// levels of a tree of n points whose subtrees are larger than 2^sub_log2: the
// subtrees of level l hold at most 2^(H-l) - 1 points above the last level and
// min(M, 2^(H-l)) on it
__host__ __device__ __forceinline__ int top_levels(int64_t n, int sub_log2)
{
    const Topo tp(n);
    const int l = tp.H > sub_log2 ? tp.H - sub_log2 : 0;
    const int64_t w = (int64_t)1 << (tp.H - l);
    return w - 1 + (tp.M < w ? tp.M : w) <= (int64_t)1 << sub_log2 ? l : l + 1;
}

struct Where {
    int64_t base;   // first position of the position's tree
    int64_t n;      // size of that tree
};

__device__ __forceinline__ Where locate(int64_t p, int T, const int64_t *__restrict__ off,
                                        const int32_t *__restrict__ tree_of, int64_t total)
{
    if (T == 1)
        return {0, total};
    int i = tree_of[p];
    int64_t b = off[i];
    return {b, off[i + 1] - b};
}

// sort keys of dimensions e0 .. e0 + ne - 1, `total` apart
__global__ void prep_keys_kernel(const float *__restrict__ pts, int64_t total, int D, int e0, int ne,
                                 uint32_t *__restrict__ keys, int *__restrict__ err)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        for (int e = 0; e < ne; ++e) {
            float x = pts[i * D + e0 + e];
            if (!isfinite(x))
                atomicOr(err, ERR_NONFINITE);
            keys[e * total + i] = float_key(x);
        }
}

__global__ void tree_keys_kernel(const uint32_t *__restrict__ vals, const int32_t *__restrict__ tree_of, int64_t total,
                                 uint32_t *__restrict__ keys)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = (uint32_t)tree_of[vals[i]];
}

__global__ void tree_of_kernel(const int64_t *__restrict__ off, int T, int64_t total, int32_t *__restrict__ tree_of)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        // last tree whose offset is <= i (empty trees are skipped by taking the last)
        int lo = 0, hi = T - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= i)
                lo = mid;
            else
                hi = mid - 1;
        }
        tree_of[i] = lo;
    }
}

struct ListPtrs {
    const uint32_t *p[8];
};

// bounding box of the first min(D,3) dims of each tree: the extremes of the
// per-dimension sorted lists
__global__ void bbox_kernel(const float *__restrict__ pts, int D, ListPtrs lists, const int64_t *__restrict__ off,
                            int T, int64_t total, float *__restrict__ bbox)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T)
        return;
    int64_t a = T == 1 ? 0 : off[i], b = T == 1 ? total : off[i + 1];
    for (int e = 0; e < 3; ++e) {
        float lo = 0.f, hi = 0.f;
        if (e < D && b > a) {
            lo = pts[(int64_t)lists.p[e][a] * D + e];
            hi = pts[(int64_t)lists.p[e][b - 1] * D + e];
        }
        bbox[i * 6 + e] = lo;
        bbox[i * 6 + 3 + e] = hi;
    }
}

// a node of the tree whose first point is at `base`: the point pid as node u
__device__ __forceinline__ void emit_node(const float *__restrict__ pts, int D, int64_t base, int64_t u, uint32_t pid,
                                          uint32_t dim_bits, float4 *__restrict__ nodes, int32_t *__restrict__ ids)
{
    const float *c = pts + (int64_t)pid * D;
    const int32_t local = (int32_t)(pid - (uint32_t)base);
    const int64_t node = base + u;
    if (D <= 3) {
        nodes[node] = make_float4(c[0], D > 1 ? c[1] : 0.f, D > 2 ? c[2] : 0.f,
                                  __uint_as_float((uint32_t)local | dim_bits));
    } else if (D == 4) {
        nodes[node] = make_float4(c[0], c[1], c[2], c[3]);
        ids[node] = local;
    } else {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            v[j] = j < D ? c[j] : 0.f;
        nodes[2 * node] = make_float4(v[0], v[1], v[2], v[3]);
        nodes[2 * node + 1] = make_float4(v[4], v[5], v[6], v[7]);
        ids[node] = local;
    }
}

// Level l, split list: record each point's side and emit the level's nodes.
__global__ void assign_kernel(const uint32_t *__restrict__ list, int64_t total, int l, int sub_log2, int T,
                              const int64_t *__restrict__ off, const int32_t *__restrict__ tree_of,
                              const float *__restrict__ pts, int D, uint8_t *__restrict__ side,
                              float4 *__restrict__ nodes, int32_t *__restrict__ ids)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < total; p += (int64_t)gridDim.x * blockDim.x) {
        Where w = locate(p, T, off, tree_of, total);
        Topo tp(w.n);
        if (l >= top_levels(w.n, sub_log2))
            continue;
        int64_t u = tp.node_at(p - w.base);
        int lu = Topo::level(u);
        if (lu < l)
            continue;
        uint32_t pid = list[p];
        if (lu == l) {
            side[pid] = SIDE_NODE;
            emit_node(pts, D, w.base, u, pid, 0u, nodes, ids);
        } else {
            int bit = (int)(((u + 1) >> (lu - l - 1)) & 1);
            side[pid] = bit ? SIDE_RIGHT : SIDE_LEFT;
        }
    }
}

// ---- stored split dimension (widest extent of the node's points)

// split dimension of every node of level l: within the node's segment each
// list is sorted by its coordinate, so its first and last elements give the
// extent; the widest dimension wins, ties to the lowest index
__global__ void widest_kernel(ListPtrs lists, int64_t n, int l, const float *__restrict__ pts, int D,
                              uint8_t *__restrict__ node_dim)
{
    const int64_t first = ((int64_t)1 << l) - 1;
    const int64_t count = (first + 1 < n - first) ? first + 1 : n - first;
    const Topo tp(n);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = first + i;
        const int64_t a = tp.inorder(tp.leftmost(t));
        const int64_t b = tp.inorder(tp.rightmost(t));
        int best = 0;
        float best_ext = -1.f;
        for (int e = 0; e < D; ++e) {
            const float lo = pts[(int64_t)lists.p[e][a] * D + e];
            const float hi = pts[(int64_t)lists.p[e][b] * D + e];
            const float ext = __fsub_rn(hi, lo);
            if (ext > best_ext) {
                best_ext = ext;
                best = e;
            }
        }
        node_dim[t] = (uint8_t)best;
    }
}

// level l with per-node split dimensions: the element at in-order position p
// of its segment's split list decides the side (single tree, D <= 3)
__global__ void assign_widest_kernel(ListPtrs lists, int64_t n, int l, const uint8_t *__restrict__ node_dim,
                                     const float *__restrict__ pts, int D, uint8_t *__restrict__ side,
                                     float4 *__restrict__ nodes)
{
    const Topo tp(n);
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        if (l > tp.H)
            continue;
        const int64_t u = tp.node_at(p);
        const int lu = Topo::level(u);
        if (lu < l)
            continue;
        const int64_t t = Topo::ancestor(u, lu, l);
        const int e = node_dim[t];
        const uint32_t pid = lists.p[e][p];
        if (lu == l) {
            side[pid] = SIDE_NODE;
            emit_node(pts, D, 0, u, pid, (uint32_t)e << NODE_DIM_SHIFT, nodes, nullptr);
        } else {
            const int bit = (int)(((u + 1) >> (lu - l - 1)) & 1);
            side[pid] = bit ? SIDE_RIGHT : SIDE_LEFT;
        }
    }
}

// ---- segmented stable partition of a non-split list

struct Seg {
    uint32_t f;                 // segment head inside the range
    unsigned long long v;       // left count (low 32) | right count (high 32)
};

__device__ __forceinline__ Seg seg_op(Seg a, Seg b)
{
    Seg r;
    r.f = a.f | b.f;
    r.v = b.f ? b.v : a.v + b.v;
    return r;
}

struct Item {
    Seg s;          // value of this position
    int64_t dest;   // -1: copy through
    uint32_t pid;
    uint8_t side;
    int64_t s_t, in_t;  // segment start and node in-order position (relative)
    int64_t base, n;
};

__device__ __forceinline__ void load_item(const uint32_t *__restrict__ in, int64_t p, int64_t total, int l, int sub_log2, int T,
                                          const int64_t *__restrict__ off, const int32_t *__restrict__ tree_of,
                                          const uint8_t *__restrict__ side, Item &it)
{
    it.s.f = 1;
    it.s.v = 0;
    it.dest = -1;
    if (p >= total)
        return;
    it.pid = in[p];
    Where w = locate(p, T, off, tree_of, total);
    Topo tp(w.n);
    if (l >= top_levels(w.n, sub_log2))
        return;
    int64_t lp = p - w.base;
    int64_t u = tp.node_at(lp);
    int lu = Topo::level(u);
    if (lu < l)
        return;
    int64_t t = Topo::ancestor(u, lu, l);
    it.s_t = tp.inorder(tp.leftmost(t));
    it.in_t = tp.inorder(t);
    it.base = w.base;
    it.n = w.n;
    it.side = side[it.pid];
    it.s.f = lp == it.s_t;
    it.s.v = (it.side == SIDE_LEFT ? 1ull : 0ull) | (it.side == SIDE_RIGHT ? (1ull << 32) : 0ull);
    it.dest = 0;
}

__device__ __forceinline__ Seg shfl_up_seg(Seg x, int o)
{
    Seg r;
    r.f = __shfl_up_sync(0xffffffffu, x.f, o);
    r.v = __shfl_up_sync(0xffffffffu, x.v, o);
    return r;
}

// exclusive segmented block scan of one Seg per thread; *agg = block total
__device__ __forceinline__ Seg block_exclusive_seg(Seg x, Seg *s_warp, Seg *agg)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Seg inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        Seg y = shfl_up_seg(inc, o);
        if (lane >= o)
            inc = seg_op(y, inc);
    }
    Seg ex = shfl_up_seg(inc, 1);
    if (lane == 0)
        ex = Seg{0, 0};
    if (lane == 31)
        s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        Seg a = lane < nw ? s_warp[lane] : Seg{0, 0};
        Seg ai = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            Seg y = shfl_up_seg(ai, o);
            if (lane >= o)
                ai = seg_op(y, ai);
        }
        Seg ae = shfl_up_seg(ai, 1);
        if (lane == 0)
            ae = Seg{0, 0};
        if (lane < nw)
            s_warp[lane] = ae;
        if (lane == nw - 1)
            s_warp[32] = ai;
    }
    __syncthreads();
    Seg r = seg_op(s_warp[w], ex);
    *agg = s_warp[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(BT) part_reduce_kernel(const uint32_t *__restrict__ in, int64_t total, int l,
                                                         int sub_log2, int T,
                                                         const int64_t *__restrict__ off,
                                                         const int32_t *__restrict__ tree_of,
                                                         const uint8_t *__restrict__ side, Seg *__restrict__ tiles)
{
    __shared__ Seg s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * PTILE + (int64_t)threadIdx.x * PITEMS;
    Seg acc{0, 0};
#pragma unroll
    for (int j = 0; j < PITEMS; ++j) {
        Item it;
        load_item(in, base + j, total, l, sub_log2, T, off, tree_of, side, it);
        acc = seg_op(acc, it.s);
    }
    Seg agg;
    block_exclusive_seg(acc, s_warp, &agg);
    if (threadIdx.x == 0)
        tiles[blockIdx.x] = agg;
}

__global__ void __launch_bounds__(1024) part_tiles_kernel(Seg *__restrict__ tiles, int64_t nt)
{
    __shared__ Seg s_warp[33];
    Seg carry{0, 0};
    for (int64_t b = 0; b < nt; b += 1024) {
        int64_t i = b + threadIdx.x;
        Seg x = i < nt ? tiles[i] : Seg{0, 0};
        Seg agg;
        Seg ex = block_exclusive_seg(x, s_warp, &agg);
        if (i < nt)
            tiles[i] = seg_op(carry, ex);
        carry = seg_op(carry, agg);
    }
}

__global__ void __launch_bounds__(BT) part_scatter_kernel(const uint32_t *__restrict__ in, int64_t total, int l,
                                                          int sub_log2, int T,
                                                          const int64_t *__restrict__ off,
                                                          const int32_t *__restrict__ tree_of,
                                                          const uint8_t *__restrict__ side,
                                                          const Seg *__restrict__ tiles, uint32_t *__restrict__ out)
{
    __shared__ Seg s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * PTILE + (int64_t)threadIdx.x * PITEMS;
    Item it[PITEMS];
    Seg acc{0, 0};
#pragma unroll
    for (int j = 0; j < PITEMS; ++j) {
        load_item(in, base + j, total, l, sub_log2, T, off, tree_of, side, it[j]);
        acc = seg_op(acc, it[j].s);
    }
    Seg agg;
    Seg run = seg_op(tiles[blockIdx.x], block_exclusive_seg(acc, s_warp, &agg));
#pragma unroll
    for (int j = 0; j < PITEMS; ++j) {
        int64_t p = base + j;
        if (p >= total)
            break;
        // run is the exclusive prefix of this item within its segment (a head
        // starts from zero)
        Seg ex = it[j].s.f ? Seg{1, 0} : run;
        if (it[j].dest < 0) {
            out[p] = it[j].pid;
        } else {
            uint32_t lb = (uint32_t)(ex.v & 0xffffffffu);
            uint32_t rb = (uint32_t)(ex.v >> 32);
            int64_t d;
            if (it[j].side == SIDE_NODE)
                d = it[j].in_t;
            else if (it[j].side == SIDE_LEFT)
                d = it[j].s_t + lb;
            else
                d = it[j].in_t + 1 + rb;
            if (d >= 0 && d < it[j].n)  // always true for consistent side flags
                out[it[j].base + d] = it[j].pid;
        }
        run = seg_op(run, it[j].s);
    }
}

// ---- single trees: two kernels a level

// The in-order layout of a complete tree of n < 2^30 points in 32 bits.
struct Layout32 {
    int n, H, M;
    __device__ __forceinline__ explicit Layout32(int n_) : n(n_)
    {
        H = 31 - __clz(n_);
        M = n_ - ((1 << H) - 1);
    }
    __device__ __forceinline__ static int level(int u) { return 31 - __clz(u + 1); }
    __device__ __forceinline__ int node_at(int p) const
    {
        const int P = p < 2 * M ? p : 2 * (p - M) + 1;
        const int tz = __ffs(P + 1) - 1;
        return (1 << (H - tz)) - 1 + ((P + 1) >> (tz + 1));
    }
    __device__ __forceinline__ int inorder(int u) const
    {
        const int l = level(u);
        const int P = ((2 * (u - ((1 << l) - 1)) + 1) << (H - l)) - 1;
        const int missing = min((P + 1) >> 1, 1 << H) - M;
        return P - max(missing, 0);
    }
    // the j-th subtree of level l: w = 2^(H-l) places on the last level
    __device__ __forceinline__ int start(int l, int j) const { return (j << (H - l)) + min(M, j << (H - l)); }
    __device__ __forceinline__ int size(int l, int j) const
    {
        const int w = 1 << (H - l);
        return w - 1 + min(max(M - j * w, 0), w);
    }
    // points of its left subtree
    __device__ __forceinline__ int left(int l, int j) const
    {
        const int w = 1 << (H - l), h = w >> 1;
        return h - 1 + min(max(M - j * w, 0), h);
    }
    // points of the left subtrees of the subtrees before it on the level
    __device__ __forceinline__ int lefts_before(int l, int j) const
    {
        const int w = 1 << (H - l), h = w >> 1;
        const int full = M >= h ? min(j, ((M - h) >> (H - l)) + 1) : 0;
        return j * (h - 1) + full * h + (full < j ? min(max(M - full * w, 0), h) : 0);
    }
};

// Where the element at place p of a level's list goes: `lefts` and `ones` are
// the left elements and the level's nodes at places before p.
__device__ __forceinline__ int part_dest(const Layout32 &t, int l, int u, int lu, int p, int side, int lefts, int ones)
{
    const int j = ((u + 1) >> (lu - l)) - (1 << l);
    const int s = t.start(l, j), in = s + t.left(l, j);
    if (side == SIDE_NODE)
        return in;
    const int lb = lefts - t.lefts_before(l, j);
    if (side == SIDE_LEFT)
        return s + lb;
    return in + 1 + (p - s) - lb - (ones - j);
}

constexpr int TOP_ITEMS = 8;
constexpr int TOP_TILE = BT * TOP_ITEMS;
constexpr int TOP_WORDS = TOP_TILE / 32;  // vote words of a tile
constexpr int TOP_LISTS = 3;              // lists of one launch
constexpr int TOP_GROUP = 64;             // tiles whose counts are also summed
static_assert(TOP_WORDS <= 64 && TOP_WORDS % 32 == 0, "the words of a tile are scanned by two warps");

inline int64_t top_tiles_of(int64_t n) { return (n + TOP_TILE - 1) / TOP_TILE; }
inline int64_t top_groups_of(int64_t n) { return (top_tiles_of(n) + TOP_GROUP - 1) / TOP_GROUP; }

struct PartArgs {
    const uint32_t *in[TOP_LISTS];
    uint32_t *out[TOP_LISTS];
    const uint8_t *side;
    uint2 *votes;               // [list][tiles][TOP_WORDS]: lefts and nodes of 32 places
    unsigned long long *count;  // [list][tiles + groups]: nodes << 32 | lefts; the groups start at zero
    int n, l, tiles, groups;
    // the list that splits the next level also records that level's sides and
    // emits its nodes (-1: none does)
    int next;
    uint8_t *side_next;
    const float *pts;
    int D;
    float4 *nodes;
    int32_t *ids;
};

// Stable partition of up to three lists by the level's sides, in two kernels.
// A plain count of the left elements suffices, no segmented one: how many the
// earlier subtrees of the level hold is a closed form of the layout.
//
// part_votes_kernel gathers the sides once and keeps them as vote words, with
// the counts of tiles and of groups of tiles; part_move_kernel sums the counts
// before its tile (a group's and a tile's count a thread) and moves the elements.
//
// Bound: the random bytes, a gather an element and list in the first and a
// store an element for the next level's sides in the second, beside 12 bytes
// an element of list traffic.  One kernel with a look-back took 0.42 ms a level
// of 2^24 points (its blocks waited for the look-back with the gathers of two
// blocks an SM in flight; windows of 32 and of 256 tiles alike), the
// count, scan, scatter and assign kernels before it 0.71.
__global__ void __launch_bounds__(BT) part_votes_kernel(const PartArgs a)
{
    __shared__ uint32_t s_cnt;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, y = blockIdx.y, tile = blockIdx.x;
    if (tid == 0)
        s_cnt = 0;
    __syncthreads();
    const uint32_t *in = y == 0 ? a.in[0] : (y == 1 ? a.in[1] : a.in[2]);
    const Layout32 t(a.n);
    const int first = tile * TOP_TILE + w * 32 * TOP_ITEMS + lane;
    uint32_t pid[TOP_ITEMS], side[TOP_ITEMS];
#pragma unroll
    for (int j = 0; j < TOP_ITEMS; ++j) {
        const int p = first + 32 * j;
        pid[j] = p < a.n && Layout32::level(t.node_at(p)) >= a.l ? in[p] : 0xffffffffu;
    }
#pragma unroll
    for (int j = 0; j < TOP_ITEMS; ++j)
        side[j] = pid[j] != 0xffffffffu ? a.side[pid[j]] : 3u;  // 3: not in a subtree of the level
    uint32_t run = 0;
    uint2 words = make_uint2(0, 0);
#pragma unroll
    for (int j = 0; j < TOP_ITEMS; ++j) {
        const uint32_t bl = __ballot_sync(0xffffffffu, side[j] == SIDE_LEFT);
        const uint32_t bn = __ballot_sync(0xffffffffu, side[j] == SIDE_NODE);
        if (lane == j)
            words = make_uint2(bl, bn);
        run += __popc(bl) | __popc(bn) << 16;
    }
    if (lane < TOP_ITEMS)
        a.votes[((size_t)y * a.tiles + tile) * TOP_WORDS + w * TOP_ITEMS + lane] = words;
    if (lane == 0)
        atomicAdd(&s_cnt, run);  // at most TOP_TILE of each
    __syncthreads();
    if (tid == 0) {
        const unsigned long long c = (unsigned long long)(s_cnt >> 16) << 32 | (s_cnt & 0xffffu);
        unsigned long long *count = a.count + (size_t)y * (a.tiles + a.groups);
        count[tile] = c;
        atomicAdd(count + a.tiles + tile / TOP_GROUP, c);
    }
}

__global__ void __launch_bounds__(BT) part_move_kernel(const PartArgs a)
{
    __shared__ unsigned long long s_sum[BT / 32];
    __shared__ uint2 s_vote[TOP_WORDS];
    __shared__ uint32_t s_before[TOP_WORDS + 1];  // nodes << 16 | lefts of the words before, halves apart
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, y = blockIdx.y, tile = blockIdx.x;
    const uint32_t *in = y == 0 ? a.in[0] : (y == 1 ? a.in[1] : a.in[2]);
    uint32_t *out = y == 0 ? a.out[0] : (y == 1 ? a.out[1] : a.out[2]);
    const Layout32 t(a.n);
    const int first = tile * TOP_TILE + w * 32 * TOP_ITEMS + lane;
    uint32_t pid[TOP_ITEMS];
#pragma unroll
    for (int j = 0; j < TOP_ITEMS; ++j) {
        const int p = first + 32 * j;
        pid[j] = p < a.n ? in[p] : 0;
    }
    // the tiles before: whole groups, then the tiles of this one's
    const unsigned long long *count = a.count + (size_t)y * (a.tiles + a.groups);
    const int group = tile / TOP_GROUP;
    unsigned long long sum = 0;
    for (int i = tid; i < group; i += BT)
        sum += count[a.tiles + i];
    if (tid < tile - group * TOP_GROUP)
        sum += count[group * TOP_GROUP + tid];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0)
        s_sum[w] = sum;
    if (tid < TOP_WORDS) {
        const uint2 v = a.votes[((size_t)y * a.tiles + tile) * TOP_WORDS + tid];
        s_vote[tid] = v;
        uint32_t c = __popc(v.x) | __popc(v.y) << 16, inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
            inc += lane >= o ? x : 0;
        }
        s_before[tid] = inc - c;
        if (tid == 31)
            s_before[TOP_WORDS] = inc;  // of the first 32 words
    }
    __syncthreads();
    sum = 0;
#pragma unroll
    for (int i = 0; i < BT / 32; ++i)
        sum += s_sum[i];
    const bool next = y == a.next;
    const uint32_t lt = (1u << lane) - 1;
#pragma unroll
    for (int j = 0; j < TOP_ITEMS; ++j) {
        const int p = first + 32 * j;
        if (p >= a.n)
            break;
        const int u = t.node_at(p), lu = Layout32::level(u);
        if (lu < a.l)
            continue;
        const int word = w * TOP_ITEMS + j;
        const uint2 v = s_vote[word];
        const int s = v.x >> lane & 1u ? SIDE_LEFT : (v.y >> lane & 1u ? SIDE_NODE : SIDE_RIGHT);
        const uint32_t before = s_before[word] + (word >= 32 ? s_before[TOP_WORDS] : 0);
        const int lefts = (int)(sum & 0xffffffffu) + (int)(before & 0xffffu) + __popc(v.x & lt);
        const int ones = (int)(sum >> 32) + (int)(before >> 16) + __popc(v.y & lt);
        const int d = part_dest(t, a.l, u, lu, p, s, lefts, ones);
        if (d < 0 || d >= a.n)  // never, for consistent sides
            continue;
        out[d] = pid[j];
        if (next && s != SIDE_NODE) {
            const int x = t.node_at(d), lx = Layout32::level(x);
            if (lx == a.l + 1) {
                a.side_next[pid[j]] = SIDE_NODE;
                emit_node(a.pts, a.D, 0, x, pid[j], 0u, a.nodes, a.ids);
            } else {
                a.side_next[pid[j]] = (x + 1) >> (lx - a.l - 2) & 1 ? SIDE_RIGHT : SIDE_LEFT;
            }
        }
    }
}

// ---- the levels whose subtrees fit one block

// places a thread looks after; places and counts of a subtree fit 13 bits
constexpr int SUB_ITEMS = 4;
static_assert(SUB_LOG2_LARGE <= 12, "places and counts of a subtree are packed");

struct SubArgs {
    ListPtrs lists;
    const int64_t *off;       // T > 1: first point of every tree, [T + 1]
    const int32_t *first_job; // T > 1: first block of every tree in this launch, [T + 1], or
    bool whole_trees;         // the tree of every block
    int64_t total;
    int T, D;
    bool widest;
    const float *pts;
    uint16_t *place;          // [total] scratch: a point's place in its block
    float4 *nodes;
    int32_t *ids;
};

// bytes of sub_kernel's arrays: pid, warp counts, then 16-bit places, lists and bytes
inline size_t sub_smem(int D, int sub_log2)
{
    const size_t n = (size_t)1 << sub_log2;
    return n * (4 + 2 * (D + 1) + 2) + 2 * 32 * 4;
}

// Block b: one subtree of the first level whose subtrees fit, all its levels.
// The points are renumbered 0 .. n - 1, so the lists are 16-bit and lie in
// shared memory with the side bytes; a level is one look at the split list and
// one stable partition of the others by a block-wide count, both with the
// closed forms of the subtree's own layout, two lists at a time so that a
// place's closed forms are worked out once for both.  A node's point is noted
// by in-order place and all nodes are written at the end, a level's nodes side
// by side.
//
// Bound: instruction issue (the places' closed forms, some 60 instructions a
// place and level) between the block's barriers.  Threads with 4 / 8 / 16 places
// each: a build of 2^24 points 11.0 / 11.2 / 12.8 ms, a rebuild of 20 k 196 / 210 /
// 233 us; subtrees of 2^11 instead of 2^12 cost the large build 0.2 ms, of 2^9 or
// 2^11 instead of 2^10 the small one 2 to 6 us.
template <int SUB_LOG2>
__global__ void __launch_bounds__((1 << SUB_LOG2) / SUB_ITEMS, SUB_LOG2 == 12 ? 1 : (SUB_LOG2 == 10 ? 4 : 16)) sub_kernel(const SubArgs a)
{
    constexpr int SUB_N = 1 << SUB_LOG2;
    constexpr int THREADS = SUB_N / SUB_ITEMS;
    constexpr int WARPS = THREADS / 32;
    static_assert(WARPS <= 32, "the warp counts of two lists are summed by one warp");
    extern __shared__ uint32_t s_mem[];
    uint32_t *s_pid = s_mem;                                          // [SUB_N]
    uint32_t *s_cnt = s_pid + SUB_N;                                  // [2][32]: two lists, a warp each
    uint16_t *s_fin = reinterpret_cast<uint16_t *>(s_cnt + 64);       // [SUB_N] by in-order place
    uint16_t *s_list = s_fin + SUB_N;                                 // [D][SUB_N]
    uint8_t *s_side = reinterpret_cast<uint8_t *>(s_list + (size_t)a.D * SUB_N);  // [SUB_N]
    uint8_t *s_dim = s_side + SUB_N;                                  // [SUB_N] split dimension of a node (widest)
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, D = a.D;

    int64_t base = 0, tn = a.total;
    int job = blockIdx.x;
    if (a.T > 1) {
        int lo = 0, hi = a.T - 1;  // last tree that starts at or before the block (trees of no block have the next one's)
        if (a.whole_trees) {
            lo = hi = a.first_job[job];
            job = 0;
        }
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.first_job[mid] <= job)
                lo = mid;
            else
                hi = mid - 1;
        }
        base = a.off[lo];
        tn = a.off[lo + 1] - base;
        if (!a.whole_trees)
            job -= a.first_job[lo];
    }
    const Layout32 whole((int)tn);
    const int top = top_levels(tn, SUB_LOG2);
    const int n = whole.size(top, job);
    const int64_t seg = base + whole.start(top, job);
    const Layout32 t(n);

    const uint32_t *l0 = a.lists.p[0] + seg;
    for (int i = tid; i < n; i += THREADS) {
        const uint32_t pid = l0[i];
        s_pid[i] = pid;
        s_list[i] = (uint16_t)i;
        a.place[pid] = (uint16_t)i;
    }
    __syncthreads();
    for (int e = 1; e < D; ++e) {
        const uint32_t *le = a.lists.p[e] + seg;
        for (int i = tid; i < n; i += THREADS)
            s_list[e * SUB_N + i] = a.place[le[i]];
    }
    __syncthreads();

    // the node of a thread's places: index + 1, 0 past the end
    const int first = w * 32 * SUB_ITEMS + lane;
    uint16_t node[SUB_ITEMS];
#pragma unroll
    for (int k = 0; k < SUB_ITEMS; ++k)
        node[k] = first + 32 * k < n ? (uint16_t)(t.node_at(first + 32 * k) + 1) : (uint16_t)0;
    const uint32_t lt = (1u << lane) - 1;
    for (int l = 0; l <= t.H; ++l) {
        const int d = (top + l) % D;
        const uint32_t level = 1u << l;  // node + 1 of the level's first node
        if (a.widest) {
            const int count = min(1 << l, n - ((1 << l) - 1));
            for (int j = tid; j < count; j += THREADS) {
                const int s = t.start(l, j), z = s + t.size(l, j) - 1;
                int best = 0;
                float best_ext = -1.f;
                for (int e = 0; e < D; ++e) {
                    const float lo = a.pts[(int64_t)s_pid[s_list[e * SUB_N + s]] * D + e];
                    const float hi = a.pts[(int64_t)s_pid[s_list[e * SUB_N + z]] * D + e];
                    const float ext = __fsub_rn(hi, lo);
                    if (ext > best_ext) {
                        best_ext = ext;
                        best = e;
                    }
                }
                s_dim[(1 << l) - 1 + j] = (uint8_t)best;
            }
            __syncthreads();
        }
        // the split list: sides, and the level's nodes
#pragma unroll
        for (int k = 0; k < SUB_ITEMS; ++k) {
            const uint32_t u = node[k];
            if (u < level)
                continue;
            const int p = first + 32 * k;
            const int below = 31 - __clz(u) - l;
            const int e = a.widest ? s_dim[(u >> below) - 1] : d;
            const int id = s_list[e * SUB_N + p];
            if (below == 0) {
                s_side[id] = SIDE_NODE;
                s_fin[p] = (uint16_t)id;
            } else {
                s_side[id] = u >> (below - 1) & 1 ? SIDE_RIGHT : SIDE_LEFT;
            }
        }
        if (l == t.H)
            break;
        __syncthreads();
        // the other lists, two at a time; e1 < 0: one
        for (int e0 = !a.widest && d == 0 ? 1 : 0; e0 < D;) {
            int e1 = e0 + 1;
            if (e1 == d && !a.widest)
                ++e1;
            int e_next = e1 + 1;
            if (e_next == d && !a.widest)
                ++e_next;
            const bool two = e1 < D;
            uint16_t *la = s_list + e0 * SUB_N, *lb = s_list + (two ? e1 : e0) * SUB_N;
            // ids and sides (12 + 2 bits) of both lists; lefts and nodes at the warp's earlier places
            uint32_t item[SUB_ITEMS], before_a[SUB_ITEMS], before_b[SUB_ITEMS];
            uint32_t run_a = 0, run_b = 0;
#pragma unroll
            for (int k = 0; k < SUB_ITEMS; ++k) {
                uint32_t ia = 0, ib = 0, sa = 3, sb = 3;
                if (node[k] >= level) {
                    ia = la[first + 32 * k];
                    ib = lb[first + 32 * k];
                    sa = s_side[ia];
                    sb = s_side[ib];
                }
                item[k] = ia | sa << 14 | ib << 16 | sb << 30;
                const uint32_t al = __ballot_sync(0xffffffffu, sa == SIDE_LEFT);
                const uint32_t an = __ballot_sync(0xffffffffu, sa == SIDE_NODE);
                const uint32_t bl = __ballot_sync(0xffffffffu, sb == SIDE_LEFT);
                const uint32_t bn = __ballot_sync(0xffffffffu, sb == SIDE_NODE);
                before_a[k] = run_a + (__popc(al & lt) | __popc(an & lt) << 16);
                before_b[k] = run_b + (__popc(bl & lt) | __popc(bn & lt) << 16);
                run_a += __popc(al) | __popc(an) << 16;
                run_b += __popc(bl) | __popc(bn) << 16;
            }
            if (lane == 0) {
                s_cnt[w] = run_a;
                s_cnt[32 + w] = run_b;
            }
            __syncthreads();
            const uint32_t warps_a = __reduce_add_sync(0xffffffffu, lane < w ? s_cnt[lane] : 0);
            const uint32_t warps_b = __reduce_add_sync(0xffffffffu, lane < w ? s_cnt[32 + lane] : 0);
#pragma unroll
            for (int k = 0; k < SUB_ITEMS; ++k) {
                const uint32_t u = node[k];
                if (u < level)
                    continue;
                // as part_dest, once for both lists
                const int p = first + 32 * k;
                const int j = (int)(u >> (31 - __clz(u) - l)) - (1 << l);
                const int s = t.start(l, j), in = s + t.left(l, j), lefts = t.lefts_before(l, j);
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    if (x == 1 && !two)
                        continue;
                    const uint32_t c = x ? warps_b + before_b[k] : warps_a + before_a[k];
                    const uint32_t it = x ? item[k] >> 16 : item[k] & 0xffffu;
                    const int side = it >> 14;
                    const int lbf = (int)(c & 0xffffu) - lefts;
                    const int to = side == SIDE_NODE ? in
                                   : (side == SIDE_LEFT ? s + lbf : in + 1 + (p - s) - lbf - ((int)(c >> 16) - j));
                    if (to >= 0 && to < n)  // always, for consistent sides
                        (x ? lb : la)[to] = (uint16_t)(it & 0xfffu);
                }
            }
            __syncthreads();
            e0 = e_next;
        }
    }
    __syncthreads();
    for (int u = tid; u < n; u += THREADS) {
        const int l = Layout32::level(u), j = u - ((1 << l) - 1);
        // the subtree's root is node job of level `top`
        const int64_t at = ((int64_t)1 << (top + l)) - 1 + ((int64_t)job << l) + j;
        emit_node(a.pts, D, base, at, s_pid[s_fin[t.inorder(u)]],
                  a.widest ? (uint32_t)s_dim[u] << NODE_DIM_SHIFT : 0u, a.nodes, a.ids);
    }
}

template <int SUB_LOG2>
int launch_sub(const SubArgs &a, int64_t jobs, cudaStream_t s)
{
    const size_t smem = sub_smem(a.D, SUB_LOG2);
    // the limit is the kernel's, for all threads: the same value from every
    // call, so that none lowers it between another's setting and its launch
    KDT_CUDA(cudaFuncSetAttribute((const void *)sub_kernel<SUB_LOG2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sub_smem(8, SUB_LOG2)));
    KDT_LAUNCH sub_kernel<SUB_LOG2><<<(unsigned)jobs, (1 << SUB_LOG2) / SUB_ITEMS, smem, s>>>(a);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

// level 0 of a single tree: sides and the root from its split list
__global__ void __launch_bounds__(BT) root_kernel(const uint32_t *__restrict__ list, int n,
                                                  const float *__restrict__ pts, int D, uint8_t *__restrict__ side,
                                                  float4 *__restrict__ nodes, int32_t *__restrict__ ids)
{
    const Layout32 t(n);
    const int in = t.left(0, 0);
    for (int p = blockIdx.x * BT + threadIdx.x; p < n; p += gridDim.x * BT) {
        const uint32_t pid = list[p];
        side[pid] = p < in ? SIDE_LEFT : (p == in ? SIDE_NODE : SIDE_RIGHT);
        if (p == in)
            emit_node(pts, D, 0, 0, pid, 0u, nodes, ids);
    }
}

inline unsigned grid_for(int64_t n)
{
    int64_t b = (n + BT - 1) / BT;
    int64_t cap = (int64_t)num_sms() * 16;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

struct DevBuf {
    void *p = nullptr;
    cudaStream_t s = nullptr;
    ~DevBuf()
    {
        if (p)
            cudaFreeAsync(p, s);
    }
};

}  // namespace

int build_forest(const float *d_points, const int64_t *h_off, int T, int D, float4 *nodes, int32_t *ids, float *bbox,
                 int *err, cudaStream_t s, bool widest, int32_t *h_jobs)
{
    const int64_t total = h_off[T];
    if (total == 0)
        return KDT_OK;
    // levels built by passes over the whole lists, and the blocks of sub_kernel
    const int sub_log2 = sub_log2_of(total);
    int levels = 0;
    int64_t jobs[SUB_CLASSES] = {0, 0, 0};
    for (int i = 0; i < T; ++i) {
        const int64_t n = h_off[i + 1] - h_off[i];
        const int c = T > 1 ? sub_class_of(n, sub_log2) : SUB_CLASSES - 1;
        if (T > 1)
            h_jobs[(size_t)(SUB_CLASSES - 1) * (T + 1) + i] = (int32_t)jobs[SUB_CLASSES - 1];
        if (n < 1)
            continue;
        const int top = top_levels(n, sub_log2);
        levels = std::max(levels, top);
        if (c < SUB_CLASSES - 1)
            h_jobs[(size_t)c * (T + 1) + jobs[c]] = i;
        jobs[c] += (int64_t)1 << top;
    }
    if (T > 1)
        h_jobs[(size_t)(SUB_CLASSES - 1) * (T + 1) + T] = (int32_t)jobs[SUB_CLASSES - 1];

    // Arrays of `total` u32: lists, keys and their temporaries.  Small builds,
    // whose time is their launches, sort all dimensions at once (1.05 M points
    // of 3 dimensions: below the launch's cost from there); large ones one
    // after the other with one temporary.
    const bool together = (int64_t)total * D <= ((int64_t)1 << 21);
    const int at_once = together ? D : 1;
    const int64_t ptiles = (total + PTILE - 1) / PTILE;         // T > 1
    const int top_tiles = (int)top_tiles_of(total), top_groups = (int)top_groups_of(total);  // T == 1
    const size_t rs = radix_scratch_elems(total) * at_once;
    size_t bytes = 0;
    auto take = [&](size_t b) {
        size_t o = bytes;
        bytes += (b + 255) & ~(size_t)255;
        return o;
    };
    // lists [D], list temporaries [at_once], keys and their temporaries
    // [2 at_once]: all but the lists serve the partitions as targets
    const int spares = 3 * at_once;
    size_t o_lists = take((size_t)(D + spares) * total * 4);
    size_t o_side = take((size_t)total * 2);
    size_t o_place = take((size_t)total * 2);
    size_t o_tree = take(T > 1 ? (size_t)total * 4 : 0);
    size_t o_off = take(T > 1 ? (size_t)(T + 1) * 8 : 0);
    const size_t job_bytes = T > 1 ? (size_t)SUB_CLASSES * (T + 1) * 4 : 0;
    size_t o_job = take(job_bytes);
    size_t o_tiles = take(T > 1 ? (size_t)ptiles * sizeof(Seg) : 0);
    size_t o_rs = take(rs * 4);
    // vote words of one launch, counts of every partition
    const int parts = T == 1 ? levels * D : 0;
    const size_t count_bytes = (size_t)parts * (top_tiles + top_groups) * 8;
    size_t o_count = take(count_bytes);
    size_t o_votes = take(parts ? (size_t)TOP_LISTS * top_tiles * TOP_WORDS * sizeof(uint2) : 0);
    size_t o_dim = take(widest ? (size_t)total : 0);
    DevBuf buf;
    buf.s = s;
    KDT_CUDA(cudaMallocAsync(&buf.p, bytes, s));
    char *B = (char *)buf.p;
    uint32_t *arrays = (uint32_t *)(B + o_lists);
    uint32_t *lists[8], *spare[24];
    for (int e = 0; e < D; ++e)
        lists[e] = arrays + (size_t)e * total;
    for (int i = 0; i < spares; ++i)
        spare[i] = arrays + (size_t)(D + i) * total;
    uint8_t *side = (uint8_t *)(B + o_side), *side_next = side + total;
    int32_t *tree_of = T > 1 ? (int32_t *)(B + o_tree) : nullptr;
    int64_t *d_off = T > 1 ? (int64_t *)(B + o_off) : nullptr;
    int32_t *d_job = T > 1 ? (int32_t *)(B + o_job) : nullptr;
    Seg *tiles = (Seg *)(B + o_tiles);
    uint32_t *rscr = (uint32_t *)(B + o_rs);
    uint8_t *node_dim = (uint8_t *)(B + o_dim);

    const unsigned g = grid_for(total);
    if (T > 1) {
        KDT_CUDA(cudaMemcpyAsync(d_off, h_off, (T + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
        for (int c = 0; c < SUB_CLASSES; ++c)
            if (jobs[c])
                KDT_CUDA(cudaMemcpyAsync(d_job + (size_t)c * (T + 1), h_jobs + (size_t)c * (T + 1),
                                         (c < SUB_CLASSES - 1 ? jobs[c] : T + 1) * sizeof(int32_t),
                                         cudaMemcpyHostToDevice, s));
        KDT_LAUNCH tree_of_kernel<<<g, BT, 0, s>>>(d_off, T, total, tree_of);
    }
    int tbits = T > 1 ? floor_log2((uint64_t)(T - 1)) + 1 : 0;

    // per-dimension lists sorted by (tree, coordinate, index)
    for (int e = 0; e < D; e += at_once) {
        uint32_t *k0 = spare[at_once], *k1 = spare[2 * at_once], *v0 = lists[e], *v1 = spare[0];
        KDT_LAUNCH prep_keys_kernel<<<g, BT, 0, s>>>(d_points, total, D, e, at_once, k0, err);
        KDT_TRY(radix_sort_batch(&k0, &v0, &k1, &v1, total, at_once, total, 0, 32, true, rscr, s));
        if (T > 1) {
            for (int i = 0; i < at_once; ++i)
                KDT_LAUNCH tree_keys_kernel<<<g, BT, 0, s>>>(v0 + (size_t)i * total, tree_of, total,
                                                             k0 + (size_t)i * total);
            KDT_TRY(radix_sort_batch(&k0, &v0, &k1, &v1, total, at_once, total, 0, tbits, false, rscr, s));
        }
        // an odd number of passes leaves the result in the temporaries
        if (v0 != lists[e])
            for (int i = 0; i < at_once; ++i)
                std::swap(lists[e + i], spare[i]);
    }
    ListPtrs lp;
    auto list_ptrs = [&]() {
        for (int e = 0; e < 8; ++e)
            lp.p[e] = e < D ? lists[e] : nullptr;
    };
    list_ptrs();
    KDT_LAUNCH bbox_kernel<<<(T + 127) / 128, 128, 0, s>>>(d_points, D, lp, d_off, T, total, bbox);

    if (T == 1) {
        const int n = (int)total;
        unsigned long long *part_count = (unsigned long long *)(B + o_count);
        if (parts)
            KDT_CUDA(cudaMemsetAsync(part_count, 0, count_bytes, s));
        if (levels && !widest)
            KDT_LAUNCH root_kernel<<<g, BT, 0, s>>>(lists[0], n, d_points, D, side, nodes, ids);
        for (int l = 0; l < levels; ++l) {
            const int d = l % D;
            if (widest) {
                list_ptrs();
                KDT_LAUNCH widest_kernel<<<grid_for((int64_t)1 << l), BT, 0, s>>>(lp, total, l, d_points, D, node_dim);
                KDT_LAUNCH assign_widest_kernel<<<g, BT, 0, s>>>(lp, total, l, node_dim, d_points, D, side, nodes);
            } else if (D == 1 && l > 0) {
                // no list is partitioned that could note the next level's sides
                KDT_LAUNCH assign_kernel<<<g, BT, 0, s>>>(lists[0], total, l, sub_log2, 1, nullptr, nullptr, d_points, D, side,
                                                          nodes, ids);
            }
            // the lists to partition, TOP_LISTS or as many as there are spares at a time
            int todo[8], count = 0;
            for (int e = 0; e < D; ++e)
                if (widest || e != d)
                    todo[count++] = e;
            const int step = std::min(TOP_LISTS, spares);
            for (int c = 0; c < count; c += step) {
                const int ny = std::min(step, count - c);
                PartArgs pa;
                pa.next = -1;
                for (int i = 0; i < ny; ++i) {
                    pa.in[i] = lists[todo[c + i]];
                    pa.out[i] = spare[i];
                    if (!widest && l + 1 < levels && todo[c + i] == (l + 1) % D)
                        pa.next = i;
                }
                pa.side = side;
                pa.votes = (uint2 *)(B + o_votes);
                pa.count = part_count;
                part_count += (size_t)ny * (top_tiles + top_groups);
                pa.n = n;
                pa.l = l;
                pa.tiles = top_tiles;
                pa.groups = top_groups;
                pa.side_next = side_next;
                pa.pts = d_points;
                pa.D = D;
                pa.nodes = nodes;
                pa.ids = ids;
                const dim3 grid((unsigned)top_tiles, (unsigned)ny);
                KDT_LAUNCH part_votes_kernel<<<grid, BT, 0, s>>>(pa);
                KDT_LAUNCH part_move_kernel<<<grid, BT, 0, s>>>(pa);
                for (int i = 0; i < ny; ++i)
                    std::swap(lists[todo[c + i]], spare[i]);
            }
            if (!widest && D > 1)
                std::swap(side, side_next);
            KDT_CUDA(cudaGetLastError());
        }
    } else {
        for (int l = 0; l < levels; ++l) {
            const int d = l % D;
            KDT_LAUNCH assign_kernel<<<g, BT, 0, s>>>(lists[d], total, l, sub_log2, T, d_off, tree_of, d_points, D, side, nodes,
                                                      ids);
            for (int e = 0; e < D; ++e) {
                if (e == d)
                    continue;
                KDT_LAUNCH part_reduce_kernel<<<(unsigned)ptiles, BT, 0, s>>>(lists[e], total, l, sub_log2, T, d_off, tree_of,
                                                                              side, tiles);
                KDT_LAUNCH part_tiles_kernel<<<1, 1024, 0, s>>>(tiles, ptiles);
                KDT_LAUNCH part_scatter_kernel<<<(unsigned)ptiles, BT, 0, s>>>(lists[e], total, l, sub_log2, T, d_off, tree_of,
                                                                               side, tiles, spare[0]);
                std::swap(lists[e], spare[0]);
            }
            KDT_CUDA(cudaGetLastError());
        }
    }

    SubArgs sa;
    list_ptrs();
    sa.lists = lp;
    sa.off = d_off;
    sa.total = total;
    sa.T = T;
    sa.D = D;
    sa.widest = widest;
    sa.pts = d_points;
    sa.place = (uint16_t *)(B + o_place);
    sa.nodes = nodes;
    sa.ids = ids;
    for (int c = 0; c < SUB_CLASSES; ++c) {
        if (jobs[c] == 0)
            continue;
        sa.whole_trees = c < SUB_CLASSES - 1;
        sa.first_job = T > 1 ? d_job + (size_t)c * (T + 1) : nullptr;
        if (c == 0)
            KDT_TRY(launch_sub<SUB_LOG2_TINY>(sa, jobs[c], s));
        else if (c == 1 || sub_log2 == SUB_LOG2_SMALL)
            KDT_TRY(launch_sub<SUB_LOG2_SMALL>(sa, jobs[c], s));
        else
            KDT_TRY(launch_sub<SUB_LOG2_LARGE>(sa, jobs[c], s));
    }
    return KDT_OK;
}

}  // namespace kdt
