// Build of the box tree and the kNN kernels that walk it (layout in kdt_box.cuh).
#include <algorithm>
#include <new>

#include "kdt_box.cuh"

namespace kdt {

int grid_for_kernel(const void *fn, int threads, size_t smem);

namespace {

constexpr int BOX_BUILD_THREADS = 256;
constexpr int BOX_TINY_THREADS = 32;  // blocks of a forest's trees of at most as many buckets
constexpr int BOX_THREADS = 128;

template <int NC>
struct Box {
    float lo[NC], hi[NC];
    __device__ __forceinline__ void none()
    {
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            lo[j] = __int_as_float(0x7f800000);
            hi[j] = __int_as_float(0xff800000);
        }
    }
    __device__ __forceinline__ void add(const float (&c)[NC])
    {
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            lo[j] = fminf(lo[j], c[j]);
            hi[j] = fmaxf(hi[j], c[j]);
        }
    }
};

// box of node v into its record
template <int NC>
__device__ __forceinline__ void put_box(float4 *rec, uint32_t v, const Box<NC> &b)
{
    float *r = reinterpret_cast<float *>(rec + (size_t)(v >> 2) * BoxFormat<NC>::REC) + (v & 3u);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        r[8 * j] = b.lo[j];
        r[8 * j + 4] = b.hi[j];
    }
}

// The block's boxes (thread i: node v0 + i of one level, `count` of them, a
// power of two or a multiple of the block) into the records above, four
// levels up the record tree as far as the block holds whole subtrees.
template <int NC, int THREADS>
__device__ __forceinline__ void reduce_boxes(float4 *rec, uint32_t v, int count, Box<NC> b)
{
    __shared__ float s_box[THREADS][2 * NC + 1];
    const int tid = threadIdx.x;
    for (;;) {
        if (tid < count && v > 1)
            put_box<NC>(rec, v, b);
        if (count < 4)
            return;
        __syncthreads();
        if (tid < count) {
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                s_box[tid][j] = b.lo[j];
                s_box[tid][NC + j] = b.hi[j];
            }
        }
        __syncthreads();
        count >>= 2;
        // thread i takes nodes 4i .. 4i + 3 of the block; v of thread 0 is the first
        v = (v - tid) / 4 + tid;
        if (tid < count) {
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                b.lo[j] = fminf(fminf(s_box[4 * tid][j], s_box[4 * tid + 1][j]),
                                fminf(s_box[4 * tid + 2][j], s_box[4 * tid + 3][j]));
                b.hi[j] = fmaxf(fmaxf(s_box[4 * tid][NC + j], s_box[4 * tid + 1][NC + j]),
                                fmaxf(s_box[4 * tid + 2][NC + j], s_box[4 * tid + 3][NC + j]));
            }
        }
    }
}

// Thread i: bucket i.  Finds the node from above that the bucket holds by
// walking down from the root, writes the bucket's groups and box, and the
// block reduces its boxes.  Bound: the gathers of the tree's last four levels
// (each row of a bucket is contiguous, and neighbouring threads read
// neighbouring rows) and the latency of the walk, whose upper nodes are shared
// by the block.
struct BoxBuild {
    const float4 *nodes;
    const int32_t *ids;
    int64_t N;
    int D;
    float4 *rec, *grp;
    // forests: the trees, their first nodes and their first blocks
    int T;
    const BoxRef *trees;
    const int64_t *off;
    const int32_t *first_block;  // or, for whole_trees, the tree of every block
    bool whole_trees;
};

// the block's tree in `a` (nodes, ids, N, rec, grp) and its number within the tree
template <int LAYOUT>
__device__ __forceinline__ uint32_t box_build_tree(BoxBuild &a)
{
    if (a.T == 1)
        return blockIdx.x;
    int lo = 0, hi = a.T - 1;  // last tree that starts at or before the block
    if (a.whole_trees)
        lo = hi = a.first_block[blockIdx.x];
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.first_block[mid] <= (int)blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    const int64_t base = a.off[lo];
    a.N = a.off[lo + 1] - base;
    a.nodes += base * LayoutTraits<LAYOUT>::NF;
    a.ids = a.ids ? a.ids + base : nullptr;
    a.rec = const_cast<float4 *>(a.trees[lo].rec);
    a.grp = const_cast<float4 *>(a.trees[lo].grp);
    return a.whole_trees ? 0 : blockIdx.x - a.first_block[lo];
}

template <int LAYOUT, int THREADS>
__global__ void __launch_bounds__(THREADS) box_leaf_kernel(BoxBuild a)
{
    constexpr int NC = LayoutTraits<LAYOUT>::NC;
    const uint32_t block = box_build_tree<LAYOUT>(a);
    const float4 *__restrict__ nodes = a.nodes;
    const int32_t *__restrict__ ids = a.ids;
    float4 *rec = a.rec, *grp = a.grp;
    const int N = (int)a.N, D = a.D;
    const BoxShape sh(N);
    const uint32_t first = block * THREADS, i = first + threadIdx.x;
    const int count = (int)min((int64_t)THREADS, sh.buckets - (int64_t)first);
    Box<NC> box;
    box.none();
    if ((int64_t)i < sh.buckets) {
        const float nan = __int_as_float(0x7fffffff);
        // the point handed down to this bucket
        float hand[NC];
        uint32_t hand_id = 0xffffffffu;
        bool held = false;
        int dim = 0;
        for (int l = 0; l < sh.LB; ++l) {
            const int t = (int)(((1u << sh.LB) + i) >> (sh.LB - l)) - 1;
            const NodeVal<LAYOUT> nd = fetch<LAYOUT, false>(nodes, nullptr, 0, t);
            const int sd = split_dim_of<LAYOUT>(nd, dim);
            const bool right = i >> (sh.LB - l - 1) & 1u;
            const bool to_right = held && select_dim<NC>(hand, sd) > select_dim<NC>(nd.c, sd);
            if (!held || to_right != right) {
                // the node's own point: to the other side than the one from
                // above, or to the left
                held = held || !right;
                if (held) {
#pragma unroll
                    for (int j = 0; j < NC; ++j)
                        hand[j] = nd.c[j];
                    hand_id = LAYOUT == 0 ? nd.id : (LAYOUT == 3 ? nd.id & NODE_ID_MASK : (uint32_t)ids[t]);
                }
            }
            dim = dim + 1 == D ? 0 : dim + 1;
        }
        const int root = (1 << sh.LB) - 1 + (int)i;
        const int groups = sh.count(i);
        float4 *g = grp + (size_t)sh.group(i) * BoxFormat<NC>::GRP;
        for (int k = 0; k < groups; ++k, g += BoxFormat<NC>::GRP) {
            float c[NC][BOX_GROUP];
            uint32_t id[BOX_GROUP];
#pragma unroll
            for (int m = 0; m < BOX_GROUP; ++m) {
                const int node = bucket_node(root, k, m);
                const bool above = k == 0 && m == 7;
                const bool ok = above ? held : node < N;
                if (!above && ok) {
                    const NodeVal<LAYOUT> nd = fetch<LAYOUT, false>(nodes, nullptr, 0, node);
#pragma unroll
                    for (int j = 0; j < NC; ++j)
                        c[j][m] = nd.c[j];
                    id[m] = LAYOUT == 0 ? nd.id : (LAYOUT == 3 ? nd.id & NODE_ID_MASK : (uint32_t)ids[node]);
                } else {
#pragma unroll
                    for (int j = 0; j < NC; ++j)
                        c[j][m] = ok ? hand[j] : nan;
                    id[m] = ok ? hand_id : 0xffffffffu;
                }
                // fminf / fmaxf pass over the NaN of an empty place
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    box.lo[j] = fminf(box.lo[j], c[j][m]);
                    box.hi[j] = fmaxf(box.hi[j], c[j][m]);
                }
            }
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                g[2 * j] = make_float4(c[j][0], c[j][1], c[j][2], c[j][3]);
                g[2 * j + 1] = make_float4(c[j][4], c[j][5], c[j][6], c[j][7]);
            }
            uint4 *gi = reinterpret_cast<uint4 *>(g + 2 * NC);
            gi[0] = make_uint4(id[0], id[1], id[2], id[3]);
            gi[1] = make_uint4(id[4], id[5], id[6], id[7]);
        }
    }
    if (sh.LB > 0)
        reduce_boxes<NC, THREADS>(rec, (uint32_t)sh.buckets + i, count, box);
}

// Thread i: node i of the level `up` levels above the buckets, whose records
// are complete
template <int LAYOUT>
__global__ void __launch_bounds__(BOX_BUILD_THREADS) box_upper_kernel(BoxBuild a, int up)
{
    constexpr int NC = LayoutTraits<LAYOUT>::NC;
    const uint32_t block = box_build_tree<LAYOUT>(a);
    float4 *rec = a.rec;
    const uint32_t v0 = 1u << (BoxShape(a.N).LB - up);
    const uint32_t first = block * BOX_BUILD_THREADS, i = first + threadIdx.x;
    const int count = (int)min((uint32_t)BOX_BUILD_THREADS, v0 - first);
    Box<NC> box;
    box.none();
    if (i < v0) {
        const float4 *r = rec + (size_t)(v0 + i) * BoxFormat<NC>::REC;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const float4 lo = r[2 * j], hi = r[2 * j + 1];
            box.lo[j] = fminf(fminf(lo.x, lo.y), fminf(lo.z, lo.w));
            box.hi[j] = fmaxf(fmaxf(hi.x, hi.y), fmaxf(hi.z, hi.w));
        }
    }
    reduce_boxes<NC, BOX_BUILD_THREADS>(rec, v0 + i, count, box);
}

// ---- kNN
//
// Persistent lanes, a query each, as in the state machine's kernel; a warp
// alternates between records (while more than BOX_RECORD_LANES of its lanes
// are on one) and the buckets that its lanes have reached, and takes new
// queries when BOX_FREE_LANES lanes are free.  Both are sweet spots of a sweep
// on all kNN cases (records 0 / 4 / 8 / 16 / 24, free 1 / 4 / 8 / 16 / 24): a
// bucket costs several records, so few lanes should be kept from it, and the
// claim, the row's store and the new query's first bucket run best with most
// lanes taking part (free 8 -> 24: surface k = 16 4.17 -> 3.78 ms, closest
// point in 4-D 6.81 -> 6.58 ms).
//
// Bound: the arithmetic and selects of buckets and lists in 3-D with k >= 8
// (12 to 14 of 32 lanes active), L1 wavefronts in 4-D with incoherent queries
// (98 %).  Whole passes against the state machine's kernel: clustered 2^24, k = 8
// 1060 -> 19.2 ms (13.3 k processed nodes a query -> 56 records and 14 buckets),
// surface 4 M, k = 16 10.3 -> 2.76 ms, 8-D k = 10 24.4 -> 4.49 ms, 10^7 closest
// points in 4-D 8.76 -> 5.24 ms, a scan of 5003 closest points 46 -> 25 us.  The
// state machine is not faster on any of them.
constexpr int BOX_RECORD_LANES = 4;
constexpr int BOX_FREE_LANES = 24;
// With the heap (K > 16), whose set-up and final sort cost most, nearly the
// whole warp (k = 40 2.60 -> 2.47 ms); in 5 to 8 dimensions, where a walk is 470
// steps and a lane that waits is the dearer part, a quarter (8-D 4.81 -> 4.61).
__host__ __device__ constexpr int box_free_lanes(int layout, int k) { return k > MAX_REG_K ? 31 : (layout == 2 ? 8 : BOX_FREE_LANES); }

// Resident blocks to build for.  Closest points in 4-D, bound by L1 wavefronts
// whose latency more warps cover: 10 (10^7 of them 5.58 -> 5.33 ms against 8; in
// 3-D 10 costs a scan of 5003 24.5 -> 27 us).  3-D: 7 to k = 8 (forest 2.32 -> 2.28
// ms against 6), 6 at k = 16 (surface 2.85 -> 2.77 ms against 5).  Elsewhere the
// registers that more blocks leave are too few (spills).
constexpr int box_blocks_per_sm(int layout, int k)
{
    return k <= 1 ? (layout == 1 ? 10 : (layout == 0 ? 8 : 6)) : (k <= 8 ? (layout == 0 ? 7 : 6) : (k <= 16 && layout == 0 ? 6 : 1));
}

// No distance to a NaN query passes a test, but every box's would: the maximum
// that clamps its coordinates at 0 drops the NaN.  Such a query is not walked.
template <int NC>
__device__ __forceinline__ bool is_nan(const float (&q)[NC])
{
    bool nan = false;
#pragma unroll
    for (int j = 0; j < NC; ++j)
        nan = nan || q[j] != q[j];
    return nan;
}

// FOREST: a lane's query finds its tree by its place in the query offsets.
template <int LAYOUT, int K, int MODE, bool FOREST>
__global__ void __launch_bounds__(BOX_THREADS, box_blocks_per_sm(LAYOUT, K)) box_knn_kernel(const QueryArgs a, const BoxArgs b)
{
    constexpr int NC = LayoutTraits<LAYOUT>::NC;
    using List = typename std::conditional<(K <= MAX_REG_K), RegList<K <= MAX_REG_K ? K : 1>, SmemList>::type;
    extern __shared__ float4 s_dyn[];
    constexpr int FREE_LANES = box_free_lanes(LAYOUT, K);
    const int64_t ngate = (MODE == MODE_BOUNDED && a.n_gate) ? (int64_t)*a.n_gate : INT64_MAX;
    uint32_t cap = a.step_cap ? a.step_cap : 3u * (uint32_t)a.N + 3u;
    BoxRef tree = b.tree;
    bool gated = false;
    double ratio = 0.0;
    float q[NC];
    float r2 = 0.f;
    List list;
    float *const s_far = reinterpret_cast<float *>(s_dyn) + threadIdx.x;
    const int stride = blockDim.x;
    const f32x2 one = pair(b.one, b.one);
    if constexpr (K > MAX_REG_K) {
        if (a.heap) {
            list.s = a.heap + ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * (size_t)a.k;
            list.stride = 1;
        } else {
            list.s = reinterpret_cast<unsigned long long *>(s_dyn) + BoxWalk::MAX_RECORDS / 2 * stride + threadIdx.x;
            list.stride = stride;
        }
    }
    BoxWalk w;
    w.v = 0;
    uint32_t steps = 0;
    // the first query of a lane is its place in the grid, the next ones are claimed
    int64_t qi = -1;
    bool busy = false, first = true, exhausted = false;
    const int64_t lanes = (int64_t)gridDim.x * blockDim.x;
    for (;;) {
        const unsigned free_lanes = __ballot_sync(0xffffffffu, !busy && !exhausted);
        const unsigned busy_lanes = __ballot_sync(0xffffffffu, busy);
        if (!busy_lanes || __popc(free_lanes) >= FREE_LANES) {
            // write the finished rows, take the next queries
            if (!busy && qi >= 0) {
                bool again = false;
                if constexpr (MODE == MODE_BOUNDED) {
                    const bool full = list.full(a.k);
                    // exact when the list is full or the proposal did not
                    // shrink the radius; else once more with the caller's
                    again = steps <= cap && !(full || r2 == a.r2);
                    if (again) {
                        atomicAdd(a.fb_count, 1ull);
                        gated = false;
                        r2 = a.r2;
                        list.init(a.k, r2);
                        w.start(tree.leaf, s_far);
                        steps = 0;
                        busy = again = !is_nan(q);
                    } else if (gated && full && list.cull() > 0.f && r2 < __int_as_float(0x7f800000)) {
                        ratio += sqrt((double)r2 / (double)list.cull());
                    }
                }
                if (!again) {
                    if (steps > cap)
                        atomicOr(a.err, ERR_TRAVERSAL);
                    list.store(a.k, a.out_ids + qi * a.k, a.out_d2 + qi * a.k);
                    qi = -1;
                }
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
                    gated = MODE == MODE_BOUNDED && slot < ngate;
                    r2 = gated ? a.r2q[qi] : a.r2;
                    if constexpr (FOREST) {
                        int lo = 0, hi = a.T - 1;  // last tree whose queries start at or before qi
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (a.q_off[mid] <= qi)
                                lo = mid;
                            else
                                hi = mid - 1;
                        }
                        tree = b.trees[lo];
                        cap = 3u * (uint32_t)(a.node_off[lo + 1] - a.node_off[lo]) + 3u;
                    }
                    load_query<LAYOUT>(a.queries, qi, a.D, q);
                    list.init(a.k, r2);
                    w.start(tree.leaf, s_far);
                    steps = 0;
                    busy = !is_nan(q) && (!FOREST || tree.leaf > 0);
                } else {
                    exhausted = true;
                }
            }
            first = false;
            if (__all_sync(0xffffffffu, !busy && exhausted && qi < 0))
                break;
        }
        // records, until few lanes are left on them
        for (;;) {
            if (busy && w.v < tree.leaf) {
                ++steps;
                busy = w.template step<NC>(tree.rec, q, one, list.cull(), stride);
            }
            if (__popc(__ballot_sync(0xffffffffu, busy && w.v < tree.leaf)) <= BOX_RECORD_LANES)
                break;
        }
        if (busy && w.v >= tree.leaf) {
            ++steps;
            box_bucket<NC, K>(tree, w.v - tree.leaf, q, one, list);
            busy = w.pop(list.cull(), stride);
        }
        if (steps > cap)
            busy = false;
    }
    if (MODE == MODE_BOUNDED) {
        for (int o = 16; o > 0; o >>= 1)
            ratio += __shfl_down_sync(0xffffffffu, ratio, o);
        if ((threadIdx.x & 31) == 0 && ratio != 0.0)
            atomicAdd(a.ratio_sum, ratio);
    }
}

template <int LAYOUT, int K, int MODE, bool FOREST>
int launch_box_one(const QueryArgs &a, const BoxArgs &b, cudaStream_t s)
{
    const void *fn = (const void *)box_knn_kernel<LAYOUT, K, MODE, FOREST>;
    // few queries: small blocks, so that they spread over the SMs; heaps in
    // shared memory: half blocks fill it better (k = 40 2.47 -> 2.40 ms)
    int threads = K > MAX_REG_K ? BOX_THREADS / 2 : BOX_THREADS;
    while (threads > 32 && a.Q < (int64_t)num_sms() * threads)
        threads >>= 1;
    const size_t smem = (size_t)threads * (4 * BoxWalk::MAX_RECORDS + (K > MAX_REG_K && !a.heap ? 8 * a.k : 0));
    static_assert(BOX_THREADS / 2 * (4 * BoxWalk::MAX_RECORDS + 8 * 64) <= 48 * 1024 &&
                      BOX_THREADS * 4 * BoxWalk::MAX_RECORDS <= 48 * 1024,
                  "the lists fit without a raised limit");
    int64_t grid = grid_for_kernel(fn, threads, smem);
    if (a.heap)
        grid = std::max<int64_t>(1, std::min<int64_t>(grid, a.heap_threads / threads));
    grid = std::min<int64_t>(grid, (a.Q + threads - 1) / threads);
    if (grid * threads < a.Q)
        KDT_CUDA(cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s));
    KDT_LAUNCH box_knn_kernel<LAYOUT, K, MODE, FOREST><<<(unsigned)grid, threads, smem, s>>>(a, b);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

template <int LAYOUT, int MODE, bool FOREST>
int launch_box_k(const QueryArgs &a, const BoxArgs &b, cudaStream_t s)
{
    if (a.k <= 1)
        return launch_box_one<LAYOUT, 1, MODE, FOREST>(a, b, s);
    if (a.k <= 2)
        return launch_box_one<LAYOUT, 2, MODE, FOREST>(a, b, s);
    if (a.k <= 4)
        return launch_box_one<LAYOUT, 4, MODE, FOREST>(a, b, s);
    if (a.k <= 8)
        return launch_box_one<LAYOUT, 8, MODE, FOREST>(a, b, s);
    if (a.k <= 16)
        return launch_box_one<LAYOUT, 16, MODE, FOREST>(a, b, s);
    return launch_box_one<LAYOUT, 64, MODE, FOREST>(a, b, s);
}

// A block writes the boxes of five levels of the record tree (256 nodes and
// their 64, 16, 4 and 1 ancestors), the next launch starts above them; `blocks`
// and `first` (device, T > 1) of each launch.  Launch BOX_TINY is for a forest's
// trees of at most 32 buckets: a warp holds the whole of one (100 000 clouds of
// 10 points: 587 us in blocks of 256 that search their tree, 57 in warps that are given it).
constexpr int BOX_LAUNCH_LEVELS = 10;
constexpr int BOX_TINY = BOX_LAUNCHES - 1;

// adds the blocks of every launch for a tree of n points, one of a forest's or
// the only one
void add_box_blocks(int64_t n, bool forest, int64_t *blocks)
{
    const BoxShape sh(n);
    if (n < 1)
        return;
    if (forest && sh.buckets <= BOX_TINY_THREADS) {
        ++blocks[BOX_TINY];
        return;
    }
    for (int r = 0, level = sh.LB; r == 0 || level >= 1; ++r, level -= BOX_LAUNCH_LEVELS)
        blocks[r] += (((int64_t)1 << level) + BOX_BUILD_THREADS - 1) / BOX_BUILD_THREADS;
}

template <int LAYOUT>
int build_box_layout(BoxBuild a, const int64_t *blocks, const int32_t *const *first, cudaStream_t s)
{
    for (int r = 0; r < BOX_LAUNCHES; ++r) {
        if (blocks[r] == 0)
            continue;
        a.first_block = first[r];
        a.whole_trees = r == BOX_TINY;
        if (r == BOX_TINY)
            KDT_LAUNCH box_leaf_kernel<LAYOUT, BOX_TINY_THREADS><<<(unsigned)blocks[r], BOX_TINY_THREADS, 0, s>>>(a);
        else if (r == 0)
            KDT_LAUNCH box_leaf_kernel<LAYOUT, BOX_BUILD_THREADS><<<(unsigned)blocks[r], BOX_BUILD_THREADS, 0, s>>>(a);
        else
            KDT_LAUNCH box_upper_kernel<LAYOUT><<<(unsigned)blocks[r], BOX_BUILD_THREADS, 0, s>>>(
                a, BOX_LAUNCH_LEVELS * r);
        KDT_CUDA(cudaGetLastError());
    }
    return KDT_OK;
}

int build_boxes(int layout, const BoxBuild &a, const int64_t *blocks, const int32_t *const *first, cudaStream_t s)
{
    switch (layout) {
    case 0: return build_box_layout<0>(a, blocks, first, s);
    case 1: return build_box_layout<1>(a, blocks, first, s);
    case 3: return build_box_layout<3>(a, blocks, first, s);
    default: return build_box_layout<2>(a, blocks, first, s);
    }
}

// float4s of a tree's records, rounded up to a 128-byte line, and of its groups
size_t box_rec_size(int64_t n, int D) { return ((size_t)BoxShape(n).records() * 2 * box_coords(D) + 7) & ~(size_t)7; }
size_t box_grp_size(int64_t n, int D) { return (size_t)BoxShape(n).groups() * 2 * (box_coords(D) + 1); }
// of a forest's tree: the next one starts on a 128-byte line too
size_t box_tree_size(int64_t n, int D) { return (box_rec_size(n, D) + box_grp_size(n, D) + 7) & ~(size_t)7; }

}  // namespace

size_t box_tree_bytes(int64_t n, int D) { return (box_rec_size(n, D) + box_grp_size(n, D)) * sizeof(float4); }

void box_tree_place(kdt_tree *t, void *p)
{
    t->box_rec = (float4 *)p;
    t->box_grp = t->box_rec + box_rec_size(t->N, t->D);
}

int build_box_tree(const kdt_tree *t, cudaStream_t s)
{
    BoxBuild a = {t->nodes, t->ids, t->N, t->D, t->box_rec, t->box_grp, 1, nullptr, nullptr, nullptr, false};
    int64_t blocks[BOX_LAUNCHES] = {};
    const int32_t *first[BOX_LAUNCHES] = {};
    add_box_blocks(t->N, false, blocks);
    return build_boxes(t->layout, a, blocks, first, s);
}

int build_box_forest(kdt_forest *f, cudaStream_t s)
{
    const int T = f->f.T, D = f->f.D;
    // [records and groups of every tree][BoxRef of every tree][first blocks of every launch]
    BoxRef *ref = new (std::nothrow) BoxRef[T];
    if (!ref)
        return set_error(KDT_ENOMEM, "host allocation failed");
    f->box_host = ref;
    int32_t *first = f->h_first + (size_t)SUB_CLASSES * (T + 1);  // behind the builder's
    size_t at = 0;
    int64_t blocks[BOX_LAUNCHES] = {};
    for (int i = 0; i < T; ++i) {
        const int64_t n = f->h_offsets[i + 1] - f->h_offsets[i];
        for (int r = 0; r < BOX_TINY; ++r)
            first[(size_t)r * (T + 1) + i] = (int32_t)blocks[r];
        first[(size_t)BOX_TINY * (T + 1) + blocks[BOX_TINY]] = i;  // stands if the tree is such a one
        add_box_blocks(n, true, blocks);
        at += n ? box_tree_size(n, D) : 0;
    }
    for (int r = 0; r < BOX_TINY; ++r)
        first[(size_t)r * (T + 1) + T] = (int32_t)blocks[r];
    const size_t first_bytes = (size_t)BOX_LAUNCHES * (T + 1) * sizeof(int32_t);
    const size_t data = at * sizeof(float4), refs = (size_t)T * sizeof(BoxRef);
    char *p = nullptr;
    const size_t bytes = data + refs + first_bytes;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        // the builder's scratch, freed but kept by the stream-ordered pool, may
        // be what is missing: give it back and try again
        cudaGetLastError();
        KDT_CUDA(cudaStreamSynchronize(s));
        cudaMemPool_t pool;
        int dev = 0;
        KDT_CUDA(cudaGetDevice(&dev));
        KDT_CUDA(cudaDeviceGetDefaultMemPool(&pool, dev));
        KDT_CUDA(cudaMemPoolTrimTo(pool, 0));
        e = cudaMalloc(&p, bytes);
    }
    KDT_CUDA(e);
    f->box_data = (float4 *)p;
    f->box_refs = p + data;
    at = 0;
    for (int i = 0; i < T; ++i) {
        const int64_t n = f->h_offsets[i + 1] - f->h_offsets[i];
        ref[i] = n ? box_ref(n, f->box_data + at, f->box_data + at + box_rec_size(n, D)) : BoxRef{nullptr, nullptr, 0, 0};
        at += n ? box_tree_size(n, D) : 0;
    }
    KDT_CUDA(cudaMemcpyAsync(p + data, ref, refs, cudaMemcpyHostToDevice, s));
    BoxBuild a = {f->nodes, f->ids, f->f.total, D, nullptr, nullptr, T, (const BoxRef *)f->box_refs, f->f.d_offsets,
                  nullptr, false};
    if (T == 1 && f->f.total) {
        a.rec = const_cast<float4 *>(ref[0].rec);
        a.grp = const_cast<float4 *>(ref[0].grp);
    }
    int32_t *d_first[BOX_LAUNCHES];
    for (int r = 0; r < BOX_LAUNCHES; ++r) {
        d_first[r] = (int32_t *)(p + data + refs) + (size_t)r * (T + 1);
        if (blocks[r])
            KDT_CUDA(cudaMemcpyAsync(d_first[r], first + (size_t)r * (T + 1),
                                     (r == BOX_TINY ? blocks[r] : T + 1) * sizeof(int32_t), cudaMemcpyHostToDevice,
                                     s));
    }
    return build_boxes(layout_of(D), a, blocks, d_first, s);
}

int launch_box_query(int layout, const BoxRef &tree, const QueryArgs &a, int mode, cudaStream_t s)
{
    BoxArgs b;
    b.tree = tree;
    const bool bounded = mode == MODE_BOUNDED;
    // the groups hold coordinates and ids alike for layouts 0 and 3
    switch (layout) {
    case 0:
    case 3:
        return bounded ? launch_box_k<0, MODE_BOUNDED, false>(a, b, s) : launch_box_k<0, MODE_RESULTS, false>(a, b, s);
    case 1: return launch_box_k<1, MODE_RESULTS, false>(a, b, s);
    default: return launch_box_k<2, MODE_RESULTS, false>(a, b, s);
    }
}

int launch_box_forest(const kdt_forest *f, const QueryArgs &a, cudaStream_t s)
{
    BoxArgs b;
    b.trees = (const BoxRef *)f->box_refs;
    switch (layout_of(f->f.D)) {
    case 0: return launch_box_k<0, MODE_RESULTS, true>(a, b, s);
    case 1: return launch_box_k<1, MODE_RESULTS, true>(a, b, s);
    default: return launch_box_k<2, MODE_RESULTS, true>(a, b, s);
    }
}

}  // namespace kdt
