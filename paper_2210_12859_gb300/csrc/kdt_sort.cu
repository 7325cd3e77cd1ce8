// Device-wide primitives used by the builder and the query reordering:
// an exclusive prefix sum (three-phase: per-tile reduce, scan of the tile
// totals, per-tile scan) and a stable LSD radix sort of (u32 key, u32 value)
// pairs, 8 bits and one kernel per pass.
#include <algorithm>

#include "kdt_internal.cuh"

namespace kdt {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
static_assert(SCAN_TILE == SCAN_TILE_ELEMS, "scan tile and the scratch-size formula disagree");

constexpr int RADIX_THREADS = 256;
static_assert(RADIX_THREADS == RADIX_BLOCK, "radix tile and the scratch-size formula disagree");
constexpr int RADIX_WARPS = RADIX_THREADS / 32;

template <typename T>
__device__ __forceinline__ T warp_inclusive_sum(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o)
            v += u;
    }
    return v;
}

// exclusive block scan of one value per thread; returns the exclusive prefix
// and writes the block total to *total (all threads)
template <typename T>
__device__ __forceinline__ T block_exclusive_sum(T v, T *s_warp, T *total)
{
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T inc = warp_inclusive_sum(v);
    if (lane == 31)
        s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        T x = lane < nw ? s_warp[lane] : T(0);
        T xi = warp_inclusive_sum(x);
        if (lane < nw)
            s_warp[lane] = xi - x;
        if (lane == nw - 1)
            s_warp[32] = xi;
    }
    __syncthreads();
    T r = s_warp[w] + inc - v;
    *total = s_warp[32];
    __syncthreads();
    return r;
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) scan_reduce_kernel(const T *__restrict__ data, int64_t n,
                                                                     T *__restrict__ partials)
{
    __shared__ T s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    T sum = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        int64_t i = base + (int64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n)
            sum += data[i];
    }
    T total;
    block_exclusive_sum(sum, s_warp, &total);
    if (threadIdx.x == 0)
        partials[blockIdx.x] = total;
}

// single block: exclusive scan of the tile totals, in chunks
template <typename T>
__global__ void __launch_bounds__(1024) scan_partials_kernel(T *__restrict__ partials, int64_t np)
{
    __shared__ T s_warp[33];
    T carry = 0;
    for (int64_t base = 0; base < np; base += 1024) {
        int64_t i = base + threadIdx.x;
        T v = i < np ? partials[i] : T(0);
        T total;
        T ex = block_exclusive_sum(v, s_warp, &total);
        if (i < np)
            partials[i] = carry + ex;
        carry += total;
    }
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) scan_downsweep_kernel(T *__restrict__ data, int64_t n,
                                                                        const T *__restrict__ partials)
{
    __shared__ T s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T v[SCAN_ITEMS];
    T sum = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        int64_t i = base + j;
        v[j] = i < n ? data[i] : T(0);
        sum += v[j];
    }
    T total;
    T run = block_exclusive_sum(sum, s_warp, &total) + partials[blockIdx.x];
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        int64_t i = base + j;
        if (i < n)
            data[i] = run;
        run += v[j];
    }
}

template <typename T>
int exclusive_scan_t(T *data, int64_t n, T *scratch, cudaStream_t s)
{
    if (n <= 0)
        return KDT_OK;
    int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    KDT_LAUNCH scan_reduce_kernel<T><<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(data, n, scratch);
    KDT_LAUNCH scan_partials_kernel<T><<<1, 1024, 0, s>>>(scratch, tiles);
    KDT_LAUNCH scan_downsweep_kernel<T><<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(data, n, scratch);
    KDT_CUDA(cudaGetLastError());
    return KDT_OK;
}

// ---- radix sort
//
// Stable LSD sort, 8 bits a pass.  One kernel reads the keys once and counts
// the digits of all passes; then every pass is one kernel that reads each
// (key, value) pair once and writes it once: a block ranks its tile in
// registers and shared memory, learns how many equal digits the tiles before
// it hold by looking back through their published counts, and writes the tile
// through shared memory so that equal digits leave in runs.
//
// Bound: memory, 16 bytes a pair and pass, for large sorts; the latency of a
// pass's chain (load, rank, look-back, write) for small ones.  Against the
// passes it replaced (a histogram kernel, three scan kernels and a scatter
// that wrote every pair by itself, 20 launches a sort), the order of
// 10^7 queries takes 0.54 ms instead of 0.85 and that of 2^14 queries 43 us
// instead of 115.

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Digit counts of all passes, one read of the keys.  blockIdx.y: the array.
__global__ void __launch_bounds__(RADIX_THREADS) radix_hist_kernel(const uint32_t *__restrict__ keys, int64_t n,
                                                                     int64_t stride, int lo_bit, int passes,
                                                                     uint32_t *__restrict__ hist)
{
    __shared__ uint32_t s_cnt[RADIX_MAX_PASSES * 256];
    for (int i = threadIdx.x; i < passes * 256; i += RADIX_THREADS)
        s_cnt[i] = 0;
    __syncthreads();
    const uint32_t *k = keys + blockIdx.y * stride;
    const int64_t step = (int64_t)gridDim.x * RADIX_THREADS;
    for (int64_t i = (int64_t)blockIdx.x * RADIX_THREADS + threadIdx.x; i < n; i += step) {
        const uint32_t key = k[i] >> lo_bit;
        for (int p = 0; p < passes; ++p)
            atomicAdd(&s_cnt[p * 256 + ((key >> (8 * p)) & 255u)], 1u);
    }
    __syncthreads();
    uint32_t *h = hist + (int64_t)blockIdx.y * RADIX_MAX_PASSES * 256;
    for (int i = threadIdx.x; i < passes * 256; i += RADIX_THREADS)
        if (s_cnt[i])
            atomicAdd(&h[i], s_cnt[i]);
}

// A tile's published count of one digit: nothing yet, the tile's own count, or
// the count over the tile and all before it.
constexpr unsigned long long ST_NONE = 0, ST_OWN = 1ull << 62, ST_ALL = 2ull << 62, ST_VALUE = (1ull << 62) - 1;
// polls of one predecessor before its count is taken from its keys instead
constexpr int RADIX_POLLS = 1 << 16;

// Tiles are numbered by the order in which their blocks start, so every
// predecessor of a running tile is running or done and publishes without
// waiting for a later one.  A predecessor that has still published nothing
// after RADIX_POLLS reads is counted from its keys: the wait is bounded and
// the result does not depend on it.
// IOTA: the values of the first pass are the positions.
template <int ITEMS, bool IOTA>
__global__ void __launch_bounds__(RADIX_THREADS, 4) radix_pass_kernel(
    const uint32_t *__restrict__ keys_, const uint32_t *__restrict__ vals_, uint32_t *__restrict__ keys_out_,
    uint32_t *__restrict__ vals_out_, int64_t n, int64_t stride, int shift, int64_t tiles,
    const uint32_t *__restrict__ hist_, unsigned long long *__restrict__ state_, uint32_t *__restrict__ ticket)
{
    constexpr int TILE = RADIX_THREADS * ITEMS;
    __shared__ uint32_t s_warp[RADIX_WARPS][256];
    __shared__ uint32_t s_key[TILE], s_val[TILE];
    __shared__ unsigned long long s_to[256];  // where the tile's run of a digit goes, less its start in the tile
    __shared__ uint32_t s_scan[33];
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (tid == 0)
        s_tile = atomicAdd(ticket + blockIdx.y, 1u);
    for (int i = tid; i < RADIX_WARPS * 256; i += RADIX_THREADS)
        (&s_warp[0][0])[i] = 0;
    __syncthreads();
    const int64_t tile = s_tile;
    const uint32_t *keys = keys_ + blockIdx.y * stride;
    const uint32_t *vals = IOTA ? nullptr : vals_ + blockIdx.y * stride;
    unsigned long long *state = state_ + (int64_t)blockIdx.y * tiles * 256;
    const int64_t base = tile * TILE;
    const int count = (int)(n - base < TILE ? n - base : TILE);

    // a warp owns 32 ITEMS consecutive pairs, item j of lane i at 32 j + i
    const int first = w * 32 * ITEMS + lane;
    uint32_t key[ITEMS], val[ITEMS];
    uint32_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int i = first + 32 * j;
        key[j] = i < count ? keys[base + i] : 0xffffffffu;
        if constexpr (IOTA)
            val[j] = (uint32_t)(base + i);
        else
            val[j] = i < count ? vals[base + i] : 0;
    }
    // rank among the warp's equal digits, in order
    const uint32_t lt = lanemask_lt();
    // (equal digits by eight votes: 16 in a row overlap, where match_any waits;
    // with the bound of four blocks an SM a pass of 2^24 pairs 0.20 -> 0.15 ms)
    uint32_t peer[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
    {
        const bool valid = first + 32 * j < count;
        const uint32_t d = key[j] >> shift;
        uint32_t m = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int bit = 0; bit < 8; ++bit) {
            const bool one = d >> bit & 1u;
            const uint32_t v = __ballot_sync(0xffffffffu, one);
            m &= one ? v : ~v;
        }
        peer[j] = m;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool valid = first + 32 * j < count;
        const uint32_t d = (key[j] >> shift) & 255u;
        uint32_t at = 0;
        if (valid)
            at = s_warp[w][d];
        __syncwarp();
        if (valid && (peer[j] & lt) == 0)
            s_warp[w][d] = at + __popc(peer[j]);
        __syncwarp();
        rank[j] = at + __popc(peer[j] & lt);
    }
    __syncthreads();
    // thread tid: digit tid.  Counts of the warps before each warp, the
    // tile's count, and the digit's first place in the sorted tile
    uint32_t mine = 0;
#pragma unroll
    for (int v = 0; v < RADIX_WARPS; ++v) {
        const uint32_t c = s_warp[v][tid];
        s_warp[v][tid] = mine;
        mine += c;
    }
    volatile unsigned long long *st = state;
    st[tile * 256 + tid] = (tile ? ST_OWN : ST_ALL) | mine;
    uint32_t total;
    const uint32_t in_tile = block_exclusive_sum(mine, s_scan, &total);
    const uint32_t all = hist_[(int64_t)blockIdx.y * RADIX_MAX_PASSES * 256 + tid];
    // pairs with a smaller digit (below n < 2^32), then pairs of this digit in earlier tiles
    const uint32_t smaller = block_exclusive_sum(all, s_scan, &total);
    unsigned long long before = 0;
    for (int64_t t = tile - 1; t >= 0; --t) {
        unsigned long long v = ST_NONE;
        for (int polls = 0; polls < RADIX_POLLS; ++polls) {
            v = st[t * 256 + tid];
            if (v != ST_NONE)
                break;
        }
        if (v == ST_NONE) {
            unsigned long long c = 0;
            for (int64_t i = t * TILE; i < (t + 1) * TILE; ++i)
                c += ((keys[i] >> shift) & 255u) == (uint32_t)tid;
            v = ST_OWN | c;
        }
        before += v & ST_VALUE;
        if (v & ST_ALL)
            break;
    }
    if (tile)
        st[tile * 256 + tid] = ST_ALL | (before + mine);
    s_to[tid] = smaller + before - in_tile;
#pragma unroll
    for (int v = 0; v < RADIX_WARPS; ++v)
        s_warp[v][tid] += in_tile;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
        if (first + 32 * j < count) {
            const uint32_t r = s_warp[w][(key[j] >> shift) & 255u] + rank[j];
            s_key[r] = key[j];
            s_val[r] = val[j];
        }
    __syncthreads();
    uint32_t *keys_out = keys_out_ + blockIdx.y * stride, *vals_out = vals_out_ + blockIdx.y * stride;
    for (int i = tid; i < count; i += RADIX_THREADS) {
        const uint32_t k = s_key[i];
        const unsigned long long dst = s_to[(k >> shift) & 255u] + (uint32_t)i;
        if (dst < (unsigned long long)n) {  // always, for a consistent histogram
            keys_out[dst] = k;
            vals_out[dst] = s_val[i];
        }
    }
}

}  // namespace

size_t scan_scratch_elems(int64_t n)
{
    return scan_scratch_elems_of(n);
}

int exclusive_scan_u64(unsigned long long *data, int64_t n, unsigned long long *scratch, cudaStream_t s)
{
    return exclusive_scan_t<unsigned long long>(data, n, scratch, s);
}

size_t radix_scratch_elems(int64_t n)
{
    return radix_scratch_elems_of(n);
}

namespace {

template <int ITEMS>
int radix_passes(uint32_t *&ka, uint32_t *&va, uint32_t *&kb, uint32_t *&vb, int64_t n, int batch, int64_t stride,
                 int lo_bit, int passes, bool iota, const uint32_t *hist, unsigned long long *state,
                 uint32_t *ticket, cudaStream_t s)
{
    const int64_t tiles = radix_tiles_of(n);
    const dim3 grid((unsigned)tiles, (unsigned)batch);
    for (int p = 0; p < passes; ++p) {
        const uint32_t *h = hist + 256 * p;
        unsigned long long *st = state + (int64_t)p * batch * tiles * 256;
        uint32_t *tk = ticket + p * batch;
        if (iota && p == 0)
            KDT_LAUNCH radix_pass_kernel<ITEMS, true><<<grid, RADIX_THREADS, 0, s>>>(
                ka, va, kb, vb, n, stride, lo_bit + 8 * p, tiles, h, st, tk);
        else
            KDT_LAUNCH radix_pass_kernel<ITEMS, false><<<grid, RADIX_THREADS, 0, s>>>(
                ka, va, kb, vb, n, stride, lo_bit + 8 * p, tiles, h, st, tk);
        KDT_CUDA(cudaGetLastError());
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    return KDT_OK;
}

}  // namespace

int radix_sort_batch(uint32_t **keys, uint32_t **vals, uint32_t **tmp_k, uint32_t **tmp_v, int64_t n, int batch,
                     int64_t stride, int lo_bit, int bits, bool iota, uint32_t *scratch, cudaStream_t s)
{
    const int passes = std::min(RADIX_MAX_PASSES, (bits + 7) / 8);
    if (n < 1 || passes < 1)
        return KDT_OK;
    const int64_t tiles = radix_tiles_of(n);
    // [state: passes x batch x tiles x 256 (64 bits)] [digit counts] [tickets]
    unsigned long long *state = (unsigned long long *)scratch;
    uint32_t *hist = (uint32_t *)(state + (int64_t)passes * batch * tiles * 256);
    uint32_t *ticket = hist + (int64_t)batch * RADIX_MAX_PASSES * 256;
    const size_t used = (char *)(ticket + passes * batch) - (char *)scratch;
    KDT_CUDA(cudaMemsetAsync(scratch, 0, used, s));
    const unsigned hb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 8 * RADIX_THREADS - 1) /
                                                                              (8 * RADIX_THREADS),
                                                                          (int64_t)num_sms() * 8));
    KDT_LAUNCH radix_hist_kernel<<<dim3(hb, (unsigned)batch), RADIX_THREADS, 0, s>>>(*keys, n, stride, lo_bit, passes,
                                                                                  hist);
    KDT_CUDA(cudaGetLastError());
    if (radix_items_of(n) == RADIX_ITEMS_SMALL)
        return radix_passes<RADIX_ITEMS_SMALL>(*keys, *vals, *tmp_k, *tmp_v, n, batch, stride, lo_bit, passes, iota,
                                               hist, state, ticket, s);
    return radix_passes<RADIX_ITEMS_LARGE>(*keys, *vals, *tmp_k, *tmp_v, n, batch, stride, lo_bit, passes, iota, hist,
                                           state, ticket, s);
}

int num_sms()
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0)
            sms = 1;
    }
    return sms;
}

}  // namespace kdt
