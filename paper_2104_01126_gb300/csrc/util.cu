// util.cu -- device-wide primitives: exclusive prefix sum and the sorts of edges and of key-index
// pairs (the "prefix sum" and sorting primitives of Sec. 2.2, written for the GPU).
#include <algorithm>

#include "wm_internal.cuh"

namespace wm {

namespace {

constexpr int kScanBlock = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanBlock * kScanItems;

template <typename T>
__device__ inline T block_exclusive_scan(T v, T *smem_warp, T &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? smem_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) smem_warp[lane] = w;
    }
    __syncthreads();
    total = smem_warp[nw - 1];
    T r = x - v + (warp > 0 ? smem_warp[warp - 1] : 0);
    __syncthreads();
    return r;
}

template <typename T>
__global__ void scan_reduce_kernel(const T *__restrict__ in, int n, T *__restrict__ block_sums,
                                   const int *__restrict__ n_dev)
{
    if (n_dev) n = min(n, *n_dev);
    __shared__ T sw[32];
    long long base = (long long)blockIdx.x * kScanTile;
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        long long idx = base + (long long)threadIdx.x * kScanItems + i;
        if (idx < n) s += in[idx];
    }
    T total;
    block_exclusive_scan(s, sw, total);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

template <typename T>
__global__ void scan_down_kernel(const T *__restrict__ in, T *__restrict__ out, int n,
                                 const T *__restrict__ block_offs, T *total_dev, int nblocks,
                                 const int *__restrict__ n_dev)
{
    if (n_dev) n = min(n, *n_dev);
    __shared__ T sw[32];
    long long base = (long long)blockIdx.x * kScanTile;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        long long idx = base + (long long)threadIdx.x * kScanItems + i;
        v[i] = idx < n ? in[idx] : 0;
        s += v[i];
    }
    T total;
    T ex = block_exclusive_scan(s, sw, total) + (block_offs ? block_offs[blockIdx.x] : 0);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        long long idx = base + (long long)threadIdx.x * kScanItems + i;
        if (idx < n) out[idx] = ex;
        ex += v[i];
    }
    if (total_dev && blockIdx.x == nblocks - 1 && threadIdx.x == blockDim.x - 1) *total_dev = ex;
}

__global__ void fill_i32_kernel(int *p, int v, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) p[i] = v;
}

}  // namespace

void fill_i32(int *p, int v, size_t n, cudaStream_t st)
{
    if (n == 0) return;
    launch(fill_i32_kernel, grid_for((long long)n, 256), 256, 0, st, p, v, n);
}

// out[i] = sum_{j<i} in[j]; *total_dev (optional, device) = sum of all.  in may equal out.
// With n_dev, the length is min(n, *n_dev), read on the device (n is then a bound).
template <typename T>
static int scan_exclusive_t(const T *in, T *out, int n, T *total_dev, cudaStream_t st, Arena &ar,
                            const int *n_dev = nullptr)
{
    if (n <= 0) {
        if (total_dev) cudaMemsetAsync(total_dev, 0, sizeof(T), st);
        return 0;
    }
    int nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        launch(scan_down_kernel<T>, 1, kScanBlock, 0, st, in, out, n, (const T *)nullptr, total_dev, 1, n_dev);
        return 0;
    }
    size_t mark = ar.off;
    T *sums = ar.get<T>(nb);
    if (!sums) return WM_ENOMEM;
    // blocks past the device length contribute 0, so the last block still writes the total
    launch(scan_reduce_kernel<T>, nb, kScanBlock, 0, st, in, n, sums, n_dev);
    int rc = scan_exclusive_t<T>(sums, sums, nb, (T *)nullptr, st, ar);
    if (rc) return rc;
    launch(scan_down_kernel<T>, nb, kScanBlock, 0, st, in, out, n, (const T *)sums, total_dev, nb, n_dev);
    ar.off = mark;
    return 0;
}

int scan_exclusive_i32(const int *in, int *out, int n, int *total_dev, cudaStream_t st, Arena &ar)
{
    return scan_exclusive_t<int>(in, out, n, total_dev, st, ar);
}

int scan_exclusive_i64(const long long *in, long long *out, int n, long long *total_dev, cudaStream_t st, Arena &ar)
{
    return scan_exclusive_t<long long>(in, out, n, total_dev, st, ar);
}

int scan_exclusive_i32_dev(const int *in, int *out, const int *n_dev, int n_max, int *total_dev, cudaStream_t st,
                           Arena &ar)
{
    return scan_exclusive_t<int>(in, out, n_max, total_dev, st, ar, n_dev);
}

int scan_exclusive_i64_dev(const long long *in, long long *out, const int *n_dev, int n_max, long long *total_dev,
                           cudaStream_t st, Arena &ar)
{
    return scan_exclusive_t<long long>(in, out, n_max, total_dev, st, ar, n_dev);
}

// ------------------------------------------------------------------------------ sorting
// Sorts move pairs of a 32-bit key and a 32-bit index: stable LSD passes of 8 bits, three kernels each
// (digit counts per block, their prefixes, the scatter).  A pass reads 12 and writes 8 bytes per element, where
// one over the 16-byte edges themselves read 32 and wrote 16.
//
// Edges go into K order by the 32 leading bits of w2's bits, taken relative to the smallest weight, in
// four passes; edges that agree in them (few, unless weights tie) are ordered by counting inside their run.
// (EMST of 10^7 points in 3-D 21.8 -> 20.4 ms with it, HDBSCAN* of 10^6 6.24 -> 5.9.)
// The edges of runs of more than kRunMax (tied weights, which FP32 coordinates of dense points have) are
// collected, sorted by all the key bytes that differ and put back into the same places.
// Up to kSmallSort edges are sorted by one block in shared memory.
namespace {

constexpr int kRsBlock = 256, kRsItems = 8, kRsTile = kRsBlock * kRsItems;
constexpr int kRunMax = 32;
constexpr int kSmallSort = 2048;   // 32 KB of keys

// state of a sort of edges: [0] smallest hi, [1] smallest ~hi, [2] / [3] bits of hi / lo that differ from
// the first edge's, [4] edges of runs that are too long
enum { kEsMin, kEsMax, kEsHiBits, kEsLoBits, kEsLong, kEsWords };

__global__ void __launch_bounds__(256) es_range_kernel(const EdgeK *__restrict__ e, int m, unsigned long long *st)
{
    const EdgeK e0 = e[0];
    unsigned long long mn = ~0ull, mx = ~0ull, dh = 0, dl = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        const EdgeK x = e[i];
        mn = min(mn, x.hi);
        mx = min(mx, ~x.hi);
        dh |= x.hi ^ e0.hi;
        dl |= x.lo ^ e0.lo;
    }
    for (int o = 16; o; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = min(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        dh |= __shfl_xor_sync(0xffffffffu, dh, o);
        dl |= __shfl_xor_sync(0xffffffffu, dl, o);
    }
    if ((threadIdx.x & 31) == 0) {
        volatile unsigned long long *now = st;   // most warps change nothing
        if (mn < now[kEsMin]) atomicMin(st + kEsMin, mn);
        if (mx < now[kEsMax]) atomicMin(st + kEsMax, mx);
        if (dh & ~now[kEsHiBits]) atomicOr(st + kEsHiBits, dh);
        if (dl & ~now[kEsLoBits]) atomicOr(st + kEsLoBits, dl);
    }
}

// the 32 leading bits of hi - min over the range
__global__ void es_key_kernel(const EdgeK *__restrict__ e, int m, const unsigned long long *__restrict__ st,
                              unsigned *__restrict__ key, int *__restrict__ idx)
{
    const unsigned long long lo = st[kEsMin], span = ~st[kEsMax] - lo;
    const int shift = max(0, 32 - __clzll((long long)span));   // (64 - clz) bits, 32 of them kept
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        key[i] = (unsigned)((e[i].hi - lo) >> shift);
        idx[i] = i;
    }
}

// one 32-bit word of the edges in the order of idx
__global__ void es_word_kernel(const EdgeK *__restrict__ e, int m, int word, const int *__restrict__ idx,
                               unsigned *__restrict__ key)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        const int j = idx[i];
        const unsigned long long w = word < 2 ? e[j].lo : e[j].hi;
        key[i] = (unsigned)(w >> ((word & 1) * 32));
    }
}

// Edges to their places.  In a run of equal keys an edge's place is the number of smaller ones (equal
// edges keep the order of idx).
__global__ void es_place_kernel(const EdgeK *__restrict__ e, int m, const unsigned *__restrict__ key,
                                const int *__restrict__ idx, EdgeK *__restrict__ out, int *__restrict__ is_long,
                                unsigned long long *st)
{
    int n_long = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        const unsigned k = key[i];
        const EdgeK x = e[idx[i]];
        int at = i;
        if ((i > 0 && key[i - 1] == k) || (i + 1 < m && key[i + 1] == k)) {
            int b = i, t = i + 1;
            while (b > 0 && i - b <= kRunMax && key[b - 1] == k) --b;
            while (t < m && t - b <= kRunMax && key[t] == k) ++t;
            is_long[i] = t - b > kRunMax;
            if (t - b > kRunMax) {
                ++n_long;
                continue;
            }
            at = b;
            for (int j = b; j < t; ++j) {
                if (j == i) continue;
                const EdgeK y = e[idx[j]];
                at += edge_less(y, x) || (j < i && !edge_less(x, y));
            }
        } else {
            is_long[i] = 0;
        }
        out[at] = x;
    }
    n_long = __reduce_add_sync(0xffffffffu, n_long);
    if ((threadIdx.x & 31) == 0 && n_long) atomicAdd(st + kEsLong, (unsigned long long)n_long);
}

// the places and edges of long runs (at: exclusive prefixes of is_long), in order of place
__global__ void es_collect_kernel(int m, const int *__restrict__ is_long, const int *__restrict__ at,
                                  const int *__restrict__ idx, int *__restrict__ place, int *__restrict__ edge)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
        if (is_long[i]) {
            place[at[i]] = i;
            edge[at[i]] = idx[i];
        }
}

__global__ void es_put_kernel(const EdgeK *__restrict__ e, int m, const int *__restrict__ place, const int *__restrict__ idx,
                              EdgeK *__restrict__ out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) out[place[i]] = e[idx[i]];
}

// Bitonic sort of up to kSmallSort edges: one launch where the passes take a dozen and more (EMST of 10^3
// points 955 -> 780 us).
__global__ void __launch_bounds__(1024) es_small_kernel(const EdgeK *__restrict__ e, int m, EdgeK *__restrict__ out)
{
    __shared__ EdgeK k[kSmallSort];
    int p = 32;
    while (p < m) p <<= 1;
    for (int i = threadIdx.x; i < p; i += 1024) {
        EdgeK x;
        x.hi = x.lo = ~0ull;
        k[i] = i < m ? e[i] : x;
    }
    __syncthreads();
    for (int len = 2; len <= p; len <<= 1)
        for (int d = len >> 1; d; d >>= 1) {
            for (int t = threadIdx.x; t < p / 2; t += 1024) {
                const int i = 2 * t - (t & (d - 1)), j = i + d;
                const EdgeK x = k[i], y = k[j];
                if (edge_less(y, x) == ((i & len) == 0)) {
                    k[i] = y;
                    k[j] = x;
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < m; i += 1024) out[i] = k[i];
}

// digit counts of a block's chunk: bh[digit * G + block]
__global__ void __launch_bounds__(kRsBlock) rs_count_kernel(const unsigned *__restrict__ key, int m, int bit, int chunk,
                                                            int *__restrict__ bh)
{
    __shared__ int h[8][256];
    const int warp = threadIdx.x >> 5;
    for (int w = 0; w < 8; ++w) h[w][threadIdx.x] = 0;
    __syncthreads();
    const long long beg = (long long)blockIdx.x * chunk, end = min(beg + chunk, (long long)m);
    for (long long i = beg + threadIdx.x; i < end; i += kRsBlock) atomicAdd(&h[warp][(key[i] >> bit) & 0xffu], 1);
    __syncthreads();
    int s = 0;
    for (int w = 0; w < 8; ++w) s += h[w][threadIdx.x];
    bh[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
}

// exclusive prefixes of a digit's counts over the blocks, and the digit's total; one block per digit
__global__ void __launch_bounds__(kRsBlock) rs_prefix_kernel(int *bh, int G, int *__restrict__ total)
{
    __shared__ int sw[32];
    int *row = bh + (size_t)blockIdx.x * G, run = 0;
    for (int b0 = 0; b0 < G; b0 += kRsBlock * 4) {
        int v[4], s = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = b0 + threadIdx.x * 4 + t;
            v[t] = i < G ? row[i] : 0;
            s += v[t];
        }
        int all;
        int x = run + block_exclusive_scan(s, sw, all);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = b0 + threadIdx.x * 4 + t;
            if (i < G) row[i] = x;
            x += v[t];
        }
        run += all;
    }
    if (threadIdx.x == 0) total[blockIdx.x] = run;
}

// Stable scatter of a block's chunk, a tile of kRsTile elements at a time: a warp takes 256 consecutive ones and
// counts the digits on the way, so its elements' ranks need no barrier.
__global__ void __launch_bounds__(kRsBlock) rs_move_kernel(const unsigned *__restrict__ key, const int *__restrict__ idx, int m,
                                                           int bit, int chunk, const int *__restrict__ bh,
                                                           const int *__restrict__ total, unsigned *__restrict__ key_out,
                                                           int *__restrict__ idx_out)
{
    __shared__ int base[256], cnt[8][256], sw[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        int all;
        const int first = block_exclusive_scan(total[threadIdx.x], sw, all);   // of the digit
        base[threadIdx.x] = first + bh[(size_t)threadIdx.x * gridDim.x + blockIdx.x];
    }
    const long long beg = (long long)blockIdx.x * chunk, end = min(beg + chunk, (long long)m);
    for (long long t0 = beg; t0 < end; t0 += kRsTile) {
        for (int w = 0; w < 8; ++w) cnt[w][threadIdx.x] = 0;
        __syncthreads();
        unsigned k[kRsItems];
        int v[kRsItems], r[kRsItems];
        const long long i0 = t0 + warp * (kRsTile / 8) + lane;
#pragma unroll
        for (int t = 0; t < kRsItems; ++t) {
            const long long i = i0 + 32 * t;
            k[t] = i < end ? key[i] : 0;
            v[t] = i < end ? idx[i] : 0;
        }
#pragma unroll
        for (int t = 0; t < kRsItems; ++t) {
            const bool in = i0 + 32 * t < end;
            const unsigned d = in ? (k[t] >> bit) & 0xffu : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            r[t] = in ? cnt[warp][d] + __popc(peers & lanemask_lt()) : 0;
            __syncwarp();
            if (in && lane == __ffs(peers) - 1) cnt[warp][d] += __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        {   // a digit's counts to the warps' first places
            int s = base[threadIdx.x];
            for (int w = 0; w < 8; ++w) {
                const int c = cnt[w][threadIdx.x];
                cnt[w][threadIdx.x] = s;
                s += c;
            }
            base[threadIdx.x] = s;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < kRsItems; ++t) {
            if (i0 + 32 * t >= end) continue;
            const int o = cnt[warp][(k[t] >> bit) & 0xffu] + r[t];
            key_out[o] = k[t];
            idx_out[o] = v[t];
        }
        __syncthreads();
    }
}

}  // namespace

int sort_pairs_begin(SortPairs &P, int m, Arena &ar, int *room)
{
    P.m = m;
    P.cur = 0;
    for (int t = 0; t < 2; ++t) {
        P.key[t] = room ? (unsigned *)room + (size_t)(2 * t) * m : ar.get<unsigned>(m);
        P.idx[t] = room ? room + (size_t)(2 * t + 1) * m : ar.get<int>(m);
    }
    // whole tiles, at most 2048 blocks
    const long long tiles = ((long long)m + kRsTile - 1) / kRsTile, per = std::max(1LL, (tiles + 2047) / 2048);
    P.chunk = (int)(per * kRsTile);
    P.G = (int)std::max(1LL, (tiles + per - 1) / per);
    P.bh = ar.get<int>(256 * (size_t)P.G);
    P.total = ar.get<int>(256);
    return ar.failed ? WM_ENOMEM : 0;
}

void sort_pairs_pass(SortPairs &P, int bit, cudaStream_t st)
{
    const int c = P.cur;
    launch(rs_count_kernel, P.G, kRsBlock, 0, st, P.key[c], P.m, bit, P.chunk, P.bh);
    launch(rs_prefix_kernel, 256, kRsBlock, 0, st, P.bh, P.G, P.total);
    launch(rs_move_kernel, P.G, kRsBlock, 0, st, P.key[c], P.idx[c], P.m, bit, P.chunk, P.bh, P.total, P.key[c ^ 1], P.idx[c ^ 1]);
    P.cur ^= 1;
}

void sort_pairs(SortPairs &P, unsigned max_key, cudaStream_t st)
{
    for (int bit = 0; bit < 32 && (max_key >> bit); bit += 8) sort_pairs_pass(P, bit, st);
}

int sort_edges(const EdgeK *in, EdgeK *out, int m, cudaStream_t st, Arena &ar, void *pin)
{
    if (m <= 0) return 0;
    if (m <= kSmallSort) {
        launch(es_small_kernel, 1, 1024, 0, st, in, m, out);
        return 0;
    }
    const size_t mark = ar.off;
    unsigned long long *state = ar.get<unsigned long long>(kEsWords), *h = (unsigned long long *)pin;
    SortPairs P;
    if (sort_pairs_begin(P, m, ar) || !state) {
        ar.off = mark;
        return WM_ENOMEM;
    }
    const int g = grid_for(m, 256);
    cudaMemsetAsync(state, 0xff, 2 * sizeof *state, st);
    cudaMemsetAsync(state + 2, 0, (kEsWords - 2) * sizeof *state, st);
    launch(es_range_kernel, grid_for(m, 256, num_sms() * 4), 256, 0, st, in, m, state);
    launch(es_key_kernel, g, 256, 0, st, in, m, state, P.key[0], P.idx[0]);
    sort_pairs(P, 0xffffffffu, st);
    int *is_long = (int *)P.key[P.cur ^ 1], *at = P.idx[P.cur ^ 1];   // (free now)
    launch(es_place_kernel, g, 256, 0, st, in, m, P.key[P.cur], P.idx[P.cur], out, is_long, state);
    cudaMemcpyAsync(h, state, kEsWords * sizeof *state, cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) {
        ar.off = mark;
        return WM_ECUDA;
    }
    const int ml = (int)h[kEsLong];
    if (ml > 0) {
        SortPairs Q;
        int *place = ar.get<int>(ml);
        if (sort_pairs_begin(Q, ml, ar) || scan_exclusive_i32(is_long, at, m, nullptr, st, ar)) {
            ar.off = mark;
            return WM_ENOMEM;
        }
        launch(es_collect_kernel, g, 256, 0, st, m, is_long, at, P.idx[P.cur], place, Q.idx[0]);
        const unsigned long long diff[2] = {h[kEsLoBits], h[kEsHiBits]};
        const int gl = grid_for(ml, 256);
        for (int word = 0; word < 4; ++word) {
            const unsigned w = (unsigned)(diff[word >> 1] >> ((word & 1) * 32));
            if (!w) continue;
            launch(es_word_kernel, gl, 256, 0, st, in, ml, word, Q.idx[Q.cur], Q.key[Q.cur]);
            for (int bit = 0; bit < 32; bit += 8)
                if ((w >> bit) & 0xffu) sort_pairs_pass(Q, bit, st);
        }
        launch(es_put_kernel, gl, 256, 0, st, in, ml, place, Q.idx[Q.cur], out);
    }
    ar.off = mark;
    return 0;
}

}  // namespace wm
