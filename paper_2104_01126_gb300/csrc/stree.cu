// stree.cu -- ingest of the input points and construction of the search tree (stree.cuh): a spatial-median
// k-d tree (Sec. 2.3) down to buckets of at most kBucket points.
//
// A node splits its tight bounding box at the midpoint of the widest dimension; if every point falls on
// one side (equal points, an extent of one ulp) it splits its points by count instead.  The walks need
// no node below a bucket, so about 0.4 nodes per point are made instead of the 2 of the traversals' tree
// (kdtree.cu), and each is written once, in the form the walks read.
//
// A point travels as one row: its FP32 coordinates (less a centre, see centre()) and its input id, 16 bytes up to 3 dimensions and 32
// up to 7, moved by vector loads and stores.  Nodes above M points are split level by level over the
// whole GPU in one pass per level: a block takes 256 x R rows into registers, splits them with one pair
// of atomics on the node's two ends (left points fill the range upwards, right points downwards, so no
// counting pass is needed) and accumulates the children's boxes on the way.  A node of at most M points
// is finished by one block in shared memory, a warp per segment and level.
#include <algorithm>
#include <cstring>

#include "stree.cuh"

namespace wm {

namespace {

// float <-> unsigned key of the same order
__device__ inline unsigned f2key(float f)
{
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}
__host__ __device__ inline float key2f(unsigned k)
{
    const unsigned u = (k & 0x80000000u) ? k & 0x7fffffffu : ~k;
    float f;
    memcpy(&f, &u, sizeof f);
    return f;
}

constexpr int kStThreads = 256;
template <int S> constexpr int rows_per_thread() { return S == 4 ? 8 : S == 8 ? 4 : 2; }
template <int S> constexpr int block_points() { return S <= 8 ? 1024 : 512; }   // M

// device scalars of a build
struct BuildState {
    int next_id;      // first free node row
    int active;       // nodes of the current level
    int units;        // their work units
    int subs;         // entries of the block list
    int sub_next;     // its dispenser
    int depth;        // levels below a block's root
    unsigned bad;     // non-finite or too large coordinate
    unsigned delta;   // bits of max |x64 - x32|
    unsigned delta_c; // the same of the centred copy
    int centred;      // 1: it replaces the other
    int buckets;      // of more than kBucket / 2 points, made by the blocks
    int coarse;       // those whose widest extent is below kCoarse times that
};

constexpr size_t kStateBytes = 64;   // of a BuildState; root_acc follows, and one fill clears both
static_assert(sizeof(BuildState) <= kStateBytes, "BuildState has outgrown its place");

// A bucket's extent of two spacings or so, in units of the FP32 copy's largest error, below which most of its
// points' distances are in one band of the screen.
constexpr float kCoarse = 32.f;

// Where the FP32 copy is inexact, a box side is widened so that it bounds exact distances from a rounded query:
// rounding moves a coordinate of the box by half an ulp of the side's larger magnitude m at most, and the query
// by as much, by twice that where it lies in the next binade, or, farther out, by 2^-23 of its distance from
// the box, which the margin of lower_w2 holds.  (The widening follows the side, not the largest error of any
// point: one coordinate of 10^6 would else blur all points within 0.1.)
__device__ inline float widening(float lo, float hi)
{
    const unsigned e = __float_as_uint(fmaxf(fabsf(lo), fabsf(hi))) >> 23;   // biased exponent of m
    const float half_ulp = __uint_as_float(e > 24 ? (e - 24) << 23 : 1u << max((int)e - 2, 0));
    return __fmul_ru(3.f + 1.0f / 1048576.0f, half_ulp);   // (more than 3, for centred copies)
}

struct LNode {
    int node, b, e, dim;
    float val;
};

struct StArgs {
    int n, d, dtype, layout;
    const void *src;
    float *buf[2];           // point rows, ping-pong; buf[0] becomes the final array
    float *nodes;
    int2 *range;
    int *parent;
    BuildState *state;
    LNode *act[2];
    int *unit_off[2];
    int *lr;                 // per active node: points placed left, right
    unsigned *acc;           // per active node: [2][d][2] box keys of the children (max of ~key, key)
    unsigned *root_acc;      // [d][2] of all points; then the same of the centred copy
    int4 *sub;               // block list: node, first point, size | dim << 16 | buffer << 31, split value
    int *pid, *pos;
    double *x64;
};

__device__ inline double src_coord(const StArgs &a, int i, int k)
{
    const size_t at = a.layout == WM_SOA ? (size_t)k * a.n + i : (size_t)i * a.d + k;
    return a.dtype == WM_F32 ? (double)((const float *)a.src)[at] : ((const double *)a.src)[at];
}

// Rows from the input; validation, delta and the box of all points.
template <int S>
__global__ void __launch_bounds__(kStThreads) st_ingest_kernel(StArgs a)
{
    __shared__ unsigned sk[2 * S];
    if (threadIdx.x < 2 * S) sk[threadIdx.x] = 0;
    __syncthreads();
    const int d = a.d, lane = threadIdx.x & 31;
    float dmax = 0.f;
    bool bad = false;
    float mn[S], mx[S];
#pragma unroll
    for (int k = 0; k < S; ++k) { mn[k] = INFINITY; mx[k] = -INFINITY; }
    for (int i = blockIdx.x * kStThreads + threadIdx.x; i < a.n; i += gridDim.x * kStThreads) {
        float v[S];
#pragma unroll
        for (int k = 0; k < S; ++k) {
            v[k] = 0.f;
            if (k < d) {
                const double x = src_coord(a, i, k);
                v[k] = __double2float_rn(x);
                if (a.dtype != WM_F32) {
                    // the error rounded up: above 0 wherever the copy is inexact, however small (the FP64
                    // coordinates are kept only then)
                    dmax = fmaxf(dmax, __double2float_ru(fabs(x - (double)v[k])));
                }
                bad = bad || !(fabsf(v[k]) <= 1152921504606846976.0f) || fabs(x) > 1152921504606846976.0;
                mn[k] = fminf(mn[k], v[k]);
                mx[k] = fmaxf(mx[k], v[k]);
            }
        }
        v[S - 1] = __int_as_float(i);
        float4 *r = (float4 *)(a.buf[0] + (size_t)i * S);
#pragma unroll
        for (int c = 0; c < S / 4; ++c) r[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    }
#pragma unroll
    for (int k = 0; k < S - 1; ++k) {
        if (k >= d) break;
        const unsigned lo = __reduce_max_sync(0xffffffffu, ~f2key(mn[k]));
        const unsigned hi = __reduce_max_sync(0xffffffffu, f2key(mx[k]));
        if (lane == 0) {
            atomicMax(&sk[2 * k], lo);
            atomicMax(&sk[2 * k + 1], hi);
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&a.state->bad, 1u);
    for (int o = 16; o; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0 && dmax > 0.f) atomicMax(&a.state->delta, __float_as_uint(dmax));
    __syncthreads();
    if (threadIdx.x < 2 * d && sk[threadIdx.x] > *(volatile unsigned *)(a.root_acc + threadIdx.x))
        atomicMax(a.root_acc + threadIdx.x, sk[threadIdx.x]);
}

// The centre of a dimension whose FP64 coordinates lie far from 0 beside their range (timestamps, map coordinates),
// else 0.  The rows then hold coordinates less that, rounded: distances are what the walks need, and the copy of
// 1.6x10^9 + [0, 10^5] errs by 0.004 instead of 64.  (The FP64 subtraction adds 2^-53 of the result.)
__device__ inline float centre(const StArgs &a, int k)
{
    const float lo = key2f(~a.root_acc[2 * k]), hi = key2f(a.root_acc[2 * k + 1]), mid = lo + (hi - lo) * 0.5f;
    return fabsf(mid) > 4.f * (hi - lo) ? mid : 0.f;
}

// The centred copy, its error and box; nothing where no dimension needs it.
template <int S>
__global__ void __launch_bounds__(kStThreads) st_centre_kernel(StArgs a)
{
    __shared__ unsigned sk[2 * S];
    const int d = a.d, lane = threadIdx.x & 31;
    if (threadIdx.x < 2 * S) sk[threadIdx.x] = 0;
    const bool away = threadIdx.x < d && centre(a, threadIdx.x) != 0.f, inexact = a.state->delta != 0 && !a.state->bad;
    if (!__syncthreads_or(away && inexact)) return;   // the same for every block
    if (blockIdx.x == 0 && threadIdx.x == 0) a.state->centred = 1;
    unsigned *acc = a.root_acc + 2 * S;
    float dmax = 0.f, mn[S], mx[S], c[S];
#pragma unroll
    for (int k = 0; k < S; ++k) {
        mn[k] = INFINITY;
        mx[k] = -INFINITY;
        c[k] = k < d ? centre(a, k) : 0.f;
    }
    for (int i = blockIdx.x * kStThreads + threadIdx.x; i < a.n; i += gridDim.x * kStThreads) {
        float *row = a.buf[0] + (size_t)i * S;
#pragma unroll
        for (int k = 0; k < S - 1; ++k) {
            if (k >= d) break;
            const double x = __dsub_rn(src_coord(a, i, k), (double)c[k]);
            const float v = __double2float_rn(x);
            float e = __double2float_ru(fabs(x - (double)v));
            if (c[k] != 0.f) e = __fmaf_ru(fabsf(v), 1.0f / 4503599627370496.0f, e);
            dmax = fmaxf(dmax, e);
            mn[k] = fminf(mn[k], v);
            mx[k] = fmaxf(mx[k], v);
            row[k] = v;
        }
    }
#pragma unroll
    for (int k = 0; k < S - 1; ++k) {
        if (k >= d) break;
        const unsigned lo = __reduce_max_sync(0xffffffffu, ~f2key(mn[k]));
        const unsigned hi = __reduce_max_sync(0xffffffffu, f2key(mx[k]));
        if (lane == 0) {
            atomicMax(&sk[2 * k], lo);
            atomicMax(&sk[2 * k + 1], hi);
        }
    }
    for (int o = 16; o; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0 && dmax > 0.f) atomicMax(&a.state->delta_c, __float_as_uint(dmax));
    __syncthreads();
    if (threadIdx.x < 2 * d && sk[threadIdx.x] > *(volatile unsigned *)(acc + threadIdx.x)) atomicMax(acc + threadIdx.x, sk[threadIdx.x]);
}

// the split of a box: its widest dimension, at the midpoint
__device__ inline void choose_split(const unsigned *acc, int d, int &dim, float &val)
{
    float ext = -1.f;
    dim = 0;
    val = 0.f;
    for (int k = 0; k < d; ++k) {
        const float lo = key2f(~acc[2 * k]), hi = key2f(acc[2 * k + 1]);
        if (hi - lo > ext) {
            ext = hi - lo;
            dim = k;
            val = lo + (hi - lo) * 0.5f;
        }
    }
}

// box of a node row, widened where the copy is inexact
template <int S>
__device__ inline void write_box(float *row, const unsigned *acc, int d, bool inexact)
{
    for (int k = 0; k < S; ++k) {
        float lo = 0.f, hi = 0.f;
        if (k < d) {
            lo = key2f(~acc[2 * k]);
            hi = key2f(acc[2 * k + 1]);
            if (inexact) {
                const float w = widening(lo, hi);
                lo = __fsub_rd(lo, w);
                hi = __fadd_ru(hi, w);
            }
        }
        row[box_lo(k)] = lo;
        row[box_hi(k)] = k == S - 1 ? __int_as_float(-1) : hi;
    }
}

__device__ inline int4 sub_entry(int node, int b, int size, int dim, int buffer, float val)
{
    return make_int4(node, b, (int)((unsigned)size | (unsigned)dim << 16 | (unsigned)buffer << 31), __float_as_int(val));
}

template <int S>
__global__ void st_root_kernel(StArgs a)
{
    BuildState &s = *a.state;
    if (s.centred) {
        for (int k = 0; k < 2 * a.d; ++k) a.root_acc[k] = a.root_acc[2 * S + k];
        s.delta = s.delta_c;
    }
    write_box<S>(a.nodes, a.root_acc, a.d, s.delta != 0);
    a.range[0] = make_int2(0, a.n);
    a.parent[0] = -1;
    int dim;
    float val;
    choose_split(a.root_acc, a.d, dim, val);
    s.next_id = 1;
    s.active = 0;
    s.units = 0;
    if (a.n > block_points<S>()) {
        a.act[0][0] = LNode{0, 0, a.n, dim, val};
        a.unit_off[0][0] = 0;
        s.active = 1;
        s.units = (a.n + kStThreads * rows_per_thread<S>() - 1) / (kStThreads * rows_per_thread<S>());
    } else {
        a.sub[0] = sub_entry(0, 0, a.n, dim, 0, val);
        s.subs = 1;
    }
}

// One level: every unit's rows to their side of the node's range in the other buffer.
template <int S>
__global__ void __launch_bounds__(kStThreads) st_scatter_kernel(StArgs a, int level)
{
    constexpr int R = rows_per_thread<S>(), U = kStThreads * R, W = kStThreads / 32;
    __shared__ int s_node, s_l[W], s_r[W], s_base[2];
    __shared__ unsigned sk[4 * S];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, d = a.d;
    const int A = a.state->active, TU = a.state->units, cur = level & 1;
    const LNode *act = a.act[cur];
    const int *uoff = a.unit_off[cur];
    const float *src = a.buf[cur];
    float *dst = a.buf[cur ^ 1];
    for (int u = blockIdx.x; u < TU; u += gridDim.x) {
        if (threadIdx.x == 0) {
            int lo = 0, hi = A - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (uoff[mid] <= u) lo = mid; else hi = mid - 1;
            }
            s_node = lo;
        }
        if (threadIdx.x < 4 * S) sk[threadIdx.x] = 0;
        __syncthreads();
        const int j = s_node;
        const LNode nd = act[j];
        const int b = nd.b + (u - uoff[j]) * U, e = min(b + U, nd.e);
        float4 row[R][S / 4];
        unsigned left = 0, in = 0;   // bit r: row r is a left point / a point
        int wl = 0, wr = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = b + r * kStThreads + threadIdx.x;
            if (i < e) {
                in |= 1u << r;
                const float4 *p = (const float4 *)(src + (size_t)i * S);
#pragma unroll
                for (int c = 0; c < S / 4; ++c) row[r][c] = p[c];
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float x = 0.f;
#pragma unroll
            for (int c = 0; c < S / 4; ++c) {
                const float v[4] = {row[r][c].x, row[r][c].y, row[r][c].z, row[r][c].w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (4 * c + k == nd.dim) x = v[k];
            }
            const bool is = (in >> r) & 1u, l = is && x < nd.val;
            if (l) left |= 1u << r;
            wl += __popc(__ballot_sync(0xffffffffu, l));
            wr += __popc(__ballot_sync(0xffffffffu, is && !l));
        }
        if (lane == 0) { s_l[wid] = wl; s_r[wid] = wr; }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tl = 0, tr = 0;
            for (int w = 0; w < W; ++w) {
                const int x = s_l[w], y = s_r[w];
                s_l[w] = tl;
                s_r[w] = tr;
                tl += x;
                tr += y;
            }
            s_base[0] = tl ? atomicAdd(&a.lr[2 * j], tl) : 0;
            s_base[1] = tr ? atomicAdd(&a.lr[2 * j + 1], tr) : 0;
        }
        __syncthreads();
        int pl = nd.b + s_base[0] + s_l[wid], pr = nd.e - 1 - s_base[1] - s_r[wid];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const bool is = (in >> r) & 1u, l = (left >> r) & 1u;
            const unsigned bl = __ballot_sync(0xffffffffu, l), br = __ballot_sync(0xffffffffu, is && !l);
            if (is) {
                float4 *p = (float4 *)(dst + (size_t)(l ? pl + __popc(bl & lanemask_lt()) : pr - __popc(br & lanemask_lt())) * S);
#pragma unroll
                for (int c = 0; c < S / 4; ++c) p[c] = row[r][c];
            }
            pl += __popc(bl);
            pr -= __popc(br);
        }
        // children's boxes
#pragma unroll
        for (int k = 0; k < S - 1; ++k) {
            if (k >= d) break;
            unsigned q[4] = {0, 0, 0, 0};   // left ~min, left max, right ~min, right max
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 v = row[r][k / 4];
                const float x = (k & 3) == 0 ? v.x : (k & 3) == 1 ? v.y : (k & 3) == 2 ? v.z : v.w;
                if ((in >> r) & 1u) {
                    const unsigned key = f2key(x);
                    if ((left >> r) & 1u) { q[0] = max(q[0], ~key); q[1] = max(q[1], key); }
                    else { q[2] = max(q[2], ~key); q[3] = max(q[3], key); }
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const unsigned m = __reduce_max_sync(0xffffffffu, q[t]);
                if (lane == 0) atomicMax(&sk[(t >> 1) * 2 * d + 2 * k + (t & 1)], m);
            }
        }
        __syncthreads();
        if (threadIdx.x < 4 * d) {
            unsigned *g = a.acc + (size_t)j * 4 * d + threadIdx.x;
            const unsigned v = sk[threadIdx.x];
            if (v > *(volatile unsigned *)g) atomicMax(g, v);   // most units cannot widen the box
        }
        __syncthreads();
    }
}

// Children of the level's nodes: rows, the next level's list, the block list.  One block.
template <int S>
__global__ void __launch_bounds__(1024) st_level_kernel(StArgs a, int level)
{
    constexpr int M = block_points<S>(), U = kStThreads * rows_per_thread<S>();
    __shared__ int sh[32];
    __shared__ int s_act, s_units;
    const int A = a.state->active, id0 = a.state->next_id, d = a.d, cur = level & 1;
    const bool inexact = a.state->delta != 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) { s_act = 0; s_units = 0; }
    __syncthreads();
    for (int j0 = 0; j0 < A; j0 += 1024) {
        const int j = j0 + threadIdx.x;
        int units[2] = {0, 0};   // of a child that stays active
        LNode ch[2];
        if (j < A) {
            const LNode nd = a.act[cur][j];
            const unsigned *acc = a.acc + (size_t)j * 4 * d;
            int L = a.lr[2 * j];
            const int sz = nd.e - nd.b;
            const bool by_count = L == 0 || L == sz;   // all points on one side: both halves keep its box
            const int full = L == 0 ? 1 : 0;
            if (by_count) L = sz / 2;
            const int c0 = id0 + 2 * j;
            a.nodes[(size_t)nd.node * 2 * S + box_lo(S - 1)] = __int_as_float(c0);
            for (int s = 0; s < 2; ++s) {
                const unsigned *box = acc + (by_count ? full : s) * 2 * d;
                LNode c;
                c.node = c0 + s;
                c.b = s ? nd.b + L : nd.b;
                c.e = s ? nd.e : nd.b + L;
                choose_split(box, d, c.dim, c.val);
                write_box<S>(a.nodes + (size_t)c.node * 2 * S, box, d, inexact);
                a.range[c.node] = make_int2(c.b, c.e);
                a.parent[c.node] = nd.node;
                const int m = c.e - c.b;
                if (m > M) units[s] = (m + U - 1) / U;
                else a.sub[atomicAdd(&a.state->subs, 1)] = sub_entry(c.node, c.b, m, c.dim, cur ^ 1, c.val);
                ch[s] = c;
            }
        }
        // slots of the active children in the next list and their unit offsets
        const int na = (units[0] > 0) + (units[1] > 0), nu = units[0] + units[1];
        long long x = (long long)na << 32 | (long long)nu, t = x;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        __shared__ long long wt[32];
        if (lane == 31) wt[wid] = t;
        __syncthreads();
        if (wid == 0) {
            long long y = wt[lane], z = y;
            for (int o = 1; o < 32; o <<= 1) {
                const long long q = __shfl_up_sync(0xffffffffu, z, o);
                if (lane >= o) z += q;
            }
            wt[lane] = z - y;
            if (lane == 31) sh[0] = (int)(z >> 32), sh[1] = (int)(z & 0xffffffffLL);
        }
        __syncthreads();
        t += wt[wid] - x;
        int slot = s_act + (int)(t >> 32), uo = s_units + (int)(t & 0xffffffffLL);
        for (int s = 0; s < 2; ++s) {
            if (units[s] == 0) continue;
            a.act[cur ^ 1][slot] = ch[s];
            a.unit_off[cur ^ 1][slot] = uo;
            ++slot;
            uo += units[s];
        }
        __syncthreads();
        if (threadIdx.x == 0) { s_act += sh[0]; s_units += sh[1]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.state->next_id = id0 + 2 * A;
        a.state->active = s_act;
        a.state->units = s_units;
    }
}

// A node of at most M points, finished by a block in shared memory.  Every level, a warp takes a segment
// (a node above kBucket points): it moves the points to their side in the other buffer, computes both
// children's boxes from them and writes the children's rows; a child that is a bucket goes to its final
// place, the others form the next level.
template <int S>
__global__ void __launch_bounds__(kStThreads) st_block_kernel(StArgs a)
{
    constexpr int M = block_points<S>(), W = kStThreads / 32, C = S / 4;
    extern __shared__ float4 st_smem[];
    float *buf0 = (float *)st_smem, *buf1 = buf0 + (size_t)M * S;
    int4 *seg = (int4 *)(buf1 + (size_t)M * S);      // [2][M / 8]: first, end, node, dim
    float *sval = (float *)(seg + 2 * (M / 8));      // [2][M / 8]
    __shared__ int s_entry, s_next, s_base, s_buckets, s_coarse;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, d = a.d;
    const float delta = __uint_as_float(a.state->delta);
    if (threadIdx.x == 0) s_buckets = s_coarse = 0;
    const int nsub = a.state->subs;
    while (true) {
        if (threadIdx.x == 0) s_entry = atomicAdd(&a.state->sub_next, 1);
        __syncthreads();
        const int entry = s_entry;
        if (entry >= nsub) {   // the same for every thread
            if (threadIdx.x == 0 && s_coarse) atomicAdd(&a.state->coarse, s_coarse);
            if (threadIdx.x == 0 && s_buckets) atomicAdd(&a.state->buckets, s_buckets);
            return;
        }
        const int4 E = a.sub[entry];
        const int node = E.x, gb = E.y, m = E.z & 0xffff, dim = (E.z >> 16) & 0x7fff;
        const float4 *src = (const float4 *)(a.buf[(unsigned)E.z >> 31] + (size_t)gb * S);
        if (m <= kBucket) {   // (block-uniform)
            if (threadIdx.x == 0)
                a.nodes[(size_t)node * 2 * S + box_lo(S - 1)] = __uint_as_float(bucket_ref(gb, m));
            if ((unsigned)E.z >> 31)
                for (int t = threadIdx.x; t < m * C; t += kStThreads) ((float4 *)(a.buf[0] + (size_t)gb * S))[t] = src[t];
            __syncthreads();
            continue;
        }
        for (int t = threadIdx.x; t < m * C; t += kStThreads) ((float4 *)buf0)[t] = src[t];
        if (threadIdx.x == 0) {
            seg[0] = make_int4(0, m, node, dim);
            sval[0] = __int_as_float(E.w);
        }
        int nseg = 1, cur = 0, depth = 0;
        __syncthreads();
        while (nseg > 0) {
            if (threadIdx.x == 0) {
                s_base = atomicAdd(&a.state->next_id, 2 * nseg);
                s_next = 0;
            }
            __syncthreads();
            const int base = s_base;
            const float *sb = cur ? buf1 : buf0;
            float *db = cur ? buf0 : buf1;
            for (int s = wid; s < nseg; s += W) {
                const int4 g = seg[cur * (M / 8) + s];
                const float val = sval[cur * (M / 8) + s];
                const int b = g.x, e = g.y;
                if (lane == 0) a.nodes[(size_t)g.z * 2 * S + box_lo(S - 1)] = __int_as_float(base + 2 * s);
                int L = 0, Rt = 0;
                for (int i0 = b; i0 < e; i0 += 32) {
                    const int i = i0 + lane;
                    const bool in = i < e, l = in && sb[(size_t)i * S + g.w] < val;
                    const unsigned bl = __ballot_sync(0xffffffffu, l), br = __ballot_sync(0xffffffffu, in && !l);
                    if (in) {
                        const int t = l ? b + L + __popc(bl & lanemask_lt()) : e - 1 - Rt - __popc(br & lanemask_lt());
#pragma unroll
                        for (int c = 0; c < C; ++c) ((float4 *)db)[t * C + c] = ((const float4 *)sb)[i * C + c];
                    }
                    L += __popc(bl);
                    Rt += __popc(br);
                }
                if (L == 0 || Rt == 0) L = (e - b) / 2;   // all points on one side: split by count
                __syncwarp();
                for (int side = 0; side < 2; ++side) {
                    const int cb = side ? b + L : b, ce = side ? e : b + L, sz = ce - cb;
                    const int id = base + 2 * s + side;
                    // box, split and row
                    float v[(2 * S + 31) / 32];   // the words of the row that this lane writes
#pragma unroll
                    for (int w = 0; w < (2 * S + 31) / 32; ++w) v[w] = 0.f;
                    float ext = -1.f, cval = 0.f;
                    int cdim = 0;
                    unsigned klo[S], khi[S];
#pragma unroll
                    for (int k = 0; k < S; ++k) klo[k] = khi[k] = 0;
                    for (int i = cb + lane; i < ce; i += 32) {
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const float4 q = ((const float4 *)db)[i * C + c];
                            const float x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if (4 * c + k >= S - 1) continue;
                                const unsigned key = f2key(x[k]);
                                klo[4 * c + k] = max(klo[4 * c + k], ~key);
                                khi[4 * c + k] = max(khi[4 * c + k], key);
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < S - 1; ++k) {
                        if (k >= d) break;
                        float lo = key2f(~__reduce_max_sync(0xffffffffu, klo[k]));
                        float hi = key2f(__reduce_max_sync(0xffffffffu, khi[k]));
                        if (hi - lo > ext) {
                            ext = hi - lo;
                            cdim = k;
                            cval = lo + (hi - lo) * 0.5f;
                        }
                        if (delta > 0.f) {
                            const float w = widening(lo, hi);
                            lo = __fsub_rd(lo, w);
                            hi = __fadd_ru(hi, w);
                        }
                        if (lane == (box_lo(k) & 31)) v[box_lo(k) >> 5] = lo;
                        if (lane == (box_hi(k) & 31)) v[box_hi(k) >> 5] = hi;
                    }
                    if (lane == (box_hi(S - 1) & 31)) v[box_hi(S - 1) >> 5] = __int_as_float(-1);
                    if (lane == (box_lo(S - 1) & 31)) v[box_lo(S - 1) >> 5] = __uint_as_float(bucket_ref(gb + cb, min(sz, kBucket)));
#pragma unroll
                    for (int w = 0; w < (2 * S + 31) / 32; ++w)
                        if (32 * w + lane < 2 * S) a.nodes[(size_t)id * 2 * S + 32 * w + lane] = v[w];
                    if (lane == 0) {
                        a.range[id] = make_int2(gb + cb, gb + ce);
                        a.parent[id] = g.z;
                    }
                    if (sz <= kBucket) {
                        if (delta > 0.f && lane == 0 && sz > kBucket / 2) {   // (a few points have no extent)
                            atomicAdd(&s_buckets, 1);
                            if (ext < kCoarse * delta) atomicAdd(&s_coarse, 1);
                        }
                        for (int t = lane; t < sz * C; t += 32)
                            ((float4 *)(a.buf[0] + (size_t)(gb + cb) * S))[t] = ((const float4 *)db)[cb * C + t];
                    } else if (lane == 0) {
                        const int t = atomicAdd(&s_next, 1);   // segments above 8 points: fewer than M / 8
                        seg[(cur ^ 1) * (M / 8) + t] = make_int4(cb, ce, id, cdim);
                        sval[(cur ^ 1) * (M / 8) + t] = cval;
                    }
                }
            }
            __syncthreads();
            nseg = s_next;
            cur ^= 1;
            ++depth;
            __syncthreads();
        }
        if (threadIdx.x == 0) atomicMax(&a.state->depth, depth);
    }
}

// ids out of the rows, labels in; the FP64 coordinates in tree order where the FP32 copy is inexact
template <int S>
__global__ void st_finish_kernel(StArgs a)
{
    const bool exact = a.state->delta == 0 || a.x64 == nullptr;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        float *w = a.buf[0] + (size_t)i * S + S - 1;
        const int id = __float_as_int(*w);
        *w = __int_as_float(i);
        a.pid[i] = id;
        a.pos[id] = i;
        if (!exact)
            for (int k = 0; k < a.d; ++k) a.x64[(size_t)k * a.n + i] = src_coord(a, id, k);
    }
}

template <int S>
int build(StArgs &a, SearchTree &X, Points &P, Arena &ar, cudaStream_t st, int *pin)
{
    constexpr int M = block_points<S>(), U = kStThreads * rows_per_thread<S>();
    constexpr int smem = 2 * M * S * 4 + 2 * (M / 8) * (16 + 4);
    const int n = a.n;
    if (cudaFuncSetAttribute(st_block_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return WM_ECUDA;
    const int cap = n / M + 2;   // active nodes of a level (each above M points)
    for (int i = 0; i < 2; ++i) {
        a.act[i] = ar.get<LNode>(cap);
        a.unit_off[i] = ar.get<int>(cap);
    }
    a.lr = ar.get<int>(2 * (size_t)cap);
    a.acc = ar.get<unsigned>((size_t)cap * 4 * a.d);
    a.sub = ar.get<int4>(n > M ? n : 1);
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(a.state, 0, kStateBytes + sizeof(unsigned) * 4 * S, st);   // (and root_acc)
    launch(st_ingest_kernel<S>, grid_for(n, kStThreads, num_sms() * 8), kStThreads, 0, st, a);
    if (a.dtype != WM_F32) launch(st_centre_kernel<S>, grid_for(n, kStThreads, num_sms() * 8), kStThreads, 0, st, a);
    launch(st_root_kernel<S>, 1, 1, 0, st, a);
    // levels: at least log2(n / M) are needed; the host then learns every two levels whether more are
    int level = 0, want = 0;
    while ((long long)M << want < (long long)n) ++want;
    const int grid = (int)std::min<long long>((long long)num_sms() * 8, ((long long)n + U - 1) / U + 1);
    while (want > 0) {
        for (; want > 0; --want, ++level) {
            cudaMemsetAsync(a.lr, 0, sizeof(int) * 2 * cap, st);
            cudaMemsetAsync(a.acc, 0, sizeof(unsigned) * (size_t)cap * 4 * a.d, st);
            launch(st_scatter_kernel<S>, grid, kStThreads, 0, st, a, level);
            launch(st_level_kernel<S>, 1, 1024, 0, st, a, level);
        }
        cudaMemcpyAsync(pin, &a.state->active, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
        if (pin[0] > 0) want = 2;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, st_block_kernel<S>, kStThreads, smem) != cudaSuccess || per_sm < 1)
        return WM_ECUDA;
    launch(st_block_kernel<S>, n > M ? num_sms() * per_sm : 1, kStThreads, smem, st, a);
    launch(st_finish_kernel<S>, grid_for(n, 256), 256, 0, st, a);
    cudaMemcpyAsync(pin, a.state, sizeof(BuildState), cudaMemcpyDeviceToHost, st);
    if (cudaPeekAtLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    BuildState h;
    memcpy(&h, pin, sizeof h);
    if (h.bad) return WM_EINVAL;
    float delta;
    memcpy(&delta, &h.delta, sizeof delta);
    P.delta = delta;
    X.coarse = h.buckets > 0 ? (double)h.coarse / h.buckets : 0.0;
    X.Ns = h.next_id;
    X.depth = level + h.depth + 1;
    return 0;
}

}  // namespace

// Search tree and tree-order points of the input (device memory); n < 2^28 (28-bit positions in a
// bucket's reference).  P.x64 is set when the FP32 copy is inexact (FP64 input); P.x32 is not.
int build_search_tree(const void *src, int n, int d, int dtype, int layout, Points &P, SearchTree &X, Arena &ar,
                      cudaStream_t st, int *pin)
{
    P.n = n;
    P.d = d;
    X.S = row_floats(d);
    StArgs a;
    memset(&a, 0, sizeof a);
    a.n = n;
    a.d = d;
    a.dtype = dtype;
    a.layout = layout;
    a.src = src;
    X.rows = a.buf[0] = ar.get<float>((size_t)n * X.S);
    X.nodes = a.nodes = ar.get<float>((size_t)(2LL * n) * 2 * X.S);
    X.range = a.range = ar.get<int2>(2LL * n);
    X.parent = a.parent = ar.get<int>(2LL * n);
    P.pid = a.pid = ar.get<int>(n);
    P.pos = a.pos = ar.get<int>(n);
    a.x64 = dtype == WM_F64 ? ar.get<double>((size_t)n * d) : nullptr;
    if (ar.failed) return WM_ENOMEM;
    const size_t mark = ar.off;
    a.buf[1] = ar.get<float>((size_t)n * X.S);
    a.state = (BuildState *)ar.take(kStateBytes + sizeof(unsigned) * 4 * X.S);
    a.root_acc = (unsigned *)((char *)a.state + kStateBytes);   // (not used before the check below)
    if (ar.failed) return WM_ENOMEM;
    int rc;
    switch (X.S) {
    case 4: rc = build<4>(a, X, P, ar, st, pin); break;
    case 8: rc = build<8>(a, X, P, ar, st, pin); break;
    case 16: rc = build<16>(a, X, P, ar, st, pin); break;
    default: rc = build<24>(a, X, P, ar, st, pin); break;
    }
    if (rc) return rc;
    P.x64 = P.delta > 0.f ? a.x64 : nullptr;
    ar.off = mark;
    // stacks of the walks
    X.root = n > kBucket ? 1u : bucket_ref(0, n);
    X.stack_cap = X.depth + 4;
    X.deep_levels = std::max(1, X.stack_cap - kWalkStack);
    X.walk_blocks = (int)std::min<long long>((long long)num_sms() * (2048 / kWalkThreads),
                                             ((long long)n + kWalkThreads - 1) / kWalkThreads);
    // a very deep tree (hundreds of levels) of few points gets fewer blocks rather than larger stacks
    const long long per_block = (long long)kWalkThreads * X.deep_levels * (long long)sizeof(uint2);
    X.walk_blocks = (int)std::min<long long>(X.walk_blocks, std::max(1LL, std::max(8LL << 20, 256LL * n) / per_block));
    X.deep = ar.get<uint2>((size_t)X.walk_blocks * kWalkThreads * X.deep_levels);
    return ar.failed ? WM_ENOMEM : 0;
}

}  // namespace wm
