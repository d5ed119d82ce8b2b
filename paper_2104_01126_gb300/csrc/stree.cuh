// stree.cuh -- the search tree that the k-NN pass (knn.cu) and the nearest-component search
// (boruvka.cu) walk with one thread per query point.
//
// It is a spatial-median k-d tree down to buckets of at most kBucket points, siblings adjacent: about
// 0.4 nodes per point instead of the 2 of a tree with single-point leaves, so that the levels a walk
// visits most stay in L2.  A node row holds its box in groups of four dimensions (lo then hi, box_lo / box_hi, each
// group one 256-bit load) and, in the last padded dimension, a reference (lo slot) and a component
// label or -1 (hi slot): a visit reads the two child rows and nothing else.  A reference is the row of
// the left child, or for a bucket kBucketBit | (size - 1) << 28 | first point.  A point row holds the
// FP32 coordinates (of FP64 ones far from 0: less a centre) and, in its last slot, the point's component label.
#pragma once

#include "wm_internal.cuh"

namespace wm {

constexpr int kBucket = 8;        // points of a subtree that is scanned directly (3 bits in a reference)
constexpr int kWalkThreads = 128; // threads per block of the walking kernels
constexpr int kWalkStack = 16;    // stack entries of a thread in shared memory (the rest in global memory)
constexpr unsigned kBucketBit = 0x80000000u, kWalkDone = 0xffffffffu;

struct SearchTree {
    int S = 0;                    // floats per point row; a node row has 2 S
    int Ns = 0;                   // nodes
    unsigned root = 0;            // reference of the root
    float *rows = nullptr;        // [n][S]
    float *nodes = nullptr;       // [Ns][2 S]
    int2 *range = nullptr;        // [Ns] point range
    int *parent = nullptr;        // [Ns] (-1 at the root)
    uint2 *deep = nullptr;        // stack entries beyond kWalkStack, [deep_levels][walk_threads]
    int deep_levels = 0;
    int walk_blocks = 0;          // the largest grid the stacks are sized for
    int stack_cap = 0;            // entries of a thread's stack: one per tree level
    int depth = 0;                // levels
    double coarse = 0.0;          // share of the buckets whose extent the FP32 copy's largest error blurs
};

// rows of d coordinates and one more slot
__host__ __device__ constexpr int row_floats(int d) { return d <= 3 ? 4 : d <= 7 ? 8 : d <= 15 ? 16 : 24; }

// the compile-time dimension of the walks for d coordinates: d itself, or one above it whose rows have
// the same width (a padded coordinate is 0 in every row and box and adds nothing)
__host__ __device__ constexpr int walk_dim(int d) { return d <= 2 ? 2 : d <= 8 ? d : d <= 15 ? 15 : 16; }
constexpr bool walk_dims_fit(int d) { return d > 16 || (walk_dim(d) >= d && row_floats(walk_dim(d)) == row_floats(d) && walk_dims_fit(d + 1)); }
static_assert(walk_dims_fit(1), "a walk's rows must be as wide as the search tree's");

int build_search_tree(const void *src, int n, int d, int dtype, int layout, Points &P, SearchTree &X, Arena &ar,
                      cudaStream_t st, int *pin);

__host__ __device__ inline unsigned bucket_ref(int first, int size) { return kBucketBit | (unsigned)(size - 1) << 28 | (unsigned)first; }

#ifdef __CUDACC__
__device__ __forceinline__ float next_up(float x) { return x < INFINITY ? __uint_as_float(__float_as_uint(x) + 1u) : x; }

// 256-bit load of walk data.  A walk of many points touches far more rows between two uses of one than
// L1 holds (3.9 % of the sectors hit in 7-D), and every missed sector then costs L1 a second pass to
// fill it: with kStream the rows bypass L1 (EMST search of 10^7 points: 7-D 112.9 -> 94.6 ms, 5-D 30.4 ->
// 25.2).  Rows of up to 3 dimensions and the short HDBSCAN* searches do hit, and stay cached.
template <bool kStream>
__device__ __forceinline__ void ld_walk(const float *p, float4 &a, float4 &b)
{
    if (kStream)
        asm("ld.global.nc.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
            : "l"(p));
    else
        ldg256(p, a, b);
}

template <int S, bool kStream = false>
__device__ __forceinline__ void load_row(const float *__restrict__ rows, int i, float (&v)[S])
{
    if (S == 4) {
        const float4 p = *(const float4 *)(rows + (size_t)i * 4);
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
    } else {
#pragma unroll
        for (int c = 0; c < S / 8; ++c) {
            float4 p, q;
            ld_walk<kStream>(rows + (size_t)i * S + 8 * c, p, q);
            v[8 * c] = p.x; v[8 * c + 1] = p.y; v[8 * c + 2] = p.z; v[8 * c + 3] = p.w;
            v[8 * c + 4] = q.x; v[8 * c + 5] = q.y; v[8 * c + 6] = q.z; v[8 * c + 7] = q.w;
        }
    }
}

// FP32 squared distance of q to a point row
template <int D, int S>
__device__ __forceinline__ float row_dist(const float (&q)[S], const float (&x)[S])
{
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float t = q[k] - x[k];
        s = fmaf(t, t, s);
    }
    return s;
}

// exact FP64 squared distance of positions i and j: from the FP64 coordinates where the rows are rounded
// copies (x64 not null), else from the rows, which then hold the coordinates themselves
template <int D, int S>
__device__ inline double walk_dist64(const double *__restrict__ x64, int n, int d, const float *__restrict__ rows, int i, int j)
{
    double s = 0.0;
    if (x64) {
        for (int k = 0; k < d; ++k) {
            const double t = __dsub_rn(x64[(size_t)k * n + i], x64[(size_t)k * n + j]);
            s = __dadd_rn(s, __dmul_rn(t, t));
        }
    } else {
        float x[S], y[S];
        load_row<S>(rows, i, x);
        load_row<S>(rows, j, y);
#pragma unroll
        for (int k = 0; k < D; ++k) {   // a padded coordinate is 0 on both sides and adds exactly 0
            const double t = __dsub_rn((double)x[k], (double)y[k]);
            s = __dadd_rn(s, __dmul_rn(t, t));
        }
    }
    return s;
}

// True when no FP32 operation of the squared distance s of two rows rounds, so that every FP64 one gives the same.
// (Differences and sums by their errors after Knuth, squares by the fused remainder, which is exact above 2^-60.)
template <int D, int S>
__device__ __forceinline__ bool dist32_is_exact(const float (&x)[S], const float (&y)[S], float &s)
{
    s = 0.f;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float t = __fsub_rn(x[k], y[k]), u = __fsub_rn(t, x[k]);
        ok = ok && __fsub_rn(x[k], __fsub_rn(t, u)) == __fadd_rn(y[k], u);
        const float p = __fmul_rn(t, t);
        ok = ok && (t == 0.f || (p > 8.7e-19f && __fmaf_rn(t, t, -p) == 0.f));
        const float r = __fadd_rn(s, p), v = __fsub_rn(r, s);
        ok = ok && __fsub_rn(s, __fsub_rn(r, v)) == __fsub_rn(v, p);
        s = r;
        if (!ok) break;
    }
    return ok;
}

// walk_dist64 of two positions that may tie with others: rows of few significant bits, which is what ties
// (lattices), need no FP64 operation, whose rate is a 64th.  (EMST of a 7-D lattice of 280,000 points 7.6 -> 6.3 ms, FP64
// form 10.4 -> 8.6; on rows whose operations round the test ends with the first dimension.)
template <int D, int S>
__device__ inline double tie_dist64(const double *__restrict__ x64, int n, int d, const float *__restrict__ rows, int i, int j)
{
    if (!x64) {
        float x[S], y[S], s;
        load_row<S>(rows, i, x);
        load_row<S>(rows, j, y);
        if (dist32_is_exact<D, S>(x, y, s)) return (double)s;
    }
    return walk_dist64<D, S>(x64, n, d, rows, i, j);
}

// screened distance of positions i (row q) and j (row x): the FP32 distance of the rows, or in the plain
// form the FP64 distance rounded to FP32 (which only orders lists and bounds; decisions compare FP64)
template <int D, int S, bool F64>
__device__ inline float screen_dist(const double *__restrict__ x64, int n, int d, const float *__restrict__ rows, int i, int j,
                                    const float (&q)[S], const float (&x)[S])
{
    return F64 ? __double2float_rn(walk_dist64<D, S>(x64, n, d, rows, i, j)) : row_dist<D>(q, x);
}

// Relative error of a coordinate difference of two rounded rows, for point_bound (0: exact rows): both round by
// at most 2^-24 of the larger magnitude.
__host__ __device__ constexpr float row_error(float delta) { return delta > 0.f ? 1.2e-7f : 0.f; }   // > 2^-23

// rigorous lower bound of the FP64 squared distance from two rows: the node bound of visit_children for a
// single point
template <int D, int S>
__device__ __forceinline__ float point_bound(const float (&q)[S], const float (&x)[S], float rel)
{
    float g = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float t = fmaxf(fmaf(-rel, fmaxf(fabsf(q[k]), fabsf(x[k])), fabsf(q[k] - x[k])), 0.f);
        g = fmaf(t, t, g);
    }
    return lower_w2(g);
}

// One visit: rigorous lower bounds of the FP64 squared distance from q to the boxes of the children
// cur and cur + 1, their references and labels.
template <int D, int S, bool kStream>
__device__ __forceinline__ void visit_children(const float *__restrict__ nodes, unsigned cur, const float (&q)[S],
                                               float &g0, float &g1, unsigned &r0, unsigned &r1, int &l0, int &l1)
{
    const float *bx = nodes + (size_t)cur * 2 * S;
    g0 = 0.f;
    g1 = 0.f;
#pragma unroll
    for (int g = 0; g < S / 4; ++g) {
        float4 lo0, hi0, lo1, hi1;
        ld_walk<kStream>(bx + 8 * g, lo0, hi0);
        ld_walk<kStream>(bx + 2 * S + 8 * g, lo1, hi1);
        const float a0[4] = {lo0.x, lo0.y, lo0.z, lo0.w}, z0[4] = {hi0.x, hi0.y, hi0.z, hi0.w};
        const float a1[4] = {lo1.x, lo1.y, lo1.z, lo1.w}, z1[4] = {hi1.x, hi1.y, hi1.z, hi1.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (4 * g + k < D) {
                const float u = fmaxf(fmaxf(a0[k] - q[4 * g + k], q[4 * g + k] - z0[k]), 0.f);
                const float v = fmaxf(fmaxf(a1[k] - q[4 * g + k], q[4 * g + k] - z1[k]), 0.f);
                g0 = fmaf(u, u, g0);
                g1 = fmaf(v, v, g1);
            }
        }
        if (g == S / 4 - 1) {
            r0 = __float_as_uint(lo0.w);
            r1 = __float_as_uint(lo1.w);
            l0 = __float_as_int(hi0.w);
            l1 = __float_as_int(hi1.w);
        }
    }
    g0 = lower_w2(g0);
    g1 = lower_w2(g1);
}

// The walk of a warp whose lanes answer one query each.  A lane either stands at an internal node, at a
// bucket, or is idle; every step the warp runs the phase (visit the children / scan the bucket) that
// more of its lanes wait for, and once walk_refill(D) lanes are idle they finish their queries and take
// the next ones together.  As a plain loop per thread the same walk kept 4 (7-D) to 7 (3-D) of 32 lanes
// active per instruction, since the descents of neighbouring queries differ in length; now 16 (7-D, first
// search of 2x10^6 points: 25.2 -> 14.8 ms).  Taking two or four neighbouring queries along one path was
// slower: the union of their paths is 1.6 and 2.5 times one's.
//   begin(t)       sets the lane up for query t (in [0, m))
//   bound(c, g..)  may raise the lower bounds of the children c and c + 1
//   need(g, l)     true when a child with lower bound g and label l has to be visited
//   pending(g)     the same for a pending node, against the bound as it is now
//   scan(j0, sz)   the points [j0, j0 + sz) of a bucket; called by a subset of the warp's lanes
//   finish()       the lane's query is answered
__host__ __device__ constexpr int walk_refill(int D) { return D <= 3 ? 32 : 16; }

template <int D, int S, bool kStream, class Begin, class Bound, class Need, class Pending, class Scan, class Finish>
__device__ __forceinline__ void walk_queries(const SearchTree &X, int m, int *next, uint2 *stk, int stk_stride, uint2 *deep,
                                             size_t deep_stride, int *err, int err_bit, const float (&q)[S],
                                             const Begin &begin, const Bound &bound, const Need &need,
                                             const Pending &pending, const Scan &scan, const Finish &finish)
{
    const int lane = threadIdx.x & 31;
    unsigned cur = kWalkDone;
    int sp = 0;
    bool live = false, more = true;
    auto pop = [&] {
        cur = kWalkDone;
        while (sp > 0) {
            --sp;
            const uint2 e = sp < kWalkStack ? stk[sp * stk_stride] : deep[(size_t)(sp - kWalkStack) * deep_stride];
            if (pending(__uint_as_float(e.y))) { cur = e.x; break; }
        }
    };
    while (true) {
        const unsigned idle = __ballot_sync(0xffffffffu, cur == kWalkDone);
        if (idle == 0xffffffffu || (more && __popc(idle) >= walk_refill(D))) {
            if (cur == kWalkDone && live) {
                finish();
                live = false;
            }
            __syncwarp();
            if (more) {
                int base = 0;
                if (lane == __ffs(idle) - 1) base = atomicAdd(next, __popc(idle));
                base = __shfl_sync(0xffffffffu, base, __ffs(idle) - 1);
                const int t = base + __popc(idle & lanemask_lt());
                if (cur == kWalkDone && t < m) {
                    begin(t);
                    live = true;
                    cur = X.root;
                    sp = 0;
                }
                more = base + __popc(idle) < m;
                __syncwarp();
            }
            if (!__any_sync(0xffffffffu, live)) break;
        }
        const bool inner = !(cur & kBucketBit);
        const unsigned ni = __ballot_sync(0xffffffffu, inner);
        const unsigned nb = __ballot_sync(0xffffffffu, !inner && cur != kWalkDone);
        if (__popc(ni) >= __popc(nb)) {
            if (inner) {
                float g0, g1;
                unsigned r0, r1;
                int l0, l1;
                visit_children<D, S, kStream>(X.nodes, cur, q, g0, g1, r0, r1, l0, l1);
                bound(cur, g0, g1);
                const bool n0 = need(g0, l0), n1 = need(g1, l1);
                if (n0 || n1) {
                    const bool sw = !n0 || (n1 && g1 < g0);   // true: child 1 next
                    if (n0 && n1) {
                        const uint2 far = sw ? make_uint2(r0, __float_as_uint(g0)) : make_uint2(r1, __float_as_uint(g1));
                        if (sp < kWalkStack) stk[sp * stk_stride] = far;
                        else if (sp < X.stack_cap) deep[(size_t)(sp - kWalkStack) * deep_stride] = far;
                        else { atomicOr(err, err_bit); --sp; }   // cannot happen: one entry per level
                        ++sp;
                    }
                    cur = sw ? r1 : r0;
                } else {
                    pop();
                }
            }
        } else if (!inner && cur != kWalkDone) {
            scan((int)(cur & 0x0fffffffu), (int)((cur >> 28) & 7u) + 1);
            pop();
        }
        __syncwarp();
    }
}
#endif

}  // namespace wm
