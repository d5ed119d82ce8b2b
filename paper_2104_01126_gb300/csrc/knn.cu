// knn.cu -- core distances for HDBSCAN* (Sec. 2.1: cd(p) = distance to the minPts-th nearest
// neighbour, p itself counted; Sec. 2.3 / 3.1.3: computed with k-NN queries, k = minPts), the
// per-node cd_min / cd_max bounds (Table 1) and the repair edges that make the returned MST the
// canonical one under the key K.
//
// k-NN: one thread per query walks the search tree (stree.cuh), the nearer child first, and
// keeps the minPts smallest screened (FP32) values in a 4-ary max-heap in shared memory (slot-major, one bank per
// lane).  A node is skipped when its box is provably beyond the band threshold T of the heap's top, so
// every point that the walk does not evaluate screens above T.  The smallest value that the heap
// turned away or gave up (out) then tells whether the heap holds exactly the points screened within
// T(s_k): if out > T(s_k), the k-th squared distance is the largest FP64 distance of the heap's points
// and all of them (but the point itself) are its repair edges.  Otherwise (ties within the band) a warp
// collects every point within T(s_k), evaluates them in FP64 and selects the k-th; a band of more than
// kTieCap points (heavy duplicates) is answered by an exact FP64 scan of all points.
//
// The plain FP64 form is the same walk with every point distance evaluated in FP64: the heap holds them
// rounded to FP32.
//
// Repair edges: R = {(p,q), q != p : w2(p,q) <= cd2(p)}, weighted by the mutual reachability
// distance.  Under general position every edge of the K-minimum spanning tree of G_MR either has
// a weight no other edge has (then every MST contains it, the WSPD-derived candidates too) or has
// d(p,q) <= max(cd(p), cd(q)) (then it is in R); adding R to the MemoGFK batches of their weight
// range therefore yields the K-minimum tree itself.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "hdb.cuh"
#include "screen.cuh"
#include "stree.cuh"
#include "wspd.cuh"

namespace wm {

namespace {

struct KnnArgs {
    int n, d, k;
    const double *x64;   // FP64 coordinates where the rows are rounded copies, else null
    double *cd64;
    float *cd32;
    int rq;              // slots of a repair row
    int *rep_q;          // [rq][n] tree positions
    double *rep_d;       // [rq][n] FP64 squared distances
    int *rep_cnt;        // [n]
    int *slow;           // queries with ties around the k-th value
    float *slow_s;       // their screened k-th values
    int *slow_cnt;
    int *slow2;          // queries left for the full scan
    int *slow2_cnt;
    unsigned long_evals; // a walk that has evaluated more points than this is handed to the full scan,
    int *long_cnt;       // kKnnLongMax of them at most
    int *next_group;     // dispenser of 32-query groups
    int *err;            // set when a traversal stack would overflow (an internal error)
    unsigned long long *stat;   // [0] evals, [1] fp64 rechecks, [2] bits of the largest relative
                                //     error of a screened k-th value against the exact one
};

// FP64 form: a walk that has evaluated a 32nd of all points (and knn_long_evals) is an outlier, such as the
// centre of a sphere of points, which visits every node on one lane while the GPU waits: it goes to the full
// scan's blocks.  Where that is what every walk does (high dimension), the first four per SM are scanned.  Up to 5
// dimensions ordinary walks stay far below 2048 evaluations at minPts 10; above, and with long lists, they do not
// (with 4096 in 7-D, 60,000 points at minPts 256 took 89 ms instead of 60).
// (HDBSCAN* of 50,000 points on a sphere and their centre 68 -> 5.5 ms, of 10,000 14.6 -> 4.5, with the searches' own
// hand-over.  The FP32 walk is four times as fast per point, and the test cost every call 2 %.)
inline unsigned knn_long_evals(int D, int n, int k) { return std::max(D <= 5 ? std::min(2048 * (1 + k / 32), 16384) : 16384, n / 32); }
constexpr int kKnnLongMax = 608;

// -------------------------------------------------------------------------- thread per query
// Shared memory of a block of T threads: uint2 stk[kWalkStack][T], uint2 heap[k][T] (value bits,
// position), both slot-major: a lane's slots lie in its own banks, whatever slots its neighbours use.
template <int D, bool F64>
__global__ void __launch_bounds__(kWalkThreads, F64 ? 1 : D <= 3 ? 8 : 6) knn_walk_kernel(KnnArgs a, SearchTree X, TravArgs band)
{
    extern __shared__ uint2 walk_smem[];
    constexpr int S = row_floats(D);
    constexpr bool kStream = S > 4;
    const int lane = threadIdx.x & 31, T = blockDim.x;
    uint2 *heap = walk_smem + (size_t)kWalkStack * T + threadIdx.x;
    const int n = a.n, k = a.k;
    unsigned long long n_ev = 0, n_re = 0;
    float kerr = 0.f;   // largest relative error of a screened k-th value
    // the lane's query
    float q[S];
    int i = 0, cnt = 0;
    float top = 0.f;   // the heap's largest value once it is full
    float out = 0.f;   // the smallest value that is not in the heap
    float pb = 0.f;    // a node whose lower bound exceeds pb holds no point within T(top)
    unsigned ev = 0;
    auto begin = [&](int t) {
        i = t;
        load_row<S>(X.rows, i, q);
        cnt = 0;
        top = out = pb = INFINITY;
        ev = 0;
    };
    auto bound = [](unsigned, float &, float &) {};
    auto need = [&](float g, int) { return g <= pb; };
    auto pending = [&](float g) { return g <= pb; };
    auto scan = [&](int j0, int sz) {
        // screened values first, then the ones below the top enter the heap, so that the lanes of a
        // warp run their insertions together
        float s[kBucket];
        unsigned todo = 0;
#pragma unroll
        for (int h = 0; h < kBucket; h += 4) {
            if (h && h >= sz) break;
#pragma unroll
            for (int p = h; p < h + 4; ++p) {
                float x[S];
                const int j = j0 + min(p, sz - 1);
                load_row<S, kStream>(X.rows, j, x);
                if (F64) {
                    // (FP64 is slow enough that even a point is first tried against the bound)
                    if (p < sz && point_bound<D>(q, x, row_error(band.delta32)) <= pb) todo |= 1u << p;
                } else {
                    s[p] = row_dist<D>(q, x);
                    if (p < sz) {
                        if (s[p] < top) todo |= 1u << p;
                        else out = fminf(out, s[p]);
                    }
                }
            }
        }
        ev += F64 ? __popc(todo) : (unsigned)sz;
        while (todo) {
            const int p = __ffs(todo) - 1;
            todo &= todo - 1;
            float v;
            if (F64) {
                float x[S];
                load_row<S, kStream>(X.rows, j0 + p, x);
                v = screen_dist<D, S, F64>(a.x64, n, a.d, X.rows, i, j0 + p, q, x);
            } else {
                v = s[0];
#pragma unroll
                for (int r = 1; r < kBucket; ++r) v = r == p ? s[r] : v;
            }
            const uint2 mine = make_uint2(__float_as_uint(v), (unsigned)(j0 + p));
            if (cnt < k) {   // fill: sift up
                int h = cnt++;
                while (h > 0) {
                    const int u = (h - 1) >> 2;
                    const uint2 e = heap[u * T];
                    if (__uint_as_float(e.x) >= v) break;
                    heap[h * T] = e;
                    h = u;
                }
                heap[h * T] = mine;
                if (cnt == k) top = __uint_as_float(heap[0].x);
            } else if (v < top) {   // replace the top: sift down
                out = fminf(out, top);
                int h = 0;
                while (true) {
                    const int u0 = 4 * h + 1;
                    if (u0 >= k) break;
                    int u = u0;
                    uint2 e = heap[u0 * T];
#pragma unroll
                    for (int c = 1; c < 4; ++c) {
                        const int uc = min(u0 + c, k - 1);
                        const uint2 f = heap[uc * T];
                        if (__uint_as_float(f.x) > __uint_as_float(e.x)) { e = f; u = uc; }
                    }
                    if (__uint_as_float(e.x) <= v) break;
                    heap[h * T] = e;
                    h = u;
                }
                heap[h * T] = mine;
                top = __uint_as_float(heap[0].x);
            } else {
                out = fminf(out, v);
            }
        }
        pb = screen_threshold(top, band) * (1.0f + 1.0f / 131072.0f);
        if (F64 && ev > a.long_evals) {
            n_ev += ev;
            ev = 0;
            if (*(volatile int *)a.long_cnt < kKnnLongMax && atomicAdd(a.long_cnt, 1) < kKnnLongMax) {
                a.slow2[atomicAdd(a.slow2_cnt, 1)] = i;
                pb = -1.f;   // nothing left to visit
            }
        }
    };
    auto finish = [&] {
        n_ev += ev;
        if (F64 && pb < 0.f) return;   // handed over
        if (cnt < k || !(out > screen_threshold(top, band))) {
            const int t = atomicAdd(a.slow_cnt, 1);
            a.slow[t] = i;
            a.slow_s[t] = top;
            return;
        }
        // the k points of the heap are the k nearest; all but the point itself are repair edges
        unsigned long long cd = 0;
        int r = 0;
        for (int h = 0; h < k; ++h) {
            const int j = (int)heap[h * T].y;
            if (j == i) continue;
            const double w = walk_dist64<D, S>(a.x64, n, a.d, X.rows, i, j);
            cd = max(cd, (unsigned long long)__double_as_longlong(w));
            if (r < a.rq) {
                a.rep_q[(size_t)r * n + i] = j;
                a.rep_d[(size_t)r * n + i] = w;
                ++r;
            }
        }
        n_re += (unsigned long long)k;
        const double cd2 = __longlong_as_double((long long)cd);
        a.cd64[i] = cd2;
        a.cd32[i] = __double2float_rn(cd2);
        a.rep_cnt[i] = r;
        if (!F64 && cd2 > 0.0)
            kerr = fmaxf(kerr, __fdiv_ru(__double2float_ru(fabs((double)top - cd2)), __double2float_rd(cd2)));
    };
    walk_queries<D, S, kStream>(X, n, a.next_group, walk_smem + threadIdx.x, T, X.deep + (size_t)blockIdx.x * T + threadIdx.x,
                                (size_t)gridDim.x * T, a.err, 1, q, begin, bound, need, pending, scan, finish);
    n_ev = warp_sum_u64(n_ev);
    n_re = warp_sum_u64(n_re);
    for (int o = 16; o; o >>= 1) kerr = fmaxf(kerr, __shfl_xor_sync(0xffffffffu, kerr, o));
    if (lane == 0) {
        atomicAdd(a.stat + 0, n_ev);
        atomicAdd(a.stat + 1, n_re);
        if (kerr > 0.f) atomicMax(a.stat + 2, (unsigned long long)__float_as_uint(kerr));
    }
}

// Ties around the k-th value: a warp per query collects every point within the band of the screened
// k-th value, evaluates them in FP64 and takes the k-th smallest.
constexpr int kTieCap = 512, kTieWarps = 4;

template <int D, bool F64>
__global__ void __launch_bounds__(32 * kTieWarps) knn_tie_kernel(KnnArgs a, SearchTree X, TravArgs band,
                                                                 const int *__restrict__ m_dev, int *next, int *slow2,
                                                                 int *slow2_cnt, int *extra_q, int *extra_p,
                                                                 double *extra_d, int *extra_cnt, int extra_cap,
                                                                 int *tie_overflow)
{
    __shared__ int cj_[kTieWarps][kTieCap];
    __shared__ double cw_[kTieWarps][kTieCap];
    extern __shared__ uint2 walk_smem[];
    constexpr int S = row_floats(D);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int *cj = cj_[wib];
    double *cw = cw_[wib];
    unsigned *stk = (unsigned *)walk_smem + (size_t)wib * (X.stack_cap + 2);
    const int n = a.n, k = a.k, m = *m_dev;
    unsigned long long n_re = 0;
    while (true) {
        int t = 0;
        if (lane == 0) t = atomicAdd(next, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= m) break;
        const int i = a.slow[t];
        const float Tk = screen_threshold(a.slow_s[t], band);
        const float pb = Tk * (1.0f + 1.0f / 131072.0f);
        float q[S];
        load_row<S>(X.rows, i, q);
        int c = 0, sp = 1;
        __syncwarp();
        if (lane == 0) stk[0] = X.root;
        __syncwarp();
        while (sp > 0 && c <= kTieCap) {
            const unsigned ref = stk[sp - 1];
            __syncwarp();
            --sp;
            bool take = false;
            int j = 0;
            if (ref & kBucketBit) {
                const int sz = (int)((ref >> 28) & 7u) + 1;
                if (lane < sz) {
                    j = (int)(ref & 0x0fffffffu) + lane;
                    float x[S];
                    load_row<S>(X.rows, j, x);
                    take = screen_dist<D, S, F64>(a.x64, n, a.d, X.rows, i, j, q, x) <= Tk;
                }
                const unsigned b = __ballot_sync(0xffffffffu, take);
                const int slot = c + __popc(b & lanemask_lt());
                if (take && slot < kTieCap) cj[slot] = j;
                c += __popc(b);
            } else {
                float g0, g1;
                unsigned r0, r1;
                int l0, l1;
                visit_children<D, S, false>(X.nodes, ref, q, g0, g1, r0, r1, l0, l1);
                if (sp + 2 > X.stack_cap + 2) {   // cannot happen: one entry per level and one more
                    if (lane == 0) atomicOr(a.err, 1);
                    break;
                }
                if (lane == 0) {
                    int u = sp;
                    if (g0 <= pb) stk[u++] = r0;
                    if (g1 <= pb) stk[u++] = r1;
                }
                __syncwarp();
                sp += (g0 <= pb) + (g1 <= pb);
            }
        }
        __syncwarp();
        if (c > kTieCap || c < k) {
            if (lane == 0) slow2[atomicAdd(slow2_cnt, 1)] = i;
            continue;
        }
        for (int e = lane; e < c; e += 32) cw[e] = cj[e] == i ? 0.0 : walk_dist64<D, S>(a.x64, n, a.d, X.rows, i, cj[e]);
        n_re += (unsigned long long)(lane == 0 ? c : 0);
        __syncwarp();
        // the k-th smallest: the value with fewer than k values below it and at least k at or below it
        unsigned long long kth = 0;
        for (int e = lane; e < c; e += 32) {
            const unsigned long long v = (unsigned long long)__double_as_longlong(cw[e]);
            int lt = 0, le = 0;
            for (int f = 0; f < c; ++f) {
                const unsigned long long u = (unsigned long long)__double_as_longlong(cw[f]);
                lt += u < v;
                le += u <= v;
            }
            if (lt < k && le >= k) kth = v;
        }
        for (int o = 16; o; o >>= 1) kth = max(kth, __shfl_xor_sync(0xffffffffu, kth, o));
        const double cd2 = __longlong_as_double((long long)kth);
        // its repair edges: into the row when they fit, else all into the overflow list
        int total = 0;
        for (int e = lane; e < c; e += 32)
            total += cj[e] != i && (unsigned long long)__double_as_longlong(cw[e]) <= kth;
        total = __reduce_add_sync(0xffffffffu, total);
        int xbase = 0, r = 0;
        if (total > a.rq) {
            if (lane == 0) xbase = atomicAdd(extra_cnt, total);
            xbase = __shfl_sync(0xffffffffu, xbase, 0);
        }
        for (int e0 = 0; e0 < c; e0 += 32) {
            const int e = e0 + lane;
            const bool keep = e < c && cj[e] != i && (unsigned long long)__double_as_longlong(cw[e]) <= kth;
            const unsigned b = __ballot_sync(0xffffffffu, keep);
            const int slot = r + __popc(b & lanemask_lt());
            if (keep) {
                if (total <= a.rq) {
                    a.rep_q[(size_t)slot * n + i] = cj[e];
                    a.rep_d[(size_t)slot * n + i] = cw[e];
                } else if (xbase + slot < extra_cap) {
                    extra_p[xbase + slot] = i;
                    extra_q[xbase + slot] = cj[e];
                    extra_d[xbase + slot] = cw[e];
                } else {
                    atomicOr(tie_overflow, 1);
                }
            }
            r += __popc(b);
        }
        if (lane == 0) {
            a.cd64[i] = cd2;
            a.cd32[i] = __double2float_rn(cd2);
            a.rep_cnt[i] = total <= a.rq ? total : 0;
        }
        __syncwarp();
    }
    if (lane == 0 && n_re) atomicAdd(a.stat + 1, n_re);
}

// exact squared distance from the FP64 coordinates, or (x64 null) from rows of S floats
__device__ inline double any_dist64(const double *__restrict__ x64, const float *__restrict__ rows, int S, int n, int d, int i,
                                    int j)
{
    if (x64) return dist64(x64, n, d, i, j);
    double s = 0.0;
    for (int k = 0; k < d; ++k) {
        const double t = __dsub_rn((double)rows[(size_t)i * S + k], (double)rows[(size_t)j * S + k]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// rigorous lower bound of any_dist64 from the rows (point_bound at run time)
__device__ inline float any_bound(const float *__restrict__ rows, int S, int d, int i, int j, float rel)
{
    float g = 0.f;
    for (int k = 0; k < d; ++k) {
        const float q = rows[(size_t)i * S + k], x = rows[(size_t)j * S + k];
        const float t = fmaxf(fmaf(-rel, fmaxf(fabsf(q), fabsf(x)), fabsf(q - x)), 0.f);
        g = fmaf(t, t, g);
    }
    return lower_w2(g);
}

// Exact FP64 answer for one query per block (ties or duplicates overflowed the list, or a walk that does not
// end): each thread keeps the k smallest w2 of its strided share, the block merges the lists, then a
// second scan collects every q with w2 <= cd2 as repair edges.  A point whose FP32 bound is beyond the
// list costs no FP64 (whose rate is 1/64).
__global__ void __launch_bounds__(256) knn_slow_kernel(KnnArgs a, const float *__restrict__ rows, int S, float rel,
                                                       const int *__restrict__ slow, int nslow,
                                                       int *extra_q, int *extra_p, double *extra_d, int *extra_cnt,
                                                       int extra_cap, int *tie_overflow)
{
    extern __shared__ double slow_lists[];   // [k][T]
    __shared__ double s_min[8];
    __shared__ int s_who;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const int k = a.k, n = a.n, d = a.d;
    double *lw = slow_lists + tid;
    for (int t = blockIdx.x; t < nslow; t += gridDim.x) {
        const int i = slow[t];
        int cnt = 0;
        float far = INFINITY;   // the list's largest value, rounded up, once it is full
        for (int j = tid; j < n; j += T) {
            if (any_bound(rows, S, d, i, j, rel) > far) continue;
            const double w = j == i ? 0.0 : any_dist64(a.x64, rows, S, n, d, i, j);
            if (cnt < k || w < lw[(k - 1) * T]) {
                int pos = cnt < k ? cnt : k - 1;
                while (pos > 0 && lw[(pos - 1) * T] > w) { lw[pos * T] = lw[(pos - 1) * T]; --pos; }
                lw[pos * T] = w;
                if (cnt < k) ++cnt;
                if (cnt == k) far = __double2float_ru(lw[(k - 1) * T]);
            }
        }
        int head = 0;
        double kth = 0.0;
        for (int r = 0; r < k; ++r) {   // (n >= k points are in the lists)
            const double mine = head < cnt ? lw[head * T] : INFINITY;
            double mn = mine;
            for (int o = 16; o; o >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            if (lane == 0) s_min[tid >> 5] = mn;
            if (tid == 0) s_who = T;
            __syncthreads();
            for (int w = 0; w < T / 32; ++w) mn = fmin(mn, s_min[w]);
            if (mine == mn && head < cnt) atomicMin(&s_who, tid);
            __syncthreads();
            if (tid == s_who) ++head;
            kth = mn;
            __syncthreads();
        }
        if (tid == 0) {
            a.cd64[i] = kth;
            a.cd32[i] = __double2float_rn(kth);
            a.rep_cnt[i] = 0;
        }
        far = __double2float_ru(kth);
        for (int j = tid; j < n; j += T) {
            if (j == i || any_bound(rows, S, d, i, j, rel) > far) continue;
            const double w = any_dist64(a.x64, rows, S, n, d, i, j);
            if (w <= kth) {
                const int s = atomicAdd(extra_cnt, 1);
                if (s < extra_cap) { extra_p[s] = i; extra_q[s] = j; extra_d[s] = w; }
                else atomicOr(tie_overflow, 1);
            }
        }
    }
}

// node bounds of cd2, bottom-up with arrival counters
__global__ void cd_bounds_kernel(int N, const int *__restrict__ left, const int *__restrict__ right,
                                 const int *__restrict__ parent, const int *__restrict__ begin,
                                 const double *__restrict__ cd64, double *nmin, double *nmax, float *cdmin,
                                 float *cdmax, int *arrive)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        if (left[x] >= 0) continue;
        double c = cd64[begin[x]];
        nmin[x] = c; nmax[x] = c;
        cdmin[x] = __double2float_rd(c);
        cdmax[x] = __double2float_ru(c);
        int cur = x;
        for (int it = 0; it < N; ++it) {
            int p = parent[cur];
            if (p < 0) break;
            __threadfence();
            if (atomicAdd(&arrive[p], 1) == 0) break;
            __threadfence();
            double a0 = ((volatile double *)nmin)[left[p]], a1 = ((volatile double *)nmin)[right[p]];
            double b0 = ((volatile double *)nmax)[left[p]], b1 = ((volatile double *)nmax)[right[p]];
            double mn = fmin(a0, a1), mx = fmax(b0, b1);
            nmin[p] = mn; nmax[p] = mx;
            cdmin[p] = __double2float_rd(mn);
            cdmax[p] = __double2float_ru(mx);
            cur = p;
        }
    }
}

// A pair (p, q) whose distance is within both core distances is in both points' lists: only the
// endpoint with the smaller input id emits it, so every repair edge appears once.
__device__ inline bool rep_keep(int i, int j, double D, const double *__restrict__ cd64, const int *__restrict__ pid)
{
    return !(__double_as_longlong(D) <= __double_as_longlong(cd64[j]) && pid[j] < pid[i]);
}

// repair edge of positions (i, j) with FP64 squared distance D: weight max(cd2 i, cd2 j, D); appended in
// no particular order
__global__ void rep_emit_kernel(const int *__restrict__ rep_q, const double *__restrict__ rep_d,
                                const int *__restrict__ rep_cnt, int n, const double *__restrict__ cd64,
                                const int *__restrict__ pid, EdgeK *__restrict__ out, int *count)
{
    __shared__ int sh[32];
    for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
        const int i = b0 + threadIdx.x;
        const int m = i < n ? rep_cnt[i] : 0;
        int k = 0;
        for (int r = 0; r < m; ++r) k += rep_keep(i, rep_q[(size_t)r * n + i], rep_d[(size_t)r * n + i], cd64, pid);
        int o = block_append(count, k, sh);
        for (int r = 0; r < m; ++r) {
            const int j = rep_q[(size_t)r * n + i];
            const double D = rep_d[(size_t)r * n + i];
            if (!rep_keep(i, j, D, cd64, pid)) continue;
            const double c = __double_as_longlong(cd64[i]) >= __double_as_longlong(cd64[j]) ? cd64[i] : cd64[j];
            out[o++] = make_edge(__double_as_longlong(c) >= __double_as_longlong(D) ? c : D, pid[i], pid[j]);
        }
    }
}

// the exact lists of the slow queries, appended after the others (count: running total)
__global__ void rep_emit_extra_kernel(const int *__restrict__ ep, const int *__restrict__ eq,
                                      const double *__restrict__ ed, const int *__restrict__ cnt, int cap,
                                      const double *__restrict__ cd64, const int *__restrict__ pid, EdgeK *__restrict__ out,
                                      int *count)
{
    __shared__ int sh[32];
    const int m = min(*cnt, cap);
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        bool keep = false;
        int i = 0, j = 0;
        double D = 0.0;
        if (t < m) {
            i = ep[t];
            j = eq[t];
            D = ed[t];
            keep = rep_keep(i, j, D, cd64, pid);
        }
        const int slot = block_append(count, keep ? 1 : 0, sh);
        if (keep) {
            const double c = __double_as_longlong(cd64[i]) >= __double_as_longlong(cd64[j]) ? cd64[i] : cd64[j];
            out[slot] = make_edge(__double_as_longlong(c) >= __double_as_longlong(D) ? c : D, pid[i], pid[j]);
        }
    }
}

__global__ void core_out_kernel(const double *__restrict__ cd64, const int *__restrict__ pid, int n, double *out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[pid[i]] = sqrt(cd64[i]);
}

}  // namespace

// Shared memory limits of the kernels above.  They are set to the same value by every call: a limit that
// followed the call's own size could be lowered by a concurrent call (batch groups, server workers)
// between another call's setting and its launch.
constexpr int kWalkSmemMax = 100 << 10;    // (kWalkStack + minPts) entries for at least 32 threads
constexpr int kTieSmemMax = 64 << 10;      // stacks of kTieWarps warps in the deepest tree (FP32 exponents
                                           // and mantissas allow about 3800 levels in 16 dimensions)
constexpr int kSlowSmemMax = 100 << 10;    // minPts values for at least 32 threads
static_assert(kMaxMinPts * 32 * 8 <= kSlowSmemMax, "shared memory limit of the full scan");
static_assert((kWalkStack + kMaxMinPts) * 32 * 8 <= kWalkSmemMax, "shared memory limit of the k-NN walk");

// core distances and repair edges (fp64: the plain form)
int core_distances(const Points &P, const SearchTree &X, int min_pts, bool fp64, HdbState &H, Arena &ar, cudaStream_t st,
                   int *pin, wm_stats *stats)
{
    const int n = P.n, d = P.d;
    if (min_pts > kMaxMinPts) return WM_EINVAL;
    const int KL = std::min(min_pts + 8, n);   // a point's repair edges: itself left out, up to 8 more by ties
    H.cd64 = ar.get<double>(n);
    H.cd32 = ar.get<float>(n);
    if (ar.failed) return WM_ENOMEM;
    // persistent output of this function: repair edges (allocated before the scratch)
    const int RQ = KL > 1 ? KL - 1 : 1;
    const int extra_cap = 4 * n + 1024;
    EdgeK *rep = ar.get<EdgeK>((size_t)n * RQ + extra_cap);
    if (!rep) return WM_ENOMEM;
    size_t mark = ar.off;
    KnnArgs a;
    memset(&a, 0, sizeof a);
    a.n = n; a.d = d; a.k = min_pts;
    a.x64 = P.x64;
    a.cd64 = H.cd64; a.cd32 = H.cd32;
    a.rq = RQ;
    a.rep_q = ar.get<int>((size_t)n * RQ);
    a.rep_d = ar.get<double>((size_t)n * RQ);
    a.rep_cnt = ar.get<int>(n + 1);
    a.slow = ar.get<int>(n);
    a.slow_s = ar.get<float>(n);
    int *slow2 = a.slow2 = ar.get<int>(n);
    // [0] queries with ties, [1] overflow edges, [2] overflow flag, [3] repair edges, [4] dispenser of
    // the tie kernel, [5] error, [6] dispenser of the walk, [7] queries left for the full scan, [8] walks
    // handed to it
    int *cnts = ar.get<int>(9);
    a.slow_cnt = cnts;
    a.stat = ar.get<unsigned long long>(4);
    int *ex_p = ar.get<int>(extra_cap), *ex_q = ar.get<int>(extra_cap);
    double *ex_d = ar.get<double>(extra_cap);
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(cnts, 0, 9 * sizeof(int), st);
    cudaMemsetAsync(a.stat, 0, 4 * sizeof(unsigned long long), st);
    a.next_group = cnts + 6;
    a.err = cnts + 5;
    a.slow2_cnt = cnts + 7;
    a.long_cnt = cnts + 8;
    a.long_evals = knn_long_evals(walk_dim(d), n, min_pts);
    cudaEvent_t k0, k1;
    cudaEventCreate(&k0);
    cudaEventCreate(&k1);
    {
        TravArgs band;
        band.eta = fp64 ? 0.0 : 2.0 * (double)P.delta * sqrt((double)d) * (1.0 + 1e-6);
        band.exact32 = band.eta == 0.0;
        band.delta32 = P.delta;
        band.eta2_f = (float)(2.0 * band.eta);
        if ((double)band.eta2_f < 2.0 * band.eta) band.eta2_f = std::nextafter(band.eta2_f, INFINITY);
        // threads per block: four warps while two blocks of them fit an SM's shared memory
        const size_t per_thread = (size_t)(kWalkStack + min_pts) * sizeof(uint2);
        int threads = kWalkThreads;
        while (threads > 32 && per_thread * threads > (size_t)kWalkSmemMax) threads >>= 1;
        const size_t smem = per_thread * threads;
        const size_t smem_tie = (size_t)kTieWarps * (X.stack_cap + 2) * sizeof(unsigned);
        int rc = 0;
#define WM_KNN_(DM, F)                                                                                            \
    do {                                                                                                      \
        int per_sm = 0;                                                                                       \
        if (cudaFuncSetAttribute(knn_walk_kernel<DM, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWalkSmemMax) != cudaSuccess || \
            cudaFuncSetAttribute(knn_tie_kernel<DM, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTieSmemMax) != cudaSuccess || \
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, knn_walk_kernel<DM, F>, threads, smem) != cudaSuccess || \
            per_sm < 1) {                                                                                     \
            rc = WM_ECUDA;                                                                                    \
            break;                                                                                            \
        }                                                                                                     \
        const int blocks = (int)std::min<long long>(std::min<long long>((long long)num_sms() * per_sm,        \
                                                    (long long)X.walk_blocks * (kWalkThreads / threads)),    \
                                                    ((long long)n + threads - 1) / threads);                  \
        cudaEventRecord(k0, st);                                                                              \
        launch(knn_walk_kernel<DM, F>, blocks, threads, smem, st, a, X, band);                                  \
        launch(knn_tie_kernel<DM, F>, num_sms() * 4, 32 * kTieWarps, smem_tie, st, a, X, band, cnts, cnts + 4, slow2,   \
               cnts + 7, ex_q, ex_p, ex_d, cnts + 1, extra_cap, cnts + 2);                                    \
        cudaEventRecord(k1, st);                                                                              \
    } while (0)
#define WM_KNN(DM)                 \
    if (fp64) WM_KNN_(DM, true);   \
    else WM_KNN_(DM, false)
        const int wd = walk_dim(d);
        if (row_floats(wd) != X.S) rc = WM_EINTERNAL;
        else switch (wd) {
            case 2: WM_KNN(2); break;
            case 3: WM_KNN(3); break;
            case 4: WM_KNN(4); break;
            case 5: WM_KNN(5); break;
            case 6: WM_KNN(6); break;
            case 7: WM_KNN(7); break;
            case 8: WM_KNN(8); break;
            case 15: WM_KNN(15); break;
            default: WM_KNN(16); break;
            }
#undef WM_KNN
#undef WM_KNN_
        if (rc) {
            cudaGetLastError();
            cudaEventDestroy(k0);
            cudaEventDestroy(k1);
            set_error_detail("k-NN: the launch configuration was refused");
            return rc;
        }
    }
    cudaMemcpyAsync(pin, cnts, 8 * sizeof(int), cudaMemcpyDeviceToHost, st);
    if (cudaPeekAtLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
        cudaEventDestroy(k0);
        cudaEventDestroy(k1);
        return WM_ECUDA;
    }
    if (stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, k0, k1);
        stats->ms_knn_kernel = ms;
    }
    cudaEventDestroy(k0);
    cudaEventDestroy(k1);
    const int nslow = pin[7];
    if (nslow > 0) {
        int threads = 256;
        while (threads > 32 && (size_t)min_pts * threads * 8 > (size_t)kSlowSmemMax) threads >>= 1;
        cudaFuncSetAttribute(knn_slow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSlowSmemMax);
        launch(knn_slow_kernel, std::min(nslow, num_sms() * 8), threads, (size_t)min_pts * threads * 8, st, a, X.rows, X.S,
               row_error(P.delta), slow2, nslow, ex_q, ex_p, ex_d, cnts + 1, extra_cap, cnts + 2);
    }
    // repair edges: one copy of each, weighted, in no particular order (each round takes those it needs)
    launch(rep_emit_kernel, grid_for(n, 256), 256, 0, st, a.rep_q, a.rep_d, a.rep_cnt, n, H.cd64, P.pid, rep, cnts + 3);
    launch(rep_emit_extra_kernel, grid_for(extra_cap, 256), 256, 0, st, ex_p, ex_q, ex_d, cnts + 1, extra_cap, H.cd64,
           P.pid, rep, cnts + 3);
    cudaMemcpyAsync(pin, cnts, 8 * sizeof(int), cudaMemcpyDeviceToHost, st);
    unsigned long long hs[3];
    cudaMemcpyAsync(pin + 8, a.stat, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    memcpy(hs, pin + 8, sizeof hs);
    if (pin[5]) {
        set_error_detail("k-NN: a traversal stack overflowed (internal error)");
        return WM_EINTERNAL;
    }
    const int nrep = pin[3];
    if (stats) {
        stats->knn_evals = (int64_t)hs[0];
        stats->fp64_rechecks += (int64_t)hs[1];
        stats->tie_overflow = pin[2] ? 1 : 0;
        float ke;
        const unsigned kb = (unsigned)hs[2];
        memcpy(&ke, &kb, sizeof ke);
        stats->max_rel_screen_err = std::max(stats->max_rel_screen_err, (double)ke);
    }
    H.rep = rep;
    H.nrep = nrep;
    ar.off = mark;
    // keep the cd arrays (allocated before mark); drop the scratch
    return 0;
}

// node bounds of the core distances for the WSPD traversals (T.arrive is scratch)
int node_core_bounds(const Tree &T, const HdbState &H, float *cdmin, float *cdmax, Arena &ar, cudaStream_t st)
{
    const int N = T.N;
    size_t mark = ar.off;
    double *nmin = ar.get<double>(N), *nmax = ar.get<double>(N);
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(T.arrive, 0, sizeof(int) * N, st);
    launch(cd_bounds_kernel, grid_for(N, 256), 256, 0, st, N, T.left, T.right, T.parent, T.begin, H.cd64, nmin, nmax, cdmin,
           cdmax, T.arrive);
    ar.off = mark;
    return 0;
}

int write_core_distances(const Points &P, const HdbState &H, double *out, Arena &ar, cudaStream_t st)
{
    if (!out) return 0;
    cudaPointerAttributes at;
    bool dev = cudaPointerGetAttributes(&at, out) == cudaSuccess &&
               (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    double *dst = out;
    if (!dev) {
        dst = ar.get<double>(P.n);
        if (!dst) return WM_ENOMEM;
    }
    launch(core_out_kernel, grid_for(P.n, 256), 256, 0, st, H.cd64, P.pid, P.n, dst);
    if (!dev) cudaMemcpyAsync(out, dst, sizeof(double) * P.n, cudaMemcpyDeviceToHost, st);
    return cudaStreamSynchronize(st) == cudaSuccess ? 0 : WM_ECUDA;
}

}  // namespace wm
