// boruvka.cu -- nearest-component rounds: the K-minimum spanning tree by Boruvka's algorithm over the
// k-d tree (the dual-tree form is March, Ram and Gray, KDD 2010, which Sec. 5 compares with), the
// search done by warps.
//
// A round finds, for every component of the forest built so far, its K-smallest outgoing edge and
// links the components along those edges.  Under the strict key K = (w2, min id, max id) each such
// edge belongs to the one K-minimum spanning tree, so the rounds return exactly the tree that the
// MemoGFK rounds return.
//
// Every point i (tree position) keeps a list of its nearest points outside its component, with
// screened FP32 weights, and a radius R[i]: every point outside the component that is not in the
// list screens at R[i] or above.  A round then
//   refresh : drops the list heads that have joined i's component and WriteMins the first remaining
//             weight into S[c], the component's screened minimum;
//   active  : collects the points with R[i] <= T(S[c]) (T: the band threshold of the screen), i.e.
//             those that could still hold a lighter edge than the lists show, and those with a list
//             entry within T(S[c]);
//   search  : a thread per active point walks the k-d tree, the nearer child first, skipping nodes of
//             its own component and nodes beyond its bound, and rebuilds the point's list;
//   pick    : of these, the points with a list entry still within T(S[c]); FP64 evaluation of those entries
//             and the K-minimum per component by two 64-bit WriteMins; a point whose list may have
//             dropped a tie (R[i] <= T(S[c]) still) is answered by a walk that evaluates everything
//             within T(S[c]) in FP64;
//   merge   : every root links to the other endpoint's component; of a mutual choice the smaller root
//             stays and the edge is emitted once.  Then the roots left are collected and the points
//             and nodes relabelled.
// (Asking only the components of up to 1, 2 or 4 times the average size in a round was no faster on any
// of the 10^7-point sets: the others cost little to ask, and more rounds are needed.)
// The lists of the first search (all points, nothing pruned) serve the first few rounds.
//
// The plain form (WM_PREC_FP64) runs the same rounds with every point distance evaluated in FP64: a list
// holds the FP64 distances rounded to FP32, whose band then only covers that rounding.
//
// HDBSCAN*: the weights are mutual reachability distances.  All edges with D <= max(cd2 p, cd2 q)
// (the only ones that tie in general position) are in the k-NN pass's repair list, which a round
// scans edge by edge; the search only has to find lighter edges with D above both core distances,
// and R[i] starts at cd2(i).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "boruvka.cuh"
#include "screen.cuh"
#include "stree.cuh"
#include "wspd.cuh"

namespace wm {

namespace {

// List entries per point, by dimension.  A longer list serves more rounds, a shorter one has the smaller
// radius to search first: at 10^7 points 4 -> 6 entries took the search from 9.3 to 7.7 ms in 3-D and
// from 8.0 to 7.7 in 2-D, left it in 5-D (31 ms) and cost 13 % in 7-D; 2 entries were slower everywhere.
__host__ __device__ constexpr int list_len(int D) { return D <= 3 ? 6 : 4; }

// A point with R >= S cannot lower S.  Where its list is full and all of one band besides, the next list would be too,
// and the point is left to the exact search at once: such are lattice points, whose 2 D nearest neighbours a list
// of list_len(D) does not hold above 3 dimensions.  (EMST of a 7-D lattice of 280,000 points 6.3 -> 4.9 ms, FP64 form
// 8.6 -> 6.1; of a 5-D one of 100,000 2.4 -> 2.1 and 2.7 -> 2.3.  In 3-D lists get room as neighbours join the component,
// and the same rule took 2.0 -> 2.6 ms.)
__host__ __device__ constexpr bool marks_ties(int D) { return list_len(D) < 2 * D; }

// A query that has looked at long_points points (above 10^6 or two: a 1024th of all) and is still walking is handed
// to warps that share a scan of all points: the centre of a sphere of points is as far from all of them, and
// its walk visits every node on one lane while the GPU waits (EMST of 50,000 points and their centre: 83 ms, of
// which 81 on that lane; 2.7 now, FP64 form 142 and 3.7; with a limit of 2048 5.0 and 7.6.  7-D sets reach 1024 in
// ordinary walks, and were 2 % slower with it).  Points count whether they are evaluated or only bounded: in the
// FP64 form a walk that bounded most of 10^6 points went unnoticed (36 -> 13 ms).  While at most kLongMax
// queries and about kLongWork points' evaluations are waiting, such a query is handed over at once; one that
// comes later walks on, and is handed over all the same when it has looked at a kLongPart-th of all points
// (twice the limit at least), since it will hardly stop before the rest.  A query is handed over at most once a
// search, and the list has a place for every query of the search: its counter cannot pass n.  Such queries are
// rare, so the scan is launched when the host has seen one (launched every time it cost 10^4 points 6 %), for
// kLongMax of them at a time; until then the kernels behind the search hold back (held).
constexpr int kLongMax = 512, kLongPart = 16, kLongChunk = 512, kLongChunks = 1024;
constexpr int long_points(int D) { return D <= 5 ? 1024 : 2048; }
constexpr long long kLongWork = 1 << 26;

// Counters.  Those that a round starts from zero lie side by side: an even one's are [kCntEven, kCntEdges), an
// odd one's [0, kCntOddEnd).
enum {
    kCntRootsEven, kCntRepOdd,        // roots that even rounds start from; repair edges that odd rounds leave
    kCntEven,
    kCntActive = kCntEven, kCntNear, kCntSearch, kCntCand, kCntExact, kCntExactNext, kCntPicked,
    kCntLong, kCntLongExact,          // queries handed to the scan of all points
    kCntOddEnd,
    kCntRepEven = kCntOddEnd, kCntRootsOdd,
    kCntEdges,                        // tree edges so far
    kCntError,                        // error bits of the kernels
    kCntAll
};
__host__ __device__ constexpr int cnt_roots(int parity) { return parity ? kCntRootsOdd : kCntRootsEven; }
__host__ __device__ constexpr int cnt_rep(int parity) { return parity ? kCntRepOdd : kCntRepEven; }

struct NcArgs {
    int *lab;                  // component of a tree position (a tree position: the root)
    int *par;                  // links between roots
    unsigned *S;               // per root: smallest screened weight seen this round (float bits)
    unsigned long long *bhi, *blo;   // per root: K-minimum outgoing edge
    float *ls;                 // [list_len][n] list weights, ascending
    int *lj;                   // [list_len][n] list positions (-1: none)
    float *R;                  // every point outside the component and the list screens at >= |R|; the sign marks
                               // a full list of one band (see marks_ties)
    unsigned char *hd;         // first list entry that may lie outside the component
    float *low;                // smaller of the head's weight (no head: +inf) and R
    int *roots[2];             // the roots of this round and the next
    int *act, *amb, *picked;   // active points; points that need the exact scan; points with a candidate
    int *near;                 // points that may come to need the scan or have a candidate
    int *nlab;                 // labels in the node rows
    EdgeK *cand;               // candidate edges of the round and the component each serves
    int *cand_c;
    int *cnt;                  // counters, see kCnt*
    int K;                     // list_len
    const int *pos;            // input id -> tree position
    unsigned cap_bits;         // no edge at or above this weight (float bits; +inf: none)
    unsigned long long cap64;  // the same in FP64 bits
    float *rows;               // the search tree's point rows
    const float *ncd;          // HDBSCAN*: smallest core distance of a node (rounded down)
    // queries handed to the scan of all points (chunks: parts of the points; 0: no hand-over): positions in
    // amb, which the search leaves alone, or of the exact search in act
    int chunks, long_max;
    unsigned long_few, long_most;   // points after which a query is handed over: while fewer than long_max
                                    // are waiting, in any case
    int guard;                 // 1: hold back while queries of the search wait for the scan, 2: of the exact one
    int *long_done;            // [kLongMax] parts finished
    float *long_s;             // [kLongMax][chunks][K] a part's list
    int *long_j;
    KMin *long_k;              // [kLongMax][chunks] a part's K-minimum
    int first;                 // first search: components are single points, nothing is pruned by S
    int n;
};

__device__ __forceinline__ bool all_tied(float R) { return __float_as_int(R) < 0; }

// true while queries that were handed over wait for the scan of all points
__device__ __forceinline__ bool held(const NcArgs &b, int what)
{
    return (b.guard & what & 1 && b.cnt[kCntLong] > 0) || (b.guard & what & 2 && b.cnt[kCntLongExact] > 0);
}

// HDBSCAN*: true when the FP32 squared distance d32 proves D <= c for a core distance c (FP32 copy)
__device__ inline bool proven_repair(const TravArgs &a, float d32, float c)
{
    if (a.exact32) return proven_within(d32, c);
    const double r = sqrt((double)d32 * (1.0 + 1.0 / 131072.0) + kAbsTiny) + a.eta;
    return r * r * (1.0 + 1.0 / 131072.0) < (double)c * (1.0 - 1.0 / 4194304.0) - kAbsTiny;
}

// relative error of a screened weight against the exact one (an upper bound, FP32)
__device__ inline void note_err(float s, double w, float &err)
{
    if (w > 0.0) err = fmaxf(err, __fdiv_ru(__double2float_ru(fabs((double)s - w)), __double2float_rd(w)));
}

// v into an ascending list (its largest entry drops out)
template <int K>
__device__ __forceinline__ void list_insert(float (&sl)[K], int (&sj)[K], float v, int j)
{
#pragma unroll
    for (int k = K - 1; k >= 0; --k) {
        if (k > 0 && v < sl[k - 1]) {
            sl[k] = sl[k - 1];
            sj[k] = sj[k - 1];
        } else if (v < sl[k]) {
            sl[k] = v;
            sj[k] = j;
        }
    }
}

// ---------------------------------------------------------------------------------- search
// A thread per query on the search tree (stree.cuh).
// EXACT = false rebuilds the lists of the active points.  EXACT = true answers the points whose list may
// have dropped a tie: every point within T(S[c]) is evaluated in FP64 and the K-minimum becomes the
// point's candidate edge.
// Blocks per SM to compile for: 8 (64 registers) for the searches that run long; with 10 or 12 the EMST
// searches spill (7-D, 10^7 points: 91 ms at 8, 94 at will, 121 and 152 at 10 and 12), and the short HDBSCAN*
// searches above 3 dimensions are faster with all the registers they ask for.
constexpr int search_blocks(int D, bool HDB, bool F64, bool EXACT) { return EXACT || F64 || (HDB && D > 3) ? 1 : 8; }

template <int D, bool HDB, bool F64, bool EXACT>
__global__ void __launch_bounds__(kWalkThreads, search_blocks(D, HDB, F64, EXACT)) nc_search_kernel(TravArgs a, NcArgs b, SearchTree X, int m_all)
{
    __shared__ uint2 sst[kWalkStack][kWalkThreads];
    constexpr int S = row_floats(D), K = list_len(D);
    constexpr bool kStream = S > 4 && !HDB;
    const int lane = threadIdx.x & 31;
    const int n = a.n;
    const int m = EXACT ? b.cnt[kCntExact] : b.first ? m_all : b.cnt[kCntActive];
    unsigned n_ev = 0, n_re = 0;   // (a lane's share)
    float err = 0.f;
    // the lane's query
    float q[S];
    int i = 0, c = 0;
    float qcd = 0.f, qcd_lo = 0.f, Sc = 0.f;
    float sl[K];
    int sj[K];
    KMin best{~0ull, ~0ull};
    float lim = 0.f, pb = 0.f;   // a candidate screens below lim; a node is skipped when its lower bound
                                 // exceeds pb (it bounds the exact weight, within 2^-19 of the screened one)
    unsigned ev = 0;   // points of the buckets scanned
    auto begin = [&](int t) {
        i = EXACT ? b.amb[t] : b.first ? t : b.act[t];
        load_row<S>(X.rows, i, q);
        c = b.lab[i];
        if (HDB) {
            qcd = a.cd32[i];
            qcd_lo = qcd * (1.0f - 1.0f / 4194304.0f);
        }
        Sc = __uint_as_float(*(volatile unsigned *)(b.S + c));
#pragma unroll
        for (int k = 0; k < K; ++k) { sl[k] = INFINITY; sj[k] = -1; }
        best = KMin{~0ull, ~0ull};
        lim = next_up(screen_threshold(Sc, a));
        pb = lim * (1.0f + 1.0f / 131072.0f);
        ev = 0;
    };
    auto bound = [&](unsigned node, float &g0, float &g1) {
        if (HDB) {
            g0 = fmaxf(g0, fmaxf(qcd_lo, b.ncd[node]));
            g1 = fmaxf(g1, fmaxf(qcd_lo, b.ncd[node + 1]));
        }
    };
    auto need = [&](float g, int l) { return g <= pb && l != c; };
    auto pending = [&](float g) { return g <= pb; };
    auto scan = [&](int j0, int sz) {
        // screened values first, then the ones below the limit one by one: few lanes have any, and
        // they run their insertions together
        float w[kBucket];
        unsigned todo = 0;
#pragma unroll
        for (int h = 0; h < kBucket; h += 4) {
            if (h && h >= sz) break;
#pragma unroll
            for (int p = h; p < h + 4; ++p) {
                const int j = j0 + min(p, sz - 1);
                float x[S];
                load_row<S, kStream>(X.rows, j, x);
                bool take = p < sz && __float_as_int(x[S - 1]) != c;
                if (F64) {
                    // (FP64 is slow enough that even a point is first tried against the bound)
                    take = take && point_bound<D>(q, x, row_error(a.delta32)) <= pb;
                    n_ev += take;
                } else {
                    w[p] = row_dist<D>(q, x);
                    if (HDB) {
                        const float cdm = fmaxf(qcd, a.cd32[j]);
                        take = take && !proven_repair(a, w[p], cdm);
                        w[p] = fmaxf(w[p], cdm);
                    }
                    take = take && w[p] < lim;
                }
                if (take) todo |= 1u << p;
            }
        }
        ev += (unsigned)sz;
        const float was = sl[0];
        while (todo) {
            const int p = __ffs(todo) - 1;
            todo &= todo - 1;
            float v;
            double x2 = 0.0;
            if (F64) {
                x2 = EXACT ? tie_dist64<D, S>(a.x64, n, a.d, X.rows, i, j0 + p)
                           : walk_dist64<D, S>(a.x64, n, a.d, X.rows, i, j0 + p);
                v = __double2float_rn(x2);
                if (HDB) {
                    const float cdm = fmaxf(qcd, a.cd32[j0 + p]);
                    if (proven_repair(a, v, cdm)) continue;
                    v = fmaxf(v, cdm);
                }
                if (!(v < lim)) continue;
            } else {
                v = w[0];
#pragma unroll
                for (int r = 1; r < kBucket; ++r) v = r == p ? w[r] : v;
            }
            if (EXACT) {
                const int j = j0 + p;
                if (!F64) x2 = tie_dist64<D, S>(a.x64, n, a.d, X.rows, i, j);
                if (HDB) x2 = pos_dmax(x2, pos_dmax(a.cd64[i], a.cd64[j]));
                if (!F64) note_err(v, x2, err);
                kmin_update(best, x2, a.pid[i], a.pid[j]);
                ++n_re;
            } else if (v < lim) {
                list_insert<K>(sl, sj, v, j0 + p);
                lim = fminf(lim, sl[K - 1]);
            }
        }
        if (!EXACT && !b.first) {
            // the component's minimum: lowered by this point, else re-read
            float now = Sc;
            if (sl[0] < was && sl[0] < Sc)
                now = fminf(sl[0], __uint_as_float(atomicMin(b.S + c, __float_as_uint(sl[0]))));
            else if ((ev & 31u) < 8u)   // now and then
                now = __uint_as_float(*(volatile unsigned *)(b.S + c));
            if (now < Sc) {
                Sc = now;
                lim = fminf(lim, next_up(screen_threshold(Sc, a)));
            }
        }
        pb = lim * (1.0f + 1.0f / 131072.0f);
        if (ev >= b.long_few && (ev & 255u) < 8u) {   // (a bucket adds at most 8)
            int *waiting = b.cnt + (EXACT ? kCntLongExact : kCntLong);
            if (ev >= b.long_most || *(volatile int *)waiting < b.long_max) {
                (EXACT ? b.act : b.amb)[atomicAdd(waiting, 1)] = i;
                pb = -1.f;   // nothing left to visit: the query ends here
            }
        }
    };
    auto finish = [&] {
        if (!F64) n_ev += ev;
        if (pb < 0.f) return;   // handed over
        if (EXACT) {
            if (best.hi < b.cap64) {
                const int slot = atomicAdd(b.cnt + kCntCand, 1);   // at most one candidate per point: within n
                EdgeK e;
                e.hi = best.hi;
                e.lo = best.lo;
                b.cand[slot] = e;
                b.cand_c[slot] = c;
                if (best.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, best.hi);
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                b.ls[(size_t)k * n + i] = sl[k];
                b.lj[(size_t)k * n + i] = sj[k];
            }
            // (one band, and more of it may have been turned away)
            const bool tied = marks_ties(D) && sl[K - 1] < INFINITY && sl[K - 1] <= screen_threshold(sl[0], a);
            b.R[i] = tied ? -lim : lim;
            b.low[i] = fminf(sl[0], lim);
            b.hd[i] = 0;
        }
    };
    walk_queries<D, S, kStream>(X, m, b.cnt + (EXACT ? kCntExactNext : kCntSearch), &sst[0][threadIdx.x], kWalkThreads,
                                X.deep + (size_t)blockIdx.x * kWalkThreads + threadIdx.x,
                                (size_t)gridDim.x * kWalkThreads, (int *)a.overflow, 8, q, begin, bound, need, pending,
                                scan, finish);
    const unsigned long long all_ev = warp_sum_u64(n_ev);
    if (lane == 0 && all_ev) {
        atomicAdd(a.stat + 1, all_ev);
        if (!EXACT) atomicAdd(a.stat + 6, all_ev);   // (the searches that are timed)
    }
    if (EXACT) {
        err_flush(a, err);
        const unsigned long long all_re = warp_sum_u64(n_re);
        if (lane == 0 && all_re) atomicAdd(a.stat + 2, all_re);
    }
}

// the smallest K entries of the lanes' ascending lists, to every lane
template <int K>
__device__ __forceinline__ void warp_lists(float (&sl)[K], int (&sj)[K], float (&ol)[K], int (&oj)[K])
{
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const unsigned u = __float_as_uint(sl[0]), m = __reduce_min_sync(0xffffffffu, u);
        const int src = __ffs(__ballot_sync(0xffffffffu, u == m)) - 1;
        ol[r] = __uint_as_float(m);
        oj[r] = __shfl_sync(0xffffffffu, sj[0], src);
        if ((threadIdx.x & 31) == src) {
#pragma unroll
            for (int k = 0; k + 1 < K; ++k) { sl[k] = sl[k + 1]; sj[k] = sj[k + 1]; }
            sl[K - 1] = INFINITY;
            sj[K - 1] = -1;
        }
    }
}

__device__ __forceinline__ void warp_kmin(KMin &m)
{
    for (int o = 16; o; o >>= 1) {
        const unsigned long long h = __shfl_xor_sync(0xffffffffu, m.hi, o), l = __shfl_xor_sync(0xffffffffu, m.lo, o);
        if (h < m.hi || (h == m.hi && l < m.lo)) { m.hi = h; m.lo = l; }
    }
}

// The queries [first, first + kLongMax) that the search handed over: a warp per query and part of the points;
// the warp that finishes a query's last part puts the parts together.
template <int D, bool HDB, bool F64, bool EXACT>
__global__ void __launch_bounds__(kWalkThreads) nc_long_kernel(TravArgs a, NcArgs b, int first)
{
    constexpr int S = row_floats(D), K = list_len(D);
    const int lane = threadIdx.x & 31, n = a.n;
    const int *longq = (EXACT ? b.act : b.amb) + first;
    const int m = min(b.cnt[EXACT ? kCntLongExact : kCntLong] - first, kLongMax) * b.chunks;   // at most 2^19
    const int part = (n + b.chunks - 1) / b.chunks;
    unsigned long long n_ev = 0, n_re = 0;
    float err = 0.f;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < m; it += (gridDim.x * blockDim.x) >> 5) {
        const int l = it / b.chunks, ch = it % b.chunks, i = longq[l], c = b.lab[i];
        const int j1 = (int)min((long long)n, (long long)(ch + 1) * part);
        float q[S];
        load_row<S>(b.rows, i, q);
        const float qcd = HDB ? a.cd32[i] : 0.f;
        const float lim = EXACT ? next_up(screen_threshold(__uint_as_float(*(volatile unsigned *)(b.S + c)), a)) : INFINITY;
        float sl[K], ol[K];
        int sj[K], oj[K];
#pragma unroll
        for (int k = 0; k < K; ++k) { sl[k] = INFINITY; sj[k] = -1; }
        KMin best{~0ull, ~0ull};
        for (long long j0 = (long long)ch * part + lane; j0 < j1; j0 += 32) {
            const int j = (int)j0;
            float x[S];
            load_row<S>(b.rows, j, x);
            if (__float_as_int(x[S - 1]) == c) continue;
            const float now = EXACT ? lim : sl[K - 1];
            if (F64 && point_bound<D>(q, x, row_error(a.delta32)) > now * (1.0f + 1.0f / 131072.0f)) continue;
            float v = screen_dist<D, S, F64>(a.x64, n, a.d, b.rows, i, j, q, x);
            ++n_ev;
            if (HDB) {
                const float cdm = fmaxf(qcd, a.cd32[j]);
                if (proven_repair(a, v, cdm)) continue;
                v = fmaxf(v, cdm);
            }
            if (!(v < now)) continue;
            if (EXACT) {
                double x2 = tie_dist64<D, S>(a.x64, n, a.d, b.rows, i, j);
                if (HDB) x2 = pos_dmax(x2, pos_dmax(a.cd64[i], a.cd64[j]));
                if (!F64) note_err(v, x2, err);
                kmin_update(best, x2, a.pid[i], a.pid[j]);
                ++n_re;
            } else {
                list_insert<K>(sl, sj, v, j);
            }
        }
        __syncwarp();
        if (EXACT) {
            warp_kmin(best);
            if (lane == 0) b.long_k[it] = best;
        } else {
            warp_lists<K>(sl, sj, ol, oj);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    b.long_s[(size_t)it * K + k] = ol[k];
                    b.long_j[(size_t)it * K + k] = oj[k];
                }
            }
        }
        int done = 0;
        if (lane == 0) {
            __threadfence();
            done = atomicAdd(b.long_done + l, 1);
            __threadfence();
        }
        if (__shfl_sync(0xffffffffu, done, 0) != b.chunks - 1) continue;
        const size_t at = (size_t)l * b.chunks;
        if (EXACT) {
            best = KMin{~0ull, ~0ull};
            for (int p = lane; p < b.chunks; p += 32) {
                const unsigned long long h = __ldcg(&b.long_k[at + p].hi), w = __ldcg(&b.long_k[at + p].lo);
                if (h < best.hi || (h == best.hi && w < best.lo)) { best.hi = h; best.lo = w; }
            }
            __syncwarp();
            warp_kmin(best);
            if (lane == 0 && best.hi < b.cap64) {
                const int slot = atomicAdd(b.cnt + kCntCand, 1);   // at most one candidate per point: within n
                EdgeK e;
                e.hi = best.hi;
                e.lo = best.lo;
                b.cand[slot] = e;
                b.cand_c[slot] = c;
                if (best.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, best.hi);
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) { sl[k] = INFINITY; sj[k] = -1; }
            for (int p = lane; p < b.chunks * K; p += 32) {
                const float v = __ldcg(b.long_s + at * K + p);
                if (v < sl[K - 1]) list_insert<K>(sl, sj, v, __ldcg(b.long_j + at * K + p));
            }
            __syncwarp();
            warp_lists<K>(sl, sj, ol, oj);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    b.ls[(size_t)k * n + i] = ol[k];
                    b.lj[(size_t)k * n + i] = oj[k];
                }
                b.R[i] = ol[K - 1];
                b.low[i] = ol[0];
                b.hd[i] = 0;
                if (!b.first && ol[0] < INFINITY) atomicMin(b.S + c, __float_as_uint(ol[0]));
            }
        }
        if (lane == 0) b.long_done[l] = 0;
    }
    n_ev = warp_sum_u64(n_ev);
    if (lane == 0 && n_ev) {
        atomicAdd(a.stat + 1, n_ev);
        if (!EXACT) atomicAdd(a.stat + 6, n_ev);
    }
    if (EXACT) {
        err_flush(a, err);
        n_re = warp_sum_u64(n_re);
        if (lane == 0 && n_re) atomicAdd(a.stat + 2, n_re);
    }
}

// HDBSCAN*: smallest core distance (rounded down) of every search tree node: buckets from their
// points, the rest bottom-up, the second child to arrive composing the parent
__global__ void nc_core_min_kernel(int Ns, const int2 *__restrict__ range, const int *__restrict__ parent,
                                   const double *__restrict__ cd64, float *ncd, int *arrive)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < Ns; x += gridDim.x * blockDim.x) {
        const int2 r = range[x];
        if (r.y - r.x > kBucket) continue;
        double m = cd64[r.x];
        for (int i = r.x + 1; i < r.y; ++i) m = fmin(m, cd64[i]);
        float f = __double2float_rd(m);
        *(volatile float *)(ncd + x) = f;
        int cur = x;
        for (int it = 0; it < Ns; ++it) {
            const int p = parent[cur];
            if (p < 0) break;
            __threadfence();
            if (atomicAdd(arrive + p, 1) == 0) break;   // the sibling composes the parent
            __threadfence();
            // the sibling shares the pair that starts at an odd row (the root is row 0)
            f = fminf(f, *(volatile float *)(ncd + (((cur - 1) ^ 1) + 1)));
            *(volatile float *)(ncd + p) = f;
            cur = p;
        }
    }
}

// ------------------------------------------------------------------------- round bookkeeping
__global__ void nc_init_kernel(TravArgs a, NcArgs b, bool hdb)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        b.lab[i] = i;
        b.par[i] = i;
        b.roots[0][i] = i;
        b.S[i] = b.cap_bits;
        b.bhi[i] = ~0ull;
        b.blo[i] = ~0ull;
        if (hdb) {   // no list yet: an edge outside the repair list is longer than the core distance
            b.hd[i] = (unsigned char)b.K;
            b.R[i] = b.low[i] = __double2float_rd(a.cd64[i]);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) b.cnt[cnt_roots(0)] = a.n;
}

// WriteMin of a weight into a component's slot; a value that cannot lower it is not issued
__device__ __forceinline__ void s_min(unsigned *S, int c, float v)
{
    const unsigned u = __float_as_uint(v);
    if (u < *(volatile unsigned *)(S + c)) atomicMin(S + c, u);
}

// Advances the list heads past entries that joined the component; the first entry left bounds the
// component's minimum.  A point without one offers its neighbours in tree order.  Nothing is looked up where
// neither the head's weight nor the radius beyond the list can lower the minimum as it stands: such a head
// may lie inside the component (it is looked at again once it matters).  In the late rounds most points stop
// there; in the early ones a component's points are read together, before its minimum has come down (10^7
// points in 3-D: 200 us in the second round, 80 in the tenth, bound by the gather of the heads' labels).
template <int D, bool HDB, bool F64>
__device__ __forceinline__ void refresh_points(const TravArgs &a, const NcArgs &b)
{
    if (b.first && held(b, 1)) return;   // (lists are missing)
    constexpr int S = row_floats(D);
    const int n = a.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = b.lab[i];
        if (__float_as_uint(b.low[i]) >= *(volatile unsigned *)(b.S + c)) continue;
        int h = b.hd[i];
        if (h < b.K) {
            const int h0 = h;
            int j = -1;
            for (; h < b.K; ++h) {
                j = b.lj[(size_t)h * n + i];
                if (j >= 0 && b.lab[j] != c) break;
            }
            const float s = h < b.K ? b.ls[(size_t)h * n + i] : INFINITY;
            if (h != h0) {
                b.hd[i] = (unsigned char)h;
                b.low[i] = fminf(s, fabsf(b.R[i]));
            }
            if (h < b.K) s_min(b.S, c, s);
        }
        if (h >= b.K) {
#pragma unroll
            for (int o = -1; o <= 1; o += 2) {
                const int j = i + o;
                if (j < 0 || j >= n || b.lab[j] == c) continue;
                float x[S], y[S];
                load_row<S>(b.rows, i, x);
                load_row<S>(b.rows, j, y);
                float acc = screen_dist<D, S, F64>(a.x64, n, a.d, b.rows, i, j, x, y);
                if (HDB) acc = fmaxf(acc, fmaxf(a.cd32[i], a.cd32[j]));
                s_min(b.S, c, acc);
            }
        }
    }
}

// HDBSCAN*: repair edges between two components WriteMin their exact weight; the others are dropped
__global__ void nc_repair_kernel(NcArgs b, const EdgeK *__restrict__ in, const int *__restrict__ m_dev, int m_first,
                                 EdgeK *__restrict__ out, int *out_n)
{
    __shared__ int sh[32];
    const int m = m_dev ? *m_dev : m_first;
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        bool keep = false;
        EdgeK e;
        e.hi = 0;
        e.lo = 0;
        if (t < m) {
            e = in[t];
            const int cu = b.lab[b.pos[edge_u(e)]], cv = b.lab[b.pos[edge_v(e)]];
            keep = cu != cv;
            if (keep && e.hi < b.cap64) {
                const float s = __double2float_ru(edge_w2(e));
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const int c = side ? cv : cu;
                    s_min(b.S, c, s);
                    if (e.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, e.hi);
                }
            }
        }
        const int slot = block_append(out_n, keep ? 1 : 0, sh);
        if (keep) out[slot] = e;
    }
}

// HDBSCAN*: a component whose repair edges reach down to cd2(i) needs nothing from i's other edges
// (each is longer than cd2(i)).  (bhi may only fall: a stale value costs time, not the result.)
__device__ __forceinline__ bool settled(const TravArgs &a, const NcArgs &b, int i, int c)
{
    return *(volatile unsigned long long *)(b.bhi + c) <= (unsigned long long)__double_as_longlong(a.cd64[i]);
}

// The active points, and those that pick_points has to look at: S only falls until then, and T with it.
// (Eight points per thread between two appends: an append per 256 points, which most of those have a point
// for, made the pass wait for one counter, 120 us for 10^7 points against 37 now.  With the list, this pass
// and the one that picks take 0.67 ms a call where two passes over all points took 1.40.)
template <bool HDB, bool MARK>
__device__ __forceinline__ void active_points(const TravArgs &a, const NcArgs &b, int *sh)
{
    const int n = a.n, items = 8 * blockDim.x;
    for (long long b0 = (long long)blockIdx.x * items; b0 < n; b0 += (long long)gridDim.x * items) {
        unsigned on = 0, near = 0;
        int c[8];
        float low[8], T[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const long long at = b0 + t * blockDim.x + threadIdx.x;
            c[t] = at < n ? b.lab[at] : -1;
            low[t] = at < n ? b.low[at] : 0.f;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) T[t] = c[t] >= 0 ? __uint_as_float(b.S[c[t]]) : 0.f;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            T[t] = screen_threshold(T[t], a);
            if (c[t] >= 0 && low[t] <= T[t]) near |= 1u << t;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            if (!((near >> t) & 1u)) continue;
            const int i = (int)(b0 + t * blockDim.x + threadIdx.x);
            const float R = b.R[i];
            if (fabsf(R) <= T[t] && !(MARK && all_tied(R) && fabsf(R) >= __uint_as_float(b.S[c[t]])) &&
                !(HDB && settled(a, b, i, c[t])))
                on |= 1u << t;
        }
        if (!__syncthreads_or(near)) continue;
        int slot = block_append(b.cnt + kCntNear, __popc(near), sh);
        for (unsigned m = near; m; m &= m - 1) b.near[slot++] = (int)(b0 + (__ffs(m) - 1) * blockDim.x + threadIdx.x);
        if (!__syncthreads_or(on)) continue;
        slot = block_append(b.cnt + kCntActive, __popc(on), sh);
        for (unsigned m = on; m; m &= m - 1) b.act[slot++] = (int)(b0 + (__ffs(m) - 1) * blockDim.x + threadIdx.x);
    }
}

// Points with a list entry inside the band of their component's screened minimum, and points whose list
// may have dropped one
template <bool HDB>
__device__ __forceinline__ void pick_points(const TravArgs &a, const NcArgs &b, int *sh)
{
    if (held(b, 1)) return;
    const int n = a.n, m = b.first ? n : b.cnt[kCntNear];
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        bool exact = false, has = false;
        int i = 0;
        if (t < m) {
            i = b.first ? t : b.near[t];
            const int c = b.lab[i];
            const float T = screen_threshold(__uint_as_float(b.S[c]), a);
            exact = fabsf(b.R[i]) <= T;
            if (HDB && exact) exact = !settled(a, b, i, c);
            const int h = b.hd[i];
            has = !exact && h < b.K && b.ls[(size_t)h * n + i] <= T;
        }
        if (__syncthreads_or(has)) {
            const int slot = block_append(b.cnt + kCntPicked, has ? 1 : 0, sh);
            if (has) b.picked[slot] = i;
        }
        if (exact) b.amb[atomicAdd(b.cnt + kCntExact, 1)] = i;
    }
}

// K-minimum of a picked point's list entries inside the band, in FP64 (on a dense list: an FP64
// instruction costs a warp the same however few of its lanes need it)
template <int D, bool HDB, bool F64>
__device__ __forceinline__ void candidates(const TravArgs &a, const NcArgs &b, int *sh)
{
    constexpr int S = row_floats(D);
    const int n = a.n, m = b.cnt[kCntPicked];
    unsigned long long n_re = 0;
    float err = 0.f;
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        int c = -1;
        KMin best{~0ull, ~0ull};
        if (t < m) {
            const int i = b.picked[t];
            c = b.lab[i];
            const float T = screen_threshold(__uint_as_float(b.S[c]), a);
            for (int h = b.hd[i]; h < b.K; ++h) {
                const float s = b.ls[(size_t)h * n + i];
                if (s > T) break;
                const int j = b.lj[(size_t)h * n + i];
                if (j < 0 || b.lab[j] == c) continue;
                double w = walk_dist64<D, S>(a.x64, n, a.d, b.rows, i, j);
                if (HDB) w = pos_dmax(w, pos_dmax(a.cd64[i], a.cd64[j]));
                if (!F64) note_err(s, w, err);
                kmin_update(best, w, a.pid[i], a.pid[j]);
                ++n_re;
            }
        }
        const bool has = best.hi < b.cap64;
        const int slot = block_append(b.cnt + kCntCand, has ? 1 : 0, sh);
        if (has) {
            EdgeK e;
            e.hi = best.hi;
            e.lo = best.lo;
            b.cand[slot] = e;
            b.cand_c[slot] = c;
            if (best.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, best.hi);
        }
    }
    err_flush(a, err);
    n_re = warp_sum_u64(n_re);
    if ((threadIdx.x & 31) == 0 && n_re) atomicAdd(a.stat + 2, n_re);
}

// Among the candidates with their component's smallest weight: WriteMin of the id pair
__device__ __forceinline__ void low_ids(const NcArgs &b)
{
    if (held(b, 3)) return;
    const int m = b.cnt[kCntCand];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) {
        const EdgeK e = b.cand[t];
        const int c = b.cand_c[t];
        if (e.hi == b.bhi[c]) atomicMin(b.blo + c, e.lo);
    }
}

__global__ void nc_low_repair_kernel(NcArgs b, const EdgeK *__restrict__ rep, const int *__restrict__ m_dev)
{
    if (held(b, 3)) return;
    const int m = *m_dev;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) {
        const EdgeK e = rep[t];
        const int cu = b.lab[b.pos[edge_u(e)]], cv = b.lab[b.pos[edge_v(e)]];
        if (e.hi == b.bhi[cu]) atomicMin(b.blo + cu, e.lo);
        if (e.hi == b.bhi[cv]) atomicMin(b.blo + cv, e.lo);
    }
}

// Every root with an edge links to the component at its other end; of two roots that chose the same
// edge the smaller stays a root.  (The keys along a chain of choices strictly fall, so there is no
// longer cycle.)
__device__ __forceinline__ void merge_roots(const TravArgs &a, const NcArgs &b, int cur, EdgeK *out, int out_cap, int *sh)
{
    if (held(b, 3)) return;
    const int m = b.cnt[cnt_roots(cur)];
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        bool emit = false;
        EdgeK e;
        e.hi = 0;
        e.lo = 0;
        if (t < m) {
            const int i = b.roots[cur][t];
            e.hi = b.bhi[i];
            e.lo = b.blo[i];
            if (e.hi != ~0ull) {
                const int cu = b.lab[b.pos[edge_u(e)]], cv = b.lab[b.pos[edge_v(e)]];
                const int o = cu == i ? cv : cu;
                if (o == i || (cu != i && cv != i)) {
                    atomicOr(a.overflow, 16u);   // not an outgoing edge: an internal error, reported
                } else {
                    const bool mutual = b.bhi[o] == e.hi && b.blo[o] == e.lo;
                    emit = !mutual || i < o;
                    if (!(emit && mutual)) b.par[i] = o;
                }
            }
        }
        const int slot = block_append(b.cnt + kCntEdges, emit ? 1 : 0, sh);
        if (emit) {
            if (slot < out_cap) out[slot] = e;
            else atomicOr(a.overflow, 16u);
        }
    }
}

// After the links: every root of the round is linked to its component's root; the roots left are collected and
// their slots reset for the next round.
__device__ __forceinline__ void collect_roots(const NcArgs &b, int cur, int *sh)
{
    if (held(b, 3)) return;
    const int m = b.cnt[cnt_roots(cur)];
    const int *roots = b.roots[cur];
    link_to_roots(b.par, m, [roots](int t) { return roots[t]; });
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        bool stays = false;
        int i = 0;
        if (t < m) {
            i = roots[t];
            stays = *(volatile int *)(b.par + i) == i;
            if (stays) {
                b.S[i] = b.cap_bits;
                b.bhi[i] = ~0ull;
                b.blo[i] = ~0ull;
            }
        }
        const int slot = block_append(b.cnt + cnt_roots(cur ^ 1), stays ? 1 : 0, sh);
        if (stays) b.roots[cur ^ 1][slot] = i;
    }
}

// The root above x: x itself or, for a root that linked in this round, where collect_roots has linked it.
__device__ __forceinline__ int root_of(const int *__restrict__ par, int x, int n)
{
    for (int it = 0; it < n; ++it) {
        const int p = par[x];
        if (p == x) break;
        x = p;
    }
    return x;
}

// New labels, and per tile of positions the number of label changes along tree order (a node is in one
// component when none falls inside its range).  A warp takes kTileItems times 32 consecutive positions, so that
// labels and rows are read and written by neighbouring lanes (10^7 points in 3-D: 52 us a round, where eight
// consecutive positions per thread took 130, and 15 for the prefixes instead of 40).
constexpr int kTileItems = 8, kTile = 256 * kTileItems;

// Up to this many points the steps between the searches are run by one block each, see nc_small_back_kernel.  The line
// lies where one block takes as long as the launches it saves (ms, one block / launches, EMST in 2-D: 1000 points 0.66 /
// 0.78, 2000 0.77 / 0.83, 3000 0.92 / 0.93, 4096 1.04 / 0.96; in 7-D 1.27 / 1.33, 2.07 / 2.15, 2.53 / 2.48, 3.21 / 3.05;
// HDBSCAN* in 2-D 1.09 / 1.18, 1.26 / 1.29, 1.41 / 1.41, 1.66 / 1.59).
constexpr int kSmallThreads = 512, kSmallPoints = 3072;
static_assert(kSmallPoints <= kSmallThreads * kTileItems, "one tile (change_prefixes)");

// Once a single component is left nobody reads a label again, and the steps below return at once.
__device__ __forceinline__ void relabel_points(const NcArgs &b, int S, const int *roots, int *sums)
{
    __shared__ int s_chg;
    const int n = b.n, lane = threadIdx.x & 31, tile_items = blockDim.x * kTileItems;
    if (*roots == 1) return;
    const int *par = b.par;
    for (int tile = blockIdx.x; tile * (long long)tile_items < n; tile += gridDim.x) {
        if (threadIdx.x == 0) s_chg = 0;
        __syncthreads();
        const int i0 = tile * tile_items + (threadIdx.x >> 5) * (32 * kTileItems) + lane;
        // (the label before may be replaced already: a root points at itself)
        int last = lane == 0 && i0 > 0 && i0 < n ? root_of(par, *(volatile int *)(b.lab + i0 - 1), n) : -1;
        int chg = 0, c[kTileItems], x[kTileItems];
        // (the loads of all positions first: most roots are two links away)
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) c[t] = i0 + 32 * t < n ? b.lab[i0 + 32 * t] : -1;
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) x[t] = c[t] >= 0 ? par[c[t]] : -1;
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) {
            const int up = x[t] >= 0 ? par[x[t]] : -1;
            if (up != x[t]) x[t] = root_of(par, up, n);
        }
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) {
            const int i = i0 + 32 * t;
            if (x[t] != c[t]) {
                *(volatile int *)(b.lab + i) = x[t];
                b.rows[(size_t)i * S + S - 1] = __int_as_float(x[t]);
            }
            const int before = __shfl_up_sync(0xffffffffu, x[t], 1);
            chg += i > 0 && i < n && x[t] != (lane ? before : last);
            last = __shfl_sync(0xffffffffu, x[t], 31);
        }
        chg = __reduce_add_sync(0xffffffffu, chg);
        if (lane == 0 && chg) atomicAdd(&s_chg, chg);
        __syncthreads();
        if (threadIdx.x == 0) sums[tile] = s_chg;
    }
}

// E[i] = label changes in (0, i), from the tiles' prefixes (null: there is one tile); E[n] all of them
__device__ __forceinline__ void change_prefixes(int n, const int *lab, const int *sums, const int *roots, int *E)
{
    if (*roots == 1) return;
    __shared__ int sw[kSmallThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tile_items = blockDim.x * kTileItems;
    for (int tile = blockIdx.x; tile * (long long)tile_items < n; tile += gridDim.x) {
        const int i0 = tile * tile_items + wid * (32 * kTileItems) + lane;
        int last = lane == 0 && i0 > 0 && i0 < n ? lab[i0 - 1] : -1;
        unsigned chg[kTileItems];
        int s = 0;
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) {
            const int i = i0 + 32 * t;
            const int x = i < n ? lab[i] : -1;
            const int before = __shfl_up_sync(0xffffffffu, x, 1);
            chg[t] = __ballot_sync(0xffffffffu, i > 0 && i < n && x != (lane ? before : last));
            last = __shfl_sync(0xffffffffu, x, 31);
            s += __popc(chg[t]);
        }
        if (lane == 0) sw[wid] = s;
        __syncthreads();
        int at = sums ? sums[tile] : 0;
        for (int w = 0; w < wid; ++w) at += sw[w];
#pragma unroll
        for (int t = 0; t < kTileItems; ++t) {
            const int i = i0 + 32 * t, e = at + __popc(chg[t] & lanemask_lt());
            if (i < n) E[i] = e;
            if (i == n - 1) E[n] = e + (int)((chg[t] >> lane) & 1u);
            at += __popc(chg[t]);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void node_labels(int Ns, int S, const int2 *__restrict__ range, float *nodes, int *nlab, const int *lab,
                                            const int *E, const int *roots)
{
    if (*roots == 1) return;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < Ns; x += gridDim.x * blockDim.x) {
        const int2 r = range[x];
        if (E[r.y] != E[r.x + 1]) continue;   // mixed: the label is -1 from the start
        const int c = lab[r.x];
        if (nlab[x] == c) continue;
        nlab[x] = c;
        nodes[(size_t)x * 2 * S + box_hi(S - 1)] = __int_as_float(c);
    }
}

template <int D, bool HDB, bool F64>
__global__ void nc_refresh_kernel(TravArgs a, NcArgs b) { refresh_points<D, HDB, F64>(a, b); }

template <bool HDB, bool MARK>
__global__ void nc_active_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    active_points<HDB, MARK>(a, b, sh);
}

template <bool HDB>
__global__ void nc_pick_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    pick_points<HDB>(a, b, sh);
}

template <int D, bool HDB, bool F64>
__global__ void nc_cand_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    candidates<D, HDB, F64>(a, b, sh);
}

__global__ void nc_low_kernel(NcArgs b) { low_ids(b); }

__global__ void nc_merge_kernel(TravArgs a, NcArgs b, int cur, EdgeK *out, int out_cap)
{
    __shared__ int sh[32];
    merge_roots(a, b, cur, out, out_cap, sh);
}

__global__ void __launch_bounds__(256) nc_roots_kernel(NcArgs b, int cur)
{
    __shared__ int sh[32];
    collect_roots(b, cur, sh);
}

__global__ void __launch_bounds__(256) nc_relabel_kernel(NcArgs b, int S, const int *roots, int *sums)
{
    relabel_points(b, S, roots, sums);
}

__global__ void __launch_bounds__(256) nc_prefix_kernel(int n, const int *lab, const int *sums, const int *roots, int *E)
{
    change_prefixes(n, lab, sums, roots, E);
}

__global__ void nc_node_labels_kernel(int Ns, int S, const int2 *range, float *nodes, int *nlab, const int *lab, const int *E,
                                      const int *roots)
{
    node_labels(Ns, S, range, nodes, nlab, lab, E, roots);
}

// Few points: the steps before, between and after the searches by one block, with barriers for the ends of the
// kernels.  Each of them is then shorter than the gap between two launches (figures at kSmallPoints).
template <int D, bool HDB, bool F64>
__global__ void __launch_bounds__(kSmallThreads) nc_small_front_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    refresh_points<D, HDB, F64>(a, b);
    __syncthreads();
    active_points<HDB, marks_ties(D)>(a, b, sh);
}

template <int D, bool HDB, bool F64>
__global__ void __launch_bounds__(kSmallThreads) nc_small_mid_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    if (b.first) {
        refresh_points<D, HDB, F64>(a, b);
        __syncthreads();
    }
    pick_points<HDB>(a, b, sh);
    __syncthreads();
    candidates<D, HDB, F64>(a, b, sh);
}

__global__ void __launch_bounds__(kSmallThreads) nc_small_back_kernel(TravArgs a, NcArgs b, int cur, EdgeK *out, int out_cap, int Ns,
                                                                      int S, const int2 *range, float *nodes, int *sums, int *E)
{
    __shared__ int sh[32];
    const int *roots = b.cnt + cnt_roots(cur ^ 1);
    low_ids(b);
    __syncthreads();
    merge_roots(a, b, cur, out, out_cap, sh);
    __syncthreads();
    collect_roots(b, cur, sh);
    __syncthreads();
    relabel_points(b, S, roots, sums);
    __syncthreads();
    change_prefixes(b.n, b.lab, nullptr, roots, E);
    __syncthreads();
    node_labels(Ns, S, range, nodes, b.nlab, b.lab, E, roots);
}

template <int D, bool HDB, bool F64>
int rounds(NcCall &C, TravArgs &a, NcArgs &b)
{
    cudaStream_t st = C.st;
    const int n = a.n;
    const int g = grid_for(n, 256), gt = grid_for(n, kTile);
    constexpr int S = row_floats(D);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nc_search_kernel<D, HDB, F64, false>, kWalkThreads, 0) != cudaSuccess ||
        per_sm < 1)
        return WM_ECUDA;
    const int gs = std::min(num_sms() * per_sm, C.X->walk_blocks);
    const SearchTree &X = *C.X;
    Arena &ar = *C.ar;
    b.nlab = ar.get<int>(X.Ns);
    const int tiles = (n + kTile - 1) / kTile;
    int *sums = ar.get<int>(tiles), *E = ar.get<int>((size_t)n + 1);
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(b.nlab, 0xff, sizeof(int) * X.Ns, st);
    if (HDB) {
        float *ncd = ar.get<float>(X.Ns);
        int *arrive = ar.get<int>(X.Ns);
        if (ar.failed) return WM_ENOMEM;
        cudaMemsetAsync(arrive, 0, sizeof(int) * X.Ns, st);
        launch(nc_core_min_kernel, grid_for(X.Ns, 256), 256, 0, st, X.Ns, X.range, X.parent, a.cd64, ncd, arrive);
        b.ncd = ncd;
    }
    launch(nc_init_kernel, g, 256, 0, st, a, b, HDB);
    const bool small = n <= kSmallPoints;
    const EdgeK *rin = C.rep;
    EdgeK *rbuf[2] = {C.rep_tmp0, C.rep_tmp1};
    long long edges = 0;
    // every component that can still grow links in a round: their number at least halves
    for (int r = 0; r < 64 && edges < C.target; ++r) {
        const int cur = r & 1;
        cudaMemsetAsync(b.cnt + (cur ? 0 : kCntEven), 0, (cur ? kCntOddEnd : kCntEdges - kCntEven) * sizeof(int), st);
        const int *roots = b.cnt + cnt_roots(cur ^ 1);
        const EdgeK *rnow = nullptr;
        const int *rn = nullptr;
        if (HDB) {
            launch(nc_repair_kernel, grid_for(C.nrep, 256), 256, 0, st, b, rin, r ? b.cnt + cnt_rep(cur ^ 1) : (const int *)nullptr,
                   C.nrep, rbuf[cur], b.cnt + cnt_rep(cur));
            rin = rnow = rbuf[cur];
            rn = b.cnt + cnt_rep(cur);
        }
        b.first = !HDB && r == 0;
        if (!b.first) {
            if (small) {
                launch(nc_small_front_kernel<D, HDB, F64>, 1, kSmallThreads, 0, st, a, b);
            } else {
                launch(nc_refresh_kernel<D, HDB, F64>, g, 256, 0, st, a, b);
                launch(nc_active_kernel<HDB, marks_ties(D)>, gt, 256, 0, st, a, b);
            }
        }
        auto middle = [&] {
            if (small) {
                launch(nc_small_mid_kernel<D, HDB, F64>, 1, kSmallThreads, 0, st, a, b);
            } else {
                if (b.first) launch(nc_refresh_kernel<D, HDB, F64>, g, 256, 0, st, a, b);   // the lists' minima into S
                launch(nc_pick_kernel<HDB>, g, 256, 0, st, a, b);
                launch(nc_cand_kernel<D, HDB, F64>, g, 256, 0, st, a, b);
            }
            launch(nc_search_kernel<D, HDB, F64, true>, gs, kWalkThreads, 0, st, a, b, X, n);
        };
        auto back = [&]() -> int {
            if (HDB) launch(nc_low_repair_kernel, grid_for(C.nrep, 256), 256, 0, st, b, rnow, rn);
            if (small) {
                launch(nc_small_back_kernel, 1, kSmallThreads, 0, st, a, b, cur, C.out, n - 1, X.Ns, S, X.range, X.nodes, sums, E);
            } else {
                launch(nc_low_kernel, g, 256, 0, st, b);
                launch(nc_merge_kernel, g, 256, 0, st, a, b, cur, C.out, n - 1);
                launch(nc_roots_kernel, std::min(g, num_sms() * kLinkBlocks), 256, 0, st, b, cur);
                launch(nc_relabel_kernel, gt, 256, 0, st, b, S, roots, sums);
                const int rc = scan_exclusive_i32(sums, sums, tiles, nullptr, st, ar);
                if (rc) return rc;
                launch(nc_prefix_kernel, gt, 256, 0, st, n, b.lab, sums, roots, E);
                launch(nc_node_labels_kernel, grid_for(X.Ns, 256), 256, 0, st, X.Ns, S, X.range, X.nodes, b.nlab, b.lab, E, roots);
            }
            cudaMemcpyAsync(C.pin, b.cnt, kCntAll * sizeof(int), cudaMemcpyDeviceToHost, st);
            return cudaStreamSynchronize(st) == cudaSuccess ? 0 : WM_ECUDA;
        };
        b.guard = 3;
        C.mark(C.ctx);
        launch(nc_search_kernel<D, HDB, F64, false>, gs, kWalkThreads, 0, st, a, b, X, n);
        C.mark(C.ctx);
        middle();
        int rc = back();
        if (rc == 0 && C.pin[kCntLong] > 0) {
            b.guard = 2;
            C.mark(C.ctx);
            for (int f = 0; f < C.pin[kCntLong]; f += kLongMax)
                launch(nc_long_kernel<D, HDB, F64, false>, num_sms() * 8, kWalkThreads, 0, st, a, b, f);
            C.mark(C.ctx);
            cudaMemsetAsync(b.cnt + kCntExactNext, 0, sizeof(int), st);   // (the search with nothing to do drew from it)
            middle();
            rc = back();
        }
        if (rc == 0 && C.pin[kCntLongExact] > 0) {
            b.guard = 0;
            for (int f = 0; f < C.pin[kCntLongExact]; f += kLongMax)
                launch(nc_long_kernel<D, HDB, F64, true>, num_sms() * 8, kWalkThreads, 0, st, a, b, f);
            rc = back();
        }
        if (rc) return rc;
        ++C.rounds;
        C.candidates += C.pin[kCntCand] + (HDB ? C.pin[cnt_rep(cur)] : 0);
        // (every edge takes one root)
        if (C.pin[kCntError] || C.pin[cnt_roots(cur ^ 1)] != n - C.pin[kCntEdges]) {
            set_error_detail("nearest-component rounds: an internal check failed");
            return WM_EINTERNAL;
        }
        if (C.pin[kCntEdges] == edges) break;   // cannot happen while an edge is missing; the caller checks
        edges = C.pin[kCntEdges];
    }
    C.done = edges;
    return 0;
}

}  // namespace

int nearest_component_rounds(NcCall &C, TravArgs &a)
{
    const int n = a.n;
    Arena &ar = *C.ar;
    size_t mark = ar.off;
    NcArgs b;
    memset(&b, 0, sizeof b);
    b.lab = ar.get<int>(n);
    b.par = ar.get<int>(n);
    b.S = ar.get<unsigned>(n);
    b.bhi = ar.get<unsigned long long>(n);
    b.blo = ar.get<unsigned long long>(n);
    b.K = list_len(walk_dim(a.d));
    b.ls = ar.get<float>((size_t)b.K * n);
    b.lj = ar.get<int>((size_t)b.K * n);
    b.R = ar.get<float>(n);
    b.hd = ar.get<unsigned char>(n);
    b.low = ar.get<float>(n);
    b.act = ar.get<int>(n);
    b.amb = ar.get<int>(n);
    b.cand = ar.get<EdgeK>(n);
    b.cand_c = ar.get<int>(n);
    b.cnt = ar.get<int>(kCntAll);
    b.roots[0] = ar.get<int>(n);
    b.roots[1] = ar.get<int>(n);
    b.picked = ar.get<int>(n);
    b.near = b.cand_c;   // (read before the candidates are written)
    a.overflow = (unsigned *)b.cnt + kCntError;
    b.n = n;
    b.long_few = ~0u;            // (of few points even a walk of all is short)
    const int few = long_points(walk_dim(a.d));
    if (n >= 2 * few) {
        b.long_few = (unsigned)std::max(few, n / 1024);
        b.long_most = std::max(2 * b.long_few, (unsigned)n / kLongPart);
        b.chunks = std::min(kLongChunks, n / kLongChunk);
        b.long_max = (int)std::min<long long>(kLongMax, std::max<long long>(4, kLongWork / n));
        b.long_done = ar.get<int>(kLongMax);
        b.long_s = ar.get<float>((size_t)kLongMax * b.chunks * b.K);
        b.long_j = ar.get<int>((size_t)kLongMax * b.chunks * b.K);
        b.long_k = ar.get<KMin>((size_t)kLongMax * b.chunks);
    }
    if (C.rep) {
        C.rep_tmp0 = ar.get<EdgeK>(C.nrep);
        C.rep_tmp1 = ar.get<EdgeK>(C.nrep);
    }
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(b.cnt, 0, kCntAll * sizeof(int), C.st);
    if (b.chunks) cudaMemsetAsync(b.long_done, 0, kLongMax * sizeof(int), C.st);
    b.pos = C.pos;
    b.rows = C.X->rows;
    const float cf = C.cap < INFINITY ? C.cap_f : INFINITY;
    memcpy(&b.cap_bits, &cf, sizeof cf);
    memcpy(&b.cap64, &C.cap, sizeof C.cap);
    if (!(C.cap < INFINITY)) b.cap64 = ~0ull;
    int rc;
    const bool hdb = a.cd64 != nullptr;
#define WM_NC(DV)                                                                          \
    rc = a.fp64 ? (hdb ? rounds<DV, true, true>(C, a, b) : rounds<DV, false, true>(C, a, b)) \
                : (hdb ? rounds<DV, true, false>(C, a, b) : rounds<DV, false, false>(C, a, b))
    const int wd = walk_dim(a.d);
    if (row_floats(wd) != C.X->S) { ar.off = mark; return WM_EINTERNAL; }
    switch (wd) {
    case 2: WM_NC(2); break;
    case 3: WM_NC(3); break;
    case 4: WM_NC(4); break;
    case 5: WM_NC(5); break;
    case 6: WM_NC(6); break;
    case 7: WM_NC(7); break;
    case 8: WM_NC(8); break;
    case 15: WM_NC(15); break;
    default: WM_NC(16); break;
    }
#undef WM_NC
    ar.off = mark;
    return rc;
}

}  // namespace wm
