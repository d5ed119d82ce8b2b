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
//             those that could still hold a lighter edge than the lists show;
//   search  : a thread per active point walks the k-d tree, the nearer child first, skipping nodes of
//             its own component and nodes beyond its bound, and rebuilds the point's list;
//   pick    : FP64 evaluation of the list entries within T(S[c]); the K-minimum per component by
//             two 64-bit WriteMins; a point whose list may have dropped a tie (R[i] <= T(S[c])
//             still) is answered by a walk that evaluates everything within T(S[c]) in FP64;
//   merge   : every component's root links to the other endpoint's component; of a mutual choice
//             the smaller root stays and the edge is emitted once.
// The lists of the first search (all points, nothing pruned) serve the first few rounds.
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
#include "wspd.cuh"

namespace wm {

namespace {

constexpr int kNcK = 4;         // list entries per point
constexpr int kNcBucket = 8;    // a subtree of at most this many points is scanned directly
constexpr int kNcThreads = 128; // threads per block of the search
constexpr int kNcStack = 16;    // stack entries of a thread in shared memory (the rest in global memory)
constexpr unsigned kBucketBit = 0x80000000u, kDone = 0xffffffffu;

struct NcArgs {
    int *lab;                  // component of a tree position (a tree position: the root)
    int *par;                  // links between roots
    unsigned *S;               // per root: smallest screened weight seen this round (float bits)
    unsigned long long *bhi, *blo;   // per root: K-minimum outgoing edge
    float *ls;                 // [kNcK][n] list weights, ascending
    int *lj;                   // [kNcK][n] list positions (-1: none)
    float *R;                  // every point outside the component and the list screens at >= R
    unsigned char *hd;         // first list entry that may lie outside the component
    int *act, *amb;            // active points; points that need the exact scan
    EdgeK *cand;               // candidate edges of the round and the component each serves
    int *cand_c;
    int *cnt;                  // [0] active, [1] search dispenser, [2] candidates, [3] exact scans,
                               // [4] their dispenser, [5] tree edges, [6] repair edges left
    const int *pos;            // input id -> tree position
    unsigned cap_bits;         // no edge at or above this weight (float bits; +inf: none)
    unsigned long long cap64;  // the same in FP64 bits
    const float4 *rows;        // point rows: coordinates, label in the last slot
    const float4 *nodes;       // search tree rows
    const int2 *range;         // their point ranges
    const float *ncd;          // HDBSCAN*: their smallest core distance (rounded down)
    unsigned root;             // reference of the root
    int Ns;                    // nodes of the search tree
    uint2 *deep;               // stack entries beyond kNcStack, [stack_cap - kNcStack][threads]
    int first;                 // first search: components are single points, nothing is pruned by S
    int stack_cap;
};

__device__ __forceinline__ float next_up(float x) { return x < INFINITY ? __uint_as_float(__float_as_uint(x) + 1u) : x; }

// one point of the point-major copy into registers (rows of 4, 8 or 16 floats)
template <int S>
__device__ __forceinline__ void load_row(const float4 *__restrict__ x4, int i, float (&v)[S])
{
    if (S == 4) {
        const float4 p = x4[i];
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
    } else {
#pragma unroll
        for (int c = 0; c < S / 8; ++c) {
            float4 p, q;
            ldg256((const float *)x4 + (size_t)i * S + 8 * c, p, q);
            v[8 * c] = p.x; v[8 * c + 1] = p.y; v[8 * c + 2] = p.z; v[8 * c + 3] = p.w;
            v[8 * c + 4] = q.x; v[8 * c + 5] = q.y; v[8 * c + 6] = q.z; v[8 * c + 7] = q.w;
        }
    }
}

// floats per point row: the coordinates and, in the last slot, the component label
template <int D>
__device__ __host__ __forceinline__ constexpr int row_floats() { return D <= 3 ? 4 : D <= 7 ? 8 : D <= 15 ? 16 : 24; }

// HDBSCAN*: true when the FP32 squared distance d32 proves D <= c for a core distance c (FP32 copy)
__device__ inline bool proven_repair(const TravArgs &a, float d32, float c)
{
    if (a.exact32) return d32 * (1.0f + 1.0f / 131072.0f) < c * (1.0f - 1.0f / 4194304.0f);
    const double r = sqrt((double)d32 * (1.0 + 1.0 / 131072.0)) + a.eta;
    return r * r * (1.0 + 1.0 / 131072.0) < (double)c * (1.0 - 1.0 / 4194304.0);
}

// relative error of a screened weight against the exact one (an upper bound, FP32)
__device__ inline void note_err(float s, double w, float &err)
{
    if (w > 0.0) err = fmaxf(err, __fdiv_ru(__double2float_ru(fabs((double)s - w)), __double2float_rd(w)));
}

// ---------------------------------------------------------------------------------- search
// The search tree: the nodes of the k-d tree down to the subtrees of at most kNcBucket points, siblings
// adjacent.  A node row holds its box in groups of four dimensions (lo then hi, as the traversals'
// packed boxes) and, in the last padded dimension, a reference (lo slot) and the component label or -1
// (hi slot).  A reference is the row of the left child, or for a bucket
// kBucketBit | (size - 1) << 28 | first point.
//
// EXACT = false rebuilds the lists of the active points.  EXACT = true answers the points whose list may
// have dropped a tie: every point within T(S[c]) is evaluated in FP64 and the K-minimum becomes the
// point's candidate edge.
template <int D, bool HDB, bool EXACT>
__global__ void __launch_bounds__(kNcThreads) nc_search_kernel(TravArgs a, NcArgs b, int m_all)
{
    __shared__ uint2 sst[kNcStack][kNcThreads];
    constexpr int S = row_floats<D>(), G = S / 4, K = kNcK;
    const int lane = threadIdx.x & 31;
    const int n = a.n;
    const int m = EXACT ? b.cnt[3] : b.first ? m_all : b.cnt[0];
    const size_t nthr = (size_t)gridDim.x * kNcThreads;
    uint2 *deep = b.deep + (size_t)blockIdx.x * kNcThreads + threadIdx.x;
    unsigned long long n_ev = 0, n_re = 0;
    float err = 0.f;
    while (true) {
        int base = 0;
        if (lane == 0) base = atomicAdd(b.cnt + (EXACT ? 4 : 1), 32);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= m) break;
        const bool valid = base + lane < m;
        const int t = valid ? base + lane : base;
        const int i = EXACT ? b.amb[t] : b.first ? t : b.act[t];
        float q[S];
        load_row<S>(b.rows, i, q);
        const int c = b.lab[i];
        const float qcd = HDB ? a.cd32[i] : 0.f;
        const float qcd_lo = HDB ? qcd * (1.0f - 1.0f / 4194304.0f) : 0.f;
        float Sc = __uint_as_float(*(volatile unsigned *)(b.S + c));
        float sl[K];
        int sj[K];
#pragma unroll
        for (int k = 0; k < K; ++k) { sl[k] = INFINITY; sj[k] = -1; }
        KMin best{~0ull, ~0ull};
        // a candidate screens below lim; a node is skipped when its lower bound exceeds pb (the
        // bound is on the exact weight, which is within 2^-19 of the screened one)
        float lim = next_up(screen_threshold(Sc, a));
        float pb = lim * (1.0f + 1.0f / 131072.0f);
        int sp = 0, since = 0;
        unsigned cur = valid ? b.root : kDone;
        unsigned ev = 0;
        for (unsigned guard = 0; guard < 2u * (unsigned)a.N + 2u; ++guard) {
            // ---- down to the next bucket within the bound
            while (!(cur & kBucketBit)) {
                const float *bx = (const float *)b.nodes + (size_t)cur * 2 * S;
                float g0 = 0.f, g1 = 0.f;
                unsigned r0 = 0, r1 = 0;
                int l0 = 0, l1 = 0;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    float4 lo0, hi0, lo1, hi1;
                    ldg256(bx + 8 * g, lo0, hi0);
                    ldg256(bx + 2 * S + 8 * g, lo1, hi1);
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
                    if (g == G - 1) {
                        r0 = __float_as_uint(lo0.w);
                        r1 = __float_as_uint(lo1.w);
                        l0 = __float_as_int(hi0.w);
                        l1 = __float_as_int(hi1.w);
                    }
                }
                g0 = lower_w2(g0);
                g1 = lower_w2(g1);
                if (HDB) {
                    g0 = fmaxf(g0, fmaxf(qcd_lo, b.ncd[cur]));
                    g1 = fmaxf(g1, fmaxf(qcd_lo, b.ncd[cur + 1]));
                }
                const bool n0 = g0 <= pb && l0 != c, n1 = g1 <= pb && l1 != c;
                if (n0 && n1) {
                    const bool sw = g1 < g0;
                    const uint2 far = sw ? make_uint2(r0, __float_as_uint(g0)) : make_uint2(r1, __float_as_uint(g1));
                    if (sp < kNcStack) sst[sp][threadIdx.x] = far;
                    else if (sp < b.stack_cap) deep[(size_t)(sp - kNcStack) * nthr] = far;
                    else { atomicOr(a.overflow, 8u); cur = kDone; break; }   // cannot happen: one entry per level
                    ++sp;
                    cur = sw ? r1 : r0;
                } else if (n0 || n1) {
                    cur = n0 ? r0 : r1;
                } else {
                    cur = kDone;
                    while (sp > 0) {
                        --sp;
                        const uint2 e = sp < kNcStack ? sst[sp][threadIdx.x] : deep[(size_t)(sp - kNcStack) * nthr];
                        if (__uint_as_float(e.y) <= pb) { cur = e.x; break; }
                    }
                }
            }
            if (cur == kDone) break;
            // ---- scan the bucket
            const int j0 = (int)(cur & 0x0fffffffu), sz = (int)((cur >> 28) & 7u) + 1;
            const float was = sl[0];
            for (int p = 0; p < sz; ++p) {
                float x[S];
                load_row<S>(b.rows, j0 + p, x);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    const float dx = q[k] - x[k];
                    s = fmaf(dx, dx, s);
                }
                float w = s, cdm = 0.f;
                if (HDB) {
                    cdm = fmaxf(qcd, a.cd32[j0 + p]);
                    w = fmaxf(s, cdm);
                }
                if (w < lim && __float_as_int(x[S - 1]) != c && (!HDB || !proven_repair(a, s, cdm))) {
                    if (EXACT) {
                        const int j = j0 + p;
                        double x2 = dist64(a.x64, n, a.d, i, j);
                        if (HDB) x2 = pos_dmax(x2, pos_dmax(a.cd64[i], a.cd64[j]));
                        note_err(w, x2, err);
                        kmin_update(best, x2, a.pid[i], a.pid[j]);
                        ++n_re;
                        continue;
                    }
#pragma unroll
                    for (int k = K - 1; k >= 0; --k) {
                        if (k > 0 && w < sl[k - 1]) {
                            sl[k] = sl[k - 1];
                            sj[k] = sj[k - 1];
                        } else if (w < sl[k]) {
                            sl[k] = w;
                            sj[k] = j0 + p;
                        }
                    }
                    lim = fminf(lim, sl[K - 1]);
                }
            }
            ev += (unsigned)sz;
            if (!EXACT && !b.first) {
                // the component's minimum: lowered by this point, else re-read now and then
                ++since;
                float now = Sc;
                if (sl[0] < was && sl[0] < Sc)
                    now = fminf(sl[0], __uint_as_float(atomicMin(b.S + c, __float_as_uint(sl[0]))));
                else if ((since & 3) == 0)
                    now = __uint_as_float(*(volatile unsigned *)(b.S + c));
                if (now < Sc) {
                    Sc = now;
                    lim = fminf(lim, next_up(screen_threshold(Sc, a)));
                }
            }
            pb = lim * (1.0f + 1.0f / 131072.0f);
            // ---- next pending node within the bound
            cur = kDone;
            while (sp > 0) {
                --sp;
                const uint2 e = sp < kNcStack ? sst[sp][threadIdx.x] : deep[(size_t)(sp - kNcStack) * nthr];
                if (__uint_as_float(e.y) <= pb) { cur = e.x; break; }
            }
            if (cur == kDone) break;
        }
        n_ev += ev;
        if (EXACT && valid && best.hi < b.cap64) {
            const int slot = atomicAdd(b.cnt + 2, 1);   // at most one candidate per point: within n
            EdgeK e;
            e.hi = best.hi;
            e.lo = best.lo;
            b.cand[slot] = e;
            b.cand_c[slot] = c;
            if (best.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, best.hi);
        }
        if (!EXACT && valid) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                b.ls[(size_t)k * n + i] = sl[k];
                b.lj[(size_t)k * n + i] = sj[k];
            }
            b.R[i] = lim;
            b.hd[i] = 0;
        }
        __syncwarp();
    }
    n_ev = warp_sum_u64(n_ev);
    if (lane == 0 && n_ev) {
        atomicAdd(a.stat + 1, n_ev);
        atomicAdd(a.stat + 6, n_ev);
    }
    if (EXACT) {
        err_flush(a, err);
        n_re = warp_sum_u64(n_re);
        if (lane == 0 && n_re) atomicAdd(a.stat + 2, n_re);
    }
}

// ---------------------------------------------------------------------------- search tree
// flag of the nodes the search tree keeps: the root and every child of a node above kNcBucket points
__global__ void nc_flag_kernel(int N, const int *__restrict__ begin, const int *__restrict__ end,
                               const int *__restrict__ parent, int *__restrict__ flag)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const int p = parent[x];
        flag[x] = p < 0 || end[p] - begin[p] > kNcBucket;
    }
}

// rows of the kept nodes (idx: exclusive prefix of the flags)
template <int S>
__global__ void nc_nodes_kernel(int N, int d, const int *__restrict__ begin, const int *__restrict__ end,
                                const int *__restrict__ left, const int *__restrict__ parent,
                                const float *__restrict__ lo, const float *__restrict__ hi,
                                const float *__restrict__ cdmin, const int *__restrict__ idx, float *__restrict__ rows,
                                int2 *__restrict__ range, float *__restrict__ ncd)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const int p = parent[x];
        if (p >= 0 && end[p] - begin[p] <= kNcBucket) continue;
        const int t = idx[x], bb = begin[x], sz = end[x] - bb;
        float *r = rows + (size_t)t * 2 * S;
        const unsigned ref = sz > kNcBucket ? (unsigned)idx[left[x]] : kBucketBit | (unsigned)(sz - 1) << 28 | (unsigned)bb;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            r[box_lo(k)] = k < d ? lo[(size_t)k * N + x] : k == S - 1 ? __uint_as_float(ref) : 0.f;
            r[box_hi(k)] = k < d ? hi[(size_t)k * N + x] : k == S - 1 ? __int_as_float(-1) : 0.f;
        }
        range[t] = make_int2(bb, bb + sz);
        if (ncd) ncd[t] = cdmin[x];
    }
}

template <int S>
__global__ void nc_rows_kernel(int n, int d, const float *__restrict__ x32, float *__restrict__ rows)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float4 *r = (float4 *)(rows + (size_t)i * S);
#pragma unroll
        for (int c = 0; c < S / 4; ++c) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                v[k] = 4 * c + k < d ? x32[(size_t)(4 * c + k) * n + i] : 4 * c + k == S - 1 ? __int_as_float(i) : 0.f;
            r[c] = make_float4(v[0], v[1], v[2], v[3]);
        }
    }
}

// ------------------------------------------------------------------------- round bookkeeping
__global__ void nc_init_kernel(TravArgs a, NcArgs b, bool hdb)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        b.lab[i] = i;
        b.par[i] = i;
        b.S[i] = b.cap_bits;
        b.bhi[i] = ~0ull;
        b.blo[i] = ~0ull;
        if (hdb) {   // no list yet: an edge outside the repair list is longer than the core distance
            b.hd[i] = (unsigned char)kNcK;
            b.R[i] = __double2float_rd(a.cd64[i]);
        }
    }
}

// WriteMin of a weight into a component's slot; a value that cannot lower it is not issued
__device__ __forceinline__ void s_min(unsigned *S, int c, float v)
{
    const unsigned u = __float_as_uint(v);
    if (u < *(volatile unsigned *)(S + c)) atomicMin(S + c, u);
}

// Advances the list heads past entries that joined the component; the first entry left bounds the
// component's minimum.  A point without one offers its neighbours in tree order.
template <int D, bool HDB>
__global__ void nc_refresh_kernel(TravArgs a, NcArgs b)
{
    constexpr int S = row_floats<D>();
    const int n = a.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = b.lab[i];
        int h = b.hd[i];
        if (h < kNcK) {
            const int h0 = h;
            int j = -1;
            for (; h < kNcK; ++h) {
                j = b.lj[(size_t)h * n + i];
                if (j >= 0 && b.lab[j] != c) break;
            }
            if (h != h0) b.hd[i] = (unsigned char)h;
            if (h < kNcK) s_min(b.S, c, b.ls[(size_t)h * n + i]);
        }
        if (h >= kNcK) {
#pragma unroll
            for (int o = -1; o <= 1; o += 2) {
                const int j = i + o;
                if (j < 0 || j >= n || b.lab[j] == c) continue;
                float x[S], y[S];
                load_row<S>(b.rows, i, x);
                load_row<S>(b.rows, j, y);
                float acc = 0.f;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    const float dx = x[k] - y[k];
                    acc = fmaf(dx, dx, acc);
                }
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
                s_min(b.S, cu, s);
                s_min(b.S, cv, s);
                if (e.hi < *(volatile unsigned long long *)(b.bhi + cu)) atomicMin(b.bhi + cu, e.hi);
                if (e.hi < *(volatile unsigned long long *)(b.bhi + cv)) atomicMin(b.bhi + cv, e.hi);
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

template <bool HDB>
__global__ void nc_active_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    const int n = a.n;
    for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
        const int i = b0 + threadIdx.x;
        bool on = false;
        if (i < n) {
            const int c = b.lab[i];
            on = b.R[i] <= screen_threshold(__uint_as_float(b.S[c]), a);
            if (HDB && on) on = !settled(a, b, i, c);
        }
        const int slot = block_append(b.cnt + 0, on ? 1 : 0, sh);
        if (on) b.act[slot] = i;
    }
}

// K-minimum of a point's list entries inside the band of its component's screened minimum
template <bool HDB>
__global__ void nc_pick_kernel(TravArgs a, NcArgs b)
{
    __shared__ int sh[32];
    const int n = a.n;
    unsigned long long n_re = 0;
    float err = 0.f;
    for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
        const int i = b0 + threadIdx.x;
        bool exact = false;
        int c = -1;
        KMin best{~0ull, ~0ull};
        if (i < n) {
            c = b.lab[i];
            const float T = screen_threshold(__uint_as_float(b.S[c]), a);
            exact = b.R[i] <= T;
            if (HDB && exact) exact = !settled(a, b, i, c);
            if (!exact) {
                for (int h = b.hd[i]; h < kNcK; ++h) {
                    const float s = b.ls[(size_t)h * n + i];
                    if (s > T) break;
                    const int j = b.lj[(size_t)h * n + i];
                    if (j < 0 || b.lab[j] == c) continue;
                    double w = dist64(a.x64, n, a.d, i, j);
                    if (HDB) w = pos_dmax(w, pos_dmax(a.cd64[i], a.cd64[j]));
                    note_err(s, w, err);
                    kmin_update(best, w, a.pid[i], a.pid[j]);
                    ++n_re;
                }
            }
        }
        const bool has = best.hi < b.cap64;
        int slot = block_append(b.cnt + 2, has ? 1 : 0, sh);
        if (has) {
            EdgeK e;
            e.hi = best.hi;
            e.lo = best.lo;
            b.cand[slot] = e;
            b.cand_c[slot] = c;
            if (best.hi < *(volatile unsigned long long *)(b.bhi + c)) atomicMin(b.bhi + c, best.hi);
        }
        slot = block_append(b.cnt + 3, exact ? 1 : 0, sh);
        if (exact) b.amb[slot] = i;
    }
    err_flush(a, err);
    n_re = warp_sum_u64(n_re);
    if ((threadIdx.x & 31) == 0 && n_re) atomicAdd(a.stat + 2, n_re);
}

// Among the candidates with their component's smallest weight: WriteMin of the id pair
__global__ void nc_low_kernel(NcArgs b)
{
    const int m = b.cnt[2];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) {
        const EdgeK e = b.cand[t];
        const int c = b.cand_c[t];
        if (e.hi == b.bhi[c]) atomicMin(b.blo + c, e.lo);
    }
}

__global__ void nc_low_repair_kernel(NcArgs b, const EdgeK *__restrict__ rep, const int *__restrict__ m_dev)
{
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
__global__ void nc_merge_kernel(TravArgs a, NcArgs b, EdgeK *__restrict__ out, int out_cap)
{
    __shared__ int sh[32];
    const int n = a.n;
    for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
        const int i = b0 + threadIdx.x;
        bool emit = false;
        EdgeK e;
        e.hi = 0;
        e.lo = 0;
        if (i < n && b.lab[i] == i) {
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
                    if (emit && mutual) b.par[i] = i;
                    else b.par[i] = o;
                }
            }
        }
        const int slot = block_append(b.cnt + 5, emit ? 1 : 0, sh);
        if (emit) {
            if (slot < out_cap) out[slot] = e;
            else atomicOr(a.overflow, 16u);
        }
    }
}

// New labels; the per-round slots are reset on the way
__global__ void nc_relabel_kernel(NcArgs b, int n, int S)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = b.lab[i];
        int x = c;
        for (int it = 0; it < n; ++it) {
            const int p = *(volatile int *)(b.par + x);
            if (p == x) break;
            const int g = *(volatile int *)(b.par + p);
            if (g != p) *(volatile int *)(b.par + x) = g;   // path halving (the forest is static)
            x = p;
        }
        if (x != c) {
            b.lab[i] = x;
            const_cast<float *>((const float *)b.rows)[(size_t)i * S + S - 1] = __int_as_float(x);
        }
        if (x == i) {   // only roots' slots are read
            b.S[i] = b.cap_bits;
            b.bhi[i] = ~0ull;
            b.blo[i] = ~0ull;
        }
    }
}

__global__ void nc_change_kernel(const int *__restrict__ lab, int n, int *__restrict__ chg)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        chg[i] = i > 0 && lab[i] != lab[i - 1];
}

__global__ void nc_node_labels_kernel(int Ns, int S, const int2 *__restrict__ range, float *__restrict__ nodes,
                                      const int *__restrict__ lab, const int *__restrict__ E)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < Ns; x += gridDim.x * blockDim.x) {
        const int2 r = range[x];
        if (E[r.y] != E[r.x + 1]) continue;   // mixed: the label is -1 from the start
        nodes[(size_t)x * 2 * S + box_hi(S - 1)] = __int_as_float(lab[r.x]);
    }
}

// the union-find over input ids that the MemoGFK rounds continue from
__global__ void nc_export_kernel(const int *__restrict__ lab, const int *__restrict__ pid, int n, int *__restrict__ uf)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) uf[pid[i]] = pid[lab[i]];
}

template <int D, bool HDB>
int rounds(NcCall &C, TravArgs &a, NcArgs &b)
{
    cudaStream_t st = C.st;
    const int n = a.n;
    const int g = grid_for(n, 256);
    constexpr int S = row_floats<D>();
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nc_search_kernel<D, HDB, false>, kNcThreads, 0) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        return 0;
    }
    const int gs = (int)std::min<long long>((long long)num_sms() * per_sm, ((long long)n + kNcThreads - 1) / kNcThreads);
    // ---- the search tree and the point rows
    const Tree &T = *C.T;
    float *rows = C.ar->get<float>((size_t)n * S);
    b.deep = C.ar->get<uint2>((size_t)gs * kNcThreads * std::max(1, b.stack_cap - kNcStack));
    int *idx = C.ar->get<int>((size_t)a.N + 1);
    if (C.ar->failed) return WM_ENOMEM;
    const int gN = grid_for(a.N, 256);
    launch(nc_flag_kernel, gN, 256, 0, st, a.N, T.begin, T.end, T.parent, idx);
    int rc0 = scan_exclusive_i32(idx, idx, a.N, idx + a.N, st, *C.ar);
    if (rc0) return rc0;
    cudaMemcpyAsync(C.pin, idx + a.N, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    b.Ns = C.pin[0];
    float *nodes = C.ar->get<float>((size_t)b.Ns * 2 * S);
    int2 *range = C.ar->get<int2>(b.Ns);
    float *ncd = HDB ? C.ar->get<float>(b.Ns) : nullptr;
    if (C.ar->failed) return WM_ENOMEM;
    launch(nc_nodes_kernel<S>, gN, 256, 0, st, a.N, a.d, T.begin, T.end, T.left, T.parent, T.lo, T.hi, a.cdmin, idx, nodes,
           range, ncd);
    launch(nc_rows_kernel<S>, g, 256, 0, st, n, a.d, a.x32, rows);
    b.rows = (const float4 *)rows;
    b.nodes = (const float4 *)nodes;
    b.range = range;
    b.ncd = ncd;
    b.root = n > kNcBucket ? 1u : kBucketBit | (unsigned)(n - 1) << 28;
    launch(nc_init_kernel, g, 256, 0, st, a, b, HDB);
    const EdgeK *rin = C.rep;
    EdgeK *rbuf[2] = {C.rep_tmp0, C.rep_tmp1};
    long long done = 0;
    for (int r = 0; r < 64 && done < C.target; ++r) {
        cudaMemsetAsync(b.cnt, 0, 5 * sizeof(int), st);
        cudaMemsetAsync(b.cnt + 6 + (r & 1), 0, sizeof(int), st);
        const EdgeK *rnow = nullptr;
        const int *rn = nullptr;
        if (HDB) {
            launch(nc_repair_kernel, grid_for(C.nrep, 256), 256, 0, st, b, rin, r ? b.cnt + 6 + ((r & 1) ^ 1) : (const int *)nullptr,
                   C.nrep, rbuf[r & 1], b.cnt + 6 + (r & 1));
            rin = rnow = rbuf[r & 1];
            rn = b.cnt + 6 + (r & 1);
        }
        b.first = !HDB && r == 0;
        if (!b.first) {
            launch(nc_refresh_kernel<D, HDB>, g, 256, 0, st, a, b);
            launch(nc_active_kernel<HDB>, g, 256, 0, st, a, b);
        }
        const int e0 = C.mark(C.ctx);
        launch(nc_search_kernel<D, HDB, false>, gs, kNcThreads, 0, st, a, b, n);
        const int e1 = C.mark(C.ctx);
        C.span(C.ctx, e0, e1);
        if (b.first) launch(nc_refresh_kernel<D, HDB>, g, 256, 0, st, a, b);   // the lists' minima into S
        launch(nc_pick_kernel<HDB>, g, 256, 0, st, a, b);
        launch(nc_search_kernel<D, HDB, true>, gs, kNcThreads, 0, st, a, b, n);
        launch(nc_low_kernel, g, 256, 0, st, b);
        if (HDB) launch(nc_low_repair_kernel, grid_for(C.nrep, 256), 256, 0, st, b, rnow, rn);
        launch(nc_merge_kernel, g, 256, 0, st, a, b, C.out, n - 1);
        launch(nc_relabel_kernel, g, 256, 0, st, b, n, S);
        launch(nc_change_kernel, g, 256, 0, st, b.lab, n, C.E);
        int rc = scan_exclusive_i32(C.E, C.E, n, C.E + n, st, *C.ar);
        if (rc) return rc;
        launch(nc_node_labels_kernel, grid_for(b.Ns, 256), 256, 0, st, b.Ns, S, range, nodes, b.lab, C.E);
        cudaMemcpyAsync(C.pin, b.cnt, 8 * sizeof(int), cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(C.pin + 8, a.overflow, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
        ++C.rounds;
        C.candidates += C.pin[2] + (HDB ? C.pin[6 + (r & 1)] : 0);
        if (C.pin[8]) {
            set_error_detail("nearest-component rounds: an internal check failed");
            return WM_EINTERNAL;
        }
        if (C.pin[5] <= done) break;   // no progress: the caller's other path takes over
        done = C.pin[5];
    }
    C.done = done;
    launch(nc_export_kernel, g, 256, 0, st, b.lab, a.pid, n, C.uf);
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
    b.ls = ar.get<float>((size_t)kNcK * n);
    b.lj = ar.get<int>((size_t)kNcK * n);
    b.R = ar.get<float>(n);
    b.hd = ar.get<unsigned char>(n);
    b.act = ar.get<int>(n);
    b.amb = ar.get<int>(n);
    b.cand = ar.get<EdgeK>(n);
    b.cand_c = ar.get<int>(n);
    b.cnt = ar.get<int>(16);
    C.E = ar.get<int>((size_t)n + 1);
    if (C.rep) {
        C.rep_tmp0 = ar.get<EdgeK>(C.nrep);
        C.rep_tmp1 = ar.get<EdgeK>(C.nrep);
    }
    if (ar.failed) return WM_ENOMEM;
    cudaMemsetAsync(b.cnt, 0, 16 * sizeof(int), C.st);
    b.pos = C.pos;
    b.stack_cap = C.depth + 4;
    const float cf = C.cap < INFINITY ? C.cap_f : INFINITY;
    memcpy(&b.cap_bits, &cf, sizeof cf);
    memcpy(&b.cap64, &C.cap, sizeof C.cap);
    if (!(C.cap < INFINITY)) b.cap64 = ~0ull;
    int rc;
    const bool hdb = a.cd64 != nullptr;
#define WM_NC(DV) rc = hdb ? rounds<DV, true>(C, a, b) : rounds<DV, false>(C, a, b)
    if (a.d == 2) WM_NC(2);
    else if (a.d == 3) WM_NC(3);
    else if (a.d <= 4) WM_NC(4);
    else if (a.d == 5) WM_NC(5);
    else if (a.d == 6) WM_NC(6);
    else if (a.d == 7) WM_NC(7);
    else if (a.d <= 8) WM_NC(8);
    else WM_NC(16);
#undef WM_NC
    ar.off = mark;
    return rc;
}

}  // namespace wm
