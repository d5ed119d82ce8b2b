// dendro.cu -- ordered dendrogram and reachability plot of a weighted spanning tree (Sec. 4).
//
// Input: the n-1 tree edges sorted by K (rank i = position).  Dendrogram node n+i is the merge
// of edge i; leaves are the points.  The parents come from contracting the tree bottom-up (after
// Sao, Prokopenko and Lebrun-Grandie, PANDORA, 2024; the output is that of Sec. 4): a level contracts the
// lightest edge P(v) of every vertex v, as a Boruvka round does, and the contracted components are the
// vertices of the next level, at most half as many.  An edge that is the lightest at one of its ends has
// a vertex below it, so it does not branch, and contracting it only shortens a chain of the dendrogram.
// Let V be the vertex that an edge e is contracted into.  While P(V) is lighter than e, e lies above P(V)
// and V is replaced by the next level's vertex that contains it; the V at which this stops names the
// chain of e: the edges that stop at V, in rank order, hang below one another, and the last of them
// below P(V).  Every leaf hangs below its lightest incident edge.  (The heavy/light recursion of Sec. 4.2
// passes over all edges once per bit of the rank; here level l has at most n / 2^l vertices.)
//
// Order (Sec. 4.2, ordering theorem): with the tree rooted at s, the child of merge (u,v) that
// contains the endpoint nearer s is the left child.  The tree is rooted by an Euler tour and list
// ranking (Sec. 2.2); a cluster lies on the far side of edge (u,v) iff a representative vertex of
// it lies in the Euler interval of the deeper endpoint.  The reachability plot is the in-order
// sequence of leaves, obtained by list ranking an Euler tour of the ordered dendrogram; the bar
// of leaf i is the height of the in-order internal node before it.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "hdb.cuh"

namespace wm {

namespace {

// ---------------------------------------------------------------------------- list ranking
// Pointer jumping (Wyllie): S[a] = sum of w from a to the end of its list.
__global__ void lr_init_kernel(const int *__restrict__ succ, const int *__restrict__ w, int m, int *__restrict__ nxt,
                               int *__restrict__ S)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x) {
        nxt[a] = succ[a];
        S[a] = w[a];
    }
}

__global__ void lr_step_kernel(const int *__restrict__ nxt, const int *__restrict__ S, int m, int *__restrict__ nxt2,
                               int *__restrict__ S2)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x) {
        int b = nxt[a];
        if (b >= 0) {
            S2[a] = S[a] + S[b];
            nxt2[a] = nxt[b];
        } else {
            S2[a] = S[a];
            nxt2[a] = -1;
        }
    }
}

// Ruling-set list ranking: every head and about one element in 16 (picked by a multiplicative
// hash of its index, so that no index pattern of the list lengthens the sublists) is a splitter.
// A splitter walks its sublist up to the next splitter (prefix sums on the way), the splitters'
// list is ranked by pointer jumping, and every element adds its splitter's rank: O(m) work, walks
// of about 16 dependent steps, pointer jumping over about m/16 elements.
__global__ void lr_mark_kernel(const int *__restrict__ succ, int m, int *__restrict__ haspred)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x)
        if (succ[a] >= 0) haspred[succ[a]] = 1;
}

__global__ void lr_flag_kernel(const int *__restrict__ haspred, int m, int *__restrict__ flag)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x)
        flag[a] = !haspred[a] || ((unsigned)a * 0x9E3779B1u) >> 28 == 0;
}

__global__ void lr_walk_kernel(const int *__restrict__ succ, const int *__restrict__ w, const int *__restrict__ flag,
                               const int *__restrict__ sid, int m, int *__restrict__ owner, int *__restrict__ pre,
                               int *__restrict__ snext, int *__restrict__ ssum)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x) {
        if (!flag[a]) continue;
        const int s = sid[a];
        int x = a, p = 0, nx = -1;
        for (int it = 0; it < m; ++it) {
            owner[x] = s;
            p += w[x];
            pre[x] = p;
            const int y = succ[x];
            if (y < 0) break;
            if (flag[y]) { nx = sid[y]; break; }
            x = y;
        }
        snext[s] = nx;
        ssum[s] = p;
    }
}

__global__ void lr_finish_kernel(const int *__restrict__ owner, const int *__restrict__ pre, const int *__restrict__ w,
                                 const int *__restrict__ SS, int m, int *__restrict__ S)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < m; a += gridDim.x * blockDim.x)
        S[a] = SS[owner[a]] - pre[a] + w[a];
}

// --------------------------------------------------------------------------- Euler tour (tree)
__global__ void degree_kernel(const EdgeK *__restrict__ E, int m, int *deg)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        atomicAdd(&deg[edge_u(E[i])], 1);
        atomicAdd(&deg[edge_v(E[i])], 1);
    }
}

__global__ void adjacency_kernel(const EdgeK *__restrict__ E, int m, const int *__restrict__ off, int *cur,
                                 int *__restrict__ adj, int *__restrict__ slot_of)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        int u = edge_u(E[i]), v = edge_v(E[i]);
        int s0 = off[u] + atomicAdd(&cur[u], 1);
        adj[s0] = 2 * i;          // arc u -> v
        slot_of[2 * i] = s0;
        int s1 = off[v] + atomicAdd(&cur[v], 1);
        adj[s1] = 2 * i + 1;      // arc v -> u
        slot_of[2 * i + 1] = s1;
    }
}

__device__ inline int arc_head(const EdgeK *__restrict__ E, int a) { return (a & 1) ? edge_u(E[a >> 1]) : edge_v(E[a >> 1]); }

__global__ void tour_succ_kernel(const EdgeK *__restrict__ E, int m, const int *__restrict__ off,
                                 const int *__restrict__ adj, const int *__restrict__ slot_of, int s,
                                 int *__restrict__ succ, int *__restrict__ w)
{
    const int start = adj[off[s]];
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < 2 * m; a += gridDim.x * blockDim.x) {
        int y = arc_head(E, a);
        int p = slot_of[a ^ 1] + 1;
        if (p == off[y + 1]) p = off[y];
        int nx = adj[p];
        succ[a] = nx == start ? -1 : nx;
        w[a] = 1;
    }
}

// child endpoint (deeper) of each edge and the Euler interval of every vertex
__global__ void rooting_kernel(const EdgeK *__restrict__ E, int m, const int *__restrict__ S, int L,
                               int *__restrict__ child, int *__restrict__ tin, int *__restrict__ tout)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        int p0 = L - S[2 * i], p1 = L - S[2 * i + 1];   // tour positions of the two arcs
        int down = p0 < p1 ? 2 * i : 2 * i + 1;
        int c = arc_head(E, down);
        child[i] = c;
        tin[c] = p0 < p1 ? p0 : p1;
        tout[c] = p0 < p1 ? p1 : p0;
    }
}

// ---------------------------------------------------------------------- contraction levels
// Vertices of all levels share one index space: level l holds [off[l], off[l] + nv[l]), level 0 the n
// points.  Per vertex: P (rank of its lightest edge, kNoRank: none left), hook (link to the other end of
// that edge, or itself at the root of its component) and next (the next level's vertex).
constexpr int kNoRank = 0x7f7f7f7f;   // above every rank; a byte pattern that cudaMemset can write
constexpr int kLevelsMax = 40;

struct Contract {
    int *cu, *cv;            // ends of an edge in the current level, by rank
    int *list[2];            // ranks of the edges left
    int *P, *hook, *next;
    int *sup;                // vertex an edge was contracted into
    int *off, *nv, *ne;      // per level
    int cap;                 // vertices of all levels
};

__global__ void ct_init_kernel(const EdgeK *__restrict__ E, int m, int n, Contract c)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        c.cu[i] = edge_u(E[i]);
        c.cv[i] = edge_v(E[i]);
        c.list[0][i] = i;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c.off[0] = 0;
        c.nv[0] = n;
        c.ne[0] = m;
    }
}

// the steps of a level, for one edge or vertex
__device__ __forceinline__ void ct_lightest(const Contract &c, int r)
{
    const int u = __ldcg(c.cu + r), v = __ldcg(c.cv + r);
    if (r < __ldcg(c.P + u)) atomicMin(c.P + u, r);
    if (r < __ldcg(c.P + v)) atomicMin(c.P + v, r);
}

// links v along its lightest edge; true at the root of a component (of a mutual choice, the smaller one)
__device__ __forceinline__ bool ct_hook(const Contract &c, int v)
{
    const int r = __ldcg(c.P + v);
    c.next[v] = -1;
    if (r == kNoRank) {   // nothing left to join
        c.hook[v] = v;
        return false;
    }
    const int a = __ldcg(c.cu + r), o = a == v ? __ldcg(c.cv + r) : a;
    const bool root = __ldcg(c.P + o) == r && v <= o;
    c.hook[v] = root ? v : o;
    return root;
}

// the next level's vertices of those that hook below a root
__device__ __forceinline__ void ct_next(const Contract &c, int off, int nv)
{
    link_to_roots(c.hook, nv, [off](int t) { return off + t; });
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nv; t += gridDim.x * blockDim.x) {
        const int x = *(volatile int *)(c.hook + off + t);
        if (x != off + t) c.next[off + t] = *(volatile int *)(c.next + x);
    }
}

// a contracted edge notes its component; another one moves to the next level
__device__ __forceinline__ bool ct_edge(const Contract &c, int r)
{
    const int u = __ldcg(c.cu + r), v = __ldcg(c.cv + r);
    const int nu = __ldcg(c.next + u);
    if (u == v || __ldcg(c.P + u) == r || __ldcg(c.P + v) == r) {
        c.sup[r] = nu;
        return false;
    }
    c.cu[r] = nu;
    c.cv[r] = __ldcg(c.next + v);
    return true;
}

__global__ void ct_lightest_kernel(Contract c, int level)
{
    const int m = c.ne[level];
    const int *list = c.list[level & 1];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) ct_lightest(c, list[t]);
}

__global__ void ct_hook_kernel(Contract c, int level, int *bad)
{
    __shared__ int sh[32];
    const int m = c.nv[level], off = c.off[level], to = off + m;
    if (blockIdx.x == 0 && threadIdx.x == 0) c.off[level + 1] = to;
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        const bool root = t < m && ct_hook(c, off + t);
        const int slot = to + block_append(c.nv + level + 1, root ? 1 : 0, sh);
        if (root) {
            if (slot < c.cap) c.next[off + t] = slot;
            else atomicOr(bad, 16);
        }
    }
}

__global__ void __launch_bounds__(256) ct_next_kernel(Contract c, int level) { ct_next(c, c.off[level], c.nv[level]); }

__global__ void ct_edge_kernel(Contract c, int level)
{
    __shared__ int sh[32];
    const int m = c.ne[level];
    const int *list = c.list[level & 1];
    int *out = c.list[(level & 1) ^ 1];
    for (int b0 = blockIdx.x * blockDim.x; b0 < m; b0 += gridDim.x * blockDim.x) {
        const int t = b0 + threadIdx.x;
        const int r = t < m ? list[t] : -1;
        const bool keep = r >= 0 && ct_edge(c, r);
        const int slot = block_append(c.ne + level + 1, keep ? 1 : 0, sh);
        if (keep) out[slot] = r;
    }
}

// The levels left, by one block (their vertices and edges are few after the levels above): the same steps
// with barriers between them.
__global__ void __launch_bounds__(1024) ct_tail_kernel(Contract c, int level, int *bad)
{
    __shared__ int sh[32];
    for (; level + 1 < kLevelsMax; ++level) {
        const int m = __ldcg(c.ne + level), nv = __ldcg(c.nv + level), off = __ldcg(c.off + level), to = off + nv;
        if (m == 0) return;   // the same for every thread
        const int *list = c.list[level & 1];
        int *out = c.list[(level & 1) ^ 1];
        for (int t = threadIdx.x; t < m; t += 1024) ct_lightest(c, __ldcg(list + t));
        if (threadIdx.x == 0) c.off[level + 1] = to;
        __syncthreads();
        for (int b0 = 0; b0 < nv; b0 += 1024) {
            const int t = b0 + threadIdx.x;
            const bool root = t < nv && ct_hook(c, off + t);
            const int slot = to + block_append(c.nv + level + 1, root ? 1 : 0, sh);
            if (root) {
                if (slot < c.cap) c.next[off + t] = slot;
                else atomicOr(bad, 16);
            }
        }
        __syncthreads();
        ct_next(c, off, nv);
        __syncthreads();
        for (int b0 = 0; b0 < m; b0 += 1024) {
            const int t = b0 + threadIdx.x;
            const int r = t < m ? __ldcg(list + t) : -1;
            const bool keep = r >= 0 && ct_edge(c, r);
            const int slot = block_append(c.ne + level + 1, keep ? 1 : 0, sh);
            if (keep) out[slot] = r;
        }
        __syncthreads();
    }
}

// the chain of every edge (the edges are in rank order already)
__global__ void ct_chain_kernel(Contract c, int m, unsigned *__restrict__ key, int *__restrict__ rank)
{
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < m; r += gridDim.x * blockDim.x) {
        int g = c.sup[r];
        for (int it = 0; it < kLevelsMax && c.P[g] < r; ++it) g = c.next[g];
        key[r] = (unsigned)g;
        rank[r] = r;
    }
}

// parents of the merges from the sorted chains, and of the leaves
__global__ void ct_parent_kernel(Contract c, const unsigned *__restrict__ key, const int *__restrict__ rank, int m, int n,
                                 int *__restrict__ par)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        par[t] = c.P[t] == kNoRank ? -1 : n + c.P[t];   // (-1: not a spanning tree)
        if (t >= m) continue;
        const unsigned k = key[t];
        const int p = t + 1 < m && key[t + 1] == k ? rank[t + 1] : c.P[k];
        par[n + rank[t]] = p == kNoRank ? -1 : n + p;
    }
}

// ------------------------------------------------------------------------ children / order
__global__ void children_kernel(const int *__restrict__ par, int total, int n, int *nch, int *__restrict__ ch,
                                int *bad)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        int p = par[x];
        if (p < 0) {
            if (x != total - 1) atomicOr(bad, 1);   // only the last merge is the root
            continue;
        }
        int s = atomicAdd(&nch[p - n], 1);
        if (s < 2) ch[2 * (p - n) + s] = x;
        else atomicOr(bad, 2);
    }
}

__global__ void order_children_kernel(const EdgeK *__restrict__ E, int m, int n, const int *__restrict__ ch,
                                      const int *__restrict__ nch, const int *__restrict__ child,
                                      const int *__restrict__ tin, const int *__restrict__ tout,
                                      int *__restrict__ lc, int *__restrict__ rc, int *bad)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        lc[i] = rc[i] = 0;
        if (nch[i] != 2) { atomicOr(bad, 4); continue; }
        int c = child[i];
        int a = ch[2 * i], b = ch[2 * i + 1];
        int ra = a < n ? a : edge_u(E[a - n]);
        int rb = b < n ? b : edge_u(E[b - n]);
        bool ina = tin[ra] >= tin[c] && tin[ra] <= tout[c];
        bool inb = tin[rb] >= tin[c] && tin[rb] <= tout[c];
        if (ina == inb) { atomicOr(bad, 8); continue; }
        lc[i] = ina ? b : a;
        rc[i] = ina ? a : b;
    }
}

// Euler tour of the ordered dendrogram: event 2x = enter x, 2x+1 = exit x.
__global__ void dtour_kernel(int total, int n, const int *__restrict__ par, const int *__restrict__ lc,
                             const int *__restrict__ rc, int *__restrict__ succ, int *__restrict__ w)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        bool leaf = x < n;
        succ[2 * x] = leaf ? 2 * x + 1 : 2 * lc[x - n];
        w[2 * x] = leaf ? 1 : 0;
        int p = par[x];
        int sx;
        if (p < 0) sx = -1;
        else if (lc[p - n] == x) sx = 2 * rc[p - n];
        else sx = 2 * p + 1;
        succ[2 * x + 1] = sx;
        w[2 * x + 1] = 0;
    }
}

__global__ void dendro_out_kernel(const EdgeK *__restrict__ E, int m, int n, const int *__restrict__ lc,
                                  const int *__restrict__ rc, const int *__restrict__ S, int key_squared,
                                  wm_dnode *__restrict__ out_d, double *__restrict__ reach)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        int x = n + i;
        double key = edge_w2(E[i]);
        double h = key_squared ? sqrt(key) : key;
        if (out_d) {
            wm_dnode o;
            o.left = lc[i];
            o.right = rc[i];
            o.height = h;
            o.size = S[2 * x] - S[2 * x + 1];
            o.reserved = 0;
            out_d[i] = o;
        }
        const int at = n - S[2 * rc[i]];
        if (reach && at >= 0 && at < n) reach[at] = h;   // (outside only when the edges are no tree: reported)
    }
}

__global__ void order_out_kernel(int n, const int *__restrict__ S, int *__restrict__ order, double *reach)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        int idx = n - S[2 * x];
        if (order && idx >= 0 && idx < n) order[idx] = x;
        if (reach && idx == 0) reach[0] = INFINITY;
    }
}

__global__ void wm_to_edgek_kernel(const wm_edge *__restrict__ src, int m, int n, EdgeK *__restrict__ out, int *bad)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        wm_edge e = src[i];
        if (e.u < 0 || e.u >= n || e.v < 0 || e.v >= n || e.u == e.v || !(e.w >= 0.0) || isinf(e.w)) {
            atomicOr(bad, 1);
            e.u = 0; e.v = 0; e.w = 0.0;
        }
        out[i] = make_edge(e.w, e.u, e.v);
    }
}

}  // namespace

int edges_from_wm(const wm_edge *src, int n, EdgeK *out, int *bad, cudaStream_t st)
{
    cudaMemsetAsync(bad, 0, sizeof(int), st);
    if (n > 1) launch(wm_to_edgek_kernel, grid_for(n - 1, 256), 256, 0, st, src, n - 1, n, out, bad);
    return 0;
}

static bool dev_ptr(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// pointer jumping over m elements (the splitter list)
static int wyllie(const int *succ, const int *w, int m, int *S, Arena &ar, cudaStream_t st)
{
    size_t mark = ar.off;
    int *n0 = ar.get<int>(m), *n1 = ar.get<int>(m), *S1 = ar.get<int>(m);
    if (ar.failed) return WM_ENOMEM;
    int g = grid_for(m, 256);
    launch(lr_init_kernel, g, 256, 0, st, succ, w, m, n0, S);
    int steps = 1;
    while ((1LL << steps) < (long long)m) ++steps;
    int *na = n0, *nb = n1, *Sa = S, *Sb = S1;
    for (int t = 0; t < steps + 1; ++t) {
        launch(lr_step_kernel, g, 256, 0, st, na, Sa, m, nb, Sb);
        int *x = na; na = nb; nb = x;
        x = Sa; Sa = Sb; Sb = x;
    }
    if (Sa != S) cudaMemcpyAsync(S, Sa, sizeof(int) * m, cudaMemcpyDeviceToDevice, st);
    ar.off = mark;
    return 0;
}

// S[a] = sum of w over the list from a to its end (inclusive), for every element of the lists
// given by succ (-1 ends a list).
static int list_rank(const int *succ, const int *w, int m, int *S, Arena &ar, cudaStream_t st, int *pin)
{
    if (m <= 0) return 0;
    size_t mark = ar.off;
    int *haspred = ar.get<int>(m), *flag = ar.get<int>(m + 1), *sid = ar.get<int>(m + 1);
    int *owner = ar.get<int>(m), *pre = ar.get<int>(m);
    int *snext = ar.get<int>(m), *ssum = ar.get<int>(m), *SS = ar.get<int>(m), *ns_d = ar.get<int>(1);
    if (ar.failed) return WM_ENOMEM;
    const int g = grid_for(m, 256);
    cudaMemsetAsync(haspred, 0, sizeof(int) * m, st);
    launch(lr_mark_kernel, g, 256, 0, st, succ, m, haspred);
    launch(lr_flag_kernel, g, 256, 0, st, haspred, m, flag);
    int rc = scan_exclusive_i32(flag, sid, m, ns_d, st, ar);
    if (rc) return rc;
    launch(lr_walk_kernel, g, 256, 0, st, succ, w, flag, sid, m, owner, pre, snext, ssum);
    cudaMemcpyAsync(pin, ns_d, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    const int ns = pin[0];
    rc = wyllie(snext, ssum, ns, SS, ar, st);
    if (rc) return rc;
    launch(lr_finish_kernel, g, 256, 0, st, owner, pre, w, SS, m, S);
    ar.off = mark;
    return 0;
}

// E: n-1 edges sorted by K on the device; key_squared: keys are squared weights (heights = sqrt)
int dendrogram_impl(const EdgeK *E, int n, int start, int key_squared, wm_dnode *out_dendro, int *out_order,
                    double *out_reach, Arena &ar, cudaStream_t st, int *pin)
{
    if (!out_dendro && !out_order && !out_reach) return 0;
    size_t mark = ar.off;
    const bool dd = dev_ptr(out_dendro), dor = dev_ptr(out_order), dre = dev_ptr(out_reach);
    if (n == 1) {
        int z = 0;
        double inf = INFINITY;
        if (out_order) {
            if (dor) cudaMemcpyAsync(out_order, &z, sizeof(int), cudaMemcpyHostToDevice, st);
            else *out_order = 0;
        }
        if (out_reach) {
            if (dre) cudaMemcpyAsync(out_reach, &inf, sizeof(double), cudaMemcpyHostToDevice, st);
            else *out_reach = inf;
        }
        return cudaStreamSynchronize(st) == cudaSuccess ? 0 : WM_ECUDA;
    }
    const int m = n - 1, total = 2 * n - 1, L = 2 * m;
    int *deg = ar.get<int>(n + 1), *cur = ar.get<int>(n), *adj = ar.get<int>(L), *slot = ar.get<int>(L);
    int *succ = ar.get<int>(2 * total), *w = ar.get<int>(2 * total), *S = ar.get<int>(2 * total);
    int *child = ar.get<int>(m), *tin = ar.get<int>(n), *tout = ar.get<int>(n);
    int *par = ar.get<int>(total);
    Contract c;
    c.cap = 2 * n + 64;
    c.cu = ar.get<int>(m);
    c.cv = ar.get<int>(m);
    c.list[0] = ar.get<int>(m);
    c.list[1] = ar.get<int>(m);
    c.P = ar.get<int>(c.cap);
    c.hook = ar.get<int>(c.cap);
    c.next = ar.get<int>(c.cap);
    c.sup = ar.get<int>(m);
    c.off = ar.get<int>(3 * kLevelsMax);
    c.nv = c.off + kLevelsMax;
    c.ne = c.nv + kLevelsMax;
    int *nch = ar.get<int>(m), *ch = ar.get<int>(2 * m), *lc = ar.get<int>(m), *rc = ar.get<int>(m);
    int *bad = ar.get<int>(1);
    if (ar.failed) return WM_ENOMEM;
    const int g = grid_for(total, 256);
    cudaMemsetAsync(bad, 0, sizeof(int), st);
    // ---- root the tree at start: Euler tour + list ranking
    cudaMemsetAsync(deg, 0, sizeof(int) * (n + 1), st);
    cudaMemsetAsync(cur, 0, sizeof(int) * n, st);
    launch(degree_kernel, g, 256, 0, st, E, m, deg);
    int rc0 = scan_exclusive_i32(deg, deg, n + 1, nullptr, st, ar);
    if (rc0) return rc0;
    launch(adjacency_kernel, g, 256, 0, st, E, m, deg, cur, adj, slot);
    launch(tour_succ_kernel, g, 256, 0, st, E, m, deg, adj, slot, start, succ, w);
    rc0 = list_rank(succ, w, L, S, ar, st, pin);
    if (rc0) return rc0;
    fill_i32(tin, -1, n, st);
    {
        int hl = L;
        cudaMemcpyAsync(tout + start, &hl, sizeof(int), cudaMemcpyHostToDevice, st);
    }
    launch(rooting_kernel, g, 256, 0, st, E, m, S, L, child, tin, tout);
    {
        int neg = -1;
        cudaMemcpyAsync(tin + start, &neg, sizeof(int), cudaMemcpyHostToDevice, st);
    }
    // ---- merge parents (contraction levels)
    cudaMemsetAsync(c.P, 0x7f, sizeof(int) * (size_t)c.cap, st);
    cudaMemsetAsync(c.off, 0, sizeof(int) * 3 * kLevelsMax, st);
    launch(ct_init_kernel, g, 256, 0, st, E, m, n, c);
    // Grid-wide levels until about a thousand vertices are left: a level keeps a third of them on the
    // trees measured (at most half in any case), and the block that finishes takes whatever is left.
    int level = 0;
    for (double v = n; v > 2048.0 && level < 24; v /= 2.7, ++level) {
        const int gl = grid_for(std::max(1, n >> level), 256);
        launch(ct_lightest_kernel, gl, 256, 0, st, c, level);
        launch(ct_hook_kernel, gl, 256, 0, st, c, level, bad);
        launch(ct_next_kernel, std::min(gl, num_sms() * kLinkBlocks), 256, 0, st, c, level);
        launch(ct_edge_kernel, gl, 256, 0, st, c, level);
    }
    launch(ct_tail_kernel, 1, 1024, 0, st, c, level, bad);
    {
        const size_t at = ar.off;
        SortPairs sp;
        rc0 = sort_pairs_begin(sp, m, ar, succ);   // (free here: 4 n - 2 ints)
        if (rc0) return rc0;
        launch(ct_chain_kernel, g, 256, 0, st, c, m, sp.key[0], sp.idx[0]);
        sort_pairs(sp, (unsigned)c.cap, st);   // (a chain is named by a vertex)
        launch(ct_parent_kernel, g, 256, 0, st, c, sp.key[sp.cur], sp.idx[sp.cur], m, n, par);
        ar.off = at;
    }
    // ---- children, left/right, in-order
    cudaMemsetAsync(nch, 0, sizeof(int) * m, st);
    launch(children_kernel, g, 256, 0, st, par, total, n, nch, ch, bad);
    launch(order_children_kernel, g, 256, 0, st, E, m, n, ch, nch, child, tin, tout, lc, rc, bad);
    launch(dtour_kernel, g, 256, 0, st, total, n, par, lc, rc, succ, w);
    rc0 = list_rank(succ, w, 2 * total, S, ar, st, pin);
    if (rc0) return rc0;
    wm_dnode *od = out_dendro;
    int *oo = out_order;
    double *orr = out_reach;
    if (out_dendro && !dd) od = ar.get<wm_dnode>(m);
    if (out_order && !dor) oo = ar.get<int>(n);
    if (out_reach && !dre) orr = ar.get<double>(n);
    if (ar.failed) return WM_ENOMEM;
    launch(dendro_out_kernel, g, 256, 0, st, E, m, n, lc, rc, S, key_squared, od, orr);
    launch(order_out_kernel, g, 256, 0, st, n, S, oo, orr);
    if (out_dendro && !dd) cudaMemcpyAsync(out_dendro, od, sizeof(wm_dnode) * m, cudaMemcpyDeviceToHost, st);
    if (out_order && !dor) cudaMemcpyAsync(out_order, oo, sizeof(int) * n, cudaMemcpyDeviceToHost, st);
    if (out_reach && !dre) cudaMemcpyAsync(out_reach, orr, sizeof(double) * n, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(pin, bad, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    ar.off = mark;
    return pin[0] ? WM_EINTERNAL : 0;
}

int dendrogram(const EdgeK *E, int n, int start, wm_dnode *out_dendro, int *out_order, double *out_reach, Arena &ar,
               cudaStream_t st, int *pin)
{
    return dendrogram_impl(E, n, start, 1, out_dendro, out_order, out_reach, ar, st, pin);
}

}  // namespace wm
