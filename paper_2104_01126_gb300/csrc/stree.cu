// stree.cu -- builds the search tree (see stree.cuh) from the k-d tree.
#include <algorithm>

#include "stree.cuh"

namespace wm {

namespace {

// flag of the nodes the search tree keeps: the root and every child of a node above kBucket points
// (siblings together, so that they stay adjacent; node ids follow the levels of the build)
__global__ void st_flag_kernel(int N, const int *__restrict__ begin, const int *__restrict__ end,
                               const int *__restrict__ parent, int *__restrict__ flag)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const int p = parent[x];
        flag[x] = p < 0 || end[p] - begin[p] > kBucket;
    }
}

// rows of the kept nodes (idx: exclusive prefix of the flags)
template <int S>
__global__ void st_nodes_kernel(int N, int d, const int *__restrict__ begin, const int *__restrict__ end,
                                const int *__restrict__ left, const int *__restrict__ parent,
                                const float *__restrict__ lo, const float *__restrict__ hi, const int *__restrict__ idx,
                                float *__restrict__ nodes, int2 *__restrict__ range, int *__restrict__ sparent)
{
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const int p = parent[x];
        if (p >= 0 && end[p] - begin[p] <= kBucket) continue;
        const int t = idx[x], bb = begin[x], sz = end[x] - bb;
        float *r = nodes + (size_t)t * 2 * S;
        const unsigned ref = sz > kBucket ? (unsigned)idx[left[x]] : kBucketBit | (unsigned)(sz - 1) << 28 | (unsigned)bb;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            r[box_lo(k)] = k < d ? lo[(size_t)k * N + x] : k == S - 1 ? __uint_as_float(ref) : 0.f;
            r[box_hi(k)] = k < d ? hi[(size_t)k * N + x] : k == S - 1 ? __int_as_float(-1) : 0.f;
        }
        range[t] = make_int2(bb, bb + sz);
        sparent[t] = p < 0 ? -1 : idx[p];
    }
}

template <int S>
__global__ void st_rows_kernel(int n, int d, const float *__restrict__ x32, float *__restrict__ rows)
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

template <int S>
void fill(const Points &P, const Tree &T, SearchTree &X, const int *idx, cudaStream_t st)
{
    launch(st_nodes_kernel<S>, grid_for(T.N, 256), 256, 0, st, T.N, P.d, T.begin, T.end, T.left, T.parent, T.lo, T.hi, idx,
           X.nodes, X.range, X.parent);
    launch(st_rows_kernel<S>, grid_for(P.n, 256), 256, 0, st, P.n, P.d, P.x32, X.rows);
}

}  // namespace

// n < 2^28 (28-bit positions in a bucket's reference)
int build_search_tree(const Points &P, const Tree &T, SearchTree &X, Arena &ar, cudaStream_t st, int *pin)
{
    const int n = P.n;
    X.S = row_floats(P.d);
    X.stack_cap = T.depth + 4;
    X.walk_blocks = (int)std::min<long long>((long long)num_sms() * (2048 / kWalkThreads),
                                             ((long long)n + kWalkThreads - 1) / kWalkThreads);
    X.deep_levels = std::max(1, X.stack_cap - kWalkStack);
    X.deep = ar.get<uint2>((size_t)X.walk_blocks * kWalkThreads * X.deep_levels);
    X.rows = ar.get<float>((size_t)n * X.S);
    int *total = ar.get<int>(1), *idx0 = ar.get<int>((size_t)T.N);
    if (ar.failed) return WM_ENOMEM;
    launch(st_flag_kernel, grid_for(T.N, 256), 256, 0, st, T.N, T.begin, T.end, T.parent, idx0);
    int rc = scan_exclusive_i32(idx0, idx0, T.N, total, st, ar);
    if (rc) return rc;
    cudaMemcpyAsync(pin, total, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return WM_ECUDA;
    X.Ns = pin[0];
    X.nodes = ar.get<float>((size_t)X.Ns * 2 * X.S);
    X.range = ar.get<int2>(X.Ns);
    X.parent = ar.get<int>(X.Ns);
    if (ar.failed) return WM_ENOMEM;
    X.root = n > kBucket ? 1u : kBucketBit | (unsigned)(n - 1) << 28;
    switch (X.S) {
    case 4: fill<4>(P, T, X, idx0, st); break;
    case 8: fill<8>(P, T, X, idx0, st); break;
    case 16: fill<16>(P, T, X, idx0, st); break;
    default: fill<24>(P, T, X, idx0, st); break;
    }
    return 0;
}

}  // namespace wm
