// Centroid update of (weighted) k-means (Sec. 2.2: k-means builds the codebook; Sec. 3.2.1: with the
// Hessian diagonal of a vector's column as its weight): with the assignment fixed, every centroid
// becomes the weighted mean of the vectors assigned to it,
//   C_i[j] = sum h_n x_j / sum h_n   over vectors (r, n) with idx[r][n] = i that have component j,
// and a component that received no weight keeps its old value.
//
// accumulate: one thread per vector.  A table of few centroids (k*v <= 4096: many vectors per address): h*x and h are added
//             to FP32 sums in a shared-memory copy per block (256 centroids of 8, 2.1 M vectors: 168 -> 113 us with one weight
//             per centroid instead of one per component).  Otherwise straight into the workspace,
//             where a centroid has a row of 16-byte aligned sums with the weight behind the v components, so that
//             four of them go out in one vector reduction: 4096 x 4096, v = 8, 65536 centroids 37 us (one reduction per
//             component for the sum and one for the weight: 160 us, bound by the reductions at L2).  Vectors of a
//             short last row weigh in on the components they have only, in an array of their own.
// finish:     one thread per (centroid, component): C = fp16(sum / weight) where weight > 0.
// FP32 atomic sums: the order of the additions is not fixed, so the result agrees with a FP64 mean
// to FP32 summation error, not bit for bit.
#include "common.cuh"

namespace vptq {

namespace {

constexpr int KM_THREADS = 256;
constexpr int KM_SMEM_ENTRIES = 4096;      // (centroid, component) pairs that fit the per-block copy: 32 KB

// floats of a centroid's row in the workspace: v sums, the weight, padded to whole 16-byte pieces
__host__ __device__ inline int row_floats(int v) { return (v + 1 + 3) / 4 * 4; }

__global__ void __launch_bounds__(KM_THREADS)
kmeans_accumulate_private_kernel(const __half *__restrict__ W, int M, int N, int v, const int *__restrict__ idx,
                                 const float *__restrict__ h, int k, float *__restrict__ sums, float *__restrict__ wsums,
                                 long long n_vectors)
{
    __shared__ float s_sum[KM_SMEM_ENTRIES];
    __shared__ float s_w[KM_SMEM_ENTRIES];            // [k] weight of the whole vectors
    const int entries = k * v;
    for (int e = threadIdx.x; e < entries; e += KM_THREADS) s_sum[e] = 0.f;
    for (int e = threadIdx.x; e < k; e += KM_THREADS) s_w[e] = 0.f;
    __syncthreads();
    for (long long g = (long long)blockIdx.x * KM_THREADS + threadIdx.x; g < n_vectors;
         g += (long long)gridDim.x * KM_THREADS) {
        const int r = (int)(g / N), n = (int)(g % N);
        const int i = __ldg(idx + g);
        if (i < 0 || i >= k) continue;                 // an index outside the table takes no part
        const float w = h != nullptr ? __ldg(h + n) : 1.f;
        const int vlen = min(v, M - r * v);
        for (int j = 0; j < vlen; j++) {
            const float x = __half2float(__ldg(W + (long long)(r * v + j) * N + n));
            atomicAdd(&s_sum[i * v + j], w * x);
            if (vlen < v) atomicAdd(wsums + (long long)i * v + j, w);
        }
        if (vlen == v) atomicAdd(&s_w[i], w);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < entries; e += KM_THREADS)
        if (s_sum[e] != 0.f) atomicAdd(sums + (long long)(e / v) * row_floats(v) + e % v, s_sum[e]);
    for (int e = threadIdx.x; e < k; e += KM_THREADS)
        if (s_w[e] != 0.f) atomicAdd(sums + (long long)e * row_floats(v) + v, s_w[e]);
}

__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

__global__ void __launch_bounds__(KM_THREADS)
kmeans_accumulate_kernel(const __half *__restrict__ W, int M, int N, int v, const int *__restrict__ idx,
                         const float *__restrict__ h, int k, float *__restrict__ sums, float *__restrict__ wsums,
                         long long n_vectors)
{
    const int rf = row_floats(v);
    for (long long g = (long long)blockIdx.x * KM_THREADS + threadIdx.x; g < n_vectors;
         g += (long long)gridDim.x * KM_THREADS) {
        const int r = (int)(g / N), n = (int)(g % N);
        const int i = __ldg(idx + g);
        if (i < 0 || i >= k) continue;                 // an index outside the table takes no part
        const float w = h != nullptr ? __ldg(h + n) : 1.f;
        const int vlen = min(v, M - r * v);
        float *row = sums + (long long)i * rf;
        const __half *col = W + (long long)r * v * N + n;
        for (int j0 = 0; j0 < rf; j0 += 4) {
            float t[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int j = j0 + u;
                t[u] = j < vlen ? w * __half2float(__ldg(col + (long long)j * N)) : (j == v && vlen == v) ? w : 0.f;
            }
            red_add4(row + j0, t[0], t[1], t[2], t[3]);
        }
        if (vlen < v)
            for (int j = 0; j < vlen; j++) atomicAdd(wsums + (long long)i * v + j, w);
    }
}

__global__ void __launch_bounds__(KM_THREADS)
kmeans_finish_kernel(const float *__restrict__ sums, const float *__restrict__ wsums, int v, long long entries,
                     __half *__restrict__ C)
{
    const long long e = (long long)blockIdx.x * KM_THREADS + threadIdx.x;
    if (e >= entries) return;
    const float *row = sums + e / v * row_floats(v);
    const float w = row[v] + wsums[e];
    if (w > 0.f) C[e] = __float2half_rn(__fdiv_rn(row[e % v], w));
}

}  // namespace

long long kmeans_update_workspace_bytes(int v, int k) 
{
    return (long long)k * (row_floats(v) + v) * (long long)sizeof(float) + 16;       // (16: the rows start on a 16-byte boundary)
}

cudaError_t launch_kmeans_update(const __half *W, int M, int N, int v, const int *idx, const float *h, int k,
                                 __half *C, void *ws, cudaStream_t st)
{
    const long long entries = (long long)k * v;
    const long long n_vectors = (long long)ceil_div(M, v) * N;
    float *sums = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(ws) + 15) / 16 * 16);
    float *wsums = sums + (long long)k * row_floats(v);
    cudaError_t e = cudaMemsetAsync(ws, 0, (size_t)kmeans_update_workspace_bytes(v, k), st);
    if (e != cudaSuccess) return e;
    if (n_vectors == 0) return cudaSuccess;
    if (entries <= KM_SMEM_ENTRIES) {
        // a block flushes its copy once: give every block many vectors
        long long blocks = (n_vectors + 16LL * KM_THREADS - 1) / (16LL * KM_THREADS);
        if (blocks > 4096) blocks = 4096;
        kmeans_accumulate_private_kernel<<<(unsigned)blocks, KM_THREADS, 0, st>>>(W, M, N, v, idx, h, k, sums, wsums, n_vectors);
    } else {
        long long blocks = (n_vectors + KM_THREADS - 1) / KM_THREADS;
        if (blocks > 65535LL * 16) blocks = 65535LL * 16;
        kmeans_accumulate_kernel<<<(unsigned)blocks, KM_THREADS, 0, st>>>(W, M, N, v, idx, h, k, sums, wsums, n_vectors);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    kmeans_finish_kernel<<<(unsigned)((entries + KM_THREADS - 1) / KM_THREADS), KM_THREADS, 0, st>>>(sums, wsums, v, entries, C);
    return cudaGetLastError();
}

}  // namespace vptq
