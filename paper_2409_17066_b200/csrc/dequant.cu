// Bit-exact restoration of the FP16 weight matrix from indices and codebooks
// (Sec. 2.2 lookup; Sec. 3.2.2 residual sum; Sec. 3.2.3 outlier columns; App. D.2 "restore
// to FP16").
//
// restore_kernel (v = 6, 8, 12): persistent grid; a warp takes (vector row, 32 x CPL columns) at a time and a lane CPL
// of those columns (8, or 4 for v = 12): it fetches their packed indices as one window of words (the next task's are in
// flight meanwhile), reads all their centroids at once, and writes the v output rows.  CPS columns of a lane are
// adjacent and go out in one store: all CPL of them (16 or 8 bytes) where rows of W start on such a boundary, else two or
// one.  Tasks are cut at multiples of CPL of W's columns, so that outlier columns in front do not misalign the stores.
// Tables that fit shared memory are staged there (SMEM; with group-wise codebooks a CTA works on the columns of one
// group and holds that group's tables), a larger main table stays in L2; a residual table of at most 256 entries has 8
// skewed copies (conflict free).  The three roundings (add, multiply, add) are those of the definition: the residual is
// added by a mixed-precision fma with factor one (f16 x 1 is exact), scale and bias are applied one
// after the other (packed f32x2 multiply and add were contracted to one rounding by the assembler, so they are not used).
// What bounds it: with the 1 MiB table the shared-memory/L1 data pipe (72 % busy: a random 16-byte read out of L2 is
// a wavefront of its own there, 29.4 M of them for 8192 x 28672, and the stores pass through it too), else the writes.
// Measured against one thread per column with 2-byte centroid loads: 8192 x 28672 over the 1 MiB table 684.6 -> 182.8 us,
// 8192 x 8192 over a 256-entry table 147.5 -> 30.8 us (4.6 TB/s), 11008 x 4096 with v = 6 / v = 12 and outlier columns
// 133 -> 43 / 191 -> 50 us.
// dequant_kernel: the same thing one column per thread and one component at a time, for every other vector length and for per-row scale.
#include "common.cuh"
#include "index_words.cuh"

namespace vptq {

namespace {

__device__ __forceinline__ float finish_value(float t, int has_scale, float s, float b)
{
    // separately rounded multiply and add: never contracted to an FMA
    return has_scale ? __fadd_rn(__fmul_rn(t, s), b) : t;
}

constexpr int RS_THREADS = 512, RS_WARPS = RS_THREADS / 32;
constexpr size_t RS_TABLE_BUDGET = 200 * 1024;           // bytes of staged tables per CTA
template <int V> constexpr int restore_cpl() { return V > 8 ? 4 : 8; }      // columns per lane

struct RestoreParams {
    LayerView L;
    __half *W;
    int chunks;            // tasks per vector row (of one group)
    int ctas_per_group;
    int cb2_rep;           // copies of the residual table (1 or 8)
};

// One table row of V values as words; `row` counts rows of STRIDE bytes in shared memory, or of 2V bytes in global memory.
template <int V> struct RowWords { uint32_t w[(V + 1) / 2]; };

template <int V>
__device__ __forceinline__ RowWords<V> row_from_global(const __half *__restrict__ tab, long long e)
{
    RowWords<V> r;
    if (V == 8) {
        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(tab) + e);
        r.w[0] = q.x; r.w[1] = q.y; r.w[2] = q.z; r.w[V / 2 - 1] = q.w;
    } else if (V % 4 == 0) {
        const uint2 *p = reinterpret_cast<const uint2 *>(tab) + e * (V / 4);
#pragma unroll
        for (int i = 0; i < V / 4; i++) { const uint2 q = __ldg(p + i); r.w[2 * i] = q.x; r.w[2 * i + 1] = q.y; }
    } else {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(tab) + e * (V / 2);
#pragma unroll
        for (int i = 0; i < V / 2; i++) r.w[i] = __ldg(p + i);
    }
    return r;
}

// shared-memory rows: V <= 8 as zero-padded 16-byte rows, V = 12 as three 8-byte words
template <int V>
__device__ __forceinline__ RowWords<V> row_from_shared(const uint8_t *tab, uint32_t e)
{
    RowWords<V> r;
    if (V <= 8) {
        const uint4 q = reinterpret_cast<const uint4 *>(tab)[e];
        const uint32_t a[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < V / 2; i++) r.w[i] = a[i];
    } else {
        const uint2 *p = reinterpret_cast<const uint2 *>(tab) + e * (V / 4);
#pragma unroll
        for (int i = 0; i < V / 4; i++) { const uint2 q = p[i]; r.w[2 * i] = q.x; r.w[2 * i + 1] = q.y; }
    }
    return r;
}

template <int V> constexpr int restore_row_bytes() { return V <= 8 ? 16 : 2 * V; }

// dense table [k][V] -> shared-memory rows, `rep` copies of every row next to each other
template <int V>
__device__ __forceinline__ void stage_table(uint8_t *dst, const __half *__restrict__ src, int k, int rep)
{
    if (V <= 8) {
        for (int i = threadIdx.x; i < k * rep; i += RS_THREADS)
            reinterpret_cast<uint4 *>(dst)[i] = load_centroid_row(src, rep == 8 ? i >> 3 : i, V);
    } else {
        // rows of 2V bytes, V a multiple of 4, 16-byte aligned table: copied as it is in 8-byte words
        const uint2 *s = reinterpret_cast<const uint2 *>(src);
        for (int i = threadIdx.x; i < k * (V / 4); i += RS_THREADS) reinterpret_cast<uint2 *>(dst)[i] = __ldg(s + i);
    }
}

// The packed bits of CPL consecutive indices, the first at stream bit `bit`: words beyond the row read as zero.
template <int CPL>
struct IndexWindow { uint32_t w[CPL / 2 + 1]; };
template <int CPL>
__device__ __forceinline__ IndexWindow<CPL> load_window(const uint8_t *__restrict__ row, unsigned bit, unsigned row_words)
{
    IndexWindow<CPL> q;
    const unsigned w0 = bit >> 5;
#pragma unroll
    for (int i = 0; i <= CPL / 2; i++) q.w[i] = w0 + i < row_words ? __ldg(reinterpret_cast<const uint32_t *>(row) + w0 + i) : 0u;
    return q;
}
// ... and index s of it, for widths of 8, 12 and 16 bits (`sh` = bit & 31), clamped to k - 1
template <int CPL>
__device__ __forceinline__ void decode_window(const IndexWindow<CPL> &q, unsigned sh, int bits, int k, int (&idx)[CPL])
{
    const uint32_t lim = (uint32_t)(k - 1);
    uint32_t a[CPL / 2 + 1];
#pragma unroll
    for (int i = 0; i < CPL / 2; i++) a[i] = __funnelshift_r(q.w[i], q.w[i + 1], sh);
    a[CPL / 2] = 0;
    if (bits == 16) {
#pragma unroll
        for (int s = 0; s < CPL; s++) idx[s] = (int)min((s & 1) ? a[s >> 1] >> 16 : a[s >> 1] & 0xFFFFu, lim);
    } else if (bits == 12) {
#pragma unroll
        for (int s = 0; s < CPL; s++)
            idx[s] = (int)min(__funnelshift_r(a[(12 * s) >> 5], a[((12 * s) >> 5) + 1], (12 * s) & 31) & 0xFFFu, lim);
    } else {
#pragma unroll
        for (int s = 0; s < CPL; s++) idx[s] = (int)min((a[s >> 2] >> (8 * (s & 3))) & 0xFFu, lim);
    }
}

// c + (the two halves of w), rounded once: w * 1 is exact
__device__ __forceinline__ float2 add_half2(float2 c, uint32_t w)
{
    asm("{\n\t.reg .b16 lo, hi, one;\n\tmov.b32 {lo, hi}, %2;\n\tmov.b16 one, 0x3C00;\n\t"
        "fma.rn.f32.f16 %0, lo, one, %0;\n\tfma.rn.f32.f16 %1, hi, one, %1;\n\t}" : "+f"(c.x), "+f"(c.y) : "r"(w));
    return c;
}

template <int V, bool RES, bool SMEM, int CPS>
__global__ void __launch_bounds__(RS_THREADS, 1)
restore_kernel(const __grid_constant__ RestoreParams P)
{
    constexpr int CPL = restore_cpl<V>(), RUNS = CPL / CPS;               // columns of a lane, runs of adjacent ones
    extern __shared__ __align__(16) uint8_t smem[];
    const LayerView &L = P.L;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = SMEM ? (int)blockIdx.x / P.ctas_per_group : 0;          // SMEM: the column group of this CTA
    const int rank = SMEM ? (int)blockIdx.x % P.ctas_per_group : (int)blockIdx.x;
    // stored columns [n_first, n_last) are this CTA's main columns; chunk 0 starts at the boundary at or before the first
    const int n_first = L.n_out + (SMEM ? g * L.cpg : 0);
    const int n_last = SMEM ? min(L.N, n_first + L.cpg) : L.N;
    const int n_base = n_first / CPL * CPL;

    constexpr int RB = restore_row_bytes<V>();
    uint8_t *t1 = smem, *t2 = SMEM ? smem + (size_t)L.k1 * RB : smem;
    if (SMEM) stage_table<V>(t1, L.c1 + (long long)g * L.k1 * V, L.k1, 1);
    const bool res_shared = RES && (SMEM || P.cb2_rep == 8);
    if (res_shared) stage_table<V>(t2, L.c2 + (long long)g * L.k2 * V, L.k2, P.cb2_rep);
    const uint32_t rep = P.cb2_rep == 8 ? (uint32_t)(lane & 7) : 0u;
    const int rshift = P.cb2_rep == 8 ? 3 : 0;
    __syncthreads();

    // tasks (row, chunk), chunk fastest, dealt out to the warps of the CTAs that share the columns
    const int step = P.ctas_per_group * RS_WARPS;
    const int step_r = step / P.chunks, step_c = step % P.chunks;
    const int first = rank * RS_WARPS + warp;
    int r = first / P.chunks, ch = first % P.chunks;
    const unsigned words1 = (unsigned)(L.s1.stride >> 2), words2 = RES ? (unsigned)(L.s2.stride >> 2) : 0u;
    const int b1 = L.s1.bits, b2 = RES ? L.s2.bits : 8;
    const bool windows = CPS == CPL && (b1 == 8 || b1 == 12 || b1 == 16) && (b2 == 8 || b2 == 12 || b2 == 16);
    // (a window may start before main column 0: it is then moved there and the lane decodes index by index)
    auto window_bit = [&](int chunk, int bits) { return (unsigned)max(0, n_base + (chunk * 32 + lane) * CPL - L.n_out) * (unsigned)bits; };
    IndexWindow<CPL> q1, q2;
    if (windows && r < L.R) {
        q1 = load_window<CPL>(L.s1.ptr + (long long)r * L.s1.stride, window_bit(ch, b1), words1);
        if (RES) q2 = load_window<CPL>(L.s2.ptr + (long long)r * L.s2.stride, window_bit(ch, b2), words2);
    }
    while (r < L.R) {
        const int n0 = n_base + ch * 32 * CPL + lane * CPS;               // this lane's first column; run u starts u * 32 * CPS further
        auto column = [&](int s) { return n0 + (s / CPS) * 32 * CPS + s % CPS; };
        const uint8_t *row1 = L.s1.ptr + (long long)r * L.s1.stride;
        const uint8_t *row2 = RES ? L.s2.ptr + (long long)r * L.s2.stride : nullptr;
        int i1[CPL], i2[CPL];
        if (windows && n0 >= L.n_out) {
            decode_window<CPL>(q1, window_bit(ch, b1) & 31u, b1, L.k1, i1);
            if (RES) decode_window<CPL>(q2, window_bit(ch, b2) & 31u, b2, L.k2, i2);
        } else {
#pragma unroll
            for (int s = 0; s < CPL; s++) {
                const int c = min(max(column(s), n_first), n_last - 1) - L.n_out;
                i1[s] = clamp_index(load_index(row1, c, b1), L.k1);
                if (RES) i2[s] = clamp_index(load_index(row2, c, b2), L.k2);
            }
        }
        const int m0 = r * V;
        // next task, and its packed words
        r += step_r; ch += step_c;
        if (ch >= P.chunks) { ch -= P.chunks; r++; }
        if (windows && r < L.R) {
            q1 = load_window<CPL>(L.s1.ptr + (long long)r * L.s1.stride, window_bit(ch, b1), words1);
            if (RES) q2 = load_window<CPL>(L.s2.ptr + (long long)r * L.s2.stride, window_bit(ch, b2), words2);
        }
        RowWords<V> w1[CPL], w2[CPL];
        // scale and bias of the columns; without them t * 1 + (-0) = t, whatever t and its sign
        float sc[CPL], bi[CPL];
#pragma unroll
        for (int s = 0; s < CPL; s++) {
            const int n = min(max(column(s), n_first), n_last - 1);
            const int gg = SMEM || L.G == 1 ? 0 : (n - L.n_out) / L.cpg;
            w1[s] = SMEM ? row_from_shared<V>(t1, (uint32_t)i1[s]) : row_from_global<V>(L.c1, (long long)gg * L.k1 + i1[s]);
            if (RES) w2[s] = res_shared ? row_from_shared<V>(t2, ((uint32_t)i2[s] << rshift) + rep)
                                        : row_from_global<V>(L.c2, (long long)gg * L.k2 + i2[s]);
            sc[s] = 1.f; bi[s] = -0.f;
        }
        if (L.has_scale) {
            if (CPS == CPL && n0 + CPL <= L.N) {
                // CPL adjacent columns from a multiple of CPL on: one load
                uint32_t q[2][CPL / 2];
                const __half *src[2] = {L.scale + n0, L.bias + n0};
#pragma unroll
                for (int d = 0; d < 2; d++) {
                    if (CPL == 8) *reinterpret_cast<uint4 *>(q[d]) = __ldg(reinterpret_cast<const uint4 *>(src[d]));
                    else *reinterpret_cast<uint2 *>(q[d]) = __ldg(reinterpret_cast<const uint2 *>(src[d]));
                }
#pragma unroll
                for (int s = 0; s < CPL; s += 2) {
                    const float2 fs = __half22float2(*reinterpret_cast<const __half2 *>(&q[0][s / 2]));
                    const float2 fb = __half22float2(*reinterpret_cast<const __half2 *>(&q[1][s / 2]));
                    sc[s] = fs.x; sc[s + 1] = fs.y; bi[s] = fb.x; bi[s + 1] = fb.y;
                }
            } else {
#pragma unroll
                for (int s = 0; s < CPL; s++) {
                    const int n = min(max(column(s), n_first), n_last - 1);
                    sc[s] = __half2float(__ldg(L.scale + n)); bi[s] = __half2float(__ldg(L.bias + n));
                }
            }
        }
        __half *dst = P.W + (long long)m0 * L.N;
#pragma unroll
        for (int i = 0; i < V / 2; i++) {
            float2 y[CPL];                                                 // components 2i, 2i + 1 of the lane's columns
#pragma unroll
            for (int s = 0; s < CPL; s++) {
                y[s] = __half22float2(*reinterpret_cast<const __half2 *>(&w1[s].w[i]));
                if (RES) y[s] = add_half2(y[s], w2[s].w[i]);
                y[s].x = __fadd_rn(__fmul_rn(y[s].x, sc[s]), bi[s]);
                y[s].y = __fadd_rn(__fmul_rn(y[s].y, sc[s]), bi[s]);
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                if (m0 + 2 * i + h < L.M) {                                // components of a partial last row beyond M are dropped
#pragma unroll
                    for (int u = 0; u < RUNS; u++) {
                        const int n = column(u * CPS);
                        __half2 o[(CPS + 1) / 2];
#pragma unroll
                        for (int t = 0; t < CPS; t += 2) {
                            const float2 &ya = y[u * CPS + t], &yb = y[u * CPS + (CPS > 1 ? t + 1 : t)];
                            o[t / 2] = __floats2half2_rn(h ? ya.y : ya.x, h ? yb.y : yb.x);
                        }
                        if (CPS > 1 && n >= n_first && n + CPS <= n_last) {
                            if (CPS == 8) *reinterpret_cast<uint4 *>(dst + n) = *reinterpret_cast<const uint4 *>(o);
                            else if (CPS == 4) *reinterpret_cast<uint2 *>(dst + n) = *reinterpret_cast<const uint2 *>(o);
                            else *reinterpret_cast<__half2 *>(dst + n) = o[0];
                        } else {
#pragma unroll
                            for (int t = 0; t < CPS; t++)
                                if (n + t >= n_first && n + t < n_last)
                                    dst[CPS == 1 ? in_col(L, n + t) : n + t] = (t & 1) ? __high2half(o[t / 2]) : __low2half(o[t / 2]);
                        }
                    }
                }
                dst += L.N;
            }
        }
    }

    // the outlier columns, shared out over the whole grid: one (outlier row, column) per thread
    const long long n_items = (long long)L.R0 * L.n_out;
    for (long long i = (long long)blockIdx.x * RS_THREADS + threadIdx.x; i < n_items; i += (long long)gridDim.x * RS_THREADS) {
        const int q = (int)(i / L.n_out), n = (int)(i % L.n_out);
        const int i0 = clamp_index(load_index(L.s0.ptr + (long long)q * L.s0.stride, n, L.s0.bits), L.k0);
        const __half *e = L.c0 + (long long)i0 * L.v0;
        float sc = 1.f, bi = 0.f;
        if (L.has_scale) { sc = __half2float(__ldg(L.scale + n)); bi = __half2float(__ldg(L.bias + n)); }
        const int f = in_col(L, n);
        for (int j = 0; j < L.v0 && q * L.v0 + j < L.M; j++) {
            const int m = q * L.v0 + j;
            P.W[(long long)m * L.N + f] = __float2half_rn(finish_value(__half2float(__ldg(e + j)), L.has_scale, sc, bi));
        }
    }
}

__global__ void __launch_bounds__(256)
dequant_kernel(LayerView L, __half *__restrict__ W)
{
    // blockIdx.y selects the region: 0 = main columns, 1 = outlier columns
    const bool outlier = (blockIdx.y == 1);
    const int cols = outlier ? L.n_out : L.Nc;
    const int vrows = outlier ? L.R0 : L.R;
    const int vlen = outlier ? L.v0 : L.v;
    long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)vrows * cols) return;
    const int r = (int)(gid / cols);
    const int c = (int)(gid % cols);
    const int n = outlier ? c : c + L.n_out;

    const __half *e1, *e2 = nullptr;
    if (outlier) {
        int i0 = clamp_index(load_index(L.s0.ptr + (long long)r * L.s0.stride, c, L.s0.bits), L.k0);
        e1 = L.c0 + (long long)i0 * vlen;
    } else {
        int i1 = clamp_index(load_index(L.s1.ptr + (long long)r * L.s1.stride, c, L.s1.bits), L.k1);
        const int g = c / L.cpg;                       // Sec. 3.1: this column's group has its own tables
        e1 = L.c1 + ((long long)g * L.k1 + i1) * vlen;
        if (L.k2 > 0) {
            int i2 = clamp_index(load_index(L.s2.ptr + (long long)r * L.s2.stride, c, L.s2.bits), L.k2);
            e2 = L.c2 + ((long long)g * L.k2 + i2) * vlen;
        }
    }
    float s = 1.f, b = 0.f;
    if (L.has_scale && !L.scale_rows) {
        s = __half2float(__ldg(L.scale + n));
        b = __half2float(__ldg(L.bias + n));
    }
    const int m0 = r * vlen;
    for (int j = 0; j < vlen; j++) {
        int m = m0 + j;
        if (m >= L.M) break;              // last vector row may be partial: extra components are dropped
        float t = __half2float(__ldg(e1 + j));
        if (e2 != nullptr) t = __fadd_rn(t, __half2float(__ldg(e2 + j)));
        if (L.has_scale && L.scale_rows) {
            s = __half2float(__ldg(L.scale + m));
            b = __half2float(__ldg(L.bias + m));
        }
        W[(long long)m * L.N + in_col(L, n)] = __float2half_rn(finish_value(t, L.has_scale, s, b));
    }
}

template <int V, bool RES, bool SMEM>
cudaError_t launch_restore(const RestoreParams &P, size_t smem, int cps, int grid, cudaStream_t st)
{
    constexpr int CPL = restore_cpl<V>();
    auto kern = cps == CPL ? restore_kernel<V, RES, SMEM, CPL> : cps == 2 ? restore_kernel<V, RES, SMEM, 2> : restore_kernel<V, RES, SMEM, 1>;
    const cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void *>(kern), smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, RS_THREADS, smem, st>>>(P);
    return cudaGetLastError();
}

template <int V>
cudaError_t restore(const LayerView &L, __half *W, cudaStream_t st)
{
    constexpr int CPL = restore_cpl<V>();
    RestoreParams P;
    P.L = L; P.W = W;
    const bool res = L.k2 > 0;
    const int G = device_sm_count();
    const int per_group = G / L.G > 0 ? G / L.G : 1;
    // staging a group's tables pays when a CTA reads more rows out of them than they have
    const size_t b1 = (size_t)L.k1 * restore_row_bytes<V>();
    const size_t b2 = res ? (size_t)L.k2 * restore_row_bytes<V>() : 0, rep2 = (V <= 8 && res && L.k2 <= 256) ? 8 : 1;
    const bool smem = b1 + b2 * rep2 <= RS_TABLE_BUDGET && (long long)L.R * L.cpg / per_group > (long long)L.k1 + L.k2;
    P.cb2_rep = (smem || L.G == 1) ? (int)rep2 : 1;
    // columns per store: what the alignment of W's rows allows; a stored column order scatters single columns
    const int cps = (L.perm == nullptr && L.N % CPL == 0) ? CPL : (L.perm == nullptr && L.N % 2 == 0) ? 2 : 1;
    // a chunk may start up to CPL - 1 columns before the CTA's first one
    P.chunks = ceil_div((smem ? L.cpg : L.Nc) + CPL - 1, 32 * CPL);
    int grid;
    size_t bytes;
    if (smem) {
        P.ctas_per_group = per_group;
        grid = P.ctas_per_group * L.G;
        bytes = b1 + b2 * rep2;
    } else {
        const long long most = ((long long)L.R * P.chunks + RS_WARPS - 1) / RS_WARPS;
        P.ctas_per_group = grid = most < G ? (int)most : G;
        bytes = P.cb2_rep == 8 ? b2 * 8 : 0;
    }
    if (smem) return res ? launch_restore<V, true, true>(P, bytes, cps, grid, st) : launch_restore<V, false, true>(P, bytes, cps, grid, st);
    return res ? launch_restore<V, true, false>(P, bytes, cps, grid, st) : launch_restore<V, false, false>(P, bytes, cps, grid, st);
}

}  // namespace

cudaError_t launch_dequant(const LayerView &L, __half *W, cudaStream_t st)
{
    if (L.Nc > 0 && !L.scale_rows) {
        if (L.v == 8) return restore<8>(L, W, st);
        if (L.v == 6) return restore<6>(L, W, st);
        if (L.v == 12) return restore<12>(L, W, st);
    }
    long long main_items = (long long)L.R * L.Nc;
    long long out_items = (long long)L.R0 * L.n_out;
    long long most = main_items > out_items ? main_items : out_items;
    if (most == 0) return cudaSuccess;
    dim3 grid((unsigned)((most + 255) / 256), L.n_out > 0 ? 2 : 1);
    dequant_kernel<<<grid, 256, 0, st>>>(L, W);
    return cudaGetLastError();
}

}  // namespace vptq
