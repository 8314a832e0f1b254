// Which kernel family runs a given (layer, batch), and the scratch it needs.
#include "paths.cuh"
#include "decode.cuh"
#include "gemm.cuh"
#include "prepared.cuh"
#include "fused_split.cuh"

namespace vptq {

namespace {
constexpr int DECODE_MAX_B = 16;
int decode_group(int B) { return B < DECODE_MAX_B ? B : DECODE_MAX_B; }
}

LinearPath choose_path(const LayerView &L, int B, int flags)
{
    if (flags & VPTQ_FLAG_FORCE_GENERIC) return PATH_GENERIC;
    if (L.deterministic) {
        // fixed summation order: the batched path with whole tiles, the L2 decode kernel in row-owner mode with
        // ordered warp partial sums, else the plain kernel (one warp per output row)
        if (B > DECODE_MAX_B && gemm_tcgen05_supported(L, B)) return PATH_GEMM_TCGEN05;
        if (l2_fma_supported(L, decode_group(B)) && l2_fma_deterministic_ok(L, decode_group(B))) return PATH_DECODE_L2_FMA;
        return PATH_GENERIC;
    }
    if (L.prep_parts > 0 && bucket_fma_supported(L, B) && L.prep_parts <= device_sm_count() &&
        ceil_div(L.R, L.prep_parts / prepared_split(L.R, ceil_div(L.k1, PREP_BUCKET), L.prep_parts)) <= PREP_MAX_ROWS)
        return PATH_DECODE_BUCKET_FMA;
    if (B > DECODE_MAX_B && gemm_tcgen05_supported(L, B)) return PATH_GEMM_TCGEN05;
    const int Bg = decode_group(B);
    if (smem_fma_supported(L, Bg)) return PATH_DECODE_SMEM_FMA;
    if (smem_mma_supported(L, Bg)) return PATH_DECODE_SMEM_MMA;
    if (l2_fma_supported(L, Bg)) return PATH_DECODE_L2_FMA;
    if (gl_fma_supported(L, Bg)) return PATH_DECODE_GL_FMA;
    return PATH_GENERIC;
}

// Whether a call of this family runs in the batched kernel.  The families whose main tables are in L2 or group-wise take at
// most four or two tokens per launch and gather every centroid again for the next ones; the batched kernel gathers it once
// whatever the batch.  4096 x 4096 over the 1 MiB table: 25 us
// at any batch up to 64, against 14-17 us per four tokens; 11008 x 4096, v = 12 in four groups: 52 us against 31 us per two.
//
// Of the family of tables in shared memory it takes, with outlier vectors of 4 or none, the calls whose tables, copies of a small
// main one among them, leave no room for all activations at once (smem_tc_tight), and of these
//   up to 8 tokens    v < 8 with a residual table and outlier columns and at most half as many rows as columns;
//   9 to 16 tokens    up to 2048 rows; v < 8 with a residual table: with outlier columns any, without them up to twice as many
//                     rows as columns where the decode kernel takes more than one slab.
// The decode kernel stages the activations slab by slab, which nothing overlaps, and reads outlier columns one after the other; the
// batched one has a set-up to pay and reads a centroid per 128 rows whatever the batch.  Both in us, decode / batched:
//   v = 6, residual, outliers, 16 tokens   4096 x 4096 27.6 / 23.1, 11008 x 4096 45.0 / 41.0, 4096 x 11008 56.6 / 40.7
//   ... 8 tokens                           2048 x 8192 27.0 / 22.7, 4096 x 11008 43.8 / 40.2; one slab, 4096 x 4096: 21.3 / 22.7
//   v = 6, residual, 16 tokens             11008 x 4096 40.4 / 39.2, 12 tokens 2048 x 6144 24.3 / 21.8; one slab, 4096 x 6400 (512 centroids): 34.7 / 35.7
//   ... 8 tokens                           4096 x 11008 36.8 / 38.1
//   v = 8, 256 centroids, 16 tokens        2048 x 8192 18.6 / 16.5, 2048 x 6600 16.2 / 15.0, 1024 x 6600 14.5 / 12.2; 4096 x 11008 26.7 / 29.3
static bool smem_takes_batched(const LayerView &L, int B)
{
    const int Bg = decode_group(B);
    if (!smem_tc_supported(L, Bg) || (L.n_out > 0 && L.v0 != 4) || !smem_tc_tight(L, Bg)) return false;
    const bool gathers = L.v < 8 && L.k2 > 0;
    if (Bg <= 8) return gathers && L.n_out > 0 && 2 * L.M <= L.N;
    return L.M <= 2048 || (gathers && (L.n_out > 0 || (L.M <= 2 * L.N && smem_tc_slabs(L, Bg) > 1)));
}

// The layer as the batched kernel takes it.  A call of one layer of the family of tables in shared memory has never had CTAs that wait
// for one another, so it may share the GPU without saying so (launches that several layers share may wait: linear_fused_waits_between_ctas).
static LayerView batched_view(LinearPath path, const LayerView &L)
{
    LayerView v = L;
    if (path == PATH_DECODE_SMEM_MMA) v.concurrent = true;
    return v;
}

static bool takes_batched(LinearPath path, const LayerView &L, int B)
{
    if (path == PATH_GEMM_TCGEN05) return true;
    if (path == PATH_DECODE_SMEM_MMA) return !L.deterministic && smem_takes_batched(L, B) && gemm_tcgen05_supported(L, B);
    return ((path == PATH_DECODE_L2_FMA && B >= 5) || (path == PATH_DECODE_GL_FMA && B >= 3)) && !L.deterministic && gemm_tcgen05_supported(L, B);
}

// (answers for the kernel that runs, whatever the family is called)
bool linear_waits_between_ctas(const LayerView &L, int B, int flags)
{
    const LinearPath path = choose_path(L, B, flags);
    const LayerView view = batched_view(path, L);
    return takes_batched(path, L, B) && gemm_tcgen05_waits_between_ctas(&view, 1, B);
}

bool linear_has_status(const LayerView &L, int B, int flags)
{
    const LinearPath path = choose_path(L, B, flags);
    return path == PATH_DECODE_BUCKET_FMA || takes_batched(path, L, B);
}

const char *linear_path_name(const LayerView &L, int B, int flags)
{
    switch (choose_path(L, B, flags)) {
    case PATH_DECODE_SMEM_FMA: return "decode_smem_fma";
    case PATH_DECODE_SMEM_MMA: return "decode_smem_mma";
    case PATH_DECODE_L2_FMA: return "decode_l2_fma";
    case PATH_DECODE_GL_FMA: return "decode_gl_fma";
    case PATH_GEMM_TCGEN05: return "gemm_tcgen05";
    case PATH_DECODE_BUCKET_FMA: return "decode_bucket_fma";
    default: return "generic";
    }
}

long long linear_workspace_bytes(const LayerView &L, int B, int flags)
{
    const LinearPath path = choose_path(L, B, flags);
    if (takes_batched(path, L, B)) {
        const LayerView view = batched_view(path, L);
        return gemm_tcgen05_workspace_bytes(&view, 1, B);
    }
    switch (path) {
    case PATH_DECODE_SMEM_FMA: return 0;
    case PATH_DECODE_SMEM_MMA: return smem_mma_workspace_bytes(L, decode_group(B));
    case PATH_DECODE_L2_FMA: return l2_fma_workspace_bytes(L, decode_group(B));
    case PATH_DECODE_GL_FMA: return 0;
    case PATH_DECODE_BUCKET_FMA: return (long long)bucket_fma_workspace_bytes(&L, &L.prep_parts, 1);
    default: return generic_workspace_bytes(L, B);
    }
}

int linear_launches(const LayerView &L, int B, int flags)
{
    const int groups = ceil_div(B, DECODE_MAX_B);
    const int last = B - (groups - 1) * DECODE_MAX_B;
    const LinearPath path = choose_path(L, B, flags);
    if (takes_batched(path, L, B)) return gemm_tcgen05_launches(L, B);
    switch (path) {
    case PATH_DECODE_SMEM_FMA:
        return (groups - 1) * smem_fma_launches(L, DECODE_MAX_B) + smem_fma_launches(L, last);
    case PATH_DECODE_SMEM_MMA: return groups * (smem_tc_supported(L, decode_group(B)) ? 2 : 1);      // pre-pass + main kernel
    case PATH_DECODE_BUCKET_FMA: return 1;
    case PATH_DECODE_L2_FMA:
        return (groups - 1) * l2_fma_launches(L, DECODE_MAX_B) + l2_fma_launches(L, last);
    case PATH_DECODE_GL_FMA:
        return (groups - 1) * gl_fma_launches(L, DECODE_MAX_B) + gl_fma_launches(L, last);
    default: return generic_launches(L, B);
    }
}

int linear_dispatch(const LayerView &L, int flags, const void *x, int B, void *out, void *ws,
                    cudaStream_t st, cudaError_t *cuda_err)
{
    cudaError_t e = cudaSuccess;
    const LinearPath path = choose_path(L, B, flags);
    if (path == PATH_GENERIC) {
        e = launch_linear_generic(L, x, B, out, ws, st);
    } else if (takes_batched(path, L, B)) {
        const LayerView view = batched_view(path, L);
        e = launch_gemm_tcgen05(&view, 1, x, B, &out, ws, st);
    } else if (path == PATH_DECODE_BUCKET_FMA) {
        const void *img = L.prepared;
        void *o = out;
        e = launch_decode_bucket_fma(&L, &img, &L.prep_parts, 1, x, &o, ws, debug_wait_limit(), st);
    } else {
        // decode kernels take up to 16 tokens per launch
        const size_t oe = (L.out_dtype == VPTQ_DTYPE_FP32) ? 4 : 2;
        for (int t0 = 0; t0 < B && e == cudaSuccess; t0 += DECODE_MAX_B) {
            const int Bg = (B - t0 < DECODE_MAX_B) ? (B - t0) : DECODE_MAX_B;
            const void *xg = reinterpret_cast<const uint8_t *>(x) + (size_t)t0 * L.N * 2;
            void *og = reinterpret_cast<uint8_t *>(out) + (size_t)t0 * L.M * oe;
            if (path == PATH_DECODE_SMEM_FMA) e = launch_decode_smem_fma(L, xg, Bg, og, st);
            else if (path == PATH_DECODE_SMEM_MMA) e = launch_decode_smem_mma(L, xg, Bg, og, ws, st);
            else if (path == PATH_DECODE_GL_FMA) e = launch_decode_gl_fma(L, xg, Bg, og, st);
            else e = launch_decode_l2_fma(L, xg, Bg, og, ws, st);
        }
    }
    *cuda_err = e;
    return e == cudaSuccess ? VPTQ_OK : VPTQ_E_CUDA;
}

// ---- several layers that read the same activations ---------------------------------------------------

// Whether layers whose own calls would take `path` are better off in one launch of the batched kernel, which costs one
// set-up for all of them: a 7B layer's q+k+v+o (1024 rows of k and v) at 16 tokens takes 50 us instead of 76 over the 1 MiB
// table, 70 instead of 100 with v = 12 in four groups.  From 17 to 64 tokens large layers, which fill the SMs on their own, keep sharing
// one layer's scratch.
// Tables in shared memory have a decode kernel that takes a weight in a little over half of the time (v = 8 over eight copies of a
// table: in half), after 8 us a layer (13 past 8 tokens, 4 more beside a residual table): shared up to 2^25 weights for each layer but one,
// twice as many past 8 tokens, twice as many with a residual table, 5/8 of all that for v = 8 with up to 256 centroids.  One by one /
// shared, us (* what is taken; of 192 calls of 5 to 16 tokens 189 are within 5 % of the better one):
//                                                     q+k+v, 4096 + 2 x 1024 rows x 4096   2 x 11008 x 4096   2 x 8192 x 3072
//   v = 6, 4096 + 256 centroids, outliers, 8 tokens   53.7 / 29.2*                         69.0* / 66.4       48.5 / 45.7*
//   ... 16 tokens                                     52.0 / 29.8*                         81.4 / 66.7*       60.5 / 46.4*
//   v = 8, 4096 centroids, 8 tokens                   33.0 / 21.6*                         41.5* / 49.5       29.7* / 33.8
//   ... 16 tokens                                     38.3 / 21.8*                         50.3* / 49.9       37.4 / 34.0*
//   v = 8, 256 centroids, 8 tokens                    30.1 / 20.5*                         31.6* / 48.3       24.1* / 32.5
//   ... 16 tokens                                     34.3 / 20.5*                         39.4* / 48.6       30.9* / 32.7
//   v = 8, 256 + 256 centroids, 8 tokens              35.2 / 22.8*                         43.0* / 52.4       31.2* / 35.3
static bool fused_batched(LinearPath path, const LayerView *Ls, int n, int B)
{
    long long weights = 0;
    for (int l = 0; l < n; l++) weights += (long long)Ls[l].M * Ls[l].N;
    if (path == PATH_DECODE_SMEM_MMA) {
        const int eighths = Ls[0].v == 8 && Ls[0].k1 <= 256 ? 5 : 8;
        return 8 * weights <= eighths * ((n - 1LL) << (25 + (B > 8) + (Ls[0].k2 > 0)));
    }
    return path != PATH_GEMM_TCGEN05 || B > 64 || weights <= ((n - 1LL) << 26);
}

// The kernel family that serves all n layers with one launch per token group, or PATH_GENERIC when there is none.
LinearPath fused_path(const LayerView *Ls, const int *flags, int n, int B)
{
    if (n < 2) return PATH_GENERIC;
    for (int l = 0; l < n; l++)
        if (Ls[l].deterministic) return PATH_GENERIC;          // one layer after the other
    const LinearPath path = choose_path(Ls[0], B, flags[0]);
    for (int l = 1; l < n; l++)
        if (choose_path(Ls[l], B, flags[l]) != path) return PATH_GENERIC;
    if (takes_batched(path, Ls[0], B) || path == PATH_DECODE_SMEM_MMA) {
        if (fused_batched(path, Ls, n, B) && gemm_tcgen05_fused_supported(Ls, n, B)) return PATH_GEMM_TCGEN05;
        if (path != PATH_DECODE_L2_FMA || B > 8) return PATH_GENERIC;
    }
    if (B > DECODE_MAX_B) return PATH_GENERIC;
    if (path == PATH_DECODE_BUCKET_FMA) {
        // prepared layers share a launch when their partitions fit the SMs side by side
        int ctas = 0;
        for (int l = 0; l < n; l++) {
            if (Ls[l].N != Ls[0].N || Ls[l].x_bf16 != Ls[0].x_bf16 || (Ls[l].k2 > 0) != (Ls[0].k2 > 0)) return PATH_GENERIC;
            ctas += Ls[l].prep_parts;
        }
        return (n <= MAX_FUSED && ctas <= device_sm_count()) ? path : PATH_GENERIC;
    }
    if (path == PATH_DECODE_L2_FMA && l2_fma_fused_supported(Ls, n, B)) return path;
    if (path == PATH_DECODE_SMEM_FMA && smem_fma_fused_supported(Ls, n, B)) return path;
    if (path == PATH_DECODE_GL_FMA && gl_fma_fused_supported(Ls, n, B)) return path;
    return PATH_GENERIC;
}

const char *linear_fused_path_name(const LayerView *Ls, const int *flags, int n, int B)
{
    const LinearPath path = fused_path(Ls, flags, n, B);
    // (a family's name, as in linear_path_name: up to 8 tokens over a table in L2 the decode family's, whichever kernel takes them;
    // linear_fused_has_status and linear_fused_waits_between_ctas answer for the kernel)
    if (path == PATH_GEMM_TCGEN05 && B <= 8 && choose_path(Ls[0], B, flags[0]) == PATH_DECODE_L2_FMA) return "fused_decode_l2_fma";
    switch (path) {
    case PATH_DECODE_L2_FMA: return "fused_decode_l2_fma";
    case PATH_DECODE_SMEM_FMA: return "fused_decode_smem_fma";
    case PATH_DECODE_GL_FMA: return "fused_decode_gl_fma";
    case PATH_DECODE_BUCKET_FMA: return "fused_decode_bucket_fma";
    case PATH_GEMM_TCGEN05: return "fused_gemm_tcgen05";
    default: return "one_by_one";
    }
}

bool linear_fused_waits_between_ctas(const LayerView *Ls, const int *flags, int n, int B)
{
    const LinearPath path = fused_path(Ls, flags, n, B);
    if (path == PATH_GEMM_TCGEN05) return gemm_tcgen05_waits_between_ctas(Ls, n, B);
    if (path != PATH_GENERIC) return false;
    for (int l = 0; l < n; l++)
        if (linear_waits_between_ctas(Ls[l], B, flags[l])) return true;
    return false;
}

// (one layer after the other: the word, if any, is the last layer's)
bool linear_fused_has_status(const LayerView *Ls, const int *flags, int n, int B)
{
    const LinearPath path = fused_path(Ls, flags, n, B);
    if (path == PATH_GENERIC) return linear_has_status(Ls[n - 1], B, flags[n - 1]);
    return path == PATH_GEMM_TCGEN05 || path == PATH_DECODE_BUCKET_FMA;
}

long long linear_fused_workspace_bytes(const LayerView *Ls, const int *flags, int n, int B)
{
    const LinearPath fp = fused_path(Ls, flags, n, B);
    if (fp == PATH_DECODE_BUCKET_FMA) {
        int parts[MAX_FUSED];
        for (int l = 0; l < n; l++) parts[l] = Ls[l].prep_parts;
        return (long long)bucket_fma_workspace_bytes(Ls, parts, n);
    }
    if (fp == PATH_GEMM_TCGEN05) return gemm_tcgen05_workspace_bytes(Ls, n, B);
    if (fp != PATH_GENERIC) return 0;
    long long need = 0;       // one layer after the other on the stream: they share the scratch
    for (int l = 0; l < n; l++) {
        const long long w = linear_workspace_bytes(Ls[l], B, flags[l]);
        if (w > need) need = w;
    }
    return need;
}

int linear_fused_launches(const LayerView *Ls, const int *flags, int n, int B)
{
    const LinearPath path = fused_path(Ls, flags, n, B);
    if (path == PATH_DECODE_L2_FMA) return l2_fma_fused_launches(B);
    if (path == PATH_DECODE_SMEM_FMA) return smem_fma_launches(Ls[0], B);      // one launch per token group
    if (path == PATH_DECODE_GL_FMA) return gl_fma_launches(Ls[0], B);
    if (path == PATH_DECODE_BUCKET_FMA) return 1;
    if (path == PATH_GEMM_TCGEN05) return gemm_tcgen05_launches(Ls[0], B);
    int total = 0;
    for (int l = 0; l < n; l++) total += linear_launches(Ls[l], B, flags[l]);
    return total;
}

int linear_fused_dispatch(const LayerView *Ls, const int *flags, int n, const void *x, int B, void *const *outs,
                          void *ws, cudaStream_t st, cudaError_t *cuda_err)
{
    const LinearPath path = fused_path(Ls, flags, n, B);
    if (path != PATH_GENERIC) {
        if (path == PATH_GEMM_TCGEN05) *cuda_err = launch_gemm_tcgen05(Ls, n, x, B, outs, ws, st);
        else if (path == PATH_DECODE_L2_FMA) *cuda_err = launch_decode_l2_fma_fused(Ls, n, x, B, outs, st);
        else if (path == PATH_DECODE_BUCKET_FMA) {
            const void *imgs[MAX_FUSED];
            int parts[MAX_FUSED];
            for (int l = 0; l < n; l++) { imgs[l] = Ls[l].prepared; parts[l] = Ls[l].prep_parts; }
            *cuda_err = launch_decode_bucket_fma(Ls, imgs, parts, n, x, outs, ws, debug_wait_limit(), st);
        }
        else if (path == PATH_DECODE_SMEM_FMA) *cuda_err = launch_decode_smem_fma_fused(Ls, n, x, B, outs, st);
        else *cuda_err = launch_decode_gl_fma_fused(Ls, n, x, B, outs, st);
        return *cuda_err == cudaSuccess ? VPTQ_OK : VPTQ_E_CUDA;
    }
    for (int l = 0; l < n; l++) {
        const int rc = linear_dispatch(Ls[l], flags[l], x, B, outs[l], ws, st, cuda_err);
        if (rc != VPTQ_OK) return rc;
    }
    return VPTQ_OK;
}

}  // namespace vptq
