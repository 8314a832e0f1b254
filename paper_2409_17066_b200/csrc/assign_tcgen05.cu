// Assignment step of the quantizer (Eq. 2) on the tensor cores, with the result of the FP32 definition.
//
// The squared distance ||x||^2 + ||c||^2 - 2 x.c is a contraction over the vector's components: D[vector][centroid] = A * B^T
//   A row (a vector):   x_0 .. x_{v-1}, 0 .., xn, 1, 2^-11           (16 FP16 values, K = 16)
//   B row (a centroid): -2c_0 .. -2c_{v-1}, 0 .., 1, hi, 2^11 lo     hi + lo = ||c||^2 split into two FP16 values
// (v = 14 has no column for lo).  xn = ||x||^2 plus a little, rounded up to FP16: the same for all centroids of a vector, so
// its rounding changes no comparison, and D stays positive.  x and c are first multiplied by a power of two 2^s that brings
// max ||c||^2 to about 2^8: FP16 keeps its 11 bits only for normal numbers, and small weights (1e-4) and their squared norms
// are far below them.  The scaling is exact for values that stay in range and leaves the order of the distances unchanged.
// One tcgen05.mma (M = 128 vectors, N = 128 centroids, K = 16) gives 16 K approximate distances, rounded once to FP16.
// They only FILTER: per vector the kernel keeps a list of the groups of 32 centroids whose minimum lay within the filter's error
// of the smallest one so far.  Those that still do at the end are evaluated with the arithmetic that defines
// the result (FP32 fma chain, lowest index wins: the same code as the plain kernel); a vector with more such groups than
// the list holds (ties), or one that leaves the FP16 range, is put on a list, and a second kernel scans all centroids for the vectors
// on the list.  The indices are therefore those of the FP32 definition, bit for bit, whatever the tensor core's summation
// order.
//   bound: before its rounding (2^-11 of the value) a filter value is off by at most E = 2^-18 (||x||^2 + max ||c||^2) (FP16
//   split of the norm, FP32 accumulation of 16 products, rounding of the fma chain; 2^-12 max ||c||^2 more without lo).  A
//   group is out when its minimum is above b (1 + 2^-10) + 2E with b the smallest; tested with half an FP16 step more and 4E.
//
// Persistent grid, one CTA per SM, 256 vectors (two A tiles) per step.  Warp 0 streams the prepared centroid tiles (8 KB for
// 256 centroids, shared-memory image with the 32-byte swizzle applied by the preparation kernel) with linear bulk copies into a
// ring; warps 0-3 issue the MMAs, each of one A tile and one half of every stage into a TMEM buffer of its own; warps 4-19 own
// a TMEM lane quarter of one A tile and one half each: a lane owns one vector, reads 128
// columns at a time as packed pairs, releases the buffer and takes minima of 64 and of its running threshold with 16
// three-input packed minima; where that is below the threshold the group joins the lane's candidates in shared memory, without a
// branch.  The next step's A tiles are written before a step's scan.
// What bounds it: the round trip of a TMEM buffer.  The accumulators of 256 vectors x 256 centroids fill TMEM, and from the
// release of a buffer to the signal of its next MMA pass about 500 clocks, whatever the MMA's size (the handshake alone, with
// nothing read or reduced, takes 640 clocks per 256 centroids; with both it is 760, where the ALU pipe needs about 400, the
// TMEM reads and the MMAs 256 each).  Buffers of 64 columns were slower (an MMA of 64 takes 48 clocks, one of 128 takes 64).
// 4096 x 4096, v = 8, 65536 centroids: 5.9 ms; with FP32 accumulators, two-input minima and a full scan of the 0.7 % of vectors
// with a second candidate group 13.7 ms.
// Every mbarrier wait is bounded; a wait that gives up sets the status word of the workspace.
#include "common.cuh"
#include "assign.cuh"
#include "tcgen05_ptx.cuh"

namespace vptq {

namespace {

using namespace tc;

constexpr int KT = 128;                       // centroids of a tile image, per MMA (N) and per accumulator buffer
constexpr int KP = 2 * KT;                    // centroids per ring stage
constexpr int ROW_BYTES = 32;                 // K = 16 FP16 values
constexpr int TILE_BYTES = KT * ROW_BYTES;    // 4 KB: an A tile (128 vectors) or half a stage (128 centroids)
constexpr int STAGE_BYTES = 2 * TILE_BYTES;
constexpr int B_STAGES = 10;
constexpr int EPI_WARP0 = 4, EPI_WARPS = 16;
constexpr int SCAN_THREADS = 32 * (EPI_WARP0 + EPI_WARPS);
constexpr int AHEAD = B_STAGES - 3;             // stages loaded ahead of the one whose MMAs are issued
constexpr int STEP_VECTORS = 256;             // two A tiles
constexpr int GROUP = 32;                     // centroids of a candidate group: every other one of 64
constexpr int LIST_LEN = 24, LIST_STRIDE = 2 * STEP_VECTORS;    // candidates kept per vector and buffer
constexpr unsigned long long NO_RESULT = 0x7F8000007FFFFFFFull;            // infinite distance, no index
// centroids from which on a lane evaluates a group by itself (16384: 2.06 -> 1.92 ms; below that the warp does: 8192 1.35 -> 1.23)
constexpr int WARP_GROUP_MAX_K = 16384;
constexpr uint32_t NO_THRESHOLD = 0x7C007C00u, GAVE_UP = 0x80008000u;      // infinity; below every value
constexpr float PAD_NORM = 60000.f;           // norm of the padding rows of the last centroid tile: never the minimum
constexpr float X_LIMIT = 3.0e4f, C_LIMIT = 1.5e4f;      // scaled ||x||^2 and max ||c||^2 up to which no real distance reaches the padding's
constexpr float ABS = 1.0f / 65536.0f;        // 2^-16: 4E of (||x||^2 + max ||c||^2)
constexpr float ABS_NO_LO = 1.0f / 1024.0f;   // 2^-10 max ||c||^2 more when the norm's low half is missing

// shared memory: A tiles [2 steps][2], B ring, candidate lists, their thresholds and lengths, results, vectors, barriers
constexpr int OFF_B = 4 * TILE_BYTES, OFF_CAND = OFF_B + B_STAGES * STAGE_BYTES, OFF_BOUND = OFF_CAND + LIST_LEN * LIST_STRIDE * 8,
              OFF_BEST = OFF_BOUND + STEP_VECTORS * 2 * 8, OFF_X = OFF_BEST + STEP_VECTORS * 8,
              OFF_BARS = OFF_X + 2 * STEP_VECTORS * 32;
constexpr int N_BARS = 2 * B_STAGES + 4 + 4 + 2 + 8;
constexpr int SCAN_SMEM = OFF_BARS + N_BARS * 8 + 16;

struct ScanParams {
    const __half *W;
    int M, N, v, k;
    const __half *C;          // [k_tiles * KT][8 or 16]: centroids padded with zeros, of every 64 the even ones first
    const uint8_t *Bimg;      // [k_tiles][TILE_BYTES]
    const float *cmax;        // max ||c||^2
    int *idx;                 // [n_vectors]
    int *list;                // vectors that need the full scan
    int *count;               // entries of the list
    int *status;
    long long n_vectors;
    int k_pairs;              // ring stages of a pass over the codebook
};

// K-major operand with 32-byte rows and the 32-byte swizzle: 8-row groups of 256 bytes
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr) { return make_smem_desc(saddr, 16, 8 * ROW_BYTES, LAYOUT_SW32); }
// kind::f16: FP16 x FP16 -> FP16 (accumulated wider, rounded once), both operands K-major, M = 128, N = 128
constexpr uint32_t SCAN_IDESC = (0u << 4) | ((uint32_t)(KT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
__device__ __forceinline__ void umma_fresh(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 0, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(SCAN_IDESC) : "memory");
}
// 128 consecutive FP16 accumulator columns of this lane's row, two to a register; the registers may be read after the wait (they
// are operands of it so that no use moves above it)
__device__ __forceinline__ void tmem_ld128(uint32_t taddr, uint32_t (&r)[64])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x64.pack::16b.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,"
                 "%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,"
                 "%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), 
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), 
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), 
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), 
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), 
                   "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), 
                   "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), 
                   "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), 
                   "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), 
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), 
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), 
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), 
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]), 
                   "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]), 
                   "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]), 
                   "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55]), "+r"(r[56]), 
                   "+r"(r[57]), "+r"(r[58]), "+r"(r[59]), "+r"(r[60]), "+r"(r[61]), "+r"(r[62]), "+r"(r[63])
                 :: "memory");
}
// Smallest of t and 32 packed pairs, low and high halves apart.  Positive FP16 values are ordered like their bit patterns, so
// these are 16-bit integer minima, three to an instruction.
template <int FIRST>
__device__ __forceinline__ uint32_t min64(uint32_t t, const uint32_t (&all)[64])
{
    const uint32_t *d = all + FIRST;
    uint32_t a[11];
    a[0] = __vimin3_s16x2(t, d[0], d[1]);
#pragma unroll
    for (int i = 1; i < 11; i++) a[i] = __vimin3_s16x2(d[3 * i - 1], d[3 * i], d[3 * i + 1]);
    const uint32_t b0 = __vimin3_s16x2(a[0], a[1], a[2]), b1 = __vimin3_s16x2(a[3], a[4], a[5]), b2 = __vimin3_s16x2(a[6], a[7], a[8]);
    return __vimin3_s16x2(__vimin3_s16x2(b0, b1, b2), a[9], a[10]);
}

// A full candidate list keeps what is still below the threshold; one that stays full gives up (no minimum is below then).
__device__ __noinline__ void compact_list(uint2 *mine, int &cnt, uint32_t &thr)
{
    int kept = 0;
    for (int i = 0; i < cnt; i++) {
        const uint2 e = mine[i * LIST_STRIDE];
        mine[kept * LIST_STRIDE] = e;
        kept += __vmins2(e.x, thr) != thr ? 1 : 0;
    }
    cnt = kept;
    if (cnt > LIST_LEN / 2) { cnt = 0; thr = GAVE_UP; }      // the full scan decides
}

// byte offset of 16-byte chunk c (0 or 1) of row r in a tile image (32-byte swizzle: bit 4 ^= bit 7)
__device__ __forceinline__ int image_offset(int r, int c) { return r * ROW_BYTES + ((c ^ ((r >> 2) & 1)) << 4); }

// The power of two that brings max ||c||^2 to [2^8, 2^10): 2^s multiplies vectors and centroids.
__device__ __forceinline__ int scale_exponent(float cmax)
{
    if (!(cmax > 0.f) || !(cmax < 3.0e38f)) return 0;
    int s = (8 - ilogbf(cmax) + 1) / 2;                 // ilogbf: floor(log2)
    return s < -12 ? -12 : (s > 24 ? 24 : s);
}

// ---- preparation, first pass: max ||c||^2; clears the list count and the status word -------------------------
__global__ void __launch_bounds__(256)
assign_norms_kernel(const __half *__restrict__ C, int k, int v, float *cmax, int *count, int *status)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i == 0) { *count = 0; *status = 0; }
    if (i >= k) return;
    float norm = 0.f;
    for (int j = 0; j < v; j++) {
        const float c = __half2float(__ldg(C + (long long)i * v + j));
        norm = __fmaf_rn(c, c, norm);
    }
    // norm >= 0: integer order = float order; a NaN norm has the largest bit pattern and so becomes the maximum
    atomicMax(reinterpret_cast<int *>(cmax), __float_as_int(norm));
}

// ---- preparation, second pass: the scaled centroid tiles as shared-memory images, and the centroids as rows of `pad` values ----
__global__ void __launch_bounds__(256)
assign_prepare_kernel(const __half *__restrict__ C, int k, int v, uint8_t *__restrict__ Bimg, __half *__restrict__ Cpad, int pad,
                      const float *cmax, int rows)
{
    const int i = blockIdx.x * 256 + threadIdx.x;          // centroid (or padding row of the last stage)
    if (i >= rows) return;
    const float scale = exp2f((float)scale_exponent(*cmax));
    __half row[16], raw[16];
#pragma unroll
    for (int j = 0; j < 16; j++) { row[j] = __float2half_rn(0.f); raw[j] = row[j]; }
    float norm = PAD_NORM;
    if (i < k) {
        norm = 0.f;
#pragma unroll
        for (int j = 0; j < 14; j++)
            if (j < v) {
                raw[j] = __ldg(C + (long long)i * v + j);
                const float c = __half2float(raw[j]) * scale;
                norm = __fmaf_rn(c, c, norm);
                row[j] = __float2half_rn(-2.f * c);         // exact while in range
            }
    }
    const __half hi = __float2half_rn(norm);
    row[14] = hi;
    if (v <= 13) {
        row[13] = __float2half_rn(1.f);
        row[15] = __float2half_rn((norm - __half2float(hi)) * 2048.f);     // the A row multiplies it by 2^-11
    } else {
        row[15] = __float2half_rn(1.f);
    }
    uint8_t *tile = Bimg + (long long)(i / KT) * TILE_BYTES;
    const uint4 *src = reinterpret_cast<const uint4 *>(row), *rsrc = reinterpret_cast<const uint4 *>(raw);
    *reinterpret_cast<uint4 *>(tile + image_offset(i % KT, 0)) = src[0];
    *reinterpret_cast<uint4 *>(tile + image_offset(i % KT, 1)) = src[1];
    // (a group's 32 centroids, the even or the odd ones of 64, next to each other)
    uint4 *dst = reinterpret_cast<uint4 *>(Cpad + (long long)((i & ~63) | ((i & 1) << 5) | ((i & 63) >> 1)) * pad);
    dst[0] = rsrc[0];
    if (pad == 16) dst[1] = rsrc[1];
}

// ---- the scan ---------------------------------------------------------------------------------------------
template <int VMAX, bool WARP_GROUP>
__global__ void __launch_bounds__(SCAN_THREADS, 1)
assign_scan_kernel(ScanParams P)
{
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    const uint32_t sA = smem_addr(sm), sB = sA + OFF_B;
    uint2 *lists = reinterpret_cast<uint2 *>(sm + OFF_CAND);               // [LIST_LEN][2 buffers][256] candidates
    int2 *bound = reinterpret_cast<int2 *>(sm + OFF_BOUND);               // [256][2 buffers] threshold, length of the list
    unsigned long long *result = reinterpret_cast<unsigned long long *>(sm + OFF_BEST);     // [256] distance bits, index below them

    uint32_t *xsave = reinterpret_cast<uint32_t *>(sm + OFF_X);           // [2 steps][256][8] components as they are

    const uint32_t bar0 = sA + OFF_BARS;
    auto bar_fullB = [&](int s) { return bar0 + 8u * s; };
    auto bar_emptyB = [&](int s) { return bar0 + 8u * (B_STAGES + s); };
    auto bar_accFull = [&](int a, int b) { return bar0 + 8u * (2 * B_STAGES + 2 * a + b); };
    auto bar_accEmpty = [&](int a, int b) { return bar0 + 8u * (2 * B_STAGES + 4 + 2 * a + b); };
    auto bar_aFull = [&](int s) { return bar0 + 8u * (2 * B_STAGES + 8 + s); };
    auto bar_pair = [&](int i) { return bar0 + 8u * (2 * B_STAGES + 10 + i); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < B_STAGES; s++) { mbar_init(bar_fullB(s), 1); mbar_init(bar_emptyB(s), 4); }
        for (int i = 0; i < 4; i++) { mbar_init(bar_accFull(i >> 1, i & 1), 1); mbar_init(bar_accEmpty(i >> 1, i & 1), 4); }
        for (int s = 0; s < 2; s++) mbar_init(bar_aFull(s), EPI_WARPS / 2);
        for (int i = 0; i < 8; i++) mbar_init(bar_pair(i), 2);
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 3) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;

    const long long n_steps = (P.n_vectors + STEP_VECTORS - 1) / STEP_VECTORS;
    bool ok = (sA & 1023u) == 0;
    if (!ok && threadIdx.x == 0) atomicExch(P.status, VPTQ_E_UNSUPPORTED);

    if (warp < EPI_WARP0) {
        // ================= MMA issue: A tile a, first or second half of every stage =================
        // (the whole warp runs the loop and an elected lane issues: see elect_one)
        if (ok) {
            const int a = warp & 1, b = warp >> 1;
            const uint64_t adesc0 = operand_desc(sA + a * TILE_BYTES), bdesc0 = operand_desc(sB + b * TILE_BYTES);
            const uint32_t d_tmem = tmem_base + (uint32_t)((b * 2 + a) * KT);
            uint32_t it = 0, step_no = 0, gave_up = 0;                     // stages used so far
            // warp 0 also streams the centroid tiles into the ring, AHEAD stages before they are needed
            const uint32_t total = blockIdx.x < n_steps ? (uint32_t)((n_steps - blockIdx.x + gridDim.x - 1) / gridDim.x) * P.k_pairs : 0u;
            uint32_t loaded = 0, load_kp = 0;
            auto load_next = [&]() {
                if (loaded >= total) return;
                const uint32_t s = loaded % B_STAGES;
                mbar_wait_uniform(bar_emptyB(s), ((loaded / B_STAGES) & 1) ^ 1u, gave_up);
                if (elect_one()) {
                    mbar_expect_tx(bar_fullB(s), STAGE_BYTES);
                    bulk_load(sB + s * STAGE_BYTES, P.Bimg + (long long)load_kp * STAGE_BYTES, STAGE_BYTES, bar_fullB(s));
                }
                loaded++;
                if (++load_kp == (uint32_t)P.k_pairs) load_kp = 0;
            };
            if (warp == 0)
                for (int i = 0; i < AHEAD; i++) load_next();
            for (long long step = blockIdx.x; step < n_steps && ok; step += gridDim.x, step_no++) {
                mbar_wait_uniform(bar_aFull(step_no & 1), (step_no >> 1) & 1, gave_up);
                const uint64_t ad = adesc0 + (uint64_t)(((step_no & 1) * 2 * TILE_BYTES) >> 4);
                for (int kp = 0; kp < P.k_pairs; kp++, it++) {
                    const uint32_t s = it % B_STAGES;
                    mbar_wait_uniform(bar_fullB(s), (it / B_STAGES) & 1, gave_up);
                    mbar_wait_uniform(bar_accEmpty(a, b), (it & 1) ^ 1u, gave_up);
                    tc_fence_after();
                    if (elect_one()) {
                        umma_fresh(d_tmem, ad, bdesc0 + (uint64_t)((s * STAGE_BYTES) >> 4));
                        umma_commit(bar_accFull(a, b));
                        // an empty buffer means that its previous MMA has read its stage
                        if (it > 0) mbar_arrive(bar_emptyB((it - 1) % B_STAGES));
                    }
                    if (warp == 0) load_next();
                }
                // some wait ran out: what was issued since is in bounds and worthless
                ok = !__any_sync(0xffffffffu, gave_up != 0 || *abort_flag != 0);
            }
            if (!ok) {
                *abort_flag = 1;
                if (lane == 0) atomicExch(P.status, VPTQ_E_TIMEOUT);
            }
            // copies still in flight (only after a wait that ran out) get a bounded time to land before the CTA exits
            if (warp == 0)
                for (uint32_t j = loaded > B_STAGES ? loaded - B_STAGES : 0; j < loaded; j++) {
                    const long long t0c = clock64();
                    while (!mbar_try(bar_fullB(j % B_STAGES), (j / B_STAGES) & 1) && clock64() - t0c < 20000000ll) {}
                }
        }
    } else {
        // ================= A tiles, then the running minima; a lane owns one vector of the step =================
        const int ew = warp - EPI_WARP0;
        const int q = warp & 3;                      // TMEM lane quarter this warp may read
        const int a = (ew >> 2) & 1, b = ew >> 3;    // A tile, accumulator buffer
        const int row = 32 * q + lane;               // row of the A tile = TMEM lane
        // the two warps that share a vector meet (twice per step: parities 0 and 1)
        auto meet = [&](uint32_t parity) {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_pair(a * 4 + q));
            return __all_sync(0xffffffffu, mbar_wait(bar_pair(a * 4 + q), parity, abort_flag, P.status)) != 0;
        };
        const float scale = exp2f((float)scale_exponent(__ldg(P.cmax)));
        const float cmax = __ldg(P.cmax) * scale * scale;      // in the filter's units
        const float abs_c = P.v <= 13 ? ABS : ABS + ABS_NO_LO;
        // this lane's column of the candidate lists
        uint2 *mine = lists + b * (LIST_STRIDE / 2) + a * 128 + row;
        // components of this lane's vector of a step, packed as they are (zeros beyond v and beyond the last vector)
        constexpr int XW = (VMAX + 1) / 2;
        auto load_x = [&](long long step, uint32_t (&xw)[XW]) {
            const long long g = step * STEP_VECTORS + a * 128 + row;
            const bool valid = step < n_steps && g < P.n_vectors;
            const int r = valid ? (int)(g / P.N) : 0, n = valid ? (int)(g % P.N) : 0;
            const unsigned short *col = reinterpret_cast<const unsigned short *>(P.W) + (long long)r * P.v * P.N + n;
#pragma unroll
            for (int w = 0; w < XW; w++) {
                const uint32_t lo = (valid && 2 * w < P.v) ? __ldg(col + (long long)(2 * w) * P.N) : 0u;
                const uint32_t hi = (valid && 2 * w + 1 < P.v) ? __ldg(col + (long long)(2 * w + 1) * P.N) : 0u;
                xw[w] = lo | (hi << 16);
            }
        };
        // ... their scaled squared norm; the lane's row of the A tile
        auto write_a = [&](uint32_t step_no, const uint32_t (&xw)[XW]) {
            __half rowv[16];
            float xn = 0.f;
#pragma unroll
            for (int j = 0; j < 14; j++) rowv[j] = __float2half_rn(0.f);
#pragma unroll
            for (int w = 0; w < XW; w++) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&xw[w]));
                const float s0 = f.x * scale, s1 = f.y * scale;
                xn = __fmaf_rn(s1, s1, __fmaf_rn(s0, s0, xn));
                rowv[2 * w] = __float2half_rn(s0); rowv[2 * w + 1] = __float2half_rn(s1);         // exact while in range
            }
            if (b == 0) {
                // the components as they are, for the evaluation at the end of the step (each step parity has a place)
                uint32_t *xr = xsave + (step_no & 1) * (STEP_VECTORS * 8) + (a * 128 + row) * 8;
                *reinterpret_cast<uint4 *>(xr) = make_uint4(xw[0], xw[XW > 1 ? 1 : 0], xw[XW > 2 ? 2 : 0], xw[XW > 3 ? 3 : 0]);
                if (XW > 4) *reinterpret_cast<uint4 *>(xr + 4) = make_uint4(xw[XW > 4 ? 4 : 0], xw[XW > 5 ? 5 : 0], xw[XW > 6 ? 6 : 0], 0u);
                // (the shift by the error bound keeps every filter value positive)
                const __half xv = __float2half_ru(xn + (xn * ABS + cmax * abs_c));
                rowv[14] = __float2half_rn(1.f);                                   // times hi
                if (P.v <= 13) { rowv[13] = xv; rowv[15] = __float2half_rn(1.f / 2048.f); }     // times 2^11 lo
                else rowv[15] = xv;
                const uint4 *src = reinterpret_cast<const uint4 *>(rowv);
                uint8_t *tile = sm + ((step_no & 1) * 2 + a) * TILE_BYTES;
                *reinterpret_cast<uint4 *>(tile + image_offset(row, 0)) = src[0];
                *reinterpret_cast<uint4 *>(tile + image_offset(row, 1)) = src[1];
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_aFull(step_no & 1));
            }
            return xn;
        };
        uint32_t it = 0, step_no = 0, gave_up = 0;
        float xn_next = 0.f;
        if (ok && blockIdx.x < n_steps) {
            uint32_t xw[XW];
            load_x(blockIdx.x, xw);
            xn_next = write_a(0, xw);
        }
        for (long long step = blockIdx.x; step < n_steps && ok; step += gridDim.x, step_no++) {
            const float xn = xn_next;
            const float err = xn * ABS + cmax * abs_c;
            // the next step's A tiles, into the buffers of the previous step (whose MMAs this pair of warps has seen complete)
            if (step + gridDim.x < n_steps) {
                uint32_t xw[XW];
                load_x(step + gridDim.x, xw);
                xn_next = write_a(step_no + 1, xw);
            }

            // Candidates go to this lane's column of the list as (packed minima of the even and odd columns, group).  The threshold,
            // in both halves of a word, is b (1 + 2^-10) + err of the smallest minimum b so far, one FP16 step up (for the
            // rounding of this sum).  No branch: lanes without a candidate store nothing.
            const uint32_t err2 = (uint32_t)__half_as_ushort(__float2half_ru(fminf(err, 65504.f))) * 0x10001u;
            const __half2 one_up = __halves2half2(__ushort_as_half(0x3C01), __ushort_as_half(0x3C01));      // 1 + 2^-10
            uint32_t thr = NO_THRESHOLD;
            int cnt = 0;
            auto keep = [&](uint32_t m, uint32_t group) {
                if (m != thr) mine[cnt * LIST_STRIDE] = make_uint2(m, group);
                cnt += m != thr ? 1 : 0;
            };
            auto lower = [&](uint32_t m) {
                const uint32_t bm = __vmins2(m, __byte_perm(m, 0, 0x1032));
                const __half2 w = __hfma2(*reinterpret_cast<const __half2 *>(&bm), one_up, *reinterpret_cast<const __half2 *>(&err2));
                thr = __vimin3_s16x2(thr, *reinterpret_cast<const uint32_t *>(&w) + 0x00010001u, NO_THRESHOLD);
            };
            // 128 distances of a stage: into registers, buffer back to the issuer, then 64 at a time
            const uint32_t t_row = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)((b * 2 + a) * KT);
            uint32_t d[64];
            for (int kp = 0; kp < P.k_pairs; kp++, it++) {
                mbar_wait_uniform(bar_accFull(a, b), it & 1, gave_up);
                tc_fence_after();
                tmem_ld128(t_row, d);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_accEmpty(a, b));
                const uint32_t group = (uint32_t)(kp * 2 + b) * 4u;
                const uint32_t m0 = min64<0>(thr, d), m1 = min64<32>(thr, d);
                keep(m0, group);
                keep(m1, group + 2u);
                lower(__vmins2(m0, m1));
                if (cnt > LIST_LEN - 2) compact_list(mine, cnt, thr);
            }
            ok = !__any_sync(0xffffffffu, gave_up != 0 || *abort_flag != 0);
            if (!ok) {
                *abort_flag = 1;
                break;
            }

            // ---- the two warps of a vector agree on the threshold; each evaluates the candidates of its own lists ----
            const int slot = a * 128 + row;
            const long long g = step * STEP_VECTORS + slot;
            bound[slot * 2 + b] = make_int2((int)(thr & 0xffff0000u), cnt);
            if (b == 0) result[slot] = NO_RESULT;
            if (!(ok = meet(0))) break;
            const int t = min((int)(thr & 0xffff0000u), bound[slot * 2 + (b ^ 1)].x);
            // (no candidate below infinity, or a vector or table out of the filter's range: the full scan decides)
            const bool full = t <= 0 || !(xn < X_LIMIT) || !(cmax < C_LIMIT);
            const bool valid = g < P.n_vectors;
            // the groups still below the common threshold, two to an entry, to the front of the lane's list
            int n = 0;
            auto put = [&](uint32_t group) { reinterpret_cast<uint32_t *>(mine + (n >> 1) * LIST_STRIDE)[n & 1] = group; n++; };
            if (valid && !full)
                for (int i = 0; i < cnt; i++) {
                    const uint2 e = mine[i * LIST_STRIDE];
                    if ((int)(e.x << 16) < t) put(e.y);
                    if ((int)(e.x & 0xffff0000u) < t) put(e.y | 1u);
                }
            // The warp's groups are numbered through, whosever they are.  A table of few centroids: the warp takes one after the other, a
            // lane a centroid, 512 bytes side by side.  Else 32 at a time, a lane a group: with 65536 centroids a vector has so many that the
            // lanes are busy that way.  (With a lane to a vector a warp took as long as its longest list, and read single centroids.
            // 4096 x 4096, one iteration, k = 65536, v = 8: 6.21 -> 6.04 ms; k = 4096, v = 8: 1.00 -> 0.89, v = 12: 0.88 -> 0.72; 65536 the first way 6.31, 4096
            // (v = 8) the second 1.07.)
            int first = n;                                             // groups of the lanes before this one
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, first, o);
                if (lane >= o) first += v;
            }
            const int total = __shfl_sync(0xffffffffu, first, 31);
            first -= n;
            __syncwarp();
            // (distances are not negative, so their bits are ordered like them; the lowest index wins a tie)
            auto pack = [](uint32_t d, int c) { return (unsigned long long)d << 32 | (unsigned)c; };
            unsigned long long best = NO_RESULT;                       // of this lane's vector (WARP_GROUP)
            for (int i0 = 0; i0 < total; i0 += 32) {
                // lane i finds the vector and the group of item i0 + i
                const int i = i0 + lane;
                int owner = 0;                                         // the last lane whose groups begin at or before i
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int v = __shfl_sync(0xffffffffu, first, owner + o);
                    if (v <= i) owner += o;
                }
                const int k = i - __shfl_sync(0xffffffffu, first, owner);
                uint32_t group = 0;
                if (i < total) group = reinterpret_cast<const uint32_t *>(lists + b * (LIST_STRIDE / 2) + a * 128 + 32 * q + owner + (k >> 1) * LIST_STRIDE)[k & 1];
                if (!WARP_GROUP) {
                    if (i >= total) continue;
                    const int os = a * 128 + 32 * q + owner, c0 = (int)(group >> 1) * 64 + (int)(group & 1u);
                    float x[VMAX];
                    const uint32_t *xr = xsave + (step_no & 1) * (STEP_VECTORS * 8) + os * 8;
#pragma unroll
                    for (int w = 0; w < XW; w++) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(xr + w));
                        x[2 * w] = f.x; x[2 * w + 1] = f.y;
                    }
                    unsigned long long least = NO_RESULT;
                    constexpr int AT_ONCE = VMAX > 8 ? 4 : 8;
#pragma unroll 1
                    for (int u0 = 0; u0 < GROUP; u0 += AT_ONCE) {
                        uint4 w[AT_ONCE][VMAX > 8 ? 2 : 1];
#pragma unroll
                        for (int u = 0; u < AT_ONCE; u++) {
                            const uint4 *cr = reinterpret_cast<const uint4 *>(P.C) + (long long)(group * GROUP + u0 + u) * (VMAX > 8 ? 2 : 1);
                            w[u][0] = __ldg(cr);
                            if (VMAX > 8) w[u][VMAX > 8 ? 1 : 0] = __ldg(cr + 1);
                        }
#pragma unroll
                        for (int u = 0; u < AT_ONCE; u++) {
                            const uint32_t *wu = reinterpret_cast<const uint32_t *>(w[u]);
                            float dd = 0.f;
#pragma unroll
                            for (int j = 0; j < VMAX; j++) {
                                const float2 cv = __half22float2(*reinterpret_cast<const __half2 *>(&wu[j >> 1]));
                                const float tt = __fsub_rn(x[j], (j & 1) ? cv.y : cv.x);
                                dd = __fmaf_rn(tt, tt, dd);
                            }
                            const int ci = c0 + 2 * (u0 + u);
                            if (ci < P.k) least = min(least, pack(__float_as_uint(dd), ci));
                        }
                    }
                    atomicMin(result + os, least);
                    continue;
                }
                const int items = min(32, total - i0);
                constexpr int AT_ONCE = 4;
#pragma unroll 1
                for (int j0 = 0; j0 < items; j0 += AT_ONCE) {
                    uint4 w[AT_ONCE][VMAX > 8 ? 2 : 1];
                    uint32_t gj[AT_ONCE];
#pragma unroll
                    for (int u = 0; u < AT_ONCE; u++) {
                        gj[u] = __shfl_sync(0xffffffffu, group, j0 + u);          // (items past the last are group 0, and dropped)
                        const uint4 *cr = reinterpret_cast<const uint4 *>(P.C) + (long long)(gj[u] * GROUP + lane) * (VMAX > 8 ? 2 : 1);
                        w[u][0] = __ldg(cr);
                        if (VMAX > 8) w[u][VMAX > 8 ? 1 : 0] = __ldg(cr + 1);
                    }
#pragma unroll
                    for (int u = 0; u < AT_ONCE; u++) {
                        const int oj = __shfl_sync(0xffffffffu, owner, j0 + u);
                        const uint32_t *xr = xsave + (step_no & 1) * (STEP_VECTORS * 8) + (a * 128 + 32 * q + oj) * 8;
                        const uint32_t *wu = reinterpret_cast<const uint32_t *>(w[u]);
                        float dd = 0.f;
#pragma unroll
                        for (int j = 0; j < XW; j++) {
                            const float2 xv = __half22float2(*reinterpret_cast<const __half2 *>(xr + j));
                            const float2 cv = __half22float2(*reinterpret_cast<const __half2 *>(&wu[j]));
                            const float t0 = __fsub_rn(xv.x, cv.x), t1 = __fsub_rn(xv.y, cv.y);
                            dd = __fmaf_rn(t0, t0, dd);
                            if (2 * j + 1 < VMAX) dd = __fmaf_rn(t1, t1, dd);
                        }
                        const int c0 = (int)(gj[u] >> 1) * 64 + (int)(gj[u] & 1u);           // the group's centroids are two apart
                        const uint32_t key = c0 + 2 * lane < P.k ? __float_as_uint(dd) : 0xffffffffu;
                        const uint32_t least = __reduce_min_sync(0xffffffffu, key);
                        const int ci = c0 + 2 * (__ffs(__ballot_sync(0xffffffffu, key == least)) - 1);     // the lowest index wins a tie
                        if (lane == oj && j0 + u < items) best = min(best, pack(least, ci));
                    }
                }
            }
            if (WARP_GROUP) atomicMin(result + slot, best);
            if (!(ok = meet(1))) break;
            if (b == 0 && valid) {
                const int nearest = (int)(unsigned)result[slot];
                if (full || nearest == 0x7fffffff) P.list[atomicAdd(P.count, 1)] = (int)g;      // the full scan decides
                else P.idx[g] = nearest;
            }
        }
    }

    tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (warp == 3) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

struct ScanLayout {
    long long off_cmax, off_count, off_bimg, off_cpad, off_list, bytes;
    int k_pairs, pad;
};

ScanLayout scan_layout(long long n_vectors, int v, int k)
{
    ScanLayout l;
    l.k_pairs = ceil_div(k, KP);
    l.pad = v <= 8 ? 8 : 16;
    l.off_cmax = 16;                    // status word at byte 0
    l.off_count = 32;
    l.off_bimg = 256;
    l.off_cpad = l.off_bimg + (long long)l.k_pairs * STAGE_BYTES;
    l.off_list = l.off_cpad + (long long)l.k_pairs * KP * l.pad * 2;
    l.bytes = l.off_list + (n_vectors * 4 + 255) / 256 * 256;
    return l;
}

}  // namespace

// vectors of at most 14 components (two or three of the 16 K columns carry the norms), whole vector rows, enough
// centroids for the filter to pay, vector numbers that fit an int
bool assign_tcgen05_supported(int M, int N, int v, int k)
{
    if (v < 1 || v > 14 || k < 1024 || k > 65536 || M % v != 0) return false;
    return (long long)(M / v) * N < 0x7fffffffLL && (long long)(M / v) * N >= 4096;
}

long long assign_tcgen05_workspace_bytes(int M, int N, int v, int k)
{
    return scan_layout((long long)ceil_div(M, v) * N, v, k).bytes;
}

cudaError_t launch_assign_tcgen05(const __half *W, int M, int N, int v, const __half *C, int k, int *idx, void *ws,
                                  cudaStream_t st)
{
    const long long n_vectors = (long long)(M / v) * N;
    const ScanLayout l = scan_layout(n_vectors, v, k);
    uint8_t *w8 = reinterpret_cast<uint8_t *>(ws);
    ScanParams P;
    P.W = W; P.M = M; P.N = N; P.v = v; P.k = k;
    P.C = reinterpret_cast<const __half *>(w8 + l.off_cpad);
    P.Bimg = w8 + l.off_bimg;
    P.cmax = reinterpret_cast<const float *>(w8 + l.off_cmax);
    P.idx = idx;
    P.list = reinterpret_cast<int *>(w8 + l.off_list);
    P.count = reinterpret_cast<int *>(w8 + l.off_count);
    P.status = reinterpret_cast<int *>(w8);
    P.n_vectors = n_vectors;
    P.k_pairs = l.k_pairs;
    cudaError_t e = cudaMemsetAsync(w8 + l.off_cmax, 0, 4, st);
    if (e != cudaSuccess) return e;
    assign_norms_kernel<<<ceil_div(k, 256), 256, 0, st>>>(C, k, v, reinterpret_cast<float *>(w8 + l.off_cmax),
                                                          P.count, P.status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    assign_prepare_kernel<<<l.k_pairs, KP, 0, st>>>(C, k, v, w8 + l.off_bimg, reinterpret_cast<__half *>(w8 + l.off_cpad), l.pad,
                                                    P.cmax, l.k_pairs * KP);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long n_steps = (n_vectors + STEP_VECTORS - 1) / STEP_VECTORS;
    const int grid = (int)(n_steps < device_sm_count() ? n_steps : device_sm_count());
    const bool warp_group = k < WARP_GROUP_MAX_K;
    auto kern = v <= 8 ? (warp_group ? assign_scan_kernel<8, true> : assign_scan_kernel<8, false>)
                       : (warp_group ? assign_scan_kernel<14, true> : assign_scan_kernel<14, false>);
    e = allow_dynamic_smem(reinterpret_cast<const void *>(kern), SCAN_SMEM);
    if (e != cudaSuccess) return e;
    kern<<<grid, SCAN_THREADS, SCAN_SMEM, st>>>(P);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the vectors with too many candidate groups: all centroids, FP32
    return launch_assign_listed(W, M, N, v, C, k, idx, P.list, P.count, device_sm_count(), st);
}

}  // namespace vptq
