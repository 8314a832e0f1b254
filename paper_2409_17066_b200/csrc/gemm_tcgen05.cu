// Batched / prefill path: out[B][M] = x[B][N] * W_hat^T as a tensor-core GEMM whose weight
// operand is dequantised on the fly into shared memory (the FP16 weight matrix never exists in
// global memory; App. D.2 describes the paper's two-phase scheme that this replaces).
//
//   D[m][t] (TMEM, FP32, 128 lanes x up to 512 columns) += A[m][k] * B[t][k]
//   A = W tile, NV whole vector rows (16 x 8, 20 x 6 or 10 x 12 output rows) x KS input columns, written by producer
//       warps from C1[i1] + C2[i2]:
//         v = 8:      KS = 32, one 16-byte store per centroid in the MN-major 128-byte-swizzled layout;
//         v = 6, 12:  KS = 64, a lane takes 8 columns of a vector row, turns them into rows in registers (one byte
//                     permute per pair) and stores 16 bytes per output row in the K-major 128-byte-swizzled layout: the
//                     MN-major form would need 4- or 8-byte stores at a time (12- and 24-byte vectors);
//   B = x*s (FP16, scale folded into the activations by a pre-pass), the tile's tokens x 32 columns per ring element,
//       K-major with the 64-byte swizzle.  The pre-pass writes the activations as the shared-memory image of these
//       elements, so one arrives by one linear bulk copy of whole 128-byte lines;
//   tcgen05.mma.cta_group::1.kind::f16, M = 128, N = the tile's tokens (16 .. 256, one or two per token tile), K = 16.
// Columns: the main columns first, then the outlier columns (a few k blocks of their own, A written from C0).
// Tables: a main codebook of at most 64 KB (16-byte rows) and a residual one of at most 16 KB sit in shared memory
// (small ones as several skewed copies); larger or group-wise ones are read out of L2, rows of 12 and 24 bytes from a copy
// with rows padded to 16 and 32 bytes that the pre-pass writes (one load instruction and one 32-byte sector per row).
//
// Warp roles: warp 0 bulk loads of B; warp 1 TMEM allocation + MMA issue (an elected lane); 10 (v = 8) or 12 producer warps in
// GROUPS groups, a k block each in turn (the next visit's packed indices in flight); 8 warps the epilogue
// (tcgen05.ld -> + bias term -> output), two per TMEM lane quarter.  A form for few tokens has more producers and one
// epilogue warp per quarter (see Tile).
// Up to 256 tokens TMEM holds two sets of accumulators, so the next piece's MMAs do not wait for the epilogue
// (8192 x 8192, v = 6, 16 tokens 54.5 -> 53.1 us).
// What bounds the k loop is the SM's shared-memory/L1 data pipe (128 bytes per clock), which everything passes: per 32
// columns at 512 tokens the MMAs read 48 KB (384 clocks) and the bulk copies write 32 KB (256), the producers' stores take 64
// and 512 gathers out of L2 a wavefront each (512) plus the residual reads: about 1280 of the 1070-1330 clocks measured
// against 512 of the MMAs alone.  More producer warps (10, 12, 16), a converged or a single-lane issue loop, a scheduler
// kept free for the MMA issuer: all the same.  CTA pairs that forward half of every activation tile into the partner's
// shared memory were slower (117 us against 88 us on 14336 x 4096 at 512 tokens).
//
// Persistent grid, one CTA per SM.  The work is the list of (tile, k block) units, tile = (token tile, row tile); every
// CTA takes an equal, contiguous share of the units, whatever tile they fall in (a deterministic call: whole tiles; a call of
// few tiles: every tile cut among CTAs of its own).
// The pieces of a split tile meet
//   - FP32 output with 16-byte rows, long shares (FLAG_ORDER_MIN_COLS columns): in the output, without a zero-fill: the
//     piece that holds the tile's last k blocks is the first thing its CTA works on, so it finishes early; it stores and
//     then raises the tile's flag in the workspace; the other pieces (the last thing their CTAs work on) wait for the flag
//     (a bounded wait that is normally over before it starts) and reduce-add;
//   - FP32 output, short shares or a call that shares the GPU: in the output, cleared by the pre-pass, every piece adds;
//   - any other output: in an FP32 scratch tile cleared by the pre-pass; every piece adds and counts itself in, and
//     whichever warp finds its part complete converts and stores it (nobody waits).  Only split tiles have one, at most one
//     per cut between two shares, so the scratch does not grow with the call.  Whole tiles per CTA, the form before,
//     left 84 of 148 SMs idle on an 8192 x 8192 layer at 333 tokens and 140 on a 1024 x 8192 one.
//
// Every mbarrier wait is bounded: after about two seconds a waiter records VPTQ_E_TIMEOUT in
// the status word of the workspace, raises a CTA-wide abort flag and every role leaves its
// loop; TMEM is freed on all paths.
#include <cuda.h>

#include "common.cuh"
#include "fused_split.cuh"
#include "gemm.cuh"
#include "index_words.cuh"
#include "tcgen05_ptx.cuh"

namespace vptq {

namespace {

using namespace tc;

constexpr int MAX_TILE_N = 512;                          // tokens of a tile: all TMEM columns
constexpr int IMG_COLS = 32;                             // columns of a B ring element
constexpr int MAX_B_STAGES = 8;
constexpr int MAX_EPI_WARPS = 8;
constexpr int EPI_TOKENS = 32;                            // tokens an epilogue warp reads out of TMEM at a time
constexpr int PIECE_TOKENS = 16;                          // ... and hands to the copy engine at a time
constexpr int EPI_BUF_BYTES = PIECE_TOKENS * 32 * 4;      // one staged piece of the output: 16 tokens x 32 rows, FP32
constexpr int B_SBO = 512;    // bytes between consecutive 8-token groups of a B element (8 x 64 B)
constexpr int WS_STATUS_BYTES = 256;
constexpr int DRAIN_COLS = 160;                          // columns of a k loop that take as long as draining 512 tokens of a tile
// ... and the columns that a piece which meets others in a scratch tile takes besides (bulk add, its completion, the count).  4096 x 11008, 16
// tokens: v = 8 without 39.7 us, with 128 38.8, 224 39.2; v = 6 41.7, 40.7, 40.1; v = 12 52.1, 50.4, 50.1.
constexpr int MEET_COLS_8 = 128, MEET_COLS = 224;
// Columns by which the longest share may grow for the sake of whole CTAs per tile: scratch tiles (plus an eighth of the tokens),
// FP32 sums.  1024 x 2048 (v = 6, 16 tokens, 16-bit results; 64 columns longer) 25.4 -> 13.0 us, 4096 x 4096 with v = 12 at 512
// tokens (105 longer) 60.4 -> 55.2; v = 8: 4096 x 4096 (138 longer) 21.4 / 21.6 at 16 tokens, 50.3 / 47.4 at 512, 8192 x 8192 (554 longer)
// 52.3 / 57.6.  Over 208 layers of v = 6, 8 and 12 at 5 to 512 tokens, all result types, the cuts taken are within 2 % of the better ones in 195, 49 of
// up to 16 tokens among them 45 (worst: v = 12, 3705 x 4728 at 5 tokens, 224 longer, 21.7 / 19.8; v = 6, 6101 x 918 at 64, 160 longer, 22.8 / 18.9).
// FP32 sums: 1024 x 8192, v = 12, 512 tokens (70 longer) 61.7 -> 45.9, 200 tokens x 1024 x 2048 (64 longer) 18.8 / 19.6.
constexpr int LONGER_COLS = 128, LONGER_COLS_SUM = 96;
// ... and where that is one CTA a tile, so that no piece meets another and nothing is cleared: that many and 5/4 of the tokens.  v = 8: 10550 x 878 at 256
// tokens (394 columns longer) 45.0 -> 25.0 us, 14463 x 397 at 32 (99) 19.7 -> 12.1, 12809 x 969 at 512 (284, v = 6) 56.5 -> 39.4, 13256 x 2119 at 512
// (638) 55.6 -> 44.9, 15702 x 2408 at 16 (411) 33.3 / 32.7, 15316 x 2793 at 64 (533) 44.3 / 46.4, 15689 x 3469 at 17 (590) 36.7 / 36.5, 13022 x 1073 at
// 64 (339) 25.8 -> 21.2; FP32 sums: 10224 x 1234 at 64 (574) 18.9 / 22.4.
constexpr int WHOLE_COLS = 400;
constexpr int FLAG_ORDER_MIN_COLS = 768;                 // columns of a share from which split tiles meet by flag order
constexpr int SMEM_LIMIT = 227 * 1024, SMEM_LIMIT_L1 = 195 * 1024;

// per vector length: geometry of the A tile and the producers
template <int V, bool FEW = false> struct Tile;
template <> struct Tile<8, false> {
    static constexpr int NV = 16, KS = 32, A_STAGES = 6, GROUP_WARPS = 2, GROUPS = 5, WARP0 = 2, WARPS = 10, EPI = 8;
};
template <> struct Tile<8, true> {
    static constexpr int NV = 16, KS = 32, A_STAGES = 8, GROUP_WARPS = 2, GROUPS = 7, WARP0 = 2, WARPS = 14, EPI = 4;
};
template <> struct Tile<6, false> {
    static constexpr int NV = 20, KS = 64, A_STAGES = 3, GROUP_WARPS = 5, GROUPS = 2, WARP0 = 4, WARPS = 12, EPI = 8;
};
template <> struct Tile<6, true> {
    static constexpr int NV = 20, KS = 64, A_STAGES = 5, GROUP_WARPS = 5, GROUPS = 4, WARP0 = 4, WARPS = 20, EPI = 4;
};
template <> struct Tile<12, false> {
    static constexpr int NV = 10, KS = 64, A_STAGES = 5, GROUP_WARPS = 3, GROUPS = 4, WARP0 = 4, WARPS = 12, EPI = 8;
};
// The form for FEW tokens (up to few_tokens() of a tile): the MMAs and the epilogue need little, and the producers are bound by the
// latency of their table reads, so there are more of them: v = 6: four groups (20 warps) in place of two, five stages of A; v = 8: seven pairs,
// eight stages; four epilogue warps.  v = 6, gate+up of 2 x 11008 x 4096 at 16 tokens 83 -> 73 us; v = 8, 1 MiB table, 8192 x 8192 at 16 48.4 -> 46.8,
// at 64 52.8 / 52.6, 4096 x 4096 at 64 22.9 / 24.0 (an epilogue of four warps).  v = 12 reads two 32-byte rows a pair out of L2, whose rate bounds it.
template <int V> constexpr int few_tokens() { return V == 8 ? 32 : V == 6 ? 64 : 0; }
// v = 6: a CTA's share from which on it is the form to take: in shorter ones four epilogue warps hold the tile's end up.  The other form / it:
// 1521 x 1024 at 48 tokens (128 columns) 12.4 / 15.1 us, 3341 x 1170 at 64 (230) 16.0 / 18.5, 1916 x 5650 at 48 (615) 20.5 / 21.8, 833 x 3843 at
// 16 (184) 13.5 / 14.6, 4096 x 4096 at 64 (983) 22.3 / 23.5; but 7488 x 2844 at 64 (1198) 28.8 / 27.3, 7232 x 5760 at 64 (2400) 42.4 / 37.8, 3 layers'
// 4500 rows x 3000 at 12 (809) 25.6 / 24.7, 5824 x 4980 at 12 (1652) 28.6 / 26.9.  Past 32 tokens not over eight copies of a small table, whose
// reads have less to wait for: 256 centroids, 11008 x 4096 at 64 (2585) 35.9 / 37.9, at 32 34.0 / 33.4.  Indices of other widths than 8, 12 and 16 bits
// are read one by one, which takes more producers at any share: 512 + 64 centroids, 2 x 3803 x 1664 at 32 tokens 29.0 / 24.2, 640 x 4014 at 21 15.7 / 14.7.
inline int few_min_cols(int tile_n) { return 18 * tile_n > 768 ? 18 * tile_n : 768; }
template <int V> constexpr int a_stage_bytes() { return 128 * Tile<V>::KS * 2; }
// Warps by role: the loader, the MMA issuer, producers from WARP0 on, then the epilogue.
// v = 6, 12: roles in whole warpgroups, between which registers move: 24 warps start with 80 registers a thread; the 12
// producers take 104, the epilogue keeps 64, loader and issuer 40: 12 x 104 + 8 x 64 + 4 x 40 = 24 x 80.  With 56 for the last two the
// epilogue spills its place in the scratch: FP16 results, v = 6, 4096 x 4096 at 512 tokens 60.5 against 59.4 us, 8192 x 8192 at 24 60.8 / 59.5.
// (16 producer warps with 96 registers fill the A ring no faster: the shared-memory pipe bounds.)
// v = 8: 20 warps with 96 registers each, five pairs of producers.  24 warps in six pairs spill some of the producers' state:
// 14336 x 4096 at 512 tokens, FP32 results, 82.2 against 80.1 us; 4096 x 14336 84.8 against 83.0; 8192 x 8192 at 333 79.7 / 77.6.
// v = 6, few tokens: 28 warps start with 72 registers: 20 x 80 + 4 x 64 + 4 x 40 = 28 x 72.
template <int V> constexpr bool split_registers() { return V != 8; }
template <int V, bool FEW> constexpr int epi_warp0() { return Tile<V, FEW>::WARP0 + Tile<V, FEW>::WARPS; }
template <int V, bool FEW> constexpr int gemm_threads() { return 32 * (epi_warp0<V, FEW>() + Tile<V, FEW>::EPI); }
template <bool FEW> constexpr int regs_producer() { return FEW ? 80 : 104; }
constexpr int REGS_EPILOGUE = 64, REGS_ISSUE = 40;

// where a table's rows come from
enum TableSource { TABLE_NONE = 0, TABLE_SHARED = 1, TABLE_GLOBAL = 2 };

// token rows of a scratch tile: whole pieces
__host__ __device__ __forceinline__ int scratch_rows(int tile_n) { return (tile_n + EPI_TOKENS - 1) / EPI_TOKENS * EPI_TOKENS; }

// How the units (k blocks of all tiles, tile by tile) are cut into one contiguous share per CTA.  Draining a tile costs a CTA
// about as much as `drain` k blocks, so the cuts are even on a line on which every tile is that much longer (a cut that
// falls into a tile's extra length is moved to the tile's end).  A v = 12 decoder layer of a 7B model at 512 tokens: 676 -> 617
// us.  whole_tiles: cuts only between tiles.
struct Shares {
    unsigned kb, len, workers, whole_tiles;      // k blocks of a tile; its length on the line, kb + drain
    unsigned per_tile;                           // not 0: that many workers for each tile, none works on two
    unsigned each, rest;                         // line (or tiles, or k blocks of a tile) per worker, and how many workers get one more
    __host__ __device__ unsigned begin(unsigned w) const        // first unit of worker w (w = workers: the end)
    {
        if (per_tile) {
            const unsigned tile = w / per_tile, part = w - tile * per_tile;
            return tile * kb + part * each + (part < rest ? part : rest);
        }
        const unsigned at = w * each + (w < rest ? w : rest);
        if (whole_tiles) return at * kb;
        const unsigned tile = at / len, off = at - tile * len;
        return tile * kb + (off < kb ? off : kb);
    }
    __host__ __device__ unsigned worker_of(unsigned u) const    // the worker whose share holds unit u
    {
        const unsigned tile = u / kb, at = whole_tiles ? tile : tile * len + (u - tile * kb);
        unsigned w = per_tile ? tile * per_tile + (u - tile * kb) / (each + 1) : at / (each + 1);
        while (w + 1 < workers && begin(w + 1) <= u) w++;
        return w;
    }
};

struct GemmParams {
    LayerView L;
    void *out;
    int B;
    int tiles_m, tiles_t, tile_n;   // row tiles, token tiles, tokens of a token tile (a multiple of 16)
    int n0;                         // tokens of the first MMA of a k step; the second takes tile_n - n0
    int kb_main, kb_total;          // k blocks of KS columns: main region, all
    Shares shares;       // how the (tile, k block) units are dealt out to the CTAs
    int b_stages;
    int cb1_shift, cb2_shift;       // log2 of the copies of a table in shared memory
    int cb1_bytes, cb2_bytes;
    int flag_order;      // split tiles: 1 = last piece stores and raises a flag, the others wait and add; 0 = all add
    int tma_out;         // FP32 output written by TMA store / reduce from shared memory (needs M % 4 == 0)
    int *status;         // workspace status word
    const float *bpart;  // [bias_parts][tiles_t * tile_n]: partial sums of x*b
    int bias_parts;
    int *tile_flags;     // [tiles][MAX_EPI_WARPS]: flag order: [tile][0] counts the epilogue warps that have stored the last
                         // piece; scratch: arrivals per epilogue warp
    float *scratch;      // [slots][4][scratch_rows(tile_n)][32] FP32 sums of split tiles, or null
    int slot_per_tile;   // a split tile's slot: 1 = its number, 0 = the worker that holds its first unit
    const uint8_t *xs;   // activation images, [tiles_t][kb_total * KS / 32][tile_n * 64 bytes]
    const uint8_t *tab1, *tab2;     // tables read from global memory: rows of 16 (v <= 8) or 32 bytes
};

// One launch: layer l is the work of CTAs [cta_begin[l], cta_begin[l + 1]).  (A launch of one layer has kernels of its own:
// parameters found by an index are loads instead of operands.  The maps are a parameter of their own for the same reason:
// their address is taken, and with them in one struct 17 tokens x 8192 columns took 26.5 us instead of 24.)
template <int NL>
struct OutMaps {
    CUtensorMap layer[NL], tail[NL];         // boxes of 32 rows; of the rows of a tile's last quarter, where it has fewer
};
template <int NL>
struct GemmLaunch {
    GemmParams layer[NL];
    int cta_begin[NL + 1];
    int n_layers;
};

// ---- PTX wrappers ----------------------------------------------------------------------------
// Bounded wait until *flag >= target (set by another CTA of this grid; all CTAs of the grid are resident).
__device__ __forceinline__ bool flag_wait(const int *flag, int target, volatile int *abort_flag, int *status)
{
    const long long t0 = clock64();
    unsigned spins = 0;
    while (true) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v >= target) return true;
        if ((++spins & 63u) == 0) {
            if (*abort_flag) return false;
            if ((unsigned long long)(clock64() - t0) > WAIT_LIMIT_CYCLES) {
                *abort_flag = 1;
                grid_dependency_wait();                  // the pre-pass clears the status word
                atomicExch(status, VPTQ_E_TIMEOUT);
                return false;
            }
        }
        __nanosleep(64);
    }
}

// kind::f16, FP16 x FP16 -> FP32, B K-major, M = 128, N = n; A MN-major or K-major
__device__ __forceinline__ uint32_t instr_desc(bool a_mn_major, int n)
{
    return (1u << 4) | ((a_mn_major ? 1u : 0u) << 15) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// (descriptors as two words: only the low one, which holds the address, changes from MMA to MMA)
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %6, 0;\n\t"
                 "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// TMA store / reduce-add of a [16 tokens][32 rows] FP32 box from shared memory into the output
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int x, int y, bool add)
{
    if (add)
        asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
    else
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// linear reduce-add of a staged piece into the scratch tile
__device__ __forceinline__ void bulk_add(float *dst, uint32_t src)
{
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;"
                 ::"l"(dst), "r"(src), "r"(EPI_BUF_BYTES) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void st_shared16(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint32_t hadd2_bits(uint32_t a, uint32_t b)
{
    const __half2 r = __hadd2(*reinterpret_cast<const __half2 *>(&a), *reinterpret_cast<const __half2 *>(&b));
    return *reinterpret_cast<const uint32_t *>(&r);
}

// One row of a table of V-component vectors as V / 2 words; the rows of a table in shared memory take 16 bytes, of one in
// global memory 16 (V <= 8) or 32.  No L1 allocation: the tensor core's operand reads share the L1 data path.
template <int V>
__device__ __forceinline__ void row_global(const uint8_t *tab, uint32_t e, uint32_t (&w)[V / 2])
{
    uint32_t r[8];
    if (V <= 8) {
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(tab + 16ull * e));
    } else {
        asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "l"(tab + 32ull * e));
    }
#pragma unroll
    for (int i = 0; i < V / 2; i++) w[i] = r[i];
}
template <int V>
__device__ __forceinline__ void row_shared(const uint4 *tab, uint32_t e, uint32_t (&w)[V / 2])
{
    const uint4 q = tab[e];
    const uint32_t r[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < V / 2; i++) w[i] = r[i < 4 ? i : 0];
}

// ---- pre-pass: xs = fp16(x * s) written as B images, partial sums of x * b per token, padded tables, and everything of the
//      workspace (and output) that has to start at zero.
// Image of (token tile, 32 columns): token row r of the tile, 16-byte chunk q (8 columns) at
//      (r / 8) * 512 + (r % 8) * 64 + ((q ^ ((r % 8) / 2)) * 16: the K-major 64-byte-swizzled operand layout.
// Block (g, y): tokens 8g .. 8g+7 of the padded range, every gridDim.y-th run of 8 images; a warp takes four tokens x two
// images (128 bytes of a row of x), a lane 8 columns of a token; tokens >= B and columns beyond a region are zeros. -------
constexpr int PRE_THREADS = 256;
constexpr long long PRE_ROWS_MIN = 1 << 20;      // activations of a launch

struct PrepassParams {
    LayerView L;
    const void *x;
    int B, tile_n;
    int img_main, img_total;        // 32-column images: main region, all
    uint8_t *xs;
    float *bpart;
    int *status;
    int *tile_flags; int n_flags;
    float *zero; long long n_zero;  // FP32 words to clear (a multiple of 4 unless the address is not 16-byte aligned)
    uint8_t *pad1, *pad2;           // null, or where the tables go with their rows padded to pad_bytes
    int pad_bytes;
};

// table [rows][v] -> rows of `pad` bytes (16 or 32), zero-filled
__device__ __forceinline__ void pad_table(uint8_t *dst, const __half *src, long long rows, int v, int pad, long long first, long long step)
{
    for (long long i = first; i < rows; i += step) {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(src + i * v);     // even v: rows are 4-byte aligned
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; k++) w[k] = 2 * k < v ? __ldg(p + k) : 0u;
        *reinterpret_cast<uint4 *>(dst + i * pad) = make_uint4(w[0], w[1], w[2], w[3]);
        if (pad == 32) *reinterpret_cast<uint4 *>(dst + i * pad + 16) = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

template <int NL>
struct PrepassLaunch {
    PrepassParams layer[NL];
};

// what has to start at zero, and the padded tables: thread tid of n_tid
__device__ __forceinline__ void prepass_clear(const PrepassParams &P, long long tid, long long n_tid)
{
    if (tid == 0) *P.status = 0;
    for (long long i = tid; i < P.n_flags; i += n_tid) P.tile_flags[i] = 0;
    if ((P.n_zero & 3) == 0) {
        for (long long i = tid; i < (P.n_zero >> 2); i += n_tid) reinterpret_cast<float4 *>(P.zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        for (long long i = tid; i < P.n_zero; i += n_tid) P.zero[i] = 0.f;
    }
    if (P.pad1) pad_table(P.pad1, P.L.c1, (long long)P.L.G * P.L.k1, P.L.v, P.pad_bytes, tid, n_tid);
    if (P.pad2) pad_table(P.pad2, P.L.c2, (long long)P.L.G * P.L.k2, P.L.v, P.pad_bytes, tid, n_tid);
}

// eight activations x their scales -> FP16 pairs; returns the sum of activation x bias
__device__ __forceinline__ float scale8(uint4 xq, uint4 sq, uint4 bq, int x_bf16, uint4 &out)
{
    const uint32_t xw[4] = {xq.x, xq.y, xq.z, xq.w}, sw[4] = {sq.x, sq.y, sq.z, sq.w}, bw[4] = {bq.x, bq.y, bq.z, bq.w};
    uint32_t o[4];
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float2 a = x_bf16 ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&xw[i]))
                                : __half22float2(*reinterpret_cast<const __half2 *>(&xw[i]));
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&sw[i]));
        const float2 h = __half22float2(*reinterpret_cast<const __half2 *>(&bw[i]));
        const __half2 y = __floats2half2_rn(a.x * f.x, a.y * f.y);
        o[i] = *reinterpret_cast<const uint32_t *>(&y);
        acc += a.x * h.x + a.y * h.y;
    }
    out = make_uint4(o[0], o[1], o[2], o[3]);
    return acc;
}
__device__ __forceinline__ uint4 pack8(const uint16_t (&e)[8])
{
    return make_uint4(e[0] | ((uint32_t)e[1] << 16), e[2] | ((uint32_t)e[3] << 16), e[4] | ((uint32_t)e[5] << 16), e[6] | ((uint32_t)e[7] << 16));
}

// words shifted down by `by` < 2^S places
template <int S, int NW>
__device__ __forceinline__ void shift_words(uint32_t (&w)[NW], int by)
{
#pragma unroll
    for (int b = S - 1; b >= 0; b--)
        if (by & (1 << b)) {
#pragma unroll
            for (int i = 0; i + (1 << b) < NW; i++) w[i] = w[i + (1 << b)];
        }
}
// Elements at .. at + 7 of p (16-byte aligned, len elements, zeros past them), which outlier columns push off 16-byte boundaries
__device__ __forceinline__ uint4 load8(const uint16_t *p, long long at, long long len)
{
    const int sh = (int)(at & 7);
    if (at - sh + (sh ? 16 : 8) <= len) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p + at - sh));
        if (sh == 0) return a;
        const uint4 b = __ldg(reinterpret_cast<const uint4 *>(p + at - sh + 8));
        uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        shift_words<2>(w, sh >> 1);
        const int h = 16 * (sh & 1);
        return make_uint4(__funnelshift_r(w[0], w[1], h), __funnelshift_r(w[1], w[2], h), __funnelshift_r(w[2], w[3], h), __funnelshift_r(w[3], w[4], h));
    }
    uint16_t e[8];
#pragma unroll
    for (int i = 0; i < 8; i++) e[i] = at + i < len ? __ldg(p + at + i) : (uint16_t)0;
    return pack8(e);
}
// input features of stored columns n .. n + 7
__device__ __forceinline__ void load_features(const LayerView &L, int n, int (&f)[8])
{
    const int sh = n & 3;
    if (n - sh + 12 <= L.N) {
        uint32_t w[12];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(L.perm + n - sh) + i);
            w[4 * i] = a.x; w[4 * i + 1] = a.y; w[4 * i + 2] = a.z; w[4 * i + 3] = a.w;
        }
        shift_words<2>(w, sh);
#pragma unroll
        for (int i = 0; i < 8; i++) f[i] = (int)(w[i] < (unsigned)L.N ? w[i] : (unsigned)(L.N - 1));
    } else {
#pragma unroll
        for (int i = 0; i < 8; i++) f[i] = in_col(L, n + i < L.N ? n + i : L.N - 1);
    }
}

// Layers with a stored column order: a block keeps T whole rows of x in shared memory and gathers from there, a lane 8
// columns for all T tokens.  2-byte gathers out of global memory take 32 L1 cycles per warp: 512 tokens x 11008 columns
// 36.6 us.  Below a million
// activations a block's rows are too many for its few columns (128 tokens x 4096: 28.6 us instead of 27.8 with the GEMM;
// 128 x 11008: 35.4 instead of 37.3, 512 x 11008: 64.6 instead of 79.8).
template <int T, int NL>
__global__ void __launch_bounds__(PRE_THREADS)
gemm_prepass_rows_kernel(const __grid_constant__ PrepassLaunch<NL> F)
{
    extern __shared__ __align__(16) uint16_t rows[];         // [T][N rounded up to 8]
    pdl_launch_dependents();
    const PrepassParams &P = F.layer[NL > 1 ? blockIdx.z : 0];
    const LayerView &L = P.L;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();          // the activations may be the previous kernel's output, and that kernel may use this workspace
    prepass_clear(P, ((long long)blockIdx.y * gridDim.x + blockIdx.x) * PRE_THREADS + threadIdx.x, (long long)gridDim.x * gridDim.y * PRE_THREADS);

    const int t0 = blockIdx.x * T, n_pad = (L.N + 7) / 8 * 8;
    for (int i = 0; i < T; i++) {
        const uint16_t *xr = reinterpret_cast<const uint16_t *>(P.x) + (long long)(t0 + i) * L.N;
        if (t0 + i >= P.B) {
            for (int n = 8 * threadIdx.x; n < n_pad; n += 8 * PRE_THREADS) *reinterpret_cast<uint4 *>(rows + i * n_pad + n) = make_uint4(0, 0, 0, 0);
        } else if ((L.N & 7) == 0) {
            for (int n = 8 * threadIdx.x; n < L.N; n += 8 * PRE_THREADS)
                *reinterpret_cast<uint4 *>(rows + i * n_pad + n) = __ldg(reinterpret_cast<const uint4 *>(xr + n));
        } else {
#pragma unroll 4
            for (int n = threadIdx.x; n < L.N; n += PRE_THREADS) rows[i * n_pad + n] = __ldg(xr + n);
        }
    }
    __syncthreads();

    const int tile = t0 / P.tile_n, row0 = t0 - tile * P.tile_n;          // (T divides tile_n)
    uint8_t *base_dst = P.xs + (long long)tile * P.img_total * (P.tile_n * 64);
    float acc[T];
#pragma unroll
    for (int i = 0; i < T; i++) acc[i] = 0.f;
    for (int ch = (blockIdx.y * (PRE_THREADS / 32) + warp) * 32 + lane; ch < P.img_total * 4; ch += gridDim.y * PRE_THREADS) {
        const int img = ch >> 2, q = ch & 3;
        const bool main_cols = img < P.img_main;
        const int c = (main_cols ? img : img - P.img_main) * IMG_COLS + q * 8;     // first column, counted in its region
        const int n_cols = main_cols ? L.Nc : L.n_out, base = main_cols ? L.n_out : 0;
        int f[8];
        load_features(L, base + c, f);
        uint4 sq = make_uint4(0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u), bq = make_uint4(0, 0, 0, 0);
        if (L.has_scale) {
            sq = load8(reinterpret_cast<const uint16_t *>(L.scale), base + c, L.N);
            bq = load8(reinterpret_cast<const uint16_t *>(L.bias), base + c, L.N);
        }
#pragma unroll
        for (int i = 0; i < T; i++) {
            uint16_t xe[8];
#pragma unroll
            for (int j = 0; j < 8; j++) xe[j] = c + j < n_cols ? rows[i * n_pad + f[j]] : (uint16_t)0;
            uint4 o;
            acc[i] += scale8(pack8(xe), sq, bq, L.x_bf16, o);
            const int row = row0 + i;
            *reinterpret_cast<uint4 *>(base_dst + (long long)img * (P.tile_n * 64) + (row >> 3) * B_SBO + (row & 7) * 64 + ((q ^ ((row & 7) >> 1)) << 4)) = o;
        }
    }
    __shared__ float red[PRE_THREADS / 32][T];
#pragma unroll
    for (int i = 0; i < T; i++) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        if (lane == 0) red[warp][i] = acc[i];
    }
    __syncthreads();
    if (threadIdx.x < T) {
        float a = 0.f;
        for (int w = 0; w < PRE_THREADS / 32; w++) a += red[w][threadIdx.x];
        P.bpart[(long long)blockIdx.y * gridDim.x * T + t0 + threadIdx.x] = a;
    }
}

template <int NL>
__global__ void __launch_bounds__(PRE_THREADS, 4)
gemm_prepass_kernel(const __grid_constant__ PrepassLaunch<NL> F)
{
    // the GEMM is launched as a programmatic dependent: its CTAs may become resident and run their set-up and
    // first centroid reads as soon as every block of this grid has started; whatever reads this kernel's
    // output waits for the whole grid (griddepcontrol.wait) first
    pdl_launch_dependents();
    const PrepassParams &P = F.layer[NL > 1 ? blockIdx.z : 0];
    const LayerView &L = P.L;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();          // the activations may be the previous kernel's output, and that kernel may use this workspace
    prepass_clear(P, ((long long)blockIdx.y * gridDim.x + blockIdx.x) * PRE_THREADS + threadIdx.x, (long long)gridDim.x * gridDim.y * PRE_THREADS);

    const int tok = 4 * (warp & 1) + (lane >> 3), q = lane & 3;
    const int tg = blockIdx.x * 8 + tok;                 // token of the padded range
    const int tile = tg / P.tile_n, row = tg - tile * P.tile_n;
    const int t = tg;                                    // token tiles are consecutive runs of tile_n tokens
    const bool live = t < P.B;
    uint8_t *dst = P.xs + (long long)tile * P.img_total * (P.tile_n * 64) + (row >> 3) * B_SBO + (row & 7) * 64 + ((q ^ ((row & 7) >> 1)) << 4);
    const uint16_t *xr = reinterpret_cast<const uint16_t *>(P.x) + (long long)(live ? t : 0) * L.N;
    const bool wide = L.perm == nullptr && (L.N & 7) == 0 && (L.n_out & 7) == 0;
    float acc = 0.f;
    constexpr int UNROLL = 2;
    const int stride = gridDim.y * 8;
    for (int img0 = blockIdx.y * 8 + (warp >> 1) * 2 + ((lane >> 2) & 1); img0 < P.img_total; img0 += UNROLL * stride) {
        uint4 xq[UNROLL], sq[UNROLL], bq[UNROLL];            // 8 activations as they are, 8 scales, 8 biases
#pragma unroll
        for (int u = 0; u < UNROLL; u++) {
            const int img = img0 + u * stride;
            const bool main_cols = img < P.img_main;
            const int c = (main_cols ? img : img - P.img_main) * IMG_COLS + q * 8;     // first column, counted in its region
            const int n_cols = img >= P.img_total ? 0 : main_cols ? L.Nc : L.n_out, base = main_cols ? L.n_out : 0;
            xq[u] = make_uint4(0, 0, 0, 0); sq[u] = make_uint4(0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u); bq[u] = xq[u];
            if (wide) {
                if (c < n_cols) {                                // (regions are multiples of 8 columns here)
                    if (live) xq[u] = __ldg(reinterpret_cast<const uint4 *>(xr + base + c));
                    if (L.has_scale) {
                        sq[u] = __ldg(reinterpret_cast<const uint4 *>(L.scale + base + c));
                        bq[u] = __ldg(reinterpret_cast<const uint4 *>(L.bias + base + c));
                    }
                }
            } else {
                uint16_t xe[8], se[8], be[8];
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const int n = base + c + i;
                    const bool in = c + i < n_cols;
                    xe[i] = (in && live) ? __ldg(xr + in_col(L, n)) : (uint16_t)0;
                    se[i] = (in && L.has_scale) ? __ldg(reinterpret_cast<const uint16_t *>(L.scale) + n) : (uint16_t)0x3C00;
                    be[i] = (in && L.has_scale) ? __ldg(reinterpret_cast<const uint16_t *>(L.bias) + n) : (uint16_t)0;
                }
                xq[u] = pack8(xe); sq[u] = pack8(se); bq[u] = pack8(be);
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; u++) {
            const int img = img0 + u * stride;
            if (img >= P.img_total) break;
            uint4 o;
            acc += scale8(xq[u], sq[u], bq[u], L.x_bf16, o);
            *reinterpret_cast<uint4 *>(dst + (long long)img * (P.tile_n * 64)) = o;
        }
    }
    __shared__ float red[PRE_THREADS / 64][8];
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((lane & 7) == 0) red[warp >> 1][tok] = acc;
    __syncthreads();
    if (threadIdx.x < 8) {
        float a = 0.f;
        for (int w = 0; w < PRE_THREADS / 64; w++) a += red[w][threadIdx.x];
        P.bpart[(long long)blockIdx.y * gridDim.x * 8 + blockIdx.x * 8 + threadIdx.x] = a;
    }
}

// ---- outlier columns (Sec. 3.2.3): value of stored column n < n_out at output row m -------------------------------------
__device__ __forceinline__ uint32_t outlier_bits(const LayerView &L, int m, int n)
{
    if (m >= L.M || n >= L.n_out) return 0u;
    const int r = m / L.v0;
    const int i = clamp_index(load_index(L.s0.ptr + (long long)r * L.s0.stride, n, L.s0.bits), L.k0);
    return __ldg(reinterpret_cast<const unsigned short *>(L.c0) + (long long)i * L.v0 + (m - r * L.v0));
}
// four output rows m0 .. m0+3 (m0 a multiple of 4) of column n as two words, for v0 = 4
__device__ __forceinline__ uint2 outlier_vector4(const LayerView &L, int m0, int n)
{
    // (a place outside reads the first one's entry and drops it: no branch, so that a caller's reads are in flight together)
    const bool in = m0 < L.M && n < L.n_out;
    const int i = clamp_index(load_index(L.s0.ptr + (long long)(in ? m0 >> 2 : 0) * L.s0.stride, in ? n : 0, L.s0.bits), L.k0);
    const uint2 c = __ldg(reinterpret_cast<const uint2 *>(L.c0) + i);
    return make_uint2(in ? c.x : 0u, in ? c.y : 0u);
}
// ... of columns 8g .. 8g + 7: the eight indices, then the eight centroids in flight at once (column by column, behind branches, a k block
// of them held the whole ring up: v = 6, gate+up and down of a 7B MLP at 16 tokens 116.5 -> 109.0 us)
__device__ __forceinline__ void outlier_vectors4(const LayerView &L, int m0, int g, uint2 (&a)[8])
{
    const int cols = m0 < L.M ? L.n_out : 0;
    uint32_t w[4];
    decode8(load_raw8(L.s0.ptr + (long long)(m0 < L.M ? m0 >> 2 : 0) * L.s0.stride, L.s0.stride, g, cols, L.s0.bits), L.s0.bits, L.k0, w);
#pragma unroll
    for (int j = 0; j < 8; j++) a[j] = __ldg(reinterpret_cast<const uint2 *>(L.c0) + ((w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu));
#pragma unroll
    for (int j = 0; j < 8; j++)
        if (8 * g + j >= cols) a[j] = make_uint2(0u, 0u);
}

// ---- the GEMM ------------------------------------------------------------------------------------
// PLAIN: no outlier columns, one group, 16-bit main and 8-bit residual indices: the same without the code for anything else in
// the producers' loop (14336 x 4096 at 512 tokens 81.3 -> 80.1 us, 4096 x 14336 84.3 -> 83.0, 5000 x 9000 at 150 48.2 -> 45.9)
template <int V, int T1, int T2, int NL, bool PLAIN, bool FEW>
__global__ void __launch_bounds__(gemm_threads<V, FEW>(), 1)
gemm_tcgen05_kernel(const __grid_constant__ OutMaps<NL> maps, const __grid_constant__ GemmLaunch<NL> F)
{
    // the layer this CTA works on, and its place among that layer's CTAs
    int li = 0;
    if (NL > 1)
        while (li + 1 < F.n_layers && (int)blockIdx.x >= F.cta_begin[li + 1]) li++;
    const GemmParams P = F.layer[NL > 1 ? li : 0];           // (a copy: through a reference gate+up of 11008 x 4096 at 300 tokens took 7 us more)
    const CUtensorMap &tmap_out = maps.layer[NL > 1 ? li : 0], &tmap_tail = maps.tail[NL > 1 ? li : 0];
    const unsigned worker = blockIdx.x - (NL > 1 ? F.cta_begin[li] : 0);
    constexpr bool MN = V == 8;                              // A layout
    using T = Tile<V, FEW>;
    constexpr int KS = T::KS, NV = T::NV, A_STAGES = T::A_STAGES, A_BYTES = a_stage_bytes<V>();
    constexpr int GROUPS = T::GROUPS, GROUP_WARPS = T::GROUP_WARPS, EPI_WARPS = T::EPI;
    constexpr int SUBS = KS / IMG_COLS, TILE_M = NV * V, W2 = V / 2;
    constexpr int A_SBO = MN ? 2048 : 1024, A_LBO = MN ? 1024 : 16;
    static_assert(A_STAGES >= GROUPS, "a producer group needs a stage of its own");
    constexpr int PRODUCER_WARP0 = T::WARP0, EPI_WARP0 = epi_warp0<V, FEW>(), GEMM_THREADS = gemm_threads<V, FEW>(), REGS_PRODUCER = regs_producer<FEW>();
    constexpr bool SPLIT_REGS = split_registers<V>();
    static_assert(GROUPS * GROUP_WARPS <= T::WARPS, "producer warps");
    static_assert(PRODUCER_WARP0 * REGS_ISSUE + T::WARPS * REGS_PRODUCER + EPI_WARPS * REGS_EPILOGUE <= 65536 / GEMM_THREADS / 8 * 8 * (GEMM_THREADS / 32) || !SPLIT_REGS,
                  "a split takes no more than the launch has");
    static_assert(!SPLIT_REGS || (PRODUCER_WARP0 % 4 == 0 && EPI_WARP0 % 4 == 0 && EPI_WARPS % 4 == 0), "whole warpgroups");
    extern __shared__ __align__(1024) uint8_t sm[];          // swizzled operand stages need 1024-byte alignment
    const LayerView &L = P.L;
    const uint32_t base = smem_addr(sm);
    if (base & 1023u) {                                      // (every thread of the grid answers alike)
        grid_dependency_wait();
        if (threadIdx.x == 0) atomicExch(P.status, VPTQ_E_UNSUPPORTED);
        return;
    }
    const int b_bytes = P.tile_n * 64, b_stages = P.b_stages;
    const uint32_t sA = base;
    const uint32_t sB = sA + A_STAGES * A_BYTES;
    // Output staging, EPI_WARPS x 2 x 2 KB: before the tables, whose sizes are multiples of 16 bytes only, since a tensor copy reads
    // shared memory from a multiple of 128.
    const uint32_t sEpi = sB + b_stages * b_bytes;
    static_assert(A_BYTES % 1024 == 0 && EPI_BUF_BYTES % 128 == 0, "a piece begins on a multiple of 128 bytes (a stage of B is tile_n / 16 KB)");
    uint8_t *cb1_ptr = sm + A_STAGES * A_BYTES + b_stages * b_bytes + EPI_WARPS * 2 * EPI_BUF_BYTES;
    uint8_t *cb2_ptr = cb1_ptr + P.cb1_bytes;
    float *bias = reinterpret_cast<float *>(cb2_ptr + P.cb2_bytes);       // [tile_n] bias terms of the token tile
    uint64_t *bars = reinterpret_cast<uint64_t *>(bias + MAX_TILE_N);   // fullA[] emptyA[] fullB[] emptyB[] accum_full accum_empty
    const uint32_t bar0 = smem_addr(bars);
    auto bar_fullA = [&](int s) { return bar0 + 8u * s; };
    auto bar_emptyA = [&](int s) { return bar0 + 8u * (A_STAGES + s); };
    auto bar_fullB = [&](int s) { return bar0 + 8u * (2 * A_STAGES + s); };
    auto bar_emptyB = [&](int s) { return bar0 + 8u * (2 * A_STAGES + MAX_B_STAGES + s); };
    constexpr int N_RING_BARS = 2 * A_STAGES + 2 * MAX_B_STAGES;
    // accumulators: two sets of them, which the segments take in turn, where they fit TMEM
    const int two = P.tile_n <= MAX_TILE_N / 2;
    auto acc_set = [&](int seg) { return seg & two; };
    auto acc_parity = [&](int seg) { return (uint32_t)(seg >> two) & 1u; };
    auto bar_accum_full = [&](int set) { return bar0 + 8u * (N_RING_BARS + set); };
    auto bar_accum_empty = [&](int set) { return bar0 + 8u * (N_RING_BARS + 2 + set); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + N_RING_BARS + 4);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < A_STAGES; s++) {
            mbar_init(bar_fullA(s), GROUP_WARPS);       // one arrival per producer warp of a group
            mbar_init(bar_emptyA(s), 1);                // tcgen05.commit
        }
        for (int s = 0; s < b_stages; s++) {
            mbar_init(bar_fullB(s), 1);       // the expect_tx arrival
            mbar_init(bar_emptyB(s), 1);      // tcgen05.commit
        }
        for (int i = 0; i < 2; i++) { mbar_init(bar_accum_full(i), 1); mbar_init(bar_accum_empty(i), EPI_WARPS); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // tables -> shared memory as 16-byte rows (all threads; the loads of 4 rows are issued before the first store)
    auto stage_table = [&](uint8_t *dst, const __half *src, int k, int shift) {
        uint4 *d = reinterpret_cast<uint4 *>(dst);
        const int n = k << shift;
        for (int i0 = threadIdx.x; i0 < n; i0 += 4 * GEMM_THREADS) {
            uint4 row[4];
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (i0 + u * GEMM_THREADS < n) row[u] = load_centroid_row(src, (i0 + u * GEMM_THREADS) >> shift, V);
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (i0 + u * GEMM_THREADS < n) d[i0 + u * GEMM_THREADS] = row[u];
        }
    };
    if (T1 == TABLE_SHARED) stage_table(cb1_ptr, L.c1, L.k1, P.cb1_shift);
    if (T2 == TABLE_SHARED) stage_table(cb2_ptr, L.c2, L.k2, P.cb2_shift);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // this CTA's share of the (tile, k block) units
    const unsigned u_begin = P.shares.begin(worker), u_end = P.shares.begin(worker + 1);
    // A segment is the part of one tile inside the share: k blocks [kb0, kb1) of tile `tile`.
#define FOR_EACH_SEGMENT                                                                          \
    for (unsigned u = u_begin; u < u_end && ok; u += (unsigned)(kb1 - kb0))                         \
        if (tile = (int)(u / (unsigned)P.kb_total), kb0 = (int)(u % (unsigned)P.kb_total),          \
            kb1 = (int)min((unsigned)P.kb_total, kb0 + (u_end - u)), true)
    int tile = 0, kb0 = 0, kb1 = 0;
    bool ok = true;

    if (warp < PRODUCER_WARP0) {
        if (SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ISSUE));
        // ================= bulk copies: B ring =================
        if (warp == 0 && lane == 0) {
            grid_dependency_wait();                              // the images are the pre-pass's output
            int it = 0;
            int s = 0;
            uint32_t ps = 1;                                     // ring position, parity to wait for
            FOR_EACH_SEGMENT {
                const uint8_t *src = P.xs + ((long long)(tile / P.tiles_m) * P.kb_total * SUBS + (long long)kb0 * SUBS) * b_bytes;
                for (int i = 0; i < (kb1 - kb0) * SUBS; i++, it++, src += b_bytes) {
                    if (!(ok = mbar_wait(bar_emptyB(s), ps, abort_flag, P.status))) break;
                    mbar_expect_tx(bar_fullB(s), b_bytes);
                    bulk_load(sB + s * b_bytes, src, b_bytes, bar_fullB(s));
                    if (++s == b_stages) { s = 0; ps ^= 1u; }
                }
            }
            if (!ok) {
                // abandoned: give copies still in flight a bounded time to land before the CTA exits
                const int first = it > b_stages ? it - b_stages : 0;
                for (int j = first; j < it; j++) {
                    const long long t0c = clock64();
                    while (!mbar_try(bar_fullB(j % b_stages), (j / b_stages) & 1) && clock64() - t0c < 20000000ll) {}
                }
            }
        }
        // ================= MMA issue =================
        if (warp == 1) {
            // The whole warp runs this loop, converged, and an elected lane issues (see elect_one); the loop is a serial
            // chain, so it is kept short: descriptors are a constant plus a stage offset, stage numbers and parities are
            // running counters.
            const uint64_t adesc0 = make_smem_desc(sA, A_LBO, A_SBO, LAYOUT_SW128);
            const uint64_t bdesc0 = make_smem_desc(sB, 16, B_SBO, LAYOUT_SW64);
            const uint32_t a_lo0 = (uint32_t)adesc0, a_hi = (uint32_t)(adesc0 >> 32), b_lo0 = (uint32_t)bdesc0, b_hi = (uint32_t)(bdesc0 >> 32);
            const int n1 = P.tile_n - P.n0;
            const uint32_t id0 = instr_desc(MN, P.n0), id1 = instr_desc(MN, n1);
            const uint32_t bh = (uint32_t)((P.n0 * 64) >> 4);        // second MMA's token rows
            const uint32_t tmem_all = __shfl_sync(0xffffffffu, tmem_base, 0);
            int sa = 0, sb = 0;                                      // ring positions and their phase parities
            uint32_t pa = 0, pb = 0, gave_up = 0;
            int seg_no = 0;
            FOR_EACH_SEGMENT {
                // the accumulators must have been drained by the epilogues of the segment that had them before
                mbar_wait_uniform(bar_accum_empty(acc_set(seg_no)), acc_parity(seg_no) ^ 1u, gave_up);
                tc_fence_after();
                const uint32_t tmem0 = tmem_all + (uint32_t)(acc_set(seg_no) * (MAX_TILE_N / 2)), tmem1 = tmem0 + (uint32_t)P.n0;
                uint32_t acc = 0;
                for (int kb = kb0; kb < kb1; kb++) {
                    mbar_wait_uniform(bar_fullA(sa), pa, gave_up);
                    // (stage offsets only touch the 14-bit address field of the descriptors: no carry)
                    const uint32_t a_lo = a_lo0 + (uint32_t)((sa * A_BYTES) >> 4);
#pragma unroll
                    for (int sub = 0; sub < SUBS; sub++) {
                        mbar_wait_uniform(bar_fullB(sb), pb, gave_up);
                        const uint32_t b_lo = b_lo0 + (uint32_t)((sb * b_bytes) >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int h = 0; h < 2; h++) {                // k = 16 at a time
                                // MN-major: two 8-column groups further; K-major: 32 bytes further inside the swizzled row
                                const uint32_t ak = a_lo + (uint32_t)(MN ? (h * 2 * A_SBO) >> 4 : (sub * 2 + h) * 2);
                                const uint32_t bk = b_lo + (uint32_t)(h * 2);
                                umma_f16(tmem0, ak, a_hi, bk, b_hi, id0, acc);
                                if (n1) umma_f16(tmem1, ak, a_hi, bk + bh, b_hi, id1, acc);
                                acc = 1;
                            }
                            umma_commit(bar_emptyB(sb));      // the stages may be refilled once these MMAs have read them
                            if (sub == SUBS - 1) umma_commit(bar_emptyA(sa));
                        }
                        acc = 1;
                        if (++sb == b_stages) { sb = 0; pb ^= 1u; }
                    }
                    if (++sa == A_STAGES) { sa = 0; pa ^= 1u; }
                }
                if (__any_sync(0xffffffffu, gave_up != 0)) {         // some wait ran out: what was issued is in bounds and worthless
                    *abort_flag = 1;
                    if (lane == 0) { grid_dependency_wait(); atomicExch(P.status, VPTQ_E_TIMEOUT); }
                    ok = false;
                } else if (elect_one()) {
                    umma_commit(bar_accum_full(acc_set(seg_no)));                     // accumulators complete
                }
                __syncwarp();
                seg_no++;
            }
        }
    } else if (warp < EPI_WARP0) {
        // ================= dequant producers: A tiles =================
        if (SPLIT_REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_PRODUCER));
        const int pw = warp - PRODUCER_WARP0, group = pw / GROUP_WARPS, wi = pw % GROUP_WARPS;
        // v = 8: lane = (row chunk within the 64-row half `wi`, 8-column group of 4); else lane = (vector row of 4, group of 8)
        const int vr = MN ? 8 * wi + (lane & 7) : 4 * wi + (lane >> 3);         // vector row within the tile
        const int cg = MN ? lane >> 3 : lane & 7;
        const uint4 *cb1 = reinterpret_cast<const uint4 *>(cb1_ptr) + (lane & ((1 << P.cb1_shift) - 1));
        const uint4 *cb2 = reinterpret_cast<const uint4 *>(cb2_ptr) + (lane & ((1 << P.cb2_shift) - 1));
        const int bits1 = PLAIN ? 16 : L.s1.bits, bits2 = PLAIN ? 8 : L.s2.bits;
        if (group >= GROUPS) ok = false;                     // a warp beyond the last whole group has no work
        bool waited = false;                                 // padded tables are the pre-pass's output
        int it0 = 0;                                         // k blocks of earlier segments
        FOR_EACH_SEGMENT {
            const int mt = tile % P.tiles_m;
            const int vrow = mt * NV + vr;
            const bool row_ok = vr < NV && vrow < L.R;
            const uint8_t *row1 = L.s1.ptr + (long long)(row_ok ? vrow : 0) * L.s1.stride;
            const uint8_t *row2 = T2 ? L.s2.ptr + (long long)(row_ok ? vrow : 0) * L.s2.stride : nullptr;
            // this group's k blocks of the segment: those whose running number is = group (mod GROUPS)
            int kb = kb0 + ((group - it0 % GROUPS) + GROUPS) % GROUPS;
            // a1: packed indices of 8 columns; the next visit's are loaded one visit ahead (a column group beyond the main
            // columns reads as zeros)
            const int limit = row_ok ? L.Nc : 0;
            uint4 raw1 = make_uint4(0, 0, 0, 0), raw2 = make_uint4(0, 0, 0, 0);
            if (kb < kb1) {
                raw1 = load_raw8(row1, L.s1.stride, kb * (KS / 8) + cg, limit, bits1);
                if (T2) raw2 = load_raw8(row2, L.s2.stride, kb * (KS / 8) + cg, limit, bits2);
            }
            if ((T1 == TABLE_GLOBAL || T2 == TABLE_GLOBAL) && V != 8 && !waited) { grid_dependency_wait(); waited = true; }
            for (; kb < kb1; kb += GROUPS) {
                const int it = it0 + (kb - kb0);
                const int s = it % A_STAGES;
                const uint32_t stage = sA + s * A_BYTES;
                if (!PLAIN && kb >= P.kb_main) {
                    // a5: outlier columns; few k blocks, written element by element
                    ok = __all_sync(0xffffffffu, mbar_wait(bar_emptyA(s), ((it / A_STAGES) & 1) ^ 1, abort_flag, P.status));
                    if (!ok) break;
                    const int n0c = (kb - P.kb_main) * KS, m_tile = mt * TILE_M;
                    const bool quads = L.v0 == 4 && TILE_M % 4 == 0;
                    if (MN) {
                        // (chunk of 8 rows, column): 16 x 32 of them
                        for (int i = wi * 32 + lane; i < 16 * KS; i += GROUP_WARPS * 32) {
                            const int ch = i & 15, k = i >> 4, m0 = m_tile + 8 * ch;
                            uint32_t w[4];
                            if (quads) {
                                const uint2 a = outlier_vector4(L, m0, n0c + k), b = outlier_vector4(L, m0 + 4, n0c + k);
                                w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
                            } else {
#pragma unroll
                                for (int j = 0; j < 4; j++) w[j] = outlier_bits(L, m0 + 2 * j, n0c + k) | (outlier_bits(L, m0 + 2 * j + 1, n0c + k) << 16);
                            }
                            st_shared16(stage + (k >> 3) * 2048 + (ch >> 3) * 1024 + (k & 7) * 128 + (((ch & 7) ^ (k & 7)) << 4), w[0], w[1], w[2], w[3]);
                        }
                    } else if (quads) {
                        // (4 rows, 8 columns): 30 x 8 of them, turned into rows
                        for (int i = wi * 32 + lane; i < (TILE_M / 4) * 8; i += GROUP_WARPS * 32) {
                            const int q = i & 7, m = (i >> 3) * 4;
                            uint2 a[8];
                            outlier_vectors4(L, m_tile + m, (n0c >> 3) + q, a);
#pragma unroll
                            for (int r = 0; r < 4; r++) {
                                uint32_t w[4];
#pragma unroll
                                for (int j = 0; j < 4; j++) {
                                    const uint32_t lo = r < 2 ? a[2 * j].x : a[2 * j].y, hi = r < 2 ? a[2 * j + 1].x : a[2 * j + 1].y;
                                    w[j] = __byte_perm(lo, hi, (r & 1) ? 0x7632 : 0x5410);
                                }
                                st_shared16(stage + ((m + r) >> 3) * 1024 + ((m + r) & 7) * 128 + ((q ^ ((m + r) & 7)) << 4), w[0], w[1], w[2], w[3]);
                            }
                        }
                    } else {
                        for (int i = wi * 32 + lane; i < TILE_M * 8; i += GROUP_WARPS * 32) {
                            const int q = i & 7, m = i >> 3;
                            uint32_t w[4];
#pragma unroll
                            for (int j = 0; j < 4; j++)
                                w[j] = outlier_bits(L, m_tile + m, n0c + q * 8 + 2 * j) | (outlier_bits(L, m_tile + m, n0c + q * 8 + 2 * j + 1) << 16);
                            st_shared16(stage + (m >> 3) * 1024 + (m & 7) * 128 + ((q ^ (m & 7)) << 4), w[0], w[1], w[2], w[3]);
                        }
                    }
                } else {
                    const int col0 = kb * KS + 8 * cg;
                    // (a lane without a row or columns holds zeros and so reads entry 0 along with the others)
                    uint32_t w1[4], w2[4] = {0, 0, 0, 0};
                    decode8(raw1, bits1, L.k1, w1);
                    if (T2) decode8(raw2, bits2, L.k2, w2);
                    if (kb + GROUPS < kb1) {
                        raw1 = load_raw8(row1, L.s1.stride, (kb + GROUPS) * (KS / 8) + cg, limit, bits1);
                        if (T2) raw2 = load_raw8(row2, L.s2.stride, (kb + GROUPS) * (KS / 8) + cg, limit, bits2);
                    }
                    // Sec. 3.1: a column's tables are those of its group
                    uint32_t g = 0;
                    int g_next = 0x7fffffff;
                    // (asked in the PLAIN form too: the test between the columns keeps their reads in turn.  Without it the compiler
                    // puts all main reads before the residual ones, 8192 x 8192 at 333 tokens, FP16 results: 90.4 us against 87.3)
                    if ((T1 == TABLE_GLOBAL || T2 == TABLE_GLOBAL) && L.G > 1) { g = (uint32_t)(col0 / L.cpg); g_next = (int)(g + 1) * L.cpg; }
                    auto next_group = [&](int j) { if (col0 + j >= g_next && (int)g + 1 < L.G) { g++; g_next += L.cpg; } };
                    auto id = [&](const uint32_t (&w)[4], int j) { return (w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu; };
                    uint32_t cw[8][W2];
                    if (V <= 8 && !(FEW && V == 6)) {
                        // a3: main centroids, a4: residual centroids; all reads in flight before the wait (they do not touch the stage)
                        uint32_t rv[8][W2];
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            next_group(j);
                            if (T1 == TABLE_SHARED) row_shared<V>(cb1, id(w1, j) << P.cb1_shift, cw[j]);
                            else row_global<V>(P.tab1, g * (uint32_t)L.k1 + id(w1, j), cw[j]);
                            if (T2 == TABLE_SHARED) row_shared<V>(cb2, id(w2, j) << P.cb2_shift, rv[j]);
                            else if (T2 == TABLE_GLOBAL) row_global<V>(P.tab2, g * (uint32_t)L.k2 + id(w2, j), rv[j]);
                        }
                        // the whole warp takes the same decision: the stores below end in a warp-wide barrier
                        ok = __all_sync(0xffffffffu, mbar_wait(bar_emptyA(s), ((it / A_STAGES) & 1) ^ 1, abort_flag, P.status));
                        if (!ok) break;
                        if (T2) {            // sum in FP16 (one rounding of 2^-11)
#pragma unroll
                            for (int j = 0; j < 8; j++)
#pragma unroll
                                for (int i = 0; i < W2; i++) cw[j][i] = hadd2_bits(cw[j][i], rv[j][i]);
                        }
                    } else {
                        // v = 12: two 32-byte rows per column; few tokens: more warps with fewer registers.  Four columns in flight at a time
#pragma unroll
                        for (int j0 = 0; j0 < 8; j0 += 4) {
                            uint32_t rv[4][W2];
#pragma unroll
                            for (int u = 0; u < 4; u++) {
                                const int j = j0 + u;
                                next_group(j);
                                if (T1 == TABLE_SHARED) row_shared<V>(cb1, id(w1, j) << P.cb1_shift, cw[j]);
                                else row_global<V>(P.tab1, g * (uint32_t)L.k1 + id(w1, j), cw[j]);
                                if (T2 == TABLE_SHARED) row_shared<V>(cb2, id(w2, j) << P.cb2_shift, rv[u]);
                                else if (T2 == TABLE_GLOBAL) row_global<V>(P.tab2, g * (uint32_t)L.k2 + id(w2, j), rv[u]);
                            }
                            if (T2) {
#pragma unroll
                                for (int u = 0; u < 4; u++)
#pragma unroll
                                    for (int i = 0; i < W2; i++) cw[j0 + u][i] = hadd2_bits(cw[j0 + u][i], rv[u][i]);
                            }
                        }
                        ok = __all_sync(0xffffffffu, mbar_wait(bar_emptyA(s), ((it / A_STAGES) & 1) ^ 1, abort_flag, P.status));
                        if (!ok) break;
                    }
                    if (col0 + 8 > L.Nc) {
#pragma unroll
                        for (int j = 0; j < 8; j++)
                            if (col0 + j >= L.Nc)
#pragma unroll
                                for (int i = 0; i < W2; i++) cw[j][i] = 0u;
                    }
                    if (MN) {
                        const uint32_t dst0 = stage + cg * 2048 + wi * 1024;
#pragma unroll
                        for (int j = 0; j < 8; j++)
                            st_shared16(dst0 + j * 128 + (((lane & 7) ^ j) << 4), cw[j][0], cw[j][1], cw[j][2], cw[j][W2 - 1]);
                    } else if (vr < NV) {
                        // 8 columns x V rows -> V rows of 8 columns
#pragma unroll
                        for (int r = 0; r < V; r++) {
                            const int m = vr * V + r;
                            uint32_t w[4];
#pragma unroll
                            for (int j = 0; j < 4; j++) w[j] = __byte_perm(cw[2 * j][r >> 1], cw[2 * j + 1][r >> 1], (r & 1) ? 0x7632 : 0x5410);
                            st_shared16(stage + (m >> 3) * 1024 + (m & 7) * 128 + ((cg ^ (m & 7)) << 4), w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> visible to the MMA
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_fullA(s));
            }
            it0 += kb1 - kb0;
        }
    } else {
        // ============ epilogue: two warps per TMEM lane quarter (few tokens: one), taking turns at chunks of 32 tokens ============
        if (SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_EPILOGUE));
        const int ew = warp - EPI_WARP0, h = ew >> 2;
        const int q = warp & 3;                                  // TMEM lane quarter this warp may read
        const int padded_b = P.tiles_t * P.tile_n;
        int seg_no = 0, bias_tile = -1;
        unsigned piece = 0;                                      // staged pieces so far, over all segments: the buffers alternate
        grid_dependency_wait();                                  // bias terms, flags and cleared sums come from the pre-pass
        FOR_EACH_SEGMENT {
            const int mt = tile % P.tiles_m, tt = tile / P.tiles_m;
            const int t0 = tt * P.tile_n;
            const int m = mt * TILE_M + 32 * q + lane;
            const bool m_ok = 32 * q + lane < TILE_M && m < L.M;
            const int t_cnt = min(P.tile_n, P.B - t0);
            if (tt != bias_tile) {
                // the token tile's bias terms: the parts in order (a fixed order, whoever adds)
                asm volatile("bar.sync 1, %0;" ::"r"(EPI_WARPS * 32) : "memory");
                for (int t = ew * 32 + lane; t < P.tile_n; t += EPI_WARPS * 32) {
                    float a = 0.f;
#pragma unroll 8
                    for (int c = 0; c < P.bias_parts; c++) a += __ldg(P.bpart + (long long)c * padded_b + t0 + t);
                    bias[t] = a;
                }
                asm volatile("bar.sync 1, %0;" ::"r"(EPI_WARPS * 32) : "memory");
                bias_tile = tt;
            }
            // a split tile: the piece with the last k blocks stores and announces it, the others add afterwards
            const bool split = kb0 != 0 || kb1 != P.kb_total;
            const bool to_scratch = split && P.scratch != nullptr;
            const bool add = P.flag_order ? kb1 != P.kb_total : split;
            const bool announce = P.flag_order && kb0 != 0 && kb1 == P.kb_total;
            int pieces = 0, slot = tile;                     // shares that hold some of the tile (worked out while the MMAs run)
            if (to_scratch) {
                const unsigned first_u = (unsigned)tile * P.kb_total, end_u = first_u + P.kb_total;
                unsigned at = 0, w = P.shares.worker_of(first_u);
                // (that worker's share ends inside this tile, so no other split tile begins in it, and it is not the last one)
                if (!P.slot_per_tile) slot = (int)w;
                for (; at < end_u; w++) {
                    const unsigned next = P.shares.begin(w + 1);
                    pieces += next > at;                                     // (an empty share holds nothing)
                    at = next;
                }
            }
            ok = __all_sync(0xffffffffu, mbar_wait(bar_accum_full(acc_set(seg_no)), acc_parity(seg_no), abort_flag, P.status));
            if (!ok) break;
            tc_fence_after();
            if (add && P.flag_order) {
                ok = __all_sync(0xffffffffu, lane != 0 || flag_wait(P.tile_flags + tile * MAX_EPI_WARPS, EPI_WARPS, abort_flag, P.status));
                if (!ok) break;
                asm volatile("fence.proxy.async;" ::: "memory");     // the reduce-adds below go through the async proxy
            }
            const uint32_t ebuf = sEpi + (uint32_t)(ew * 2 * EPI_BUF_BYTES);
            const int m0 = mt * TILE_M + 32 * q;
            // A 120-row tile leaves 8 lanes of the last quarter unused, and a box of the output must not touch the next tile's rows:
            // that quarter has a map with boxes of 24 rows.  (Stored and added element by element, it held the others up:
            // 4096 x 4096 at 512 tokens, FP32 results, v = 6 61.8 us instead of 47.4, v = 12 59.1 instead of 48.0.)
            // (a quarter past the last row stages nothing: a piece without a copy would break the count of copies in flight)
            const bool box = P.tma_out && m0 < L.M;
            const bool tail = TILE_M < 128 && q == 3;
            float *sc = to_scratch ? P.scratch + ((long long)slot * 4 + q) * scratch_rows(P.tile_n) * 32 : nullptr;
            for (int c1 = EPI_TOKENS * h; c1 < t_cnt; c1 += EPI_WARPS / 4 * EPI_TOKENS) {
                uint32_t r[EPI_TOKENS];
                tmem_ld32(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc_set(seg_no) * (MAX_TILE_N / 2) + c1), r);
                if (kb0 == 0) {
                    const float4 *b4 = reinterpret_cast<const float4 *>(bias + c1);
#pragma unroll
                    for (int j = 0; j < EPI_TOKENS / 4; j++) {
                        const float4 bv = b4[j];
                        r[4 * j] = __float_as_uint(__uint_as_float(r[4 * j]) + bv.x);
                        r[4 * j + 1] = __float_as_uint(__uint_as_float(r[4 * j + 1]) + bv.y);
                        r[4 * j + 2] = __float_as_uint(__uint_as_float(r[4 * j + 2]) + bv.z);
                        r[4 * j + 3] = __float_as_uint(__uint_as_float(r[4 * j + 3]) + bv.w);
                    }
                }
                if (box || to_scratch) {
                    // through shared memory: a warp stages a [16][32] piece (lane = output row: conflict free) and one
                    // lane hands it to the copy engine (store or reduce-add); two staging buffers per warp, so the copy of
                    // one piece overlaps the next.  The buffer written two pieces ago must have been read by its copy.
#pragma unroll
                    for (int p = 0; p < EPI_TOKENS / PIECE_TOKENS; p++, piece++) {
                        const int c2 = c1 + p * PIECE_TOKENS;
                        if (c2 >= t_cnt) break;
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        __syncwarp();
                        const uint32_t buf = ebuf + (piece & 1u) * EPI_BUF_BYTES;
#pragma unroll
                        for (int j = 0; j < PIECE_TOKENS; j++)
                            if (!(tail && box) || lane < TILE_M - 96)
                                asm volatile("st.shared.b32 [%0], %1;" ::"r"(buf + j * (tail && box ? (TILE_M - 96) * 4u : 128u) + lane * 4u), "r"(r[p * PIECE_TOKENS + j]) : "memory");
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) {
                            if (to_scratch) bulk_add(sc + c2 * 32, buf);
                            else tma_store_2d(tail ? &tmap_tail : &tmap_out, buf, m0, t0 + c2, add);
                        }
                    }
                } else if (m_ok) {
                    const int nt = min(EPI_TOKENS, t_cnt - c1);                // tokens of this chunk that exist
                    const long long o0 = (long long)(t0 + c1) * L.M + m;
                    // (`add` does not come here: pieces of a tile meet in the scratch or in boxes.  Without it ptxas does worse by the rest: v = 6, FP32
                    // results, 3757 + 939 rows x 3757 at 333 tokens 59.6 -> 62.3 us, 1299 + 324 x 1299 at 65 18.9 -> 20.0; with a loop a type 62.9, 20.0.)
                    if (add) {
#pragma unroll
                        for (int j = 0; j < EPI_TOKENS; j++)
                            if (j < nt) atomicAdd(reinterpret_cast<float *>(P.out) + o0 + (long long)j * L.M, __uint_as_float(r[j]));
                    } else {
#pragma unroll
                        for (int j = 0; j < EPI_TOKENS; j++)
                            if (j < nt) store_out(P.out, o0 + (long long)j * L.M, __uint_as_float(r[j]), L.out_dtype);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_accum_empty(acc_set(seg_no)));
            if (announce) {
                // this warp's part of the tile is in memory before the flag counts it
                if (lane == 0 && P.tma_out) {
                    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                    asm volatile("fence.proxy.async;" ::: "memory");
                }
                __threadfence();
                __syncwarp();
                if (lane == 0) atomicAdd(P.tile_flags + tile * MAX_EPI_WARPS, 1);
            }
            if (to_scratch) {
                // count this warp's part in; the CTA that finds all pieces counted converts and stores the part
                int before = 0;
                if (lane == 0) {
                    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                    asm volatile("fence.proxy.async;" ::: "memory");
                    __threadfence();
                    before = atomicAdd(P.tile_flags + tile * MAX_EPI_WARPS + ew, 1);
                    __threadfence();
                }
                before = __shfl_sync(0xffffffffu, before, 0);
                if (before == pieces - 1) {
                    // eight 512-byte reads of a warp in flight: with four, 4096 x 4096 (v = 8) at 512 tokens 47.4 us instead of 45.8; the form
                    // of 72 registers keeps four (14336 x 4096 at 16 tokens 49.2 / 50.3)
                    constexpr int LOADS = SPLIT_REGS && FEW ? 4 : 8;
                    const int rq = 4 * (lane & 7), mq = m0 + rq;              // this lane's four rows
                    const bool rows4 = 32 * q + rq + 4 <= TILE_M && mq + 4 <= L.M && (L.M & 3) == 0;
                    for (int c1 = EPI_TOKENS * h; c1 < t_cnt; c1 += EPI_WARPS / 4 * EPI_TOKENS)
#pragma unroll
                    for (int c2 = c1; c2 < c1 + EPI_TOKENS; c2 += 4 * LOADS) {
                        float4 v[LOADS];
#pragma unroll
                        for (int i = 0; i < LOADS; i++) v[i] = __ldcg(reinterpret_cast<const float4 *>(sc + (c2 + 4 * i + (lane >> 3)) * 32 + rq));
#pragma unroll
                        for (int i = 0; i < LOADS; i++) {
                            const int t = c2 + 4 * i + (lane >> 3);
                            if (t >= t_cnt) continue;
                            const long long o = (long long)(t0 + t) * L.M + mq;
                            if (rows4 && L.out_dtype == VPTQ_DTYPE_FP16) {
                                __half2 p[2] = {__floats2half2_rn(v[i].x, v[i].y), __floats2half2_rn(v[i].z, v[i].w)};
                                *reinterpret_cast<uint2 *>(reinterpret_cast<__half *>(P.out) + o) = *reinterpret_cast<const uint2 *>(p);
                            } else if (rows4 && L.out_dtype == VPTQ_DTYPE_BF16) {
                                __nv_bfloat162 p[2] = {__floats2bfloat162_rn(v[i].x, v[i].y), __floats2bfloat162_rn(v[i].z, v[i].w)};
                                *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(P.out) + o) = *reinterpret_cast<const uint2 *>(p);
                            } else {
                                const float e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
                                for (int k = 0; k < 4; k++)
                                    if (32 * q + rq + k < TILE_M && mq + k < L.M) store_out(P.out, o + k, e[k], L.out_dtype);
                            }
                        }
                    }
                }
            }
            seg_no++;
        }
        // the staging buffers must outlive the copies that read them, the copies must land before the end
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
#undef FOR_EACH_SEGMENT

    // ---- teardown: everybody meets, then the allocating warp frees TMEM ---------------
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// ---- host side ----------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

struct GemmPlan {
    int t1, t2;                      // TableSource of the main and the residual table
    Shares shares;
    int tiles_m, tiles_t, tile_n, n0, ks, kb_main, kb_total, grid, any_split, flag_order, tma_out, scratch, slot_per_tile;
    int b_stages, cb1_shift, cb2_shift, cb1_bytes, cb2_bytes;
    int pre_x, pre_y;                // pre-pass grid; pre_y = parts of a bias term
    int pre_rows;                    // tokens per block of the pre-pass that keeps rows in shared memory, 0 = the other one
    long long n_scratch;
    size_t smem;
    int few;                         // the kernel for few tokens
    int plain;                       // v = 8 over a table in L2: the kernel for 16-bit main and 8-bit residual indices, nothing else
    int pad_bytes;                   // rows of padded table copies, 0 = none
    long long ws_bytes, off_flags, off_bpart, off_pad1, off_pad2, off_scratch, off_xs;
};

// `workers` CTAs at most, in a launch of n_layers layers with `rows` vector rows
template <int V>
GemmPlan plan_gemm_v(const LayerView &L, int B, int workers, int n_layers, long long rows, bool concurrent)
{
    GemmPlan p;
    memset(&p, 0, sizeof(p));
    const int ctas = workers;
    // tables: small ones of a single group in shared memory, with copies where that costs little
    p.t1 = (V <= 8 && L.G == 1 && (long long)L.k1 * 16 <= 64 * 1024) ? TABLE_SHARED : TABLE_GLOBAL;
    p.t2 = L.k2 == 0 ? TABLE_NONE : (V <= 8 && L.G == 1 && L.k2 * 16 <= 16 * 1024) ? TABLE_SHARED : TABLE_GLOBAL;
    if (p.t1 == TABLE_SHARED) {
        while (p.cb1_shift < 3 && (L.k1 * 16 << (p.cb1_shift + 1)) <= 32 * 1024) p.cb1_shift++;
        p.cb1_bytes = L.k1 * 16 << p.cb1_shift;
    }
    p.plain = V == 8 && p.t1 == TABLE_GLOBAL && L.G == 1 && L.n_out == 0 && L.s1.bits == 16 && (L.k2 == 0 || L.s2.bits == 8);
    // token tiles of equal size, at most MAX_TILE_N tokens each
    p.tiles_t = ceil_div(B, MAX_TILE_N);
    p.tile_n = (ceil_div(B, p.tiles_t) + 15) / 16 * 16;
    p.n0 = p.tile_n <= 256 ? p.tile_n : (p.tile_n / 2 + 15) / 16 * 16;
    p.tiles_m = ceil_div(L.R, Tile<V>::NV);
    p.ks = Tile<V>::KS;
    p.kb_main = ceil_div(L.Nc, p.ks);
    p.kb_total = p.kb_main + ceil_div(L.n_out, p.ks);
    // a deterministic call gets whole tiles: sums of several pieces arrive in no fixed order
    Shares &sh = p.shares;
    const unsigned tiles = (unsigned)p.tiles_m * p.tiles_t;
    sh.kb = p.kb_total; sh.whole_tiles = L.deterministic ? 1 : 0;
    p.tma_out = (L.out_dtype == VPTQ_DTYPE_FP32 && (L.M & 3) == 0) ? 1 : 0;
    // (a share of a few k blocks is not worth a CTA of its own: it costs a piece of the output and its meeting)
    const long long columns = (long long)tiles * sh.kb * p.ks;            // (of all tiles: past 32 bits for large calls)
    const long long most = L.deterministic ? tiles : (columns + 127) / 128;
    if (most < workers) workers = (int)most;
    // flag order makes CTAs wait for one another: only for a call that has the GPU to itself
    const bool in_order = p.tma_out && columns / workers >= FLAG_ORDER_MIN_COLS && !concurrent;
    const int drain_cols = DRAIN_COLS * p.tile_n / MAX_TILE_N + (p.tma_out ? 0 : V == 8 ? MEET_COLS_8 : MEET_COLS);
    sh.len = p.kb_total + drain_cols / p.ks;
    // With fewer tiles than CTAs every tile can have as many CTAs to itself (per_tile): no CTA then drains two pieces and
    // meets others twice.  Worth it while the longest share grows by less than that costs (see LONGER_COLS); under flag order
    // a second piece costs next to nothing (4096 x 4096 over the 1 MiB table, 512 tokens, FP32: 40.0 us, 41.4 per tile).
    if (!sh.whole_tiles && !in_order && tiles < (unsigned)workers) {
        const unsigned per_tile = workers / tiles;
        const long long longer = (long long)((sh.kb + per_tile - 1) / per_tile) * p.ks - columns / workers;
        const int limit = per_tile == 1 ? WHOLE_COLS + p.tile_n * 5 / 4 : p.tma_out ? LONGER_COLS_SUM : LONGER_COLS + p.tile_n / 8;
        if (longer <= limit) {
            sh.per_tile = per_tile;
            workers = (int)(tiles * per_tile);
        }
    }
    sh.workers = p.grid = workers;
    const unsigned line = sh.per_tile ? sh.kb : sh.whole_tiles ? tiles : tiles * sh.len, parts = sh.per_tile ? sh.per_tile : workers;
    sh.each = line / parts; sh.rest = line % parts;
    for (int c = 1; c < workers; c++)
        if (sh.begin(c) % p.kb_total != 0) p.any_split = 1;
    p.scratch = p.any_split && !p.tma_out;
    p.flag_order = p.any_split && in_order ? 1 : 0;
    // Shared memory: tables, A ring, then a B ring of up to 96 KB.  Three stages of it come before
    // copies of the residual table (eight copies are free of bank conflicts).  A table in L2
    // needs the L1 that is left, whose lines hold the reads in flight: past 196 KB a CTA (with the 1 KB the system keeps)
    // leaves 28 KB of L1 instead of 60 KB, and 14336 x 4096 at 512 tokens takes 101 us instead of 90.
    const int b_bytes = p.tile_n * 64;
    const int limit = p.t1 == TABLE_GLOBAL || p.t2 == TABLE_GLOBAL ? SMEM_LIMIT_L1 : SMEM_LIMIT;
    const bool copies = p.t2 == TABLE_SHARED && L.k2 <= 256;
    // (the layers of a launch take the same kernel, so by the share that a CTA has of all of them)
    const long long share = (rows + Tile<V>::NV - 1) / Tile<V>::NV * p.tiles_t * p.kb_total * p.ks / device_sm_count();
    auto quick = [](int bits) { return bits == 8 || bits == 12 || bits == 16; };
    const bool long_enough = share >= few_min_cols(p.tile_n) && (p.tile_n <= 32 || p.cb1_shift < 3);
    p.few = p.tile_n <= few_tokens<V>() && (V != 6 || (p.t1 == TABLE_SHARED && (long_enough || !quick(L.s1.bits) || (L.k2 > 0 && !quick(L.s2.bits)))));
    constexpr bool HAS_FEW = V != 12;
    const int a_stages = p.few ? Tile<V, HAS_FEW>::A_STAGES : Tile<V>::A_STAGES, epi = p.few ? Tile<V, HAS_FEW>::EPI : Tile<V>::EPI;
    p.cb2_shift = copies ? 3 : 0;
    while (true) {
        p.cb2_bytes = p.t2 == TABLE_SHARED ? L.k2 * 16 << p.cb2_shift : 0;
        const int fixed = a_stages * a_stage_bytes<V>() + p.cb1_bytes + p.cb2_bytes + epi * 2 * EPI_BUF_BYTES +
                          MAX_TILE_N * 4 + 8 * (2 * a_stages + 2 * MAX_B_STAGES + 4) + 16;
        int room = limit - fixed;
        if (room > 96 * 1024) room = 96 * 1024;
        p.b_stages = room / b_bytes < MAX_B_STAGES ? room / b_bytes : MAX_B_STAGES;
        p.smem = (size_t)fixed + (size_t)(p.b_stages > 0 ? p.b_stages : 0) * b_bytes;
        if (p.b_stages >= 3 || p.cb2_shift == 0) break;
        p.cb2_shift--;
    }
    // pre-pass: enough blocks to fill the GPU (each of them is one part of eight tokens' bias terms)
    const int images = p.kb_total * (p.ks / IMG_COLS);
    const long long row_bytes = (L.N + 7LL) / 8 * 16;
    p.pre_rows = !L.permuted || (long long)B * L.N * n_layers < PRE_ROWS_MIN ? 0 : 4 * row_bytes <= 100 * 1024 ? 4 : 2 * row_bytes <= 200 * 1024 ? 2 : 0;
    p.pre_x = p.tiles_t * p.tile_n / (p.pre_rows ? p.pre_rows : 8);
    const long long sms = device_sm_count(), blocks = (long long)p.pre_x * n_layers;
    p.pre_y = (int)(p.pre_rows ? 2 * sms / blocks : (4 * sms + blocks - 1) / blocks);
    if (p.pre_y < 1) p.pre_y = 1;
    if (p.pre_y > ceil_div(images, 8)) p.pre_y = ceil_div(images, 8);
    p.pad_bytes = (V != 8 && (p.t1 == TABLE_GLOBAL || p.t2 == TABLE_GLOBAL)) ? (V <= 8 ? 16 : 32) : 0;
    auto take = [&](long long bytes) { const long long at = p.ws_bytes; p.ws_bytes += (bytes + 255) / 256 * 256; return at; };
    take(WS_STATUS_BYTES);
    p.off_flags = take((long long)tiles * MAX_EPI_WARPS * 4);
    p.off_bpart = take((long long)p.pre_y * p.tiles_t * p.tile_n * 4);
    p.off_pad1 = take(p.pad_bytes && p.t1 == TABLE_GLOBAL ? (long long)L.G * L.k1 * p.pad_bytes : 0);
    p.off_pad2 = take(p.pad_bytes && p.t2 == TABLE_GLOBAL ? (long long)L.G * L.k2 * p.pad_bytes : 0);
    // (a slot per tile of a large call would be its whole output in FP32, cleared at every call: 28672 x 8192 at 8192 tokens
    // 1074 MB of workspace instead of 173)
    p.slot_per_tile = (long long)tiles < workers;
    p.n_scratch = p.scratch ? (p.slot_per_tile ? (long long)tiles : workers - 1) * 4 * scratch_rows(p.tile_n) * 32 : 0;
    // (as much for calls that are not cut: a workspace for a larger batch, whose tiles may be whole, serves a smaller one)
    const long long slots = L.deterministic || p.tma_out ? 0 : (long long)tiles < ctas ? (long long)tiles : ctas - 1;
    p.off_scratch = take(slots * 4 * scratch_rows(p.tile_n) * 32 * 4);
    p.off_xs = take((long long)p.tiles_t * images * b_bytes);
    return p;
}

GemmPlan plan_gemm(const LayerView &L, int B, int workers, int n_layers, long long rows, bool concurrent)
{
    return L.v == 8   ? plan_gemm_v<8>(L, B, workers, n_layers, rows, concurrent)
           : L.v == 6 ? plan_gemm_v<6>(L, B, workers, n_layers, rows, concurrent)
                      : plan_gemm_v<12>(L, B, workers, n_layers, rows, concurrent);
}

// The plans of the layers of one launch (n = 1: a launch of its own): the SMs are dealt out to the layers in proportion to
// their vector rows, at least one each, leftover SMs where the most rows per CTA remain.  Returns the workspace bytes.
long long plan_launch(const LayerView *Ls, int n, int B, GemmPlan *pl)
{
    const int G = device_sm_count();
    int ctas[MAX_FUSED], used = 0;
    long long total = 0, ws = 0;
    bool concurrent = false;                         // one layer's flag speaks for the launch
    for (int l = 0; l < n; l++) {
        total += Ls[l].R;
        concurrent = concurrent || Ls[l].concurrent;
    }
    for (int l = 0; l < n; l++) {
        ctas[l] = (int)(G * (long long)Ls[l].R / total);
        if (ctas[l] < 1) ctas[l] = 1;
        used += ctas[l];
    }
    for (; used < G; used++) {
        int most = 0;
        for (int l = 1; l < n; l++)
            if ((long long)Ls[l].R * ctas[most] > (long long)Ls[most].R * ctas[l]) most = l;
        ctas[most]++;
    }
    for (int l = 0; l < n; l++) {
        pl[l] = plan_gemm(Ls[l], B, ctas[l], n, total, concurrent);
        ws += pl[l].ws_bytes;
    }
    return ws;
}

template <int V, int T1, int T2, int NL, bool PLAIN, bool FEW>
cudaError_t launch_gemm(const GemmPlan &pl, const OutMaps<NL> &maps, const GemmLaunch<NL> &F, cudaStream_t st)
{
    const cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void *>(gemm_tcgen05_kernel<V, T1, T2, NL, PLAIN, FEW>), pl.smem);
    if (e != cudaSuccess) return e;
    // programmatic dependent launch: set-up and the producers' first reads overlap the pre-pass
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(F.cta_begin[F.n_layers], 1, 1);
    cfg.blockDim = dim3(gemm_threads<V, FEW>(), 1, 1);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_tcgen05_kernel<V, T1, T2, NL, PLAIN, FEW>, maps, F);
}

template <int V, int NL, bool FEW>
cudaError_t launch_gemm_v(const GemmPlan &pl, const OutMaps<NL> &maps, const GemmLaunch<NL> &F, cudaStream_t st)
{
    if (pl.t1 == TABLE_SHARED) {
        if (pl.t2 == TABLE_NONE) return launch_gemm<V, TABLE_SHARED, TABLE_NONE, NL, false, FEW>(pl, maps, F, st);
        if (pl.t2 == TABLE_SHARED) return launch_gemm<V, TABLE_SHARED, TABLE_SHARED, NL, false, FEW>(pl, maps, F, st);
        return launch_gemm<V, TABLE_SHARED, TABLE_GLOBAL, NL, false, FEW>(pl, maps, F, st);
    }
    constexpr bool G = FEW && V == 8;               // (v = 6 over a table in L2 has the one kernel)
    if (V == 8 && pl.plain && pl.t2 == TABLE_NONE) return launch_gemm<8, TABLE_GLOBAL, TABLE_NONE, NL, true, G>(pl, maps, F, st);
    if (V == 8 && pl.plain && pl.t2 == TABLE_SHARED) return launch_gemm<8, TABLE_GLOBAL, TABLE_SHARED, NL, true, G>(pl, maps, F, st);
    if (pl.t2 == TABLE_NONE) return launch_gemm<V, TABLE_GLOBAL, TABLE_NONE, NL, false, G>(pl, maps, F, st);
    if (pl.t2 == TABLE_SHARED) return launch_gemm<V, TABLE_GLOBAL, TABLE_SHARED, NL, false, G>(pl, maps, F, st);
    return launch_gemm<V, TABLE_GLOBAL, TABLE_GLOBAL, NL, false, G>(pl, maps, F, st);
}

template <int NL>
cudaError_t launch_layers(const LayerView *Ls, int n, const void *x, int B, void *const *outs, void *ws, cudaStream_t st)
{
    GemmPlan pls[NL];
    plan_launch(Ls, n, B, pls);
    OutMaps<NL> maps;
    GemmLaunch<NL> F;
    PrepassLaunch<NL> Q;
    memset(&maps, 0, sizeof(maps));      // not read by the kernel when tma_out == 0
    memset(&F, 0, sizeof(F));
    memset(&Q, 0, sizeof(Q));
    F.n_layers = n;
    uint8_t *w8 = reinterpret_cast<uint8_t *>(ws);
    int *status = reinterpret_cast<int *>(ws);                 // the launch's: the first layer's
    for (int l = 0; l < n; l++) {
        const GemmPlan &pl = pls[l];
        const LayerView &L = Ls[l];
        // FP32 output with 16-byte aligned rows: the epilogue goes through shared memory and TMA
        if (pl.tma_out) {
            EncodeTiledFn encode = get_encode_fn();
            if (encode == nullptr) return cudaErrorNotSupported;
            const cuuint64_t odim[2] = {(cuuint64_t)L.M, (cuuint64_t)B};
            const cuuint64_t ostride[1] = {(cuuint64_t)L.M * 4};
            const cuuint32_t tail_rows = (L.v == 8 ? Tile<8>::NV * 8 : L.v == 6 ? Tile<6>::NV * 6 : Tile<12>::NV * 12) - 96u;
            for (int k = 0; k < (tail_rows < 32 ? 2 : 1); k++) {
                const cuuint32_t obox[2] = {k ? tail_rows : 32u, PIECE_TOKENS};
                const cuuint32_t estr[2] = {1, 1};
                const CUresult r = encode(k ? &maps.tail[l] : &maps.layer[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, outs[l], odim, ostride, obox, estr,
                                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                          CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
                if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
            }
        }
        PrepassParams &q = Q.layer[l];
        q.L = L; q.x = x; q.B = B; q.tile_n = pl.tile_n;
        q.img_main = pl.kb_main * (pl.ks / IMG_COLS); q.img_total = pl.kb_total * (pl.ks / IMG_COLS);
        q.xs = w8 + pl.off_xs;
        q.bpart = reinterpret_cast<float *>(w8 + pl.off_bpart);
        q.status = status;
        q.tile_flags = reinterpret_cast<int *>(w8 + pl.off_flags); q.n_flags = pl.tiles_m * pl.tiles_t * MAX_EPI_WARPS;
        if (pl.scratch) { q.zero = reinterpret_cast<float *>(w8 + pl.off_scratch); q.n_zero = pl.n_scratch; }
        else if (pl.any_split && !pl.flag_order) { q.zero = reinterpret_cast<float *>(outs[l]); q.n_zero = (long long)B * L.M; }
        if (pl.pad_bytes && pl.t1 == TABLE_GLOBAL) q.pad1 = w8 + pl.off_pad1;
        if (pl.pad_bytes && pl.t2 == TABLE_GLOBAL) q.pad2 = w8 + pl.off_pad2;
        q.pad_bytes = pl.pad_bytes;

        GemmParams &P = F.layer[l];
        P.L = L; P.out = outs[l]; P.B = B;
        P.tiles_m = pl.tiles_m; P.tiles_t = pl.tiles_t; P.tile_n = pl.tile_n; P.n0 = pl.n0;
        P.kb_main = pl.kb_main; P.kb_total = pl.kb_total; P.shares = pl.shares;
        P.b_stages = pl.b_stages; P.cb1_shift = pl.cb1_shift; P.cb2_shift = pl.cb2_shift;
        P.cb1_bytes = pl.cb1_bytes; P.cb2_bytes = pl.cb2_bytes;
        P.flag_order = pl.flag_order; P.tma_out = pl.tma_out;
        P.status = status; P.bpart = q.bpart; P.bias_parts = pl.pre_y; P.tile_flags = q.tile_flags;
        P.scratch = pl.scratch ? reinterpret_cast<float *>(w8 + pl.off_scratch) : nullptr;
        P.slot_per_tile = pl.slot_per_tile;
        P.xs = q.xs;
        P.tab1 = q.pad1 ? q.pad1 : reinterpret_cast<const uint8_t *>(L.c1);
        P.tab2 = q.pad2 ? q.pad2 : reinterpret_cast<const uint8_t *>(L.c2);
        F.cta_begin[l + 1] = F.cta_begin[l] + pl.grid;
        w8 += pl.ws_bytes;
    }

    // (the layers of a launch have one format, so their plans differ in the tiles only)
    const GemmPlan &pl = pls[0];
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(pl.pre_x, pl.pre_y, n);
    cfg.blockDim = dim3(PRE_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)pl.pre_rows * ((Ls[0].N + 7) / 8 * 16);
    cfg.stream = st;
    cfg.attrs = attr; cfg.numAttrs = 1;
    auto pre = pl.pre_rows == 4 ? gemm_prepass_rows_kernel<4, NL> : pl.pre_rows == 2 ? gemm_prepass_rows_kernel<2, NL> : gemm_prepass_kernel<NL>;
    cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void *>(pre), cfg.dynamicSmemBytes);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, pre, Q);
    if (e != cudaSuccess) return e;
    if (Ls[0].v == 8) return pl.few ? launch_gemm_v<8, NL, true>(pl, maps, F, st) : launch_gemm_v<8, NL, false>(pl, maps, F, st);
    if (Ls[0].v == 6) return pl.few ? launch_gemm_v<6, NL, true>(pl, maps, F, st) : launch_gemm_v<6, NL, false>(pl, maps, F, st);
    return pl.t2 == TABLE_NONE ? launch_gemm<12, TABLE_GLOBAL, TABLE_NONE, NL, false, false>(pl, maps, F, st)
                               : launch_gemm<12, TABLE_GLOBAL, TABLE_GLOBAL, NL, false, false>(pl, maps, F, st);
}

}  // namespace

bool gemm_tcgen05_supported(const LayerView &L, int B)
{
    if (B < 1 || B > (1 << 30) || L.scale_rows || L.Nc <= 0) return false;       // (token numbers, padded to whole tiles, are 32-bit)
    // (so are unit numbers: more than any batch that fits the device's memory needs)
    const long long tiles = (L.M / 96 + 1LL) * (B / 256 + 1), blocks = L.N / 16 + 16;
    return (L.v == 6 || L.v == 8 || L.v == 12) && tiles <= 0x7fffffffLL / blocks;
}

long long gemm_tcgen05_workspace_bytes(const LayerView *Ls, int n, int B)
{
    GemmPlan pl[MAX_FUSED];
    return plan_launch(Ls, n, B, pl);
}

// Layers of one format (apart from M) can share a launch: q+k+v+o of a 70B layer at 333 tokens 265 -> 225 us (a 1024 x 8192
// projection alone has 8 tiles for 148 SMs, 18 pieces of each meeting in one place).
bool gemm_tcgen05_fused_supported(const LayerView *Ls, int n, int B)
{
    if (n < 2 || n > MAX_FUSED || n > device_sm_count()) return false;
    for (int l = 0; l < n; l++)
        if (!gemm_tcgen05_supported(Ls[l], B) || !same_geometry(Ls[0], Ls[l]) || Ls[l].permuted != Ls[0].permuted || Ls[l].deterministic) return false;
    return true;
}

int gemm_tcgen05_launches(const LayerView &, int) { return 2; }   // pre-pass + GEMM

bool gemm_tcgen05_waits_between_ctas(const LayerView *Ls, int n, int B)
{
    GemmPlan pl[MAX_FUSED];
    plan_launch(Ls, n, B, pl);
    for (int l = 0; l < n; l++)
        if (pl[l].flag_order) return true;
    return false;
}

cudaError_t launch_gemm_tcgen05(const LayerView *Ls, int n, const void *x, int B, void *const *outs, void *ws, cudaStream_t st)
{
    if (n < 1 || n > MAX_FUSED) return cudaErrorInvalidValue;
    return n == 1 ? launch_layers<1>(Ls, n, x, B, outs, ws, st) : launch_layers<MAX_FUSED>(Ls, n, x, B, outs, ws, st);
}

}  // namespace vptq
