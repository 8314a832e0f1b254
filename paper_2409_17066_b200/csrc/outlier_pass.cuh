// The outlier columns (Sec. 3.2.3: the first n_out stored columns, vectors of v0 rows, codebook c0) of a run of outlier rows,
// added to a CTA's partial sums.
//
// Two dependent reads of global memory (index, centroid) for a few hundred columns: nothing but latency.  So the work is cut
// into pieces of one outlier row by 16 columns, one column a lane, two pieces a warp, and every warp asks for its first four
// pieces before it waits for the activations; a warp per outlier row, reading after the wait, took 28,000 to 50,000 cycles of
// a kernel of 80,000 (4096 x 11008 with 110 outlier columns, 22016 x 4096 with 41).
#pragma once
#include "common.cuh"
#include "index_words.cuh"

namespace vptq {

struct OutlierPieces {
    static constexpr int PRE = 2;        // steps of two pieces
    int q_lo, n_seg, n_items, first, step;
    uint4 cw[PRE];                       // this lane's centroid in the pieces at hand

    // outlier rows [q_lo, q_hi), shared out over n_warps warps
    __device__ __forceinline__ OutlierPieces(const LayerView &L, int q_lo_, int q_hi, int warp, int n_warps, int lane)
        : q_lo(q_lo_), n_seg((L.n_out + 15) >> 4), n_items((q_hi - q_lo_) * ((L.n_out + 15) >> 4)), first(2 * warp + (lane >> 4)),
          step(2 * n_warps) {}

    __device__ __forceinline__ void fetch_indices(const LayerView &L, int at, int lane, int (&id)[PRE]) const
    {
#pragma unroll
        for (int p = 0; p < PRE; p++) {
            const int i = at + p * step, n = (i % n_seg) * 16 + (lane & 15);
            id[p] = i < n_items && n < L.n_out ? clamp_index(load_index(L.s0.ptr + (long long)(q_lo + i / n_seg) * L.s0.stride, n, L.s0.bits), L.k0) : -1;
        }
    }
    __device__ __forceinline__ void fetch_rows(const LayerView &L, const int (&id)[PRE])
    {
#pragma unroll
        for (int p = 0; p < PRE; p++) cw[p] = id[p] >= 0 ? load_centroid_row(L.c0, id[p], L.v0) : make_uint4(0, 0, 0, 0);
    }

    // part[row - r0][TB][VP] += outlier part of output rows [m_lo, m_hi); xs_out: scaled activations, `pitch` apart
    template <int TB, int VP>
    __device__ __forceinline__ void add(const LayerView &L, const __half *xs_out, int pitch, float *part, int r0, int m_lo, int m_hi, int lane)
    {
        for (int at = first; at - (lane >> 4) < n_items; at += PRE * step) {
            if (at != first) {
                int id[PRE];
                fetch_indices(L, at, lane, id);
                fetch_rows(L, id);
            }
#pragma unroll
            for (int p = 0; p < PRE; p++) {
                const int i = at + p * step;
                if (i - (lane >> 4) >= n_items) break;              // (the same for the whole warp)
                const int qq = q_lo + i / n_seg, n = (i % n_seg) * 16 + (lane & 15);
                const uint32_t w[4] = {cw[p].x, cw[p].y, cw[p].z, cw[p].w};
                float v[8 * TB];
#pragma unroll
                for (int t = 0; t < TB; t++) {
                    const float x = n < L.n_out ? __half2float(xs_out[t * pitch + n]) : 0.f;
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const float2 c = __half22float2(*reinterpret_cast<const __half2 *>(&w[j]));
                        v[t * 8 + 2 * j] = x * c.x; v[t * 8 + 2 * j + 1] = x * c.y;
                    }
                }
                const int vi = halving_butterfly<8 * TB, 16>(v, lane);
                constexpr int KEEP = 8 * TB >= 16 ? 8 * TB / 16 : 1, DUP = 8 * TB >= 16 ? 1 : 16 / (8 * TB);
                if (i < n_items && (lane & (DUP - 1)) == 0) {
#pragma unroll
                    for (int k = 0; k < KEEP; k++) {
                        const int t = (vi + k) >> 3, j = (vi + k) & 7, m = qq * L.v0 + j;
                        if (j < L.v0 && m >= m_lo && m < m_hi) {
                            const int rr = m / L.v;
                            atomicAdd(part + ((rr - r0) * TB + t) * VP + (m - rr * L.v), v[k]);
                        }
                    }
                }
            }
        }
    }
};

}  // namespace vptq
