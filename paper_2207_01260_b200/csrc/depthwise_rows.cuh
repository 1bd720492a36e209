// The inner loop of a depthwise convolution on the CUDA cores: a thread's output columns, row by row, from a patch in shared memory.
#pragma once

#include "common.cuh"

namespace cprune {

// x * w + a on a pair of float32 values: one instruction issues both fused multiply-adds
__device__ __forceinline__ unsigned long long fma2(unsigned long long x, unsigned long long w, unsigned long long a) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(w), "l"(a));
    return d;
}
__device__ __forceinline__ unsigned long long widen2(uint32_t v) {       // the float32 values of a bf16 pair
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(v << 16), "r"(v & 0xffff0000u));
    return r;
}
__device__ __forceinline__ float2 split2(unsigned long long a) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(a));
    return f;
}
template <int NW>
__device__ __forceinline__ void load_words(const uint32_t *p, uint32_t *v) {
    if constexpr (NW == 2) {
        const uint2 t = *reinterpret_cast<const uint2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = *p;
    }
}

// `rows` output rows of COLS columns and CH channels: `in` is the thread's first input pixel (words of two channels, `pix` from
// column to column, `row_words` from row to row), wf the taps, bf the bias.  An input row feeds all the output rows it overlaps, so
// that NACC rows of accumulators are alive; emit(column, sums) gets a finished row column by column, row_done() follows it.
template <int R, int STRIDE, int CH, int COLS, typename Emit, typename RowDone>
__device__ __forceinline__ void depthwise_rows(const uint32_t *in, uint32_t pix, uint32_t row_words, int rows, const unsigned long long (&wf)[R][R][CH / 2],
                                               const unsigned long long (&bf)[CH / 2], Emit emit, RowDone row_done) {
    constexpr int NACC = (R + STRIDE - 1) / STRIDE;      // output rows one input row can belong to
    constexpr int NPX = (COLS - 1) * STRIDE + R;         // input pixels per row of a thread's window
    constexpr int NW = CH / 2;                           // words (channel pairs) per pixel
    unsigned long long acc[NACC][COLS][NW];
#pragma unroll
    for (int a = 0; a < NACC; ++a)
#pragma unroll
        for (int c = 0; c < COLS; ++c)
#pragma unroll
            for (int k = 0; k < NW; ++k) acc[a][c][k] = 0ull;
    const int steps = rows + NACC - 1;                   // STRIDE input rows each; step t completes output row t - NACC + 1
    for (int t0 = 0; t0 < steps; t0 += NACC) {
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
            const int t = t0 + u;
            if (t >= steps) break;
#pragma unroll
            for (int j = 0; j < STRIDE; ++j) {
                if (j > 0 && t * STRIDE + j >= (rows - 1) * STRIDE + R) break;      // below the last row the segment needs
#pragma unroll
                for (int k = 0; k < NPX; ++k) {
                    uint32_t raw[NW];
                    unsigned long long xv[NW];
                    load_words<NW>(in + k * pix, raw);
#pragma unroll
                    for (int q = 0; q < NW; ++q) xv[q] = widen2(raw[q]);
#pragma unroll
                    for (int a = 0; a < NACC; ++a) {
                        const int r = a * STRIDE + j;    // this input row is tap row r of output row t - a
                        if (r < R) {
#pragma unroll
                            for (int c = 0; c < COLS; ++c) {
                                const int s = k - c * STRIDE;
                                if (s >= 0 && s < R) {
#pragma unroll
                                    for (int q = 0; q < NW; ++q) {
                                        unsigned long long &d = acc[(u - a + NACC) % NACC][c][q];
                                        d = fma2(xv[q], wf[r][s][q], (r == 0 && s == 0) ? bf[q] : d);    // an output row starts from the bias
                                    }
                                }
                            }
                        }
                    }
                }
                in += row_words;
                if (j == 0 && t >= NACC - 1) {
                    // output row t - NACC + 1 is complete (R is odd: its last tap row is the first row of a step)
#pragma unroll
                    for (int c = 0; c < COLS; ++c) emit(c, acc[(u + 1) % NACC][c]);
                    row_done();
                }
            }
        }
    }
}

}  // namespace cprune
