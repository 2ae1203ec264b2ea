// drt_synth.cuh -- H synthesis on the tensor cores: one warp's share of a tile of bins of one instant.
//
// At a fixed instant the sum over paths is a contraction once the bin index is split about the middle of
// groups of B bins, k = B u + (B - 1) / 2 +- v with v = 1/2, 3/2, .. (B - 1) / 2:  with
//   X_p[u] = a_p exp(-j 2 pi (phi0_p + (B u + (B - 1) / 2) step_p)),   Y_p[v] = exp(-j 2 pi v step_p)
// the bins at +v and -v share C = sum_p X_p Re Y_p and D = sum_p X_p Im Y_p (Y at -v is the conjugate):
//   H(+v) = C + j D,   H(-v) = C - j D,
// so two bins cost four real multiply-adds per path, as matrix products of depth P: rows (Re X, Im X),
// columns (Re Y, Im Y).  Per path only rows + B / 2 exponentials are evaluated instead of a term per bin.
//
// What bounds it: the issue slots of the exponentials and their splits.  A step of 16 paths x 512 bins takes
// 455 warp instructions on the canyon's records (about 250 on the FMA pipe, 120 at two cycles on the ALU, 32
// hardware sines and cosines at eight) and 24 MMA of 8.2 cycles, against 16 x 512 x 6.3 / 32 = 1610 term by term.  Measured
// against the term-by-term kernel: 512 paths x 2000 steps x 512 bins 112 -> 45 us, 2048 x 1237 x 256 208 -> 72 us,
// 20300 x 500 x 1024 2.40 -> 0.73 ms; error against FP64 1.7e-6 -> 0.7e-6 of the 2-norm.
//
// Precision: FP32 operands split into two FP16 parts each, x = hi + lo with 22 bits, three products
// hi hi + hi lo + lo hi into FP32 accumulators, which are added into FP32 sums every FLUSH steps (the
// tensor cores' own additions truncate: without this the 20300 paths of a highway link lose 1.8e-5).  X is
// scaled by a power of two that keeps the largest amplitude met so far in [2^11, 2^12) (a later, larger
// path rescales the sums exactly), so that paths 2^-25 of the strongest one are still normal FP16 numbers.
//
// m16n8k16 fragments (g = lane / 4, q = lane % 4): a lane evaluates the exponentials of the step's paths
// 2 q, 2 q + 1, 2 q + 8, 2 q + 9 for its own rows u = g + 8 m (row g of row tile m: Re X, row g + 8: Im X)
// and columns v = g + 8 j + 1/2 (column tile 2 j: Re Y, 2 j + 1: Im Y); no operand moves between lanes.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace drt {

// two values as packed FP16 parts hi, lo
__device__ __forceinline__ void split_f16(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// the larger of the two, NaN if one is (an amplitude that is not a number reaches every bin of its instant)
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// nearest integer of |x| < 2^22 by the rounding of an addition (rintf is a quarter-rate instruction)
constexpr float ROUND_MAGIC = 12582912.f;   // 1.5 x 2^23
// m steps of a phase step hi + lo in turns, less a whole number of turns (m hi - t is exact in one FMA)
__device__ __forceinline__ float turns(float m, float hi, float lo) {
    const float t = fmaf(m, hi, ROUND_MAGIC) - ROUND_MAGIC;
    return fmaf(m, lo, fmaf(m, hi, -t));
}
// exp(-j 2 pi ph), |ph| about 1/2 at most (hardware sine and cosine, ~4e-7 absolute)
__device__ __forceinline__ void cis_neg(float ph, float &c, float &s) {
    __sincosf(-6.28318530717958648f * ph, &s, &c);
}

// MT row tiles (u < 8 MT), NJ column groups of 8: a tile of BINS bins from k0 on
template <int MT, int NJ> struct SynthTile {
    static constexpr int B = 16 * NJ, BINS = 8 * MT * B;
    float sum[MT][2 * NJ][4];

    // the steps w0, w0 + ws, ... of 16 paths of the record rows ra, rb (n of them; a record without amplitude has
    // finite phases)
    __device__ __forceinline__ void run(const float4 *__restrict__ ra, const float *__restrict__ rb, int n, int w0,
                                        int ws, int k0) {
        constexpr int FLUSH = 8;
        const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
        float acc[MT][2 * NJ][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[m][j][e] = sum[m][j][e] = 0.f;
        float top = 0.f, scale = 1.f, unscale = 1.f;   // the scale holds for amplitudes below top
        const float m0 = (float)(k0 + B * g) + 0.5f * (B - 1);
        float4 rn[4];
        float ln[4];
        auto fetch = [&](int s) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int p = 16 * s + 2 * q + (h & 1) + 4 * (h & 2);
                rn[h] = p < n ? __ldg(ra + p) : make_float4(0.f, 0.f, 0.f, 0.f);
                ln[h] = p < n ? __ldg(rb + p) : 0.f;
            }
        };
        const int steps = (n + 15) / 16;
        if (w0 < steps) fetch(w0);
        int since = 0;
        for (int s = w0; s < steps; s += ws) {
            const float4 r[4] = {rn[0], rn[1], rn[2], rn[3]};
            const float lo[4] = {ln[0], ln[1], ln[2], ln[3]};
            if (s + ws < steps) fetch(s + ws);
            float big = 0.f;
#pragma unroll
            for (int h = 0; h < 4; ++h) big = max_nan(big, max_nan(fabsf(r[h].x), fabsf(r[h].y)));
            if (__any_sync(0xffffffffu, !(big < top))) {
                const uint32_t bits = __reduce_max_sync(0xffffffffu, __float_as_uint(big));
                if (bits == 0) continue;   // no path met so far exists at this instant
                // its power of two goes to 2^11 (bounded so that both scales are normal numbers)
                const int e = min(max((int)(bits >> 23) - 127, -100), 100);
                const float sc = __uint_as_float((uint32_t)(11 - e + 127) << 23);
                if (top != 0.f) {
                    const float down = sc * unscale;
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                acc[m][j][x] *= down;
                                sum[m][j][x] *= down;
                            }
                }
                scale = sc;
                unscale = __uint_as_float((uint32_t)(e - 11 + 127) << 23);
                top = __uint_as_float((uint32_t)(e + 1 + 127) << 23);
            }
            uint32_t ah[MT][4], al[MT][4], bh[2 * NJ][2], bl[2 * NJ][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {   // register pair h: paths 2 q + 8 h, 2 q + 8 h + 1
                float zr[2], zi[2], wr[2], wi[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float4 &R = r[2 * h + e];
                    const float l = lo[2 * h + e];
                    float ph = R.z + turns(m0, R.w, l), c, sn;
                    ph -= (ph + ROUND_MAGIC) - ROUND_MAGIC;
                    cis_neg(ph, c, sn);
                    const float ar = R.x * scale, ai = R.y * scale;
                    zr[e] = fmaf(ar, c, -ai * sn);
                    zi[e] = fmaf(ar, sn, ai * c);
                    if (MT > 1) cis_neg(turns((float)(8 * B), R.w, l), wr[e], wi[e]);   // 8 rows on
                }
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    split_f16(zr[0], zr[1], ah[m][2 * h], al[m][2 * h]);
                    split_f16(zi[0], zi[1], ah[m][2 * h + 1], al[m][2 * h + 1]);
                    if (m + 1 < MT)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float nr = fmaf(zr[e], wr[e], -zi[e] * wi[e]);
                            zi[e] = fmaf(zr[e], wi[e], zi[e] * wr[e]);
                            zr[e] = nr;
                        }
                }
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    float yr[2], yi[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        cis_neg(turns(g + 8 * j + 0.5f, r[2 * h + e].w, lo[2 * h + e]), yr[e], yi[e]);
                    split_f16(yr[0], yr[1], bh[2 * j][h], bl[2 * j][h]);
                    split_f16(yi[0], yi[1], bh[2 * j + 1][h], bl[2 * j + 1][h]);
                }
            }
            // product by product, so that consecutive MMA add to different accumulators
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int j = 0; j < 2 * NJ; ++j) mma_f16(acc[m][j], al[m], bh[j]);
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int j = 0; j < 2 * NJ; ++j) mma_f16(acc[m][j], ah[m], bl[j]);
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int j = 0; j < 2 * NJ; ++j) mma_f16(acc[m][j], ah[m], bh[j]);
            if (++since == FLUSH) {
                since = 0;
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            sum[m][j][x] += acc[m][j][x];
                            acc[m][j][x] = 0.f;
                        }
            }
        }
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
                for (int x = 0; x < 4; ++x) sum[m][j][x] = (sum[m][j][x] + acc[m][j][x]) * unscale;
    }

    // f(bin of the tile, value) for the lane's bins
    template <class F> __device__ __forceinline__ void each(F &&f) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const float cr = sum[m][2 * j][x], ci = sum[m][2 * j][2 + x];
                    const float dr = sum[m][2 * j + 1][x], di = sum[m][2 * j + 1][2 + x];
                    const int mid = B * (8 * m + g) + B / 2, v = 8 * j + 2 * q + x;
                    f(mid + v, make_float2(cr - di, ci + dr));
                    f(mid - 1 - v, make_float2(cr + di, ci - dr));
                }
    }
};

}  // namespace drt
