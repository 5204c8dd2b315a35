// One warp's share of packing a row (Sec. 6.2 centring, Eq. 8 signs, the
// |y| sum of Eq. 7), shared by the row-packing and fused front kernels.
//
// Lane l of chunk c owns feature 32c + l, so one __ballot_sync yields the
// chunk's 32-bit half-word of the packed row (LSB first). A warp takes
// chunks q, q + G, q + 2G, ... of the row (G warps share it), UNR chunks per
// batch: every load of a batch is issued before any is consumed. G and UNR
// are compile-time constants and each lane walks pointers to its own
// feature, so the batch's loads and stores carry immediate offsets; only
// the row's last batch checks bounds.
#pragma once

#include "bigcn_internal.cuh"

namespace bigcn {

// Where the centring affine y = x * scale + shift comes from: global memory
// (loaded with the batch's features, or, kGlobalLate, as each is consumed:
// fewer registers, for kernels that need full occupancy), shared memory
// (float2 pairs), or nowhere (identity).
enum class Affine { kNone, kGlobal, kGlobalLate, kShared };

template <int G, int UNR, Affine kA>
__device__ __forceinline__ float pack_share(const float *__restrict__ x, int K,
                                            const float *__restrict__ scale,
                                            const float *__restrict__ shift,
                                            const float2 *__restrict__ st,
                                            uint32_t *__restrict__ out, int64_t ld32, int q) {
    const int lane = threadIdx.x & 31;
    const int nchunks = (K + 31) >> 5;          // 32-bit half-words that carry signs
    const int full = K >> 5;                    // chunks with all 32 features inside
    constexpr int kStep = G * 32;               // features between a lane's chunks
    const int off = q * 32 + lane;
    const float *xl = x + off;
    constexpr bool kG = kA == Affine::kGlobal || kA == Affine::kGlobalLate;
    const float *sl = kG ? scale + off : nullptr;
    const float *tl = kG ? shift + off : nullptr;
    const float2 *pl = kA == Affine::kShared ? st + off : nullptr;
    uint32_t *ol = out + q;
    const bool writer = lane == 0;
    float l1 = 0.0f;
    int c0 = q;
    for (; c0 + (UNR - 1) * G < full; c0 += UNR * G) {
        float v[UNR], a[UNR], b[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            v[u] = __ldcs(xl + u * kStep);
            if (kA == Affine::kGlobal) {
                a[u] = __ldg(sl + u * kStep);
                b[u] = __ldg(tl + u * kStep);
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            float y = v[u];
            if (kA == Affine::kGlobal) y = __fmaf_rn(y, a[u], b[u]);
            if (kA == Affine::kGlobalLate)
                y = __fmaf_rn(y, __ldg(sl + u * kStep), __ldg(tl + u * kStep));
            if (kA == Affine::kShared) {
                const float2 p = pl[u * kStep];
                y = __fmaf_rn(y, p.x, p.y);
            }
            const unsigned m = __ballot_sync(kFullMask, y >= 0.0f);
            if (writer) ol[u * G] = m;
            l1 += fabsf(y);
        }
        xl += UNR * kStep;
        if (kG) {
            sl += UNR * kStep;
            tl += UNR * kStep;
        }
        if (kA == Affine::kShared) pl += UNR * kStep;
        ol += UNR * G;
    }
    if (c0 < nchunks) {                         // the last, partial batch
        float v[UNR], a[UNR], b[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const bool in = (c0 + u * G) * 32 + lane < K;
            v[u] = in ? __ldcs(xl + u * kStep) : 0.0f;
            if (kA == Affine::kGlobal) {
                a[u] = in ? __ldg(sl + u * kStep) : 0.0f;
                b[u] = in ? __ldg(tl + u * kStep) : 0.0f;
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int c = c0 + u * G;
            const bool in = c * 32 + lane < K;
            float y = v[u];
            if (kA == Affine::kGlobal) y = __fmaf_rn(y, a[u], b[u]);
            if (kA == Affine::kGlobalLate && in)
                y = __fmaf_rn(y, __ldg(sl + u * kStep), __ldg(tl + u * kStep));
            if (kA == Affine::kShared && in) {
                const float2 p = pl[u * kStep];
                y = __fmaf_rn(y, p.x, p.y);
            }
            const unsigned m = __ballot_sync(kFullMask, in && y >= 0.0f);
            if (writer && c < nchunks) ol[u * G] = m;
            l1 += in ? fabsf(y) : 0.0f;
        }
    }
    // Pad half-words past the last one that carries signs are zero.
    if (q == 0)
        for (int64_t h = nchunks + lane; h < ld32; h += 32) out[h] = 0u;
    return warp_sum(l1);
}

// R rows of X (row stride ldx, `rows` of them real) packed by one warp together:
// C chunks of each per batch, R C loads in flight, and the centring affine read
// once for all of them. Lane r C + c keeps row r's ballot of chunk c, so that a
// batch's half-words are one store. Row r's half-words go to out + r ldo, pad
// half-words up to ld32 as zeros; l1[r] receives the lane's share of its |y| sum
// (chunks in order, as pack_share's with G = 1).
template <int R, int C, Affine kA>
__device__ __forceinline__ void pack_group(const float *__restrict__ x, int64_t ldx, int rows,
                                           int K, const float *__restrict__ scale,
                                           const float *__restrict__ shift, uint32_t *out,
                                           int64_t ldo, int64_t ld32, float (&l1)[R]) {
    static_assert(R * C <= 32, "a lane per ballot");
    static_assert(kA == Affine::kNone || kA == Affine::kGlobal, "");
    const int lane = threadIdx.x & 31;
    const int nchunks = (K + 31) >> 5, full = K >> 5;
    const float *xl[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        xl[r] = x + int64_t(min(r, rows - 1)) * ldx + lane;
        l1[r] = 0.0f;
    }
    const int mr = lane / C, mc = lane % C;      // the ballot this lane keeps
    uint32_t *ol = out + int64_t(mr) * ldo + mc;
    const bool mine = mr < R && mr < rows;
    int c0 = 0;
    for (; c0 + C <= full; c0 += C) {
        float v[R][C], a[C], b[C];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) v[r][c] = __ldcs(xl[r] + 32 * c);
        if (kA == Affine::kGlobal) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                a[c] = __ldg(scale + 32 * (c0 + c) + lane);
                b[c] = __ldg(shift + 32 * (c0 + c) + lane);
            }
        }
        uint32_t word = 0;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                float y = v[r][c];
                if (kA == Affine::kGlobal) y = __fmaf_rn(y, a[c], b[c]);
                const unsigned m = __ballot_sync(kFullMask, y >= 0.0f);
                if (lane == r * C + c) word = m;
                l1[r] += fabsf(y);
            }
        if (mine) ol[c0] = word;
#pragma unroll
        for (int r = 0; r < R; ++r) xl[r] += 32 * C;
    }
    if (c0 < nchunks) {                          // the last, partial batch
        float v[R][C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const bool in = (c0 + c) * 32 + lane < K;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r][c] = in ? __ldcs(xl[r] + 32 * c) : 0.0f;
        }
        uint32_t word = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = (c0 + c) * 32 + lane;
            const bool in = k < K;
            float a = 1.0f, b = 0.0f;
            if (kA == Affine::kGlobal && in) {
                a = __ldg(scale + k);
                b = __ldg(shift + k);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float y = v[r][c];
                if (kA == Affine::kGlobal) y = __fmaf_rn(y, a, b);
                const unsigned m = __ballot_sync(kFullMask, in && y >= 0.0f);
                if (lane == r * C + c) word = m;
                l1[r] += in ? fabsf(y) : 0.0f;
            }
        }
        if (mine && c0 + mc < nchunks) ol[c0] = word;
    }
    for (int64_t h = nchunks; h < ld32; ++h)     // pad half-words (one, or a caller's extra words)
        if (lane < rows) out[int64_t(lane) * ldo + h] = 0u;
}

}  // namespace bigcn
