// The Bi-GCN layer over a weighted adjacency. The paper's notation (Sec. 3)
// takes A = [a_ij] with general entries, d_i = sum_j a_ij, A^ = A + I and
// D^_ii = sum_j a^_ij, and Eq. 1's operator D^-1/2 A^ D^-1/2 on it; the 0/1
// graphs of the other entry points are the case a_ij = 1. Here the CSR
// carries one fp32 weight per entry (finite and non-negative).
//
//   bigcn_weighted_dinv        dinv_i = 1/sqrt(1 + sum of row i's weights)
//   bigcn_spmm_norm_weighted   H_i = dinv_i (dinv_i Z_i + sum_e a_ij dinv_j Z_j)
//   bigcn_weighted_layer_forward
//       pack_rows -> pack_weights -> the degree pass (which also forms the
//       row scale s_j = alpha_j dinv_j) -> the XNOR product with s as its row
//       scale (dots kept factored when K <= 32767, in byte planes for the
//       tensor-core aggregation where they fit) -> the aggregation, which
//       weights neighbour j by a_ij s_j and multiplies the sum by dinv_i.
//
// The degrees need a pass of their own: unlike 1 + row length, a weighted
// degree is a sum over the row, and every row's is read by its neighbours.
#include "launch.cuh"

using namespace bigcn;

namespace {

constexpr int kDegThreads = 256;
constexpr int kDegWarps = kDegThreads / 32;
// Rows longer than this are summed by the whole block instead of one warp.
constexpr int64_t kDegHeavy = 2048;

// Kahan's compensated sum (a running sum and the low-order part its last
// addition lost): a row of tens of thousands of weights is summed with an
// error of a few ulps instead of one growing with its length.
struct Compensated {
    float sum = 0.0f, lost = 0.0f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - lost;
        const float t = sum + y;
        lost = (t - sum) - y;
        sum = t;
    }
    __device__ __forceinline__ float value() const { return sum - lost; }
};

// The smallest (bits, less 1) and the largest (bits) of weights other than 0, the
// self-loop's 1 among them.
struct Spread {
    uint32_t low = 0x3F800000u - 1u, high = 0x3F800000u;
    __device__ __forceinline__ void add(float v) {
        const uint32_t b = __float_as_uint(v) & 0x7fffffffu;
        low = min(low, b - 1u);
        high = max(high, b);
    }
    // So far apart (2^21 and more) that the tensor-core aggregation would take the row in
    // several passes, the row scales' own spread added.
    __device__ __forceinline__ bool far_apart() const {
        return int(high >> 23) - int((low + 1u) >> 23) > 20;
    }
};

// Sum of values[q] for q = q0, q0 + stride, ... below q1, four loads in flight.
__device__ __forceinline__ float strided_sum(const float *__restrict__ values, int64_t q0,
                                             int64_t q1, int stride, Spread &spread) {
    Compensated c;
    for (int64_t q = q0; q < q1; q += 4 * int64_t(stride)) {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t qk = q + int64_t(k) * stride;
            v[k] = qk < q1 ? __ldg(values + qk) : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c.add(v[k]);
            spread.add(v[k]);
        }
    }
    return c.value();
}

// A warp owns kDegRows consecutive rows. Rows of at most kDegShort entries go
// kDegRows at a time, kDegLanes lanes each (their loads, sums, square roots and
// stores side by side); a longer row takes the whole warp, and one of more than
// kDegHeavy entries all eight warps of the block in turn (every warp reads the
// block's row bounds, so the choice is uniform), partials added in warp order.
// One row per warp after another cost 417 instructions a row (100,003 rows of 50
// entries: 47 -> 20 us; 232,965 rows of 492: 145 -> 134 us).
constexpr int kDegRows = 4;
constexpr int kDegLanes = 32 / kDegRows;
constexpr int64_t kDegShort = 256;

__global__ void __launch_bounds__(kDegThreads)
weighted_dinv_kernel(const int64_t *__restrict__ rowptr, const float *__restrict__ values,
                     int64_t N, int64_t nnz, const float *__restrict__ alpha,
                     float *__restrict__ dinv, float *__restrict__ s,
                     uint32_t *__restrict__ spread_rows) {
    __shared__ float part[kDegWarps];
    __shared__ uint32_t part_low[kDegWarps], part_high[kDegWarps];
    constexpr int kBlockRows = kDegWarps * kDegRows;
    static_assert(kBlockRows == 32, "a lane per row of the block");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = int64_t(blockIdx.x) * kBlockRows;
    // Row bounds of the block's rows, clamped to [0, nnz] (a malformed CSR
    // gives wrong degrees, never an out-of-range read); lane r holds row r's.
    int64_t b = 0, e = 0;
    if (i0 + lane < N) {
        b = min(max(__ldg(rowptr + i0 + lane), int64_t(0)), nnz);
        e = min(max(__ldg(rowptr + i0 + lane + 1), b), nnz);
    }
    float total = 0.0f;     // of row i0 + lane, in lanes kDegRows warp .. + kDegRows - 1
    const int own = lane / kDegLanes, sub = lane % kDegLanes;
    const int row = warp * kDegRows + own;          // this lane group's row
    const int64_t rb = __shfl_sync(kFullMask, b, row), re = __shfl_sync(kFullMask, e, row);
    Spread sp;
    float v = re - rb <= kDegShort ? strided_sum(values, rb + sub, re, kDegLanes, sp) : 0.0f;
#pragma unroll
    for (int o = 1; o < kDegLanes; o <<= 1) {
        v += __shfl_xor_sync(kFullMask, v, o);
        sp.low = min(sp.low, __shfl_xor_sync(kFullMask, sp.low, o));
        sp.high = max(sp.high, __shfl_xor_sync(kFullMask, sp.high, o));
    }
    v = __shfl_sync(kFullMask, v, (lane % kDegRows) * kDegLanes);
    if (lane / kDegRows == warp) total = v;
    unsigned far = __popc(__ballot_sync(kFullMask, sub == 0 && sp.far_apart()));  // rows of the warp
    // The warp's longer rows, and the block's heaviest.
    unsigned longer = __ballot_sync(kFullMask, e - b > kDegShort && e - b <= kDegHeavy) &
                      (((1u << kDegRows) - 1u) << (warp * kDegRows));
    while (longer != 0u) {
        const int r = __ffs(longer) - 1;
        longer &= longer - 1u;
        const int64_t lb = __shfl_sync(kFullMask, b, r), le = __shfl_sync(kFullMask, e, r);
        Spread ls;
        const float t = warp_sum(strided_sum(values, lb + lane, le, 32, ls));
        if (lane == r) total = t;
        ls.low = __reduce_min_sync(kFullMask, ls.low);
        ls.high = __reduce_max_sync(kFullMask, ls.high);
        far += ls.far_apart();
    }
    unsigned heavy = __ballot_sync(kFullMask, e - b > kDegHeavy);
    while (heavy != 0u) {
        const int r = __ffs(heavy) - 1;
        heavy &= heavy - 1u;
        const int64_t lb = __shfl_sync(kFullMask, b, r), le = __shfl_sync(kFullMask, e, r);
        Spread ls;
        const float t = warp_sum(strided_sum(values, lb + threadIdx.x, le, kDegThreads, ls));
        ls.low = __reduce_min_sync(kFullMask, ls.low);
        ls.high = __reduce_max_sync(kFullMask, ls.high);
        if (lane == 0) {
            part[warp] = t;
            part_low[warp] = ls.low;
            part_high[warp] = ls.high;
        }
        __syncthreads();
        if (warp == 0) {
            for (int w = 1; w < kDegWarps; ++w) {
                ls.low = min(ls.low, part_low[w]);
                ls.high = max(ls.high, part_high[w]);
            }
            far += ls.far_apart();
        }
        if (lane == r) {
            total = 0.0f;
            for (int w = 0; w < kDegWarps; ++w) total += part[w];
        }
        __syncthreads();    // part[] is rewritten by the next heavy row
    }
    grid_dependency_wait();     // alpha is the row packing's output
    if (spread_rows != nullptr && lane == 0 && far != 0u) atomicAdd(spread_rows, far);
    const int64_t i = i0 + lane;
    if (lane / kDegRows == warp && i < N) {
        const float r = 1.0f / sqrtf(1.0f + total);
        dinv[i] = r;
        if (s != nullptr) s[i] = __ldg(alpha + i) * r;
    }
}

constexpr size_t kWAlign = 256;
size_t wround(size_t x) { return (x + kWAlign - 1) / kWAlign * kWAlign; }
constexpr int32_t kMaxDots16K = 32767;

// Workspace: A bits, alpha, B bits, beta, Z (factored or fp32), row scale,
// the tensor-core product's FP8 weight tiles, dinv, s, control words.
struct WeightedWorkspace {
    size_t a_bits, alpha, b_bits, beta, z, rowscale, bexp, bexp_bytes, dinv, s, control, total;
    bool compressed;
    bool planes;             // laid out for byte planes (rows of ldz bytes)
    int64_t ldz;
};

bool weighted_workspace(int64_t N, int32_t K, int32_t F, WeightedWorkspace *w) {
    if (N < 0 || K < 1 || F < 1) return false;
    const int64_t words = bigcn_words(K);
    w->compressed = K <= kMaxDots16K;
    w->planes = K <= kMaxPlanesK && F <= 256;
    const int64_t pad = w->planes ? 16 : 8;
    w->ldz = w->compressed ? (int64_t(F) + pad - 1) / pad * pad : F;
    if (N > kMaxElems / (words > w->ldz ? words : w->ldz)) return false;
    size_t off = 0;
    w->a_bits = off;   off = wround(off + size_t(N) * size_t(words) * 8);
    w->alpha = off;    off = wround(off + size_t(N) * 4);
    w->b_bits = off;   off = wround(off + size_t(F) * size_t(words) * 8);
    w->beta = off;     off = wround(off + size_t(F) * 4);
    w->z = off;        off = wround(off + size_t(N) * size_t(w->ldz) * (w->compressed ? 2 : 4));
    w->rowscale = off; if (w->compressed) off = wround(off + size_t(N) * 4);
    w->bexp = off;
    w->bexp_bytes = xnor_gemm_tc_bexp_bytes(K, F);
    off = wround(off + w->bexp_bytes);
    w->dinv = off;     off = wround(off + size_t(N) * 4);
    w->s = off;        off = wround(off + size_t(N) * 4);
    w->control = off;
    w->total = off + kControlBytes;
    return true;
}

}  // namespace

namespace bigcn {
void launch_weighted_dinv(const int64_t *rowptr, const float *values, int64_t N, int64_t nnz,
                          const float *alpha, float *dinv, float *s, uint32_t *spread_rows,
                          cudaStream_t stream, bool pdl) {
    if (N == 0) return;
    const int64_t rows = int64_t(kDegWarps) * kDegRows;
    const dim3 grid(unsigned((N + rows - 1) / rows));
    launch_kernel(weighted_dinv_kernel, grid, dim3(kDegThreads), 0, stream, pdl, dim3(1, 1, 1),
                  rowptr, values, N, nnz, alpha, dinv, s, spread_rows);
}
}  // namespace bigcn

extern "C" bigcn_status bigcn_weighted_dinv(const int64_t *rowptr, const float *values,
                                            int64_t N, int64_t nnz, float *dinv, void *stream) {
    if (N < 0 || N > int64_t(INT32_MAX) || nnz < 0) return BIGCN_ERR_INVALID_ARG;
    if (N == 0) return BIGCN_OK;
    if (!rowptr || !dinv || (nnz > 0 && !values)) return BIGCN_ERR_INVALID_ARG;
    if (!aligned_to(rowptr, 8) || (values && !aligned_to(values, 4)) || !aligned_to(dinv, 4))
        return BIGCN_ERR_MISALIGNED;
    if (overlaps(dinv, size_t(N) * 4, rowptr, size_t(N + 1) * 8) ||
        overlaps(dinv, size_t(N) * 4, values, size_t(nnz) * 4))
        return BIGCN_ERR_INVALID_ARG;
    DeviceInfo dev;
    const bigcn_status st = current_device(&dev);
    if (st != BIGCN_OK) return st;
    launch_weighted_dinv(rowptr, values, N, nnz, nullptr, dinv, nullptr, nullptr, as_stream(stream));
    return launch_status();
}

extern "C" bigcn_status bigcn_spmm_norm_weighted(const int64_t *rowptr, const int32_t *colidx,
                                                 const float *values, const float *dinv,
                                                 int64_t N, int64_t nnz, const float *Z,
                                                 int64_t ldz, int32_t F, float *H, int64_t ldh,
                                                 void *stream) {
    if (N < 0 || N > int64_t(INT32_MAX) || nnz < 0 || F < 1 || ldz < F || ldh < F)
        return BIGCN_ERR_INVALID_ARG;
    if (N > 0 && (N > kMaxElems / ldz || N > kMaxElems / ldh)) return BIGCN_ERR_INVALID_ARG;
    if (N == 0) return BIGCN_OK;
    if (!rowptr || !dinv || !Z || !H || (nnz > 0 && (!colidx || !values)))
        return BIGCN_ERR_INVALID_ARG;
    if (!aligned_to(rowptr, 8) || (colidx && !aligned_to(colidx, 4)) ||
        (values && !aligned_to(values, 4)) || !aligned_to(dinv, 4) || !aligned_to(Z, 4) ||
        !aligned_to(H, 4))
        return BIGCN_ERR_MISALIGNED;
    const size_t hb = span_bytes(N, F, ldh, 4);
    if (overlaps(H, hb, Z, span_bytes(N, F, ldz, 4)) ||
        overlaps(H, hb, rowptr, size_t(N + 1) * 8) || overlaps(H, hb, colidx, size_t(nnz) * 4) ||
        overlaps(H, hb, values, size_t(nnz) * 4) || overlaps(H, hb, dinv, size_t(N) * 4))
        return BIGCN_ERR_INVALID_ARG;
    DeviceInfo dev;
    const bigcn_status st = current_device(&dev);
    if (st != BIGCN_OK) return st;
    SpmmArgs a{rowptr, colidx, N, nnz, Z, ldz, F, H, ldh, false, false};
    a.agg = kAggWeighted;
    a.values = values;
    a.dinv = dinv;
    launch_spmm_norm(a, dev, as_stream(stream));
    return launch_status();
}

extern "C" size_t bigcn_weighted_layer_workspace_bytes(int64_t N, int32_t K, int32_t F) {
    WeightedWorkspace w;
    return weighted_workspace(N, K, F, &w) ? w.total : 0;
}

extern "C" bigcn_status bigcn_weighted_layer_forward(
    const float *X, int64_t N, int32_t K, int64_t ldx, const float *scale, const float *shift,
    const float *Wt, int32_t F, int64_t ldw, const int64_t *rowptr, const int32_t *colidx,
    const float *values, int64_t nnz, void *workspace, size_t ws_bytes, float *H, int64_t ldh,
    void *stream) {
    WeightedWorkspace w;
    if (N < 0 || N > int64_t(INT32_MAX) || K < 1 || F < 1 || ldx < K || ldw < F || ldh < F ||
        nnz < 0)
        return BIGCN_ERR_INVALID_ARG;
    if ((scale == nullptr) != (shift == nullptr)) return BIGCN_ERR_INVALID_ARG;
    if (!weighted_workspace(N, K, F, &w)) return BIGCN_ERR_INVALID_ARG;
    if (N > 0 && (N > kMaxElems / ldx || N > kMaxElems / ldh)) return BIGCN_ERR_INVALID_ARG;
    if (int64_t(K) > kMaxElems / ldw) return BIGCN_ERR_INVALID_ARG;
    if (N == 0) return BIGCN_OK;
    if (!X || !Wt || !rowptr || !H || !workspace || (nnz > 0 && (!colidx || !values)))
        return BIGCN_ERR_INVALID_ARG;
    if (ws_bytes < w.total) return BIGCN_ERR_INVALID_ARG;
    if (!aligned_to(X, 4) || !aligned_to(Wt, 4) || !aligned_to(rowptr, 8) ||
        (colidx && !aligned_to(colidx, 4)) || (values && !aligned_to(values, 4)) ||
        !aligned_to(H, 4) || !aligned_to(workspace, kWAlign) ||
        (scale && (!aligned_to(scale, 4) || !aligned_to(shift, 4))))
        return BIGCN_ERR_MISALIGNED;
    const size_t hb = span_bytes(N, F, ldh, 4);
    const void *inputs[] = {X, Wt, rowptr, colidx, values, scale, shift};
    const size_t in_bytes[] = {span_bytes(N, K, ldx, 4), span_bytes(K, F, ldw, 4),
                               size_t(N + 1) * 8, size_t(nnz) * 4, size_t(nnz) * 4,
                               size_t(K) * 4, size_t(K) * 4};
    for (int q = 0; q < 7; ++q) {
        if (overlaps(workspace, w.total, inputs[q], in_bytes[q])) return BIGCN_ERR_INVALID_ARG;
        if (overlaps(H, hb, inputs[q], in_bytes[q])) return BIGCN_ERR_INVALID_ARG;
    }
    if (overlaps(H, hb, workspace, w.total)) return BIGCN_ERR_INVALID_ARG;

    DeviceInfo dev;
    const bigcn_status st = current_device(&dev);
    if (st != BIGCN_OK) return st;
    char *ws = static_cast<char *>(workspace);
    uint64_t *a_bits = reinterpret_cast<uint64_t *>(ws + w.a_bits);
    float *alpha = reinterpret_cast<float *>(ws + w.alpha);
    uint64_t *b_bits = reinterpret_cast<uint64_t *>(ws + w.b_bits);
    float *beta = reinterpret_cast<float *>(ws + w.beta);
    float *dinv = reinterpret_cast<float *>(ws + w.dinv);
    float *srow = reinterpret_cast<float *>(ws + w.s);
    const int words = bigcn_words(K);
    cudaStream_t s = as_stream(stream);

    launch_pack_rows(X, N, K, ldx, scale, shift, a_bits, words, alpha, dev, s);
    uint32_t *control = reinterpret_cast<uint32_t *>(ws + w.control);
    launch_pack_weights(Wt, K, F, ldw, b_bits, words, beta, s, control);
    // Every kernel after the weights' packing may start while the one before it
    // drains (each waits for it before it reads anything the call has written).
    // Factored rows carry dinv_j in their row scale (s_j = alpha_j dinv_j);
    // fp32 rows are the plain product and the aggregation reads dinv_j.
    // (rows of very unlike weights count as wide rows do: see SpmmTcArgs)
    launch_weighted_dinv(rowptr, values, N, nnz, alpha, dinv, w.compressed ? srow : nullptr,
                         control + kWideRowsWord, s, true);
    const bool bytes = w.planes && planes_faster(N, nnz, F) &&
                       xnor_gemm_bytes_supported(N, K, F, dev);
    // (uint16 dots are padded to 8 columns even where the workspace has room for 16)
    const int64_t ldz = bytes ? w.ldz : w.compressed ? (int64_t(F) + 7) / 8 * 8 : F;
    GemmArgs g{a_bits, w.compressed ? srow : alpha, N, b_bits, beta, F, K, words, nullptr,
               ldz, nullptr, nullptr};
    if (w.bexp_bytes > 0) g.b_e4m3 = reinterpret_cast<uint8_t *>(ws + w.bexp);
    SpmmArgs a{rowptr, colidx, N, nnz, nullptr, ldz, F, H, ldh, false, false};
    a.agg = kAggWeighted;
    a.values = values;
    a.dinv = dinv;
    if (bytes) {
        g.dots8 = reinterpret_cast<uint8_t *>(ws + w.z);
        g.wide_rows = control + kWideRowsWord;
        g.ldd8 = ldz;
        g.rowscale = reinterpret_cast<float *>(ws + w.rowscale);
    } else if (w.compressed) {
        uint16_t *D16 = reinterpret_cast<uint16_t *>(ws + w.z);
        float *rowscale = reinterpret_cast<float *>(ws + w.rowscale);
        g.dots16 = D16;
        g.ldd16 = ldz;
        g.rowscale = rowscale;
        a.D16 = D16;
        a.rowscale = rowscale;
        a.colscale = beta;
    } else {
        float *Z = reinterpret_cast<float *>(ws + w.z);
        g.Z = Z;
        a.Z = Z;
    }
    launch_xnor_gemm(g, dev, s, true);
    if (bytes) {
        SpmmTcArgs t{rowptr, colidx, N, nnz, g.dots8, ldz, g.rowscale, F, K, H, ldh, beta,
                     nullptr, kAggWeighted, nullptr, nullptr, values, dinv, control,
                     g.wide_rows};
        launch_spmm_tc(t, dev, s, true);
    } else {
        launch_spmm_norm(a, dev, s, true);
    }
    return launch_status();
}
