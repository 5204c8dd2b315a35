// Step 5 of the Bi-GCN layer (Eq. 13 with the operator of Eq. 1) on the
// tensor cores, for a product kept factored as exact integer dots:
//
//   H_if = c_f * (1/sqrt(dhat_i)) * sum_{j in N(i) u {i}} s_j * dot_jf
//
// with s_j = alpha_j / sqrt(dhat_j) the row scale and c_f = beta_f the column
// scale of Eqs. 11-12. The dots come in byte planes (ByteDot): one byte per
// dot, rows of 16 * FT features; the rows marked wide in fp16, over both planes.
//
// Why tensor cores: the aggregation reads one row of dots per CSR entry. Done
// on CUDA cores, every gathered dot costs a decode and an FMA, and the kernel
// is bound by instruction issue well below what L2 delivers to random row
// gathers. Here the sum over a run of 16 CSR entries is one
// mma.sync.m16n8k16 per 16 features: A = the gathered rows (features x
// entries), B = the entries' weights s_j, D = fp32 accumulators.
//
// Why bytes: the walk is bound by latency -- rows in flight per SM, that is
// shared memory per gathered row, and the dependent steps between a block's
// arrival and the next -- not by L2's bandwidth (20 TB/s for such gathers). A
// byte per dot halves a staged row against fp16, which buys deeper rings and
// half as many copies, for one permute and one packed fma per two dots. On
// 232,965 nodes of mean degree 492 (114.8 M gathered rows): layer 1, 128
// features, 2600 -> 1590 us (9.2 TB/s of 128-byte rows; issue 57 %, ALU and the
// copies' latency bind); layer 2, 41 features, 1475 -> 980 us. On 2^20 nodes of
// mean degree 16, 64 features: 787 -> 464 us.
//
// A staged row is read with ldmatrix.trans as pairs of neighbouring features:
// a lane's register then holds features 2g and 2g + 1 of two entries, which a
// byte permute turns into two A registers (even features in matrix rows 0-7,
// odd ones in rows 8-15). The bytes u = v + 128 enter as fp16 subnormals u
// 2^-24, and one packed fma, u 2^-24 * 2^15 + ((K & 1) - 256) 2^-10, makes
// them dot * 2^-10: every step exact, and no entry's value ever leaves fp16.
// Rows marked wide weigh nothing in this walk and are added afterwards
// (rest_of_window), the few of a window 16 together, their halves as they are. That is a
// gather of twice the bytes and a pass over the window's index list more: where many rows
// are wide, a second kernel on the CUDA cores takes the whole aggregation over
// (spmm_tc_second_kernel). 232,965 nodes of mean degree 492, K = 602, F = 128, a layer: no
// wide row 1790 us, one in 1024 2150, one in 256 2560, more 2595 (16-bit dots: 2990).
//
// B carries the weights as two fp16 parts, hi = fp16(s') and lo = fp16((s' - hi) 2^11)
// with s' = s_j * 2^(14 - E) (an exact power-of-two scaling that puts the
// row's largest weight just below 2^15), and lo's sums, kept apart, are multiplied by
// 2^-11 in the end: together 23 bits or more of each weight down to 2^-24 of the
// row's largest. E is the largest exponent among the weights seen so far for
// that output row: when a later entry raises it, the row's accumulators are
// multiplied by the exact power of two that keeps them consistent. A window with
// smaller weights than that (they decide the columns in which the large neighbours'
// dots are zero) is walked again in bands of 2^24, each on a scale of its own
// (rest_of_window): as good as fp32 multiply-adds at any ratio, at the cost of one more walk
// per band.
//
// A warp takes a window of consecutive output rows whose lists (self entry
// first, then the CSR neighbours) it walks as one stream of positions, 32 to a
// block. One-row windows (long rows) put hi and lo in columns 0 and 1 of B;
// eight-row windows (short rows, so that a block is not mostly padding) give
// column r to output row r and multiply twice, by the hi and by the lo parts,
// into sums of their own (added to the same sums, the lo products would be
// rounded at the hi sums' last place: 1.3e-7 from 64 bits instead of 1.0e-7).
// Gathered rows are staged by cp.async (16 bytes per copy; positions past the
// end of the stream and out-of-range column indices copy nothing and carry
// zero weight: any stale byte is a finite fp16) in a per-warp ring,
// XOR-swizzled so that ldmatrix reads are free of bank conflicts: the copies
// of the next block(s) are in flight while block n is multiplied. The column
// indices are loaded one block ahead of the copies they name and the row scales
// along with their rows, both into registers (a lane owns one position of a
// block), so that neither is waited for.
//
// Rows with more than `heavy_degree` neighbours are each walked by all warps
// of one block, whose fp32 partial rows are added in warp order
// (deterministic); light windows go one per warp, or, when there are many,
// to the warps of one wave of persistent blocks, which first walk the heavy rows
// and then take the windows as they become free (from one counter; a fixed share
// per block left 15 % of the warps idle on power-law graphs: GraphSAGE on 232,965
// nodes 2110 -> 1808 us, weighted rows on 100,003 nodes 217 -> 178 us).
#include <cuda_fp16.h>

#include "launch.cuh"

namespace bigcn {
namespace {

constexpr int kTcThreads = 128;
constexpr int kTcWarps = kTcThreads / 32;
constexpr int kTcRows = 8;          // output rows per window of short rows
constexpr int EB = 32;              // positions per sub-block: one per lane

// Per width and window form: sub-blocks per block, blocks in a warp's ring, and
// the blocks (of 4 warps) per SM that the registers are held to. Fewer warps with
// more registers and rows in flight beat more warps: 128 features in one-row
// windows, 16 warps and three stages of 4 KB 1873 us, 20 warps and two 2245 us, 24
// warps and two 2368 us (24 in blocks of eight warps, whose windows their warps
// share less evenly, 2369 us), 12 warps and four 2084 us; 41 features, 20 warps
// and two stages of 64 rows 1160 us, 24 warps and four of 32 1249 us. Eight-row
// windows of 33 to 64 features spill at 96 registers (20 warps: 548 us, 16 warps
// 464 us on 2^20 rows).
constexpr int tc_sub(int FT, int ROWS) { return FT > 4 || ROWS > 1 ? 1 : 2; }
constexpr int tc_stages(int FT, int ROWS) { return FT > 4 ? 3 : 2; }
constexpr int tc_blocks(int FT, int ROWS) { return FT > 4 || (FT > 2 && ROWS > 1) ? 4 : 5; }

// Tiles of 16 features, sub-blocks per block, blocks in the ring.
template <int FT, int SUB, int NSTAGES>
struct TcGeom {
    static constexpr int P2 = FT <= 1 ? 1 : FT <= 2 ? 2 : FT <= 4 ? 4 : 8;   // chunks per staged row
    // Bytes per staged row, 16 P2: 8 / P2 rows to a 128-byte line, the row's
    // 16-byte chunk c stored at slot c ^ (row / (8 / P2)) mod P2. The eight rows
    // an ldmatrix reads then fall in eight different bank groups, and the two
    // halves of every 32-byte sector of a gathered row stay in one aligned
    // 32-byte slot pair (a padded pitch that splits sectors over two
    // shared-memory lines fetches them twice: 256-byte rows gathered at 13.7
    // TB/s instead of 20.6 TB/s, 96-byte rows at 8.8 instead of 13.0 TB/s).
    static constexpr int PITCH = 16 * P2;
    static constexpr int LINE = 8 / P2;            // staged rows per 128-byte line
    static constexpr int STEP = 32 / P2;           // rows covered by one copy per lane
    static constexpr int PART = EB * PITCH;        // one sub-block
    static constexpr int STAGE = SUB * PART;       // one block
    static constexpr int NS = NSTAGES;             // row ring depth (blocks)
    static constexpr int PARTS = SUB * NS;         // sub-blocks in the ring
    static constexpr int D = NS - 1;               // blocks of rows copied ahead
    // One warp's ring: NS row stages (each starting on a 128-byte line), then the
    // checked columns of the block being copied and the weights of the block
    // being multiplied (per sub-block EB hi and EB lo halves).
    static constexpr int CHECKED = NS * STAGE;
    static constexpr int HALVES = CHECKED + SUB * EB * 4;
    static constexpr int WARP = HALVES + SUB * EB * 4;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return uint32_t(__cvta_generic_to_shared(p));
}

// 16-byte global -> shared copy, skipped for j < 0 (a predicate, not a branch).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int j) {
    asm volatile(
        "{\n.reg .pred p;\n"
        "setp.ge.s32 p, %2, 0;\n"
        "@p cp.async.cg.shared.global [%0], [%1], 16;\n}" ::"r"(dst),
        "l"(src), "r"(j)
        : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void ldsm_x2_trans(uint32_t addr, uint32_t (&r)[2]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                          uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 2^e as a float for e in [-126, 127] (0 for -127).
__device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }

// Unbiased exponent of a non-negative float's bits (-127 for zero and subnormals).
__device__ __forceinline__ int exponent_of(uint32_t bits) { return int(bits >> 23) - 127; }

constexpr int kNoScale = -127;      // exponent of a row that has seen no normal weight yet
constexpr int kDotShift = 10;       // the A operands are dots times 2^-10
constexpr int kLoShift = 11;        // lo parts are kept times 2^11, and so are their sums
// Weights of a row from 2^kBandLow up (on its scale) are held to 2^-23 of themselves; a
// row that has smaller ones takes them in bands, each 2^24 below the one before.
constexpr int kBandLow = -10;
constexpr int kBandStep = 24;
// The first walk notes a weight's exponent where it lies this far below its row's: the
// row's may then rise by as much again before what it did not note could need a band.
constexpr int kLookBelow = 12;

// A row whose largest weight has exponent E multiplies its weights by 2^u, u =
// unit_exponent(E) (to just below 2^15, as far as a float's exponent goes: weights under
// 2^-113 stay smaller), and its sums by 2^(kDotShift - u) in the end; a sum begun at E
// goes on at a larger E2 times scale_change(E, E2) (0 where that is below fp32: the sum
// was made of weights under 2^-126 of the new one).
__device__ __forceinline__ int unit_exponent(int E) { return min(14 - E, 127); }
__device__ __forceinline__ float scale_change(int E, int E2) {
    return exp2i(max(unit_exponent(E2) - unit_exponent(E), -127));
}
// Unit exponent of band k of a row with unit exponent u, and the band of a weight of
// exponent e: the first in which it reaches 2^kBandLow, or the last there is.
__device__ __forceinline__ int band_unit(int u, int k) { return min(u + kBandStep * k, 127); }
__device__ __forceinline__ int band_of(int e, int u) {
    const int need = (kBandLow - e - u + kBandStep - 1) / kBandStep;
    return e + u >= kBandLow ? 0 : min(need, (127 - u + kBandStep - 1) / kBandStep);
}

struct TcParams {
    const int64_t *rowptr;
    const int32_t *colidx;
    int64_t N;
    int64_t nnz;
    const uint8_t *D;        // low plane, N x ldd bytes; the high plane follows
    int64_t ldd;             // bytes; a multiple of 16
    int width;               // bytes of a row that are gathered (<= ldd)
    const float *rowscale;   // s_j, negative for a wide row; nullptr: kept in D's rows
    int agg;                 // aggregator (kAgg...)
    const float *values;     // kAggWeighted: a_ij per CSR entry
    const float *dinv;       // kAggWeighted: 1/sqrt(dhat) per node
    uint32_t offset;         // ((K & 1) - 256) 2^-10, twice, in fp16
    uint32_t half_bias;      // what a wide row's halves lack, 2^-10 half_dot_bias(K), in fp16, twice
    int64_t heavy_degree;    // rows with more neighbours are walked by whole blocks
    uint32_t *counters;      // nullable: windows taken so far by all blocks, per column slab
    int heavy_blocks;        // blocks [0, heavy_blocks) walk the heavy rows
    int light_first;         // blocks [light_first, grid) walk the light windows
};

// A window: ROWS consecutive output rows, each contributing its list (entry 0 =
// the self-loop, entry q > 0 = CSR neighbour q - 1) or, for a part of a heavy
// row, entries [q0, q1) of it, laid out one after the other as positions.
// Row r covers positions [off[r], off[r + 1]); position p of it is the self-loop
// when p == its self position, else CSR entry cbase + p. With eight rows,
// lane r holds row r's cbase.
template <int ROWS>
struct Window {
    int64_t first;           // output row of r = 0
    int64_t cbase;           // ROWS == 1: the row's; else of row (lane & 7)
    bool self0;              // position 0 (of each row) is the self-loop
    int off[ROWS + 1];       // off[ROWS] = stream length
};

// The row that position p belongs to (zero-length rows hold none).
template <int ROWS>
__device__ __forceinline__ int row_of(const Window<ROWS> &w, int p) {
    int r = 0;
#pragma unroll
    for (int k = 1; k < ROWS; ++k) r += int(p >= w.off[k]);
    return r;
}

// What position p of the stream gathers: the CSR's column (unchecked), the
// output row's own for a self-loop, -1 past the end; with kW (a weighted A) also
// the entry's a_ij (1 for the self-loop). Called by all lanes together.
template <bool kW>
struct Entry {
    int col;
    float a;
};
template <>
struct Entry<false> {
    int col;
    static constexpr float a = 1.0f;
};

// The factor applied to row i's sum: Eq. 1's 1/sqrt(dhat_i) (read for a weighted
// A), the mean's 1/dhat_i, or GraphSAGE's 1/|N(i)| (0 without neighbours).
__device__ __forceinline__ float row_factor(const TcParams &P, int64_t i, int64_t deg) {
    return P.agg == kAggGcn        ? inv_sqrt_degree(deg)
           : P.agg == kAggWeighted ? __ldg(P.dinv + i)
           : P.agg == kAggMean     ? 1.0f / (1.0f + float(deg))
           : deg > 0               ? 1.0f / float(deg)
                                   : 0.0f;
}

template <int ROWS, bool kW>
__device__ __forceinline__ Entry<kW> fetch_entry(const TcParams &P, const Window<ROWS> &w, int p) {
    Entry<kW> q;
    q.col = -1;
    if constexpr (kW) q.a = 1.0f;
    auto take = [&](int64_t entry) {
        q.col = __ldg(P.colidx + entry);
        if constexpr (kW) q.a = __ldg(P.values + entry);
    };
    if constexpr (ROWS == 1) {
        if (p < w.off[1]) {
            if (w.self0 && p == 0) q.col = int(w.first);
            else take(w.cbase + p);
        }
    } else {
        const int r = row_of<ROWS>(w, p);
        int start = w.off[0];
#pragma unroll
        for (int k = 1; k < ROWS; ++k) start = r >= k ? w.off[k] : start;
        const int64_t entry = __shfl_sync(kFullMask, w.cbase, r) + p;
        if (p < w.off[ROWS]) {
            if (w.self0 && p == start) q.col = int(w.first) + r;
            else take(entry);
        }
    }
    return q;
}

// Per-lane sums of a window after its walk: R2 output rows (ROWS == 1: lanes
// with t = 0 hold the row; else lane (g, t) holds rows 2t and 2t + 1), features
// 16 T + 2g and 16 T + 2g + 1 (g = lane >> 2, t = lane & 3), as fp32 values.
template <int FT, int R2>
struct TcRowSums {
    float v[R2][FT][2];
};

// A lane's column j (-1: copies nothing) for copy_plane, in shared memory
// (`checked`), permuted so that a lane there reads the columns of its P2 rows at
// once: one store and one or two loads instead of P2 shuffles.
template <class G>
__device__ __forceinline__ void put_column(int *checked, int j) {
    const int lane = threadIdx.x & 31;
    checked[(lane % G::STEP) * G::P2 + lane / G::STEP] = j;
}

// The copy of one sub-block's rows of a plane to shared address `stage`.
// Copy k of a lane moves chunk `piece` of staged row r0 + k STEP to its slot,
// which for P2 = 8 alternates between two (4 rows on, bit 2 of the row flips),
// else is the same for every k. `plane` points at chunk `piece` of row 0; `mine`:
// the lane's chunk exists. kBoth: staged rows 16 to 31 come from the high plane, `high`
// bytes on (16 positions' rows, low and high).
template <class G, bool kBoth = false>
__device__ __forceinline__ void copy_plane(uint32_t stage, const int *checked,
                                           const uint8_t *plane, uint32_t row_bytes, bool mine,
                                           int64_t high = 0) {
    constexpr int P2 = G::P2;
    const int lane = threadIdx.x & 31;
    const int r0 = lane / P2, piece = lane % P2;
    const uint32_t base =
        stage + uint32_t(r0 * G::PITCH + ((piece ^ ((r0 / G::LINE) & (P2 - 1))) << 4));
    int jj[P2];
    if constexpr (P2 == 1) {
        jj[0] = checked[lane];
    } else {
        if constexpr (P2 == 2) {
            const int2 v = *reinterpret_cast<const int2 *>(checked + r0 * 2);
            jj[0] = v.x, jj[1] = v.y;
        } else {
#pragma unroll
            for (int q = 0; q < P2 / 4; ++q) {
                const int4 v = *reinterpret_cast<const int4 *>(checked + r0 * P2 + 4 * q);
                jj[4 * q] = v.x, jj[4 * q + 1] = v.y, jj[4 * q + 2] = v.z, jj[4 * q + 3] = v.w;
            }
        }
    }
    if (mine)
#pragma unroll
        for (int k = 0; k < P2; ++k)
            cp_async16((base ^ (P2 == 8 && (k & 1) ? 64u : 0u)) + uint32_t(k * G::STEP * G::PITCH),
                       plane + uint64_t(uint32_t(jj[k])) * row_bytes +
                           (kBoth && r0 + k * G::STEP >= 16 ? high : 0),
                       jj[k]);
}

// A window's sums in the MMA's accumulator layout: ROWS == 1 hi and lo in columns
// 0 and 1; else hi (v[0]) and lo (v[1]) with a column per row.
template <int FT, int ROWS>
struct TcSums {
    static constexpr int PARTS = ROWS == 1 ? 1 : 2;
    float v[PARTS][FT][4];
    // Multiplies all sums of a lane's even and odd columns.
    __device__ __forceinline__ void scale(float even, float odd) {
#pragma unroll
        for (int p = 0; p < PARTS; ++p)
#pragma unroll
            for (int T = 0; T < FT; ++T)
#pragma unroll
                for (int q = 0; q < 4; ++q) v[p][T][q] *= (q & 1) ? odd : even;
    }
};

// A lane's weight on its row's scale as its two fp16 parts in shared memory (`halves`:
// EB hi parts, then EB lo parts times 2^kLoShift), entries 2t, 2t + 1, and those 8, 16 and 24 on,
// next to one another, so that a lane's B fragments are one load.
// kBoth: 16 positions (lanes 0 to 15), hi parts and then lo parts.
template <bool kBoth = false>
__device__ __forceinline__ void put_weight(uint16_t *halves, float ws) {
    const int lane = threadIdx.x & 31;
    const __half hi = __float2half_rn(ws);
    // (the limit, far below any difference, makes an infinite weight's low part finite:
    // Inf - Inf would make its row NaN in every column, where Inf times a dot is Inf of
    // the dot's sign)
    const __half lo = __float2half_rn(
        fmaxf((ws - __half2float(hi)) * float(1 << kLoShift), -32768.0f));
    constexpr int kN = kBoth ? EB / 2 : EB;
    const int at = ((lane >> 1) & 3) * (kN / 4) + (lane >> 3) * 2 + (lane & 1);
    if (!kBoth || lane < kN) {
        halves[at] = __half_as_ushort(hi);
        halves[kN + at] = __half_as_ushort(lo);
    }
}

// One pass over a staged sub-block (shared address `rows` = the sub-block + this
// lane's ldmatrix row) with the weights in `halves`. ROWS == 1: hi in column 0
// and lo in column 1 of B; else column g holds the hi (b) or lo (c) parts of row
// g, whose positions are those with 0 <= position - glo < glen (rel = the
// sub-block's first position - glo). Per 16 features one ldmatrix (four 8-entry
// groups) feeds the MMAs of both k-steps.
template <int FT, int ROWS, class Convert>
__device__ __forceinline__ void multiply(TcSums<FT, ROWS> &acc, uint32_t rows,
                                         const uint16_t *halves, int rel, uint32_t glen,
                                         Convert convert) {
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    uint4 b = make_uint4(0u, 0u, 0u, 0u), c = b;
    if constexpr (ROWS == 1) {
        if (g < 2) b = *reinterpret_cast<const uint4 *>(halves + g * EB + t * 8);
    } else {
        b = *reinterpret_cast<const uint4 *>(halves + t * 8);
        c = *reinterpret_cast<const uint4 *>(halves + EB + t * 8);
        auto mask = [&](int e) {
            const uint32_t p = uint32_t(rel + 2 * t + e);
            return (p < glen ? 0xffffu : 0u) | (p + 1 < glen ? 0xffff0000u : 0u);
        };
        const uint32_t m0 = mask(0), m1 = mask(8), m2 = mask(16), m3 = mask(24);
        b = make_uint4(b.x & m0, b.y & m1, b.z & m2, b.w & m3);
        c = make_uint4(c.x & m0, c.y & m1, c.z & m2, c.w & m3);
    }
    const uint32_t b0[2] = {b.x, b.z}, b1[2] = {b.y, b.w};
    const uint32_t c0[2] = {c.x, c.z}, c1[2] = {c.y, c.w};
#pragma unroll
    for (int T = 0; T < FT; ++T) {
        uint32_t x[4];
        ldsm_x4_trans(rows ^ uint32_t(T << 4), x);
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            // even features (bytes 0, 2) in matrix rows 0-7, odd in 8-15
            const uint32_t a[4] = {convert(__byte_perm(x[2 * kk], 0u, 0x4240)),
                                   convert(__byte_perm(x[2 * kk], 0u, 0x4341)),
                                   convert(__byte_perm(x[2 * kk + 1], 0u, 0x4240)),
                                   convert(__byte_perm(x[2 * kk + 1], 0u, 0x4341))};
            mma_16816(acc.v[0][T], a, b0[kk], b1[kk]);
            if constexpr (ROWS > 1) mma_16816(acc.v[1][T], a, c0[kk], c1[kk]);
        }
    }
}

// Bits of entries 2t, 2t + 1 (.x) and 8 + 2t, 9 + 2t (.y) as masks of fp16 pairs.
__device__ __forceinline__ uint2 pair_masks(uint32_t bits) {
    const int t = threadIdx.x & 3;
    auto two = [](uint32_t b) {
        return (b & 1u ? 0xffffu : 0u) | (b & 2u ? 0xffff0000u : 0u);
    };
    return make_uint2(two(bits >> (2 * t)), two(bits >> (8 + 2 * t)));
}

// One pass over 16 positions whose rows are staged low plane and high plane (shared
// address `part`), some of them wide (bits of `wide`; `narrow`: of the others that weigh
// anything), weights in `halves` (put_weight<true>). Wide rows' halves go into the MMA as
// they are (staged rows 0 to 15 hold the even features, 16 to 31 the odd ones), the other
// entries' masked out (what was staged for them may be any bits); bytes as in multiply().
// ROWS > 1: the entries that belong to the lane's column g are the bits of `column`. The
// sums stay in local memory (loops over T that are not unrolled): see rest_of_window.
template <int FT, int ROWS, class G>
__device__ __forceinline__ void multiply_both(const TcParams &P, TcSums<FT, ROWS> &acc,
                                              uint32_t part, const uint16_t *halves,
                                              uint32_t wide, uint32_t narrow, uint32_t column) {
    constexpr int kN = EB / 2, P2 = G::P2;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    // ldmatrix: lane l's address is chunk T of staged row q, at slot T ^ swizzle.
    auto staged = [&](int q) {
        return part + (uint32_t(q * G::PITCH) | uint32_t(((q / G::LINE) & (P2 - 1)) << 4));
    };
    uint2 b = make_uint2(0u, 0u), c = b;
    if constexpr (ROWS == 1) {
        if (g < 2) b = *reinterpret_cast<const uint2 *>(halves + g * kN + t * 4);
    } else {
        const uint2 m = pair_masks(column);
        b = *reinterpret_cast<const uint2 *>(halves + t * 4);
        c = *reinterpret_cast<const uint2 *>(halves + kN + t * 4);
        b = make_uint2(b.x & m.x, b.y & m.y);
        c = make_uint2(c.x & m.x, c.y & m.y);
    }
    const uint2 m = pair_masks(wide);
    if (wide != 0u) {
        // entries 0-7 low, 0-7 high, 8-15 low, 8-15 high
        const uint32_t rows = staged((lane & 7) | (lane & 8) << 1 | (lane & 16) >> 1);
        const uint32_t bias = P.half_bias;
#pragma unroll 1
        for (int T = 0; T < FT; ++T) {
            uint32_t x[4];
            ldsm_x4_trans(rows ^ uint32_t(T << 4), x);
            const uint32_t a[4] = {x[0] & m.x, x[1] & m.x, x[2] & m.y, x[3] & m.y};
            const uint32_t one[4] = {bias, bias, bias, bias};       // + 1 per dot: see half_dot
            mma_16816(acc.v[0][T], a, b.x & m.x, b.y & m.y);
            if (bias != 0u) mma_16816(acc.v[0][T], one, b.x & m.x, b.y & m.y);
            if constexpr (ROWS > 1) {
                mma_16816(acc.v[1][T], a, c.x & m.x, c.y & m.y);
                if (bias != 0u) mma_16816(acc.v[1][T], one, c.x & m.x, c.y & m.y);
            }
        }
    }
    if (narrow != 0u) {
        // entries 0-7 and 8-15 of chunk T (lanes 0 to 15 give the addresses)
        const uint32_t rows = staged(lane & 15);
        const uint32_t offset = P.offset;
#pragma unroll 1
        for (int T = 0; T < FT; ++T) {
            uint32_t x[2];
            ldsm_x2_trans(rows ^ uint32_t(T << 4), x);
            const uint32_t a[4] = {bytes_to_half2(__byte_perm(x[0], 0u, 0x4240), offset),
                                   bytes_to_half2(__byte_perm(x[0], 0u, 0x4341), offset),
                                   bytes_to_half2(__byte_perm(x[1], 0u, 0x4240), offset),
                                   bytes_to_half2(__byte_perm(x[1], 0u, 0x4341), offset)};
            mma_16816(acc.v[0][T], a, b.x & ~m.x, b.y & ~m.y);
            if constexpr (ROWS > 1) mma_16816(acc.v[1][T], a, c.x & ~m.x, c.y & ~m.y);
        }
    }
}

// The columns of a window's first NS blocks, loaded before its walk begins.
template <int ROWS, bool kW, int SUB, int NS>
__device__ __forceinline__ void fetch_first(const TcParams &P, const Window<ROWS> &w,
                                            Entry<kW> (&c)[NS][SUB]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int b = 0; b < NS; ++b)
#pragma unroll
        for (int u = 0; u < SUB; ++u)
            c[b][u] = fetch_entry<ROWS, kW>(P, w, (b * SUB + u) * EB + lane);
}

// Where lane (g, t) finds the positions of row g (its column of B) in an
// eight-row window.
template <int ROWS>
struct Column {
    int lo = 0;
    uint32_t len = 0;
    __device__ __forceinline__ explicit Column(const Window<ROWS> &w) {
        if constexpr (ROWS > 1) {
            const int g = (threadIdx.x & 31) >> 2;
            int hi = w.off[1];
            lo = w.off[0];
#pragma unroll
            for (int k = 1; k < ROWS; ++k)
                if (g == k) {
                    lo = w.off[k];
                    hi = w.off[k + 1];
                }
            len = uint32_t(hi - lo);
        }
    }
};

// A window's sums as values, from band k of its rows' scales (unit exponents u: ROWS ==
// 1 the row's, else lane r holds row r's); kAdd: added to `out`.
template <bool kAdd, int FT, int ROWS>
__device__ __forceinline__ void put_sums(const TcSums<FT, ROWS> &acc, int u, int k,
                                         TcRowSums<FT, ROWS == 1 ? 1 : 2> &out) {
    constexpr float kLo = 1.0f / float(1 << kLoShift);
    constexpr int L = TcSums<FT, ROWS>::PARTS - 1;
    const int t = threadIdx.x & 3;
#pragma unroll
    for (int r = 0; r < (ROWS == 1 ? 1 : 2); ++r) {
        const int ur = ROWS == 1 ? u : __shfl_sync(kFullMask, u, 2 * t + r);
        const float back = exp2i(kDotShift - band_unit(ur, k));
        const int lo = ROWS == 1 ? 1 : r;       // columns 0 and 1, or one of each set
#pragma unroll (kAdd ? 1 : FT)
        for (int T = 0; T < FT; ++T)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float v =
                    fmaf(acc.v[L][T][2 * h + lo], kLo, acc.v[0][T][2 * h + r]) * back;
                out.v[r][T][h] = kAdd ? out.v[r][T][h] + v : v;
            }
    }
}

// What becomes of an eight-row window's results: kept for the caller.
template <int FT>
struct KeepSums {
    TcRowSums<FT, 2> *sums;
    __device__ __forceinline__ void operator()(const TcRowSums<FT, 2> &s) const { *sums = s; }
};

// What a window with wide rows or with weights far below their row's largest still
// needs (rarely) after its first walk, which left `sums` and the exponents E. last == 0:
// adds the wide rows of the 32-position sub-blocks marked in `marks` (bit q:
// sub-blocks q << shift .. ((q + 1) << shift) - 1). last > 0: the whole window again, band
// after band of its weights from `last` down to 0, the smallest first, each on its own
// scale. The results go to emit().
//
// A pass looks at every position, collects the entries it takes, a lane each, and walks
// them 16 together, as they come (a block of 32 positions that holds one wide row costs
// the index and scale of 32 and the row of one): copies of one 16 are in flight while
// the 16 before are multiplied. A function of its own, which calls none, keeps its sums
// in local memory and (one-row windows) returns nothing: the first walk's registers need
// not hold both, nor meet its results again (GraphSAGE's walk of 128 features, where no
// window came here: 1880 us with the sums returned, 2190 with them in registers here).
template <int FT, int ROWS, bool kW, class G, class Emit>
__device__ __noinline__ void rest_of_window(TcParams P, Window<ROWS> w, uint8_t *ring,
                                            TcSums<FT, ROWS> sums, int E, uint32_t marks,
                                            int shift, int last, Emit emit) {
    static_assert(G::PARTS >= 2, "one part is copied while one is multiplied");
    const int lane = threadIdx.x & 31;
    const int piece = lane % G::P2, slab = int(blockIdx.y) * FT;
    const bool mine = piece < FT && (slab + piece) * 16 < P.width;
    const uint8_t *plane = P.D + (slab + piece) * 16;
    const int64_t high = P.N * P.ldd;
    const uint32_t ring_s = smem_addr(ring);
    int *checked = reinterpret_cast<int *>(ring + G::CHECKED);
    uint16_t *halves = reinterpret_cast<uint16_t *>(ring + G::HALVES);
    float *floats = reinterpret_cast<float *>(ring + G::HALVES);
    const int nsub = (w.off[ROWS] + EB - 1) / EB;
    const int own_u = unit_exponent(E);
    int band = last;
    TcRowSums<FT, ROWS == 1 ? 1 : 2> out = {};
    auto clear = [&]() {
#pragma unroll 1
        for (int T = 0; T < FT; ++T)
#pragma unroll
            for (int q = 0; q < 4 * TcSums<FT, ROWS>::PARTS; ++q) sums.v[q / 4][T][q % 4] = 0.0f;
    };
    if (last != 0) clear();

    // Collected entries, lane q the q-th: column, weight, row (bits 0-2) and wide (bit 3).
    int count = 0, pcol = 0, pinfo = 0;
    float ps = 0.0f;
    // The 16 in flight: part, weight (on its scale) and row of lane q's, and which are
    // wide or narrow.
    int in_flight = -1, frow = 0;
    float fweight = 0.0f;
    uint32_t fwide = 0, fnarrow = 0;
    auto multiply_in_flight = [&]() {
        put_weight<true>(halves, fweight);
        uint32_t column = 0;
        if constexpr (ROWS > 1)
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t b = __ballot_sync(kFullMask, frow == r);
                if (lane >> 2 == r) column = b;
            }
        __syncwarp();
        multiply_both<FT, ROWS, G>(P, sums, ring_s + uint32_t(in_flight * G::PART), halves, fwide,
                                   fnarrow, column);
        __syncwarp();
    };
    // Starts the copies of the first 16 collected entries and multiplies the 16 before.
    auto flush = [&]() {
        const int e = lane & 15;
        const int col = __shfl_sync(kFullMask, pcol, e), info = __shfl_sync(kFullMask, pinfo, e);
        const float s = __shfl_sync(kFullMask, ps, e);
        const bool live = e < count, wide = live && (info & 8);
        const int part = in_flight == 0 ? 1 : 0;
        __syncwarp();
        put_column<G>(checked, live && (lane < 16 || wide) ? col : -1);
        __syncwarp();
        copy_plane<G, true>(ring_s + uint32_t(part * G::PART), checked, plane, uint32_t(P.ldd), mine,
                            high);
        cp_async_commit();
        if (in_flight >= 0) {
            cp_async_wait<1>();
            __syncwarp();
            multiply_in_flight();
        }
        in_flight = part;
        frow = info & 7;
        const int u = ROWS == 1 ? own_u : __shfl_sync(kFullMask, own_u, frow);
        fweight = live ? s * exp2i(band_unit(u, band)) : 0.0f;
        fwide = __ballot_sync(kFullMask, wide) & 0xffffu;
        fnarrow = __ballot_sync(kFullMask, live && !wide) & 0xffffu;
        count = max(count - 16, 0);
        pcol = __shfl_sync(kFullMask, pcol, e + 16);
        pinfo = __shfl_sync(kFullMask, pinfo, e + 16);
        ps = __shfl_sync(kFullMask, ps, e + 16);
    };
    // The first sub-block of this pass from b on (nsub: none), its entries and their scales.
    auto next = [&](int b) {
        while (last == 0 && b < nsub && !((marks >> (b >> shift)) & 1u)) ++b;
        return b;
    };
    auto entry = [&](int b) {
        Entry<kW> q;
        q.col = -1;
        if (b < nsub) q = fetch_entry<ROWS, kW>(P, w, b * EB + lane);
        return q;
    };
    auto scale_of = [&](const Entry<kW> &q) {
        if (uint32_t(q.col) >= uint32_t(P.N)) return 0.0f;
        return P.rowscale != nullptr
                   ? __ldg(P.rowscale + q.col)
                   : *reinterpret_cast<const float *>(P.D + (int64_t(q.col) + 1) * P.ldd - 4);
    };
#pragma unroll 1
    while (true) {
        int b0 = next(0), b1 = next(b0 + 1);
        Entry<kW> q0 = entry(b0), q1 = entry(b1);
        float s0 = scale_of(q0);
#pragma unroll 1
        while (true) {                              // (past the end: what is left collected)
            const bool end = b0 >= nsub;
            const int b2 = next(b1 + 1);
            const float s1 = scale_of(q1);
            const Entry<kW> q2 = entry(b2);
            const int r = ROWS == 1 ? 0 : row_of<ROWS>(w, b0 * EB + lane);
            const float s = kW ? fabsf(s0) * q0.a : fabsf(s0);
            const bool wide = __float_as_uint(s0) >> 31;
            const int u = ROWS == 1 ? own_u : __shfl_sync(kFullMask, own_u, r);
            const bool take =
                s0 != 0.0f && s != 0.0f &&          // (s0 is 0 where there is no entry)
                (last == 0 ? wide : band_of(exponent_of(__float_as_uint(fabsf(s))), u) == band);
            const unsigned taken = __ballot_sync(kFullMask, take);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {           // 16 positions more: at most 31 collected
                const unsigned m = (taken >> (16 * h)) & 0xffffu;
                if (m == 0u && !end) continue;
                const bool from = take && lane >> 4 == h;
                const int to = count + __popc(m & ((1u << (lane & 15)) - 1u));
                const bool here = lane >= count && lane < count + __popc(m);
                if (from) {
                    checked[to] = q0.col;
                    floats[to] = s;
                }
                __syncwarp();
                if (here) {
                    pcol = checked[lane];
                    ps = floats[lane];
                }
                __syncwarp();
                if (from) checked[to] = r | (wide ? 8 : 0);
                __syncwarp();
                if (here) pinfo = checked[lane];
                __syncwarp();
                count += __popc(m);
                if (count >= 16 || (end && count > 0)) flush();
            }
            if (end) break;
            b0 = b1;
            b1 = b2;
            q0 = q1;
            q1 = q2;
            s0 = s1;
        }
        cp_async_wait<0>();
        __syncwarp();
        if (in_flight >= 0) multiply_in_flight();
        in_flight = -1;
        put_sums<true>(sums, own_u, band, out);
        if (band == 0) break;
        --band;
        clear();
    }
    emit(out);
}

// Walks a window's position stream and leaves its sums in `out`, or, when that takes
// more than this walk, has them passed to emit() and returns false; c holds the
// columns of its first blocks (fetch_first). The warp's ring `ring` (shared,
// TcGeom<FT, SUB, NS>::WARP bytes) is free on entry and on exit.
//
// Pipeline (blocks of SUB x 32 positions; lane e owns position e of each
// sub-block; D = NS - 1): iteration n starts the row copies of block n + D, whose
// columns were loaded an iteration ago, loads the columns of block n + D + 1,
// then waits for block n's rows and multiplies. Block b uses row stage b mod NS.
template <int FT, int ROWS, bool kW, int SUB, int NS, class Emit>
__device__ __forceinline__ bool walk_window(const TcParams &P, const Window<ROWS> &w,
                                           uint8_t *ring, Entry<kW> (&c)[NS][SUB],
                                           TcRowSums<FT, ROWS == 1 ? 1 : 2> &out,
                                           const Emit &emit) {
    using G = TcGeom<FT, SUB, NS>;
    constexpr int P2 = G::P2, D = G::D;
    constexpr int BLOCK = SUB * EB;
    const int lane = threadIdx.x & 31;
    const int total = w.off[ROWS];
    const int nblk = (total + BLOCK - 1) / BLOCK;
    const uint32_t rows_s = smem_addr(ring);
    int *checked = reinterpret_cast<int *>(ring + G::CHECKED);
    uint16_t *halves = reinterpret_cast<uint16_t *>(ring + G::HALVES);
    const uint32_t n32 = uint32_t(P.N);     // N <= INT32_MAX
    const int piece = lane % P2;                            // this lane's chunk of a row
    const int slab = int(blockIdx.y) * FT;                  // first chunk of this column slab
    const bool mine = piece < FT && (slab + piece) * 16 < P.width;
    const uint8_t *Dbytes = P.D + (slab + piece) * 16;
    const uint32_t row_bytes = uint32_t(P.ldd);
    // ldmatrix: lane l supplies chunk T of staged row l, at slot T ^ x of it.
    const uint32_t tl =
        uint32_t(lane * G::PITCH) | uint32_t(((lane / G::LINE) & (P2 - 1)) << 4);
    // Row scales kept in D's rows: the last four bytes of the slab's last chunk.
    const uint32_t in_row = uint32_t(lane * G::PITCH) +
                            uint32_t(((FT - 1) ^ ((lane / G::LINE) & (P2 - 1))) << 4) + 12u;
    // A position's row scale (a sign bit marks a wide row) and, with kW, its a_ij.
    struct Weight {
        float s;
        float a;
        // The weight's magnitude in bits, and the weight on a scale.
        __device__ __forceinline__ uint32_t bits() const {
            return __float_as_uint(kW ? fabsf(s * a) : s) & 0x7fffffffu;
        }
        __device__ __forceinline__ float on(float unit) const {
            float v;        // (a wide row's scale is negative: 0 in this walk; NaN stays)
            asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(v) : "f"(s));
            return (kW ? v * a : v) * unit;
        }
    };
    // Starts the copies of a block's rows to the stage at `stage`; s receives this
    // lane's row scales (0 for a dead position; 1 for a live one when scales are
    // kept in the rows).
    auto start_block = [&](uint32_t stage, const Entry<kW> (&q)[SUB], Weight (&s)[SUB]) {
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
            const int col = q[u].col;
            const bool live = uint32_t(col) < n32;
            put_column<G>(checked + u * EB, live ? col : -1);
            s[u].s = !live ? 0.0f : P.rowscale == nullptr ? 1.0f : __ldg(P.rowscale + col);
            if constexpr (kW) s[u].a = q[u].a;
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < SUB; ++u)
            copy_plane<G>(stage + uint32_t(u * G::PART), checked + u * EB, Dbytes, row_bytes, mine);
    };

    TcSums<FT, ROWS> acc;
#pragma unroll
    for (int p = 0; p < TcSums<FT, ROWS>::PARTS; ++p)
#pragma unroll
        for (int T = 0; T < FT; ++T)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.v[p][T][q] = 0.0f;
    // Sub-blocks that hold wide rows, as rest_of_window takes them.
    uint32_t marks = 0;
    const int shift = max(0, 27 - __clz(max(nblk * SUB - 1, 0)));
    // The weights (bits) that a row's exponent E covers, up to 2^(E + 1): E is these bits'
    // exponent (kNoScale: 0). ROWS == 1: the row's; else of row (lane & 7).
    uint32_t bound = 0;
    auto exponent = [](uint32_t bound_) { return int(bound_ >> 23) - 127; };
    auto covers = [](int e) { return e > kNoScale ? (uint32_t(e + 127) << 23) | 0x7fffffu : 0u; };
    // Weights from here down (bits; 0 aside) are noted: kLookBelow exponents below E.
    auto look_from = [](uint32_t bound_) {
        return uint32_t(max(int(bound_) - ((kLookBelow + 1) << 23), 0));
    };
    float unit = 0.0f;          // ROWS == 1: 2^unit_exponent(E)
    int least = 127;            // no weight of the window but 0 has a smaller exponent
    const Column<ROWS> col(w);

    Weight sq[NS][SUB];         // of blocks n .. n + D
#pragma unroll
    for (int b = 0; b < NS; ++b)
#pragma unroll
        for (int u = 0; u < SUB; ++u) sq[b][u] = Weight{0.0f, 1.0f};
#pragma unroll
    for (int b = 0; b < D; ++b) {
        if (b < nblk) start_block(rows_s + uint32_t(b * G::STAGE), c[b], sq[b]);
        cp_async_commit();
        __syncwarp();           // `checked` is free again
    }
    Entry<kW> cnext[SUB];
#pragma unroll
    for (int u = 0; u < SUB; ++u) cnext[u] = c[D][u];
    uint32_t stage = rows_s;                                // block n's
    uint32_t stage_d = rows_s + uint32_t(D * G::STAGE);     // block n + D's
#pragma unroll 1
    for (int n = 0; n < nblk; ++n) {
        if (n + D < nblk) {
            start_block(stage_d, cnext, sq[D]);
#pragma unroll
            for (int u = 0; u < SUB; ++u)
                cnext[u] = fetch_entry<ROWS, kW>(P, w, ((n + D + 1) * SUB + u) * EB + lane);
        }
        cp_async_commit();              // (the count of groups goes on past the end)
        cp_async_wait<D>();             // block n's rows
        __syncwarp();

        // This block's weights (0 for dead entries) on the scale of the row they
        // belong to; a sign bit marks a wide row.
        uint32_t sb[SUB], top = 0, low = ~0u;
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
            if (!kW && P.rowscale == nullptr && sq[0][u].s != 0.0f)
                sq[0][u].s = *reinterpret_cast<const float *>(ring + (stage - rows_s) +
                                                              u * G::PART + in_row);
            sb[u] = sq[0][u].bits() | (__float_as_uint(sq[0][u].s) & 0x80000000u);
            top = max(top, sb[u]);
            low = min(low, sb[u] - 1u);
        }
        float ws[SUB];
        if constexpr (ROWS == 1) {
            // a wide row, a larger weight, or a much smaller one
            if (__any_sync(kFullMask, top > bound || low < look_from(bound))) {
                uint32_t wb = 0;
#pragma unroll
                for (int u = 0; u < SUB; ++u) {
                    if (__any_sync(kFullMask, sb[u] >> 31)) marks |= 1u << ((n * SUB + u) >> shift);
                    const uint32_t b = sb[u] & 0x7fffffffu;
                    wb = max(wb, b);
                    if (b != 0u) least = min(least, exponent_of(b));
                }
                const int E = exponent(bound), e = exponent_of(__reduce_max_sync(kFullMask, wb));
                if (e > E) {            // keep the sums on the row's current scale
                    if (E != kNoScale) least = min(least, E - kLookBelow);
                    const float f = scale_change(E, e);
                    acc.scale(f, f);
                    bound = covers(e);
                }
                unit = exp2i(unit_exponent(max(E, e)));
            }
#pragma unroll
            for (int u = 0; u < SUB; ++u) ws[u] = sq[0][u].on(unit);
        } else {
            static_assert(ROWS == 1 || SUB == 1, "");
            const int tg = row_of<ROWS>(w, n * EB + lane);
            uint32_t cover = __shfl_sync(kFullMask, bound, tg);
            if (__any_sync(kFullMask, sb[0] > cover || low < look_from(cover))) {
                const uint32_t wb = sb[0] & 0x7fffffffu;
                if (__any_sync(kFullMask, sb[0] >> 31)) marks |= 1u << (n >> shift);
                if (wb != 0u) least = min(least, exponent_of(wb));
                const int tlo = row_of<ROWS>(w, n * EB);
                const int thi = row_of<ROWS>(w, min(n * EB + EB, total) - 1);
                const int E = exponent(bound);
                int Enew = E;
                for (int r = tlo; r <= thi; ++r) {
                    const int e = exponent_of(__reduce_max_sync(kFullMask, tg == r ? wb : 0u));
                    if ((lane & 7) == r) Enew = max(Enew, e);
                }
                if (Enew > E && E != kNoScale) least = min(least, E - kLookBelow);
                const float f = scale_change(E, Enew);
                const int t = lane & 3;
                acc.scale(__shfl_sync(kFullMask, f, 2 * t), __shfl_sync(kFullMask, f, 2 * t + 1));
                bound = covers(Enew);
                cover = __shfl_sync(kFullMask, bound, tg);
            }
            ws[0] = sq[0][0].on(exp2i(unit_exponent(exponent(cover))));
        }
#pragma unroll
        for (int u = 0; u < SUB; ++u) put_weight(halves + u * 2 * EB, ws[u]);
        __syncwarp();
        const uint32_t offset = P.offset;
#pragma unroll
        for (int u = 0; u < SUB; ++u)
            multiply<FT, ROWS>(acc, stage + uint32_t(u * G::PART) + tl, halves + u * 2 * EB,
                               (n * SUB + u) * EB - col.lo, col.len,
                               [&](uint32_t h) { return bytes_to_half2(h, offset); });
        __syncwarp();           // this stage is refilled in iteration n + 1
#pragma unroll
        for (int b = 0; b < D; ++b)
#pragma unroll
            for (int u = 0; u < SUB; ++u) sq[b][u] = sq[b + 1][u];
        stage_d = stage;
        stage = stage == rows_s + uint32_t(D * G::STAGE) ? rows_s : stage + uint32_t(G::STAGE);
    }
    cp_async_wait<0>();         // the ring is idle before the next window
    __syncwarp();
    if (P.rowscale == nullptr) marks = 0u;      // (scales kept in the rows have no wide rows)
    const int E = exponent(bound);
    const int umin = ROWS == 1 ? unit_exponent(E) : __reduce_min_sync(kFullMask, unit_exponent(E));
    const int last = band_of(__reduce_min_sync(kFullMask, least), umin);
    if (last != 0 || (marks != 0u && P.rowscale != nullptr)) {
        if (P.rowscale == nullptr) marks = 0u;
        if constexpr (ROWS == 1) {
            rest_of_window<FT, ROWS, kW, G>(P, w, ring, acc, E, marks, shift, last, emit);
            return false;
        } else {
            TcRowSums<FT, 2> sums;
            rest_of_window<FT, ROWS, kW, G>(P, w, ring, acc, E, marks, shift, last,
                                            KeepSums<FT>{&sums});
            out = sums;
            return true;
        }
    }
    put_sums<false>(acc, unit_exponent(E), 0, out);
    return true;
}

// Epilogue of the plain aggregation: H_if = dinv_i * (c_f * sum_f) for f < F
// (features f0 .. f0 + 16 FT - 1 of the block's column slab), with an
// optional argmax of each row (lowest index on ties; one slab only). Called by
// all lanes for one output row per group of eight lanes (lane bits 2..4); i is
// -1 where a lane's group has none. `alone`: one row, in the lanes with t = 0.
template <int FT>
struct TcStore {
    float *H;
    int64_t ldh;
    int F;
    const float *colscale;   // nullable: 1
    int32_t *pred;           // nullable (one column slab only)
    bool vec2;               // feature pairs of H are 8-byte aligned
    // GraphSAGE (Ds non-null): the node's own product is added, from the self half
    // of its row (its bytes, or its halves in the two planes, the high one `high` bytes on)
    // with its row scale.
    const uint8_t *Ds;
    int64_t ldd;
    int64_t high;
    const float *rowscale;
    const float *colscale_s;
    int K;
    const float *sScale = nullptr;      // shared: the slab's column scales, set by prologue()
    static constexpr size_t kSmemFloats = 16 * FT;
    __device__ __forceinline__ void prologue(float *smem) {
        const int f = int(blockIdx.y) * 16 * FT + int(threadIdx.x);
        if (threadIdx.x < 16 * FT)
            smem[threadIdx.x] = colscale == nullptr ? 1.0f : f < F ? __ldg(colscale + f) : 0.0f;
        sScale = smem;
    }
    // The node's own dot with self column f.
    __device__ __forceinline__ float own_dot(int64_t i, int f, bool wide) const {
        const uint8_t *p = Ds + i * ldd;
        if (!wide) return float(2 * (int(__ldg(p + f)) - 128) + (K & 1));
        const uint16_t h = *reinterpret_cast<const uint16_t *>(p + (f & 1 ? high : 0) + (f & ~1));
        return fmaf(__half2float(__ushort_as_half(h)), 1024.0f, float(half_dot_bias(K)));
    }
    template <bool kAlone>
    __device__ __forceinline__ void row(int64_t i, float di, const float (&v)[FT][2]) const {
        const int g = (threadIdx.x & 31) >> 2;
        const int f0 = int(blockIdx.y) * 16 * FT + 2 * g;
        float bestv = 0.0f;
        int best = -1;
        if (i >= 0) {
            float *h = H + i * ldh;
            float self = 0.0f;
            bool wide = false;
            if (Ds != nullptr) {
                const float s = __ldg(rowscale + i);
                wide = __float_as_uint(s) >> 31;
                self = fabsf(s);
            }
#pragma unroll
            for (int T = 0; T < FT; ++T) {
                const int f = f0 + 16 * T;
                if (f >= F) continue;
                const bool two = f + 1 < F;
                const float2 cs = *reinterpret_cast<const float2 *>(sScale + 16 * T + 2 * g);
                float o0 = di * (cs.x * v[T][0]), o1 = di * (cs.y * v[T][1]);
                if (Ds != nullptr) {
                    o0 += self * (__ldg(colscale_s + f) * own_dot(i, f, wide));
                    if (two) o1 += self * (__ldg(colscale_s + f + 1) * own_dot(i, f + 1, wide));
                }
                if (two && vec2) {
                    *reinterpret_cast<float2 *>(h + f) = make_float2(o0, o1);
                } else {
                    h[f] = o0;
                    if (two) h[f + 1] = o1;
                }
                if (best < 0 || o0 > bestv) {
                    bestv = o0;
                    best = f;
                }
                if (two && o1 > bestv) {
                    bestv = o1;
                    best = f + 1;
                }
            }
        }
        if (pred != nullptr) {          // over the 8 lanes of the row (lane bits 2..4)
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                const float ov = __shfl_xor_sync(kFullMask, bestv, o);
                const int oi = __shfl_xor_sync(kFullMask, best, o);
                if (oi >= 0 && (best < 0 || ov > bestv || (ov == bestv && oi < best))) {
                    bestv = ov;
                    best = oi;
                }
            }
            if (i >= 0 && g == 0) pred[i] = best;
        }
    }
};

// Epilogue of layer 1 fused with layer 2's binarization and product: H1_i =
// dinv_i * beta1 . sums (optionally stored), its signs packed LSB-first,
// alpha2_i = mean |H1_i| (Eqs. 7-8), and the XNOR-popcount dots against W2's
// packed columns (Eqs. 11-12), stored as byte dots in rows of ldd2 bytes
// (|dot| <= Fh <= 128: no row is wide) with the row scale s2_i = alpha2_i *
// dinv_i, in s2 or in the row's last four bytes -- layer 2's factored product.
template <int FT>
struct TcPackGemm {
    float *H1;               // nullable N x Fh (row stride ldh1)
    int64_t ldh1;
    int Fh;
    const float *beta1;      // Fh
    const uint64_t *wbits2;  // Fo x words2
    int Fo;
    int words2;              // 1 or 2
    uint8_t *D2;             // N x ldd2 byte dots
    int64_t ldd2;
    float *s2;               // N; nullptr: the last four bytes of D2's rows
    const float *sBeta1 = nullptr;     // shared copies, set by prologue()
    const uint64_t *sW2 = nullptr;

    static constexpr size_t kSmemFloats = 128 + 2 * kMaxFusedOut * 2;
    __device__ __forceinline__ void prologue(float *smem) {
        float *b1 = smem;
        uint64_t *w2 = reinterpret_cast<uint64_t *>(smem + 128);
        for (int q = threadIdx.x; q < 128; q += kTcThreads) b1[q] = q < Fh ? __ldg(beta1 + q) : 0.0f;
        for (int q = threadIdx.x; q < Fo * words2; q += kTcThreads) w2[q] = __ldg(wbits2 + q);
        sBeta1 = b1;
        sW2 = w2;
    }
    template <bool kAlone>
    __device__ __forceinline__ void row(int64_t i, float di, const float (&v)[FT][2]) const {
        constexpr int NW = (FT + 1) / 2;        // 32-feature words
        const int lane = threadIdx.x & 31;
        const int g = lane >> 2;
        uint32_t w[NW];
        float l1 = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) w[q] = 0u;
#pragma unroll
        for (int T = 0; T < FT; ++T) {
            const int f = 16 * T + 2 * g;
            const float2 b = *reinterpret_cast<const float2 *>(sBeta1 + f);     // 0 past Fh
            const float x0 = di * (b.x * v[T][0]), x1 = di * (b.y * v[T][1]);
            if (H1 != nullptr && i >= 0) {
                if (f < Fh) H1[i * ldh1 + f] = x0;
                if (f + 1 < Fh) H1[i * ldh1 + f + 1] = x1;
            }
            if (f < Fh) l1 += fabsf(x0);
            if (f + 1 < Fh) l1 += fabsf(x1);
            if (x0 >= 0.0f && f < Fh) w[T / 2] |= 1u << (16 * (T & 1));
            if (x1 >= 0.0f && f + 1 < Fh) w[T / 2] |= 2u << (16 * (T & 1));
        }
        // Over the row's 8 lanes; the one row of a one-row window goes to all lanes.
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            w[q] <<= 2 * g;
            if (kAlone) {
                w[q] = __reduce_or_sync(kFullMask, (lane & 3) == 0 ? w[q] : 0u);
            } else {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) w[q] |= __shfl_xor_sync(kFullMask, w[q], o);
            }
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) l1 += __shfl_xor_sync(kFullMask, l1, o);
        if (i >= 0 && g == 0) {
            const float s = (l1 / float(Fh)) * di;
            if (s2 != nullptr) s2[i] = s;
            else *reinterpret_cast<float *>(D2 + (i + 1) * ldd2 - 4) = s;
        }
        if (kAlone) i = __shfl_sync(kFullMask, i, 0);
        if (i < 0) return;
        const uint64_t w0 = uint64_t(w[0]) | (NW > 1 ? uint64_t(w[NW > 1 ? 1 : 0]) << 32 : 0);
        const uint64_t w1 = NW > 2 ? uint64_t(w[NW > 2 ? 2 : 0]) |
                                         (NW > 3 ? uint64_t(w[NW > 3 ? 3 : 0]) << 32 : 0)
                                   : 0;
        uint8_t *d = D2 + i * ldd2;
        for (int o = kAlone ? lane : g; o < Fo; o += kAlone ? 32 : 8) {
            int mism = __popcll(w0 ^ sW2[o * words2]);
            if (words2 > 1) mism += __popcll(w1 ^ sW2[o * words2 + 1]);
            d[o] = uint8_t(ByteDot(Fh - 2 * mism, Fh).byte());
        }
    }
};

// What becomes of a light window's sums: the epilogue, row by row (dg: the degree of row
// (lane mod ROWS), -1 for none or a heavy block's; dinv: its factor).
template <int FT, int ROWS, class Epi>
struct LightRows {
    Epi epi;
    int64_t row;
    int dg;
    float dinv;
    __device__ __forceinline__ void operator()(
        const TcRowSums<FT, ROWS == 1 ? 1 : 2> &s) const {
        const int lane = threadIdx.x & 31;
        if constexpr (ROWS == 1) {
            if (dg >= 0) epi.template row<true>((lane & 3) == 0 ? row : -1, dinv, s.v[0]);
        } else {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int q = 2 * (lane & 3) + r;
                const bool has = __shfl_sync(kFullMask, dg, q) >= 0;
                const float di = __shfl_sync(kFullMask, dinv, q);
                epi.template row<false>(has ? row + q : -1, di, s.v[r]);
            }
        }
    }
};

// What becomes of a warp's part of a heavy row: a partial row in shared memory.
template <int FT>
struct HeavyPart {
    float *part;
    __device__ __forceinline__ void operator()(const TcRowSums<FT, 1> &s) const {
        const int lane = threadIdx.x & 31;
        if ((lane & 3) == 0) {
#pragma unroll
            for (int T = 0; T < FT; ++T)
#pragma unroll
                for (int h = 0; h < 2; ++h) part[16 * T + 2 * (lane >> 2) + h] = s.v[0][T][h];
        }
    }
};

// Light windows (heavy rows left out), which warps take in turn as they become
// free, so that no warp waits for the one with the longest rows: all blocks from
// one counter (P.counters), or a block's warps from its share of them, windows
// first, first + step, ... (`next` counts those taken). A
// warp draws its next window and loads its row pointers when it begins the one
// before, and that window's first columns before it writes the results.
template <int FT, int ROWS, bool kW, int SUB, int NS, class Epi>
__device__ __forceinline__ void light_windows(const TcParams &P, const Epi &epi, uint8_t *ring,
                                              int *next, int64_t first, int64_t step) {
    const int lane = threadIdx.x & 31;
    const int64_t windows = (P.N + ROWS - 1) / ROWS;
    auto draw = [&]() -> int64_t {          // the output row of the next window, or -1
        int64_t k = 0;
        if (lane == 0)
            k = P.counters != nullptr ? int64_t(atomicAdd(P.counters + blockIdx.y, 1u))
                                      : first + step * atomicAdd(next, 1);
        k = __shfl_sync(kFullMask, k, 0);
        return k < windows ? k * ROWS : -1;
    };
    // Row pointer `lane` of a window (rows past the end repeat the last pointer).
    auto pointer = [&](int64_t row0) -> int64_t {
        return lane <= ROWS ? __ldg(P.rowptr + min(row0 + lane, P.N)) : 0;
    };
    Window<ROWS> w;
    int64_t row0 = draw();
    if (row0 < 0) return;
    int64_t ptr = pointer(row0);
    Entry<kW> c[NS][SUB];
    const int own = P.agg == kAggSage ? 0 : 1;      // self-loop entries of a row's list
    int deg;                                // of row (lane mod ROWS); -1: none, or a heavy block's
    auto enter = [&]() {                    // row0's window from its row pointers
        w.first = row0;
        const int r = ROWS == 1 ? 0 : lane & 7;
        const int64_t b = min(max(__shfl_sync(kFullMask, ptr, r), int64_t(0)), P.nnz);
        const int64_t e = min(max(__shfl_sync(kFullMask, ptr, r + 1), b), P.nnz);
        deg = row0 + r < P.N && e - b <= P.heavy_degree ? int(e - b) : -1;
        const int len = deg < 0 ? 0 : deg + own;
        int end = len;                      // inclusive prefix sum over the window's rows
        if constexpr (ROWS > 1) {
#pragma unroll
            for (int o = 1; o < ROWS; o <<= 1) {
                const int v = __shfl_up_sync(kFullMask, end, o, ROWS);
                if (r >= o) end += v;
            }
        }
        w.off[0] = 0;
        if constexpr (ROWS == 1) {
            w.off[1] = end;
        } else {
#pragma unroll
            for (int k = 0; k < ROWS; ++k) w.off[k + 1] = __shfl_sync(kFullMask, end, k);
        }
        w.cbase = b - (end - len) - own;
        w.self0 = own != 0;
        fetch_first<ROWS, kW, SUB, NS>(P, w, c);
    };
    enter();
    while (true) {
        const int64_t row = row0;
        row0 = draw();
        if (row0 >= 0) ptr = pointer(row0);
        const int dg = deg;
        const float dinv =
            dg < 0 ? 0.0f : row_factor(P, row + (ROWS == 1 ? 0 : lane & 7), dg);
        const LightRows<FT, ROWS, Epi> emit{epi, row, dg, dinv};
        TcRowSums<FT, ROWS == 1 ? 1 : 2> s;
        const bool whole = walk_window<FT, ROWS, kW, SUB, NS>(P, w, ring, c, s, emit);
        if (row0 >= 0) enter();
        if (whole) emit(s);
        if (row0 < 0) return;
    }
}

// Heavy rows (blocks take chunks of 32 rows in turn): every warp of the block
// walks an equal part of the row's list (a one-row window), and warp 0 adds the
// partial rows in warp order. A warp's partial row goes to the start of
// its own ring, which is idle between walks.
template <int FT, bool kW, int SUB, int NS, class Epi>
__device__ __forceinline__ void heavy_rows(const TcParams &P, const Epi &epi, uint8_t *rings) {
    using G = TcGeom<FT, SUB, NS>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    uint8_t *ring = rings + warp * G::WARP;
    auto part = [&](int q) { return reinterpret_cast<float *>(rings + q * G::WARP); };
    for (int64_t base = int64_t(blockIdx.x) * 32; base < P.N;
         base += int64_t(P.heavy_blocks) * 32) {
        const int64_t r = base + lane;
        bool heavy = false;
        int64_t rb = 0, deg = 0;
        if (r < P.N) {
            const int64_t a = __ldg(P.rowptr + r), e0 = __ldg(P.rowptr + r + 1);
            rb = min(max(a, int64_t(0)), P.nnz);
            deg = min(max(e0, rb), P.nnz) - rb;
            heavy = deg > P.heavy_degree;
        }
        unsigned mm = __ballot_sync(kFullMask, heavy);
        while (mm != 0u) {
            const int bit = __ffs(mm) - 1;
            mm &= mm - 1u;
            const int64_t i = base + bit;
            const int64_t cb = __shfl_sync(kFullMask, rb, bit);
            const int64_t dg = __shfl_sync(kFullMask, deg, bit);
            const int own = P.agg == kAggSage ? 0 : 1;
            const int64_t span = dg + own;
            const int64_t q0 = span * warp / kTcWarps, q1 = span * (warp + 1) / kTcWarps;
            Window<1> w;
            w.first = i;
            w.self0 = own != 0 && q0 == 0;
            w.cbase = cb + q0 - own;
            w.off[0] = 0;
            w.off[1] = int(q1 - q0);
            TcRowSums<FT, 1> s;
            Entry<kW> c[NS][SUB];
            fetch_first<1, kW, SUB, NS>(P, w, c);
            const HeavyPart<FT> emit{part(warp)};
            if (walk_window<FT, 1, kW, SUB, NS>(P, w, ring, c, s, emit)) emit(s);
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int T = 0; T < FT; ++T)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float a = 0.0f;
                        for (int q = 0; q < kTcWarps; ++q) a += part(q)[16 * T + 2 * g + h];
                        s.v[0][T][h] = a;
                    }
                epi.template row<true>(t == 0 ? i : -1, row_factor(P, i, dg), s.v[0]);
            }
            __syncthreads();    // the rings are walked again by the next heavy row
        }
    }
}

// The second kernel that takes over where more than one row in `share` is wide (wide_rows
// nullptr: there is none), and the rows that are then made ready for it: `planes` from
// their first byte (TcParams::D may be their other half). Not part of TcParams, which
// rest_of_window takes along (there, 1790 -> 1930 us for GraphSAGE's walk).
struct SecondKernel {
    const uint32_t *wide_rows;
    int share;
    uint8_t *planes;
};

// Turns the rows that are not wide into halves too, in place, a chunk of 16 features a
// thread (the even features' halves over its bytes, the odd ones' in the high plane).
__device__ __forceinline__ void rows_to_halves(uint8_t *planes, int64_t ldd, int64_t N,
                                               const float *rowscale, uint32_t offset) {
    const int64_t chunks = ldd / 16, total = N * chunks;
    for (int64_t q = int64_t(blockIdx.x) * kTcThreads + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * kTcThreads) {
        if (__float_as_uint(__ldg(rowscale + q / chunks)) >> 31) continue;
        uint4 *low = reinterpret_cast<uint4 *>(planes) + q;
        const uint4 v = *low;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t e[4], o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            e[k] = bytes_to_half2(__byte_perm(w[k], 0u, 0x4240), offset);
            o[k] = bytes_to_half2(__byte_perm(w[k], 0u, 0x4341), offset);
        }
        *low = make_uint4(e[0], e[1], e[2], e[3]);
        low[total] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}
__device__ __noinline__ void rows_to_halves_call(uint8_t *planes, int64_t ldd, int64_t N,
                                                 const float *rowscale, uint32_t offset) {
    rows_to_halves(planes, ldd, N, rowscale, offset);
}

template <int FT, int ROWS, bool kW, int SUB, int NS, class Epi>
__global__ void __launch_bounds__(kTcThreads, tc_blocks(FT, ROWS))
spmm_tc_kernel(TcParams P, Epi epi, SecondKernel second) {
    using G = TcGeom<FT, SUB, NS>;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int next;        // windows of the block's share that its warps have taken
    if (threadIdx.x == 0) next = 0;
    // (the second kernel waits for this one's end; its launch need not)
    if (second.wide_rows != nullptr) allow_dependent_launch();
    // The rings start on a 128-byte line (the ldmatrix addressing relies on it).
    uint8_t *rings = smem + ((128u - (smem_addr(smem) & 127u)) & 127u);
    float *extra = reinterpret_cast<float *>(rings + kTcWarps * G::WARP);
    grid_dependency_wait();     // the dots and row scales come from the previous kernel
    if (second.wide_rows != nullptr && many_wide(second.wide_rows, P.N, second.share)) {
        if (blockIdx.y != 0) return;
        // (called or inlined, by which the walk below it comes out faster: 128 features in
        // one-row windows 1765 us called, 1817 inlined; 64 in eight-row windows 503, 464)
        if (ROWS == 1) rows_to_halves_call(second.planes, P.ldd, P.N, P.rowscale, P.offset);
        else rows_to_halves(second.planes, P.ldd, P.N, P.rowscale, P.offset);
        return;
    }
    epi.prologue(extra);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    uint8_t *ring = rings + warp * G::WARP;
    // Blocks [0, heavy_blocks) walk the heavy rows; blocks from light_first on
    // then walk light windows. Many windows: one wave of
    // persistent blocks does both (a block per window would hold its SM until
    // its longest row ended, most of its warps idle). Few windows: a warp per
    // window, with separate leading blocks for the heavy rows.
    if (int(blockIdx.x) < P.heavy_blocks) heavy_rows<FT, kW, SUB, NS>(P, epi, rings);
    if (int(blockIdx.x) < P.light_first) return;
    light_windows<FT, ROWS, kW, SUB, NS>(P, epi, ring, &next, int(blockIdx.x) - P.light_first,
                                int(gridDim.x) - P.light_first);
}

template <int FT, int SUB, int NS>
size_t tc_smem(size_t extra_floats) {
    using G = TcGeom<FT, SUB, NS>;
    static_assert(16 * FT * 4 <= G::WARP, "a warp's partial row must fit its ring");
    static_assert(G::WARP % 128 == 0, "stages must start on 128-byte lines");
    return 128 + size_t(kTcWarps) * G::WARP + extra_floats * 4;
}

// Heavy-row threshold: rows above max(64, 4 x the mean degree) take a whole block.
int64_t tc_heavy_degree(int64_t N, int64_t nnz) {
    const int64_t mean = N > 0 ? nnz / N : 0;
    return 4 * mean > 64 ? 4 * mean : 64;
}

template <int FT, int ROWS, bool kW, class Epi>
void launch_rows(const TcParams &P0, const Epi &epi, const SecondKernel &second, int slabs,
                 const DeviceInfo &dev, cudaStream_t s, bool pdl) {
    TcParams P = P0;
    P.heavy_degree = tc_heavy_degree(P.N, P.nnz);
    constexpr int SUB = tc_sub(FT, ROWS), NS = tc_stages(FT, ROWS);
    const size_t smem = tc_smem<FT, SUB, NS>(Epi::kSmemFloats);
    auto kernel = spmm_tc_kernel<FT, ROWS, kW, SUB, NS, Epi>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    // One wave of resident blocks, or fewer when the windows do not need them.
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kTcThreads, smem) !=
            cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const int64_t windows = (P.N + ROWS - 1) / ROWS;
    const int64_t need = (windows + kTcWarps - 1) / kTcWarps;
    const int64_t resident = int64_t(per_sm) * dev.sm_count;
    const int64_t chunks = (P.N + 31) / 32;
    int64_t blocks;
    if (need > 4 * resident) {          // persistent: every block does both
        blocks = resident;
        P.heavy_blocks = int(resident);
        P.light_first = 0;
    } else {                            // leading heavy blocks, then a warp per window
        const int64_t hb = chunks < 2 * int64_t(dev.sm_count) ? chunks : 2 * int64_t(dev.sm_count);
        P.heavy_blocks = int(hb);
        P.light_first = int(hb);
        P.counters = nullptr;           // (every block has its own windows)
        blocks = hb + need;
    }
    const dim3 grid(static_cast<unsigned>(blocks), static_cast<unsigned>(slabs));
    launch_kernel(kernel, grid, dim3(kTcThreads), smem, s, pdl, dim3(1, 1, 1), P, epi, second);
}

// Rows per window: one when rows are long (a window's blocks then all belong to
// one row; at a mean degree of 50 and 41 features 122 us against 113 us for eight
// rows, at 120 and 100 features 301 against 366 us), or too few to give many
// warps eight (1001 rows: 6.3 us against 7.8 us; 5000 rows of mean degree 6: 11.0
// against 10.0 us; 10,000 of 30: 28.7 against 30.6 us), else eight (2^20 rows of
// mean degree 16, 64 features: 442 us against 894 us).
constexpr int64_t kOneRowDegree = 64;
constexpr int64_t kFewRows = 16;        // per SM
constexpr int64_t kFewLongRows = 128;   // per SM, of mean degree kFewDegree and more
constexpr int64_t kFewDegree = 24;

bool tc_one_row(int64_t N, int64_t nnz, const DeviceInfo &dev) {
    return nnz >= kOneRowDegree * N || N < kFewRows * int64_t(dev.sm_count) ||
           (nnz >= kFewDegree * N && N < kFewLongRows * int64_t(dev.sm_count));
}

template <int FT, bool kW = false, class Epi>
void launch_ft(const TcParams &P, const Epi &epi, const SecondKernel &second,
               const DeviceInfo &dev, cudaStream_t s, bool pdl, int slabs = 1) {
    if (tc_one_row(P.N, P.nnz, dev)) launch_rows<FT, 1, kW>(P, epi, second, slabs, dev, s, pdl);
    else launch_rows<FT, kTcRows, kW>(P, epi, second, slabs, dev, s, pdl);
}

TcParams tc_params(const int64_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                   const uint8_t *D, int64_t ldd, const float *rowscale, int K) {
    // 2^-10 in fp16, as often as a wide row's halves lack 1
    const uint32_t bias = half_dot_bias(K) != 0 ? 0x1400u : 0u;
    return TcParams{rowptr, colidx, N, nnz, D, ldd, int(ldd), rowscale, kAggGcn, nullptr, nullptr,
                    byte_dot_offset(K), bias | (bias << 16), 0, nullptr, 0, 0};
}

// One wide row in how many is many, for the second kernel to take over: where it still
// beats this one's walk and the wide rows' own by what they cost there. One-row windows
// (232,965 nodes of mean degree 492, F = 128: 2690 us against 1790 without wide rows, and
// 2560 with one in 256); eight-row windows, whose wide rows cost most, over 16-bit dots
// that stay in L2 (100,003 nodes of mean degree 50, F = 100: 270 against 235, 324 with one
// in 1024) or do not (2^20 of 16, F = 64: 1270 against 950, 1330 with one in 64).
int many_wide_share(int64_t N, int64_t nnz, int F, const DeviceInfo &dev) {
    return tc_one_row(N, nnz, dev) ? 256 : N * int64_t(F) * 2 <= (int64_t(96) << 20) ? 4096 : 128;
}

// Column slabs of at most 128 features, of equal width.
template <bool kW>
void launch_store(const SpmmTcArgs &a, const DeviceInfo &dev, cudaStream_t s, bool pdl) {
    TcParams P = tc_params(a.rowptr, a.colidx, a.N, a.nnz, a.D, a.ldd, a.rowscale, a.K);
    P.agg = a.agg;
    P.values = a.values;
    P.dinv = a.dinv;
    P.counters = a.counters;
    const SecondKernel second{spmm_tc_second_kernel(a.N, a.nnz, a.K, a.F) ? a.wide_rows : nullptr,
                              many_wide_share(a.N, a.nnz, a.F, dev),
                              const_cast<uint8_t *>(a.Ds != nullptr ? a.Ds : a.D)};
    const bool vec2 = a.ldh % 2 == 0 && aligned_to(a.H, 8);
    const int tiles = (a.F + 15) / 16, slabs = (tiles + 7) / 8;
    P.width = 16 * tiles;
    switch ((tiles + slabs - 1) / slabs) {
#define BIGCN_TC_CASE(ft)                                                                      \
    case ft:                                                                                   \
        launch_ft<ft, kW>(P,                                                                   \
                          TcStore<ft>{a.H, a.ldh, a.F, a.colscale, a.pred, vec2, a.Ds, a.ldd,  \
                                      a.N * a.ldd, a.rowscale, a.colscale_s, a.K},             \
                          second, dev, s, pdl, slabs);                                         \
        break;
        BIGCN_TC_CASE(1)
        BIGCN_TC_CASE(2)
        BIGCN_TC_CASE(3)
        BIGCN_TC_CASE(4)
        BIGCN_TC_CASE(5)
        BIGCN_TC_CASE(6)
        BIGCN_TC_CASE(7)
        BIGCN_TC_CASE(8)
#undef BIGCN_TC_CASE
        default: break;
    }
    if (second.wide_rows != nullptr) launch_spmm_halves(a, second.share, dev, s, pdl);
}

}  // namespace

bool spmm_tc_second_kernel(int64_t N, int64_t nnz, int K, int F) {
    // (halves that lack a bias are rare enough to be left to the tensor cores)
    return half_dot_bias(K) == 0 && (N * int64_t(F) >= (int64_t(4) << 20) ||
                                     double(nnz) * F >= double(int64_t(128) << 20));
}

void launch_spmm_tc(const SpmmTcArgs &a, const DeviceInfo &dev, cudaStream_t s, bool pdl) {
    if (a.N == 0) return;
    if (a.agg == kAggWeighted) launch_store<true>(a, dev, s, pdl);
    else launch_store<false>(a, dev, s, pdl);
}

bool spmm_tc_pack_gemm_supported(int Fh, int Fo) {
    return Fh >= 1 && Fh <= 128 && Fo >= 1 && Fo <= kMaxFusedOut;
}

void launch_spmm_tc_pack_gemm(const SpmmTcPackGemmArgs &a, const DeviceInfo &dev,
                              cudaStream_t s, bool pdl) {
    if (a.N == 0) return;
    TcParams P = tc_params(a.rowptr, a.colidx, a.N, a.nnz, a.D1, a.ldd1, a.s1, a.K);
    P.counters = a.counters;
    const SecondKernel second{spmm_tc_second_kernel(a.N, a.nnz, a.K, a.Fh) ? a.wide_rows : nullptr,
                              many_wide_share(a.N, a.nnz, a.Fh, dev),
                              const_cast<uint8_t *>(a.D1)};
    const int words2 = (a.Fh + 63) / 64;
    switch ((a.Fh + 15) / 16) {
#define BIGCN_TCPG_CASE(ft)                                                                 \
    case ft: {                                                                              \
        TcPackGemm<ft> e{a.H1, a.ldh1, a.Fh, a.beta1, a.wbits2, a.Fo, words2, a.D2, a.ldd2, \
                         a.s2};                                                             \
        launch_ft<ft>(P, e, second, dev, s, pdl);                                           \
        break;                                                                              \
    }
        BIGCN_TCPG_CASE(1)
        BIGCN_TCPG_CASE(2)
        BIGCN_TCPG_CASE(3)
        BIGCN_TCPG_CASE(4)
        BIGCN_TCPG_CASE(5)
        BIGCN_TCPG_CASE(6)
        BIGCN_TCPG_CASE(7)
        BIGCN_TCPG_CASE(8)
#undef BIGCN_TCPG_CASE
        default: break;
    }
    if (second.wide_rows != nullptr) launch_spmm_halves_pack_gemm(a, second.share, dev, s, pdl);
}

}  // namespace bigcn
