// Internal helpers shared by the Bi-GCN CUDA translation units: argument
// checks, the per-device property cache, launch-status mapping and warp-level
// reductions. Not part of the public interface (include/bigcn.h).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "bigcn.h"

namespace bigcn {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int64_t kMaxElems = int64_t(1) << 62;

struct DeviceInfo {
    int device;
    int sm_count;
    int max_smem_optin;  // bytes of shared memory a block may opt in to
};

// Properties of the current device, queried once per device and cached.
// Returns BIGCN_ERR_UNSUPPORTED unless the device is sm_103.
bigcn_status current_device(DeviceInfo *info);

// Maps the launch result (cudaGetLastError) to a status.
bigcn_status launch_status();

inline bool aligned_to(const void *p, size_t a) {
    return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0;
}

// True when the byte ranges [a, a + na) and [b, b + nb) intersect.
inline bool overlaps(const void *a, size_t na, const void *b, size_t nb) {
    if (a == nullptr || b == nullptr || na == 0 || nb == 0) return false;
    uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
    return pa < pb + nb && pb < pa + na;
}

// Bytes spanned by a rows x cols matrix of elem-byte elements with row stride ld.
inline size_t span_bytes(int64_t rows, int64_t cols, int64_t ld, size_t elem) {
    if (rows <= 0 || cols <= 0) return 0;
    return size_t((rows - 1) * ld + cols) * elem;
}

inline cudaStream_t as_stream(void *s) { return reinterpret_cast<cudaStream_t>(s); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
    return v;
}

// Programmatic dependent launch. A kernel launched with the programmatic
// stream-serialization attribute may begin while its predecessor in the
// stream is still running; grid_dependency_wait() returns once the
// predecessor grid has completed and its memory writes are visible (at once
// when the launch has no programmatic predecessor). Every kernel calls it
// before it touches anything an earlier kernel writes; work on the call's
// own inputs may come first. allow_dependent_launch() lets the next kernel
// launch before this one finishes.
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void allow_dependent_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A word that the previous kernel of the chain wrote, read right after
// grid_dependency_wait(). A read-only (__ldg) load is free of the wait for the
// compiler, which may move it ahead of it when both are in straight line: the
// product's first operand words then came from before the packing (seen as wrong
// dots in one launch of ten). A volatile load stays behind the wait.
__device__ __forceinline__ uint64_t load_upstream(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Launches `kernel` with optional programmatic serialization (pdl) and an
// optional cluster shape; the launch error is left for launch_status().
template <typename... KArgs, typename... Args>
void launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                   cudaStream_t stream, bool pdl, dim3 cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (cluster.x * cluster.y * cluster.z > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster.x;
        attr[n].val.clusterDim.y = cluster.y;
        attr[n].val.clusterDim.z = cluster.z;
        ++n;
    }
    if (pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Records caller-supplied timing events between the kernels of an entry
// point: mark() records the next event of the array (if any is left) on the
// stream. Inside a stream capture an event must be recorded as an external
// node to be timed later; outside a capture a plain record does that.
class EventMarks {
  public:
    EventMarks(void *const *events, int32_t n, cudaStream_t s) : events_(events), n_(n), s_(s) {
        if (n_ > 0 && cudaStreamIsCapturing(s_, &capture_) != cudaSuccess) {
            cudaGetLastError();
            ok_ = false;
        }
    }
    bool ok() const { return ok_; }
    bool failed() const { return failed_; }
    void mark() {
        if (recorded_ < n_) {
            cudaEvent_t ev = static_cast<cudaEvent_t>(events_[recorded_]);
            const cudaError_t r = capture_ == cudaStreamCaptureStatusActive
                                      ? cudaEventRecordWithFlags(ev, s_, cudaEventRecordExternal)
                                      : cudaEventRecord(ev, s_);
            if (r != cudaSuccess) failed_ = true;
        }
        ++recorded_;
    }

  private:
    void *const *events_;
    int32_t n_;
    cudaStream_t s_;
    cudaStreamCaptureStatus capture_ = cudaStreamCaptureStatusNone;
    int32_t recorded_ = 0;
    bool ok_ = true;
    bool failed_ = false;
};

// A dot of Eqs. 11-12 as uint16 with a bias of 32768 (|dot| <= 32767);
// `valid` false gives the zero dot of a padding column.
__device__ __forceinline__ uint16_t encode_dot(int dot, bool valid) {
    return uint16_t(valid ? dot + 32768 : 32768);
}

// A dot in byte planes. A dot has the parity of K, so it is 2 v + (K & 1), and for dots
// of about sqrt(K) (signs that agree about half the time) v + 128 fits a byte: a row's
// bytes lie in the low plane. A row in which some dot does not -- a wide row -- is kept as
// fp16 instead, feature f's half at byte f & ~1 of the row in the low plane (even f) or
// the high plane (odd f), and the sign bit of its row scale (the scale itself is never
// negative) says so. Half the bytes of a 16-bit dot, and nothing is rounded: a half holds
// the dot times 2^-10, or, where K is odd and the dot may pass fp16's 11 bits, the dot
// less 1 (then even, and below 4096 as K <= kMaxPlanesK).
struct ByteDot {
    int b;                                          // v + 128
    __device__ __forceinline__ ByteDot(int dot, int K) : b(((dot - (K & 1)) >> 1) + 128) {}
    __device__ __forceinline__ bool wide() const { return unsigned(b) > 255u; }
    __device__ __forceinline__ uint32_t byte() const { return uint32_t(b) & 255u; }
};
__host__ __device__ constexpr int half_dot_bias(int K) { return K > 2048 ? (K & 1) : 0; }
__device__ __forceinline__ uint32_t half_dot(int dot, int K) {
    return __half_as_ushort(__float2half_rn(float(dot - half_dot_bias(K)) * (1.0f / 1024.0f)));
}

// Two bytes of such a row, each in a half-word (as fp16 subnormals u 2^-24), to two dots
// times 2^-10: u 2^-24 2^15 + ((K & 1) - 256) 2^-10, exact; byte_dot_offset is the last
// term, twice.
__host__ __device__ constexpr uint32_t byte_dot_offset(int K) {
    return (K & 1) != 0 ? 0xB3F8B3F8u : 0xB400B400u;    // -255/1024, -1/4
}
__device__ __forceinline__ uint32_t bytes_to_half2(uint32_t h, uint32_t offset) {
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(h), "r"(0x78007800u), "r"(offset));
    return r;
}
// Whether more than one row in `share` is wide (*wide_rows of N), by which two kernels
// launched one after the other agree on who does the aggregation: a load behind the
// dependency wait, as load_upstream.
__device__ __forceinline__ bool many_wide(const uint32_t *wide_rows, int64_t N, int share) {
    uint32_t n;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(n) : "l"(wide_rows) : "memory");
    return int64_t(n) * share > N;
}

// Whether column c counts for a row's wide flag: of each half of `half` columns
// the first `valid`.
__device__ __forceinline__ bool flag_column(int c, int half, int valid) {
    return (c >= half ? c - half : c) < valid;
}

// A row scale with its row's wide flag in the sign bit.
__device__ __forceinline__ float flag_scale(float s, bool wide) {
    return __uint_as_float(__float_as_uint(s) | (wide ? 0x80000000u : 0u));
}

// 1 / sqrt(1 + row length): the D^-1/2 factor of A + I (Sec. 3.1, Eq. 1),
// with IEEE-rounded sqrt and division.
__device__ __forceinline__ float inv_sqrt_degree(int64_t row_len) {
    return 1.0f / sqrtf(1.0f + float(row_len));
}

}  // namespace bigcn
