// Shared host/device helpers of the AMXFP4 CUDA library (sm_100a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "amx.h"

namespace amx {

// Group sizes: 16, 32, 64 or 128 elements, or the whole row as one group (group_size == K, K a multiple of 8:
// the grouping of the paper's worked example), which only the generic kernels take.
inline bool fixed_group_size(int gs) { return gs == 16 || gs == 32 || gs == 64 || gs == 128; }
inline bool valid_group_size(int gs, int64_t K) { return fixed_group_size(gs) || (gs > 0 && gs == K && K % 8 == 0); }

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Returns AMX_OK when the last launch was accepted, AMX_ERR_CUDA otherwise.
inline int launch_status() { return cudaGetLastError() == cudaSuccess ? AMX_OK : AMX_ERR_CUDA; }

// ---- launches ---------------------------------------------------------------------------------
// Kernels of this library are chained by programmatic dependent launch: a kernel lets its successor onto the SMs as soon
// as all of its own blocks run (grid_launch_dependents; the FP4 GEMM and the fused attention, whose blocks fill an SM, as their last
// act), and waits for its predecessors to complete before it touches memory (grid_dependency_wait; it returns at once when the launch
// carried no such dependency).  What needs no memory comes before the wait in those two: barriers, tensor memory.  The few-row kernels
// copy weights before it: the fragments kernel ahead of them lets them start only after its own wait.  The order of the stream
// is kept, the launch latency and the gap between two kernels are not: chains of ordinary launches cost about 2 us per
// kernel boundary.  A stream that is being captured gets ordinary launches (replayed from a graph the chains of short
// kernels were slower with these edges).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// First statement of the other kernels.  (Every kernel waits before it ends, so "my predecessor has completed" implies the
// same of everything before it.)
__device__ __forceinline__ void begin_kernel() {
    grid_launch_dependents();
    grid_dependency_wait();
}

inline bool programmatic_launch_ok(cudaStream_t st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return cs == cudaStreamCaptureStatusNone;
}

// One launch; programmatic: with the edge described above (never on a stream that is being captured).
template <typename... P, typename... A>
int launch_with(dim3 cluster, bool programmatic, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (programmatic) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster.x * cluster.y * cluster.z > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster.x;
        attr[n].val.clusterDim.y = cluster.y;
        attr[n].val.clusterDim.z = cluster.z;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    if (cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return AMX_ERR_CUDA;
    }
    return AMX_OK;
}

// chained = false: an ordinary launch.  For long kernels with one block per SM: started while their predecessor leaves, the
// blocks land on the SMs in another order (operands shared by neighbouring tiles cross the two halves of the L2 more often).
// That costs the longest of them up to 1 %; a call whose long kernel takes 40 us is 3-4 % faster chained.  Where the line lies was
// measured for each of the two kernels (gemm_fp4.cu, attention_fp4.cu): at 260 us (200 of one plane) and at 350 us.
template <typename... P, typename... A>
int launch_clusters(dim3 cluster, bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    return launch_with(cluster, chained && programmatic_launch_ok(st), kernel, grid, block, smem, st, static_cast<A&&>(args)...);
}

template <typename... P, typename... A>
int launch_chained(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    return launch_clusters(1, chained, kernel, grid, block, smem, st, static_cast<A&&>(args)...);
}

template <typename... P, typename... A>
int launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    return launch_chained(true, kernel, grid, block, smem, st, static_cast<A&&>(args)...);
}

// Zeroes the first n words of a workspace (the status word, the flushed-scale count) by a kernel: a memset would break
// the chain of launches (api.cu).
int clear_words(void* words, cudaStream_t st, int n = 2);

// ---- device-side number formats -------------------------------------------------------------

// fp32 value of an E5M2 byte: E5M2 is the upper byte of an IEEE half.
__device__ __forceinline__ float e5m2_to_float(uint32_t byte) {
    float f;
    unsigned short h = (unsigned short)(byte << 8);
    asm("cvt.f32.f16 %0, %1;" : "=f"(f) : "h"(h));
    return f;
}

// fp32 magnitude of a 3-bit E2M1 code EEM: 0, .5, 1, 1.5, 2, 3, 4, 6.
// For EE > 0 the bits placed at fp32 exponent/mantissa positions give 2^(EE-1) * (1 + M/2);
// EE == 0 is the subnormal M * 0.5.
__device__ __forceinline__ float e2m1_mag_to_float(uint32_t c3) {
    uint32_t bits = (c3 << 22) + (126u << 23);   // exponent field EE + 126, mantissa msb = M
    float v = __uint_as_float(bits);
    return (c3 & 6u) ? v : 0.5f * (float)(c3 & 1u);
}

// fp32 value of a scale byte without the format's special cases: its largest exponent field is read as one more power of two, as
// everywhere where scales are taken apart below (casts saturate; only a NaN among the elements leaves such a byte).
__device__ __forceinline__ float scale_value(uint32_t byte) { return __uint_as_float(byte << 21) * 5192296858534827628530496329220096.f; }   // 2^112

// An E5M2 scale byte as (key << 2) | mantissa of its normalised form: key = unbiased exponent + 17 (so that
// 2^-16 has key 1) and two mantissa bits.  Normal bytes (b >= 4) are b + 8; the subnormals 1, 2, 3 x 2^-16 are
// 1.0 x 2^-16, 1.0 x 2^-15 and 1.5 x 2^-15: 4, 8 and 10 (read from a packed table); 0 for a zero scale.
__device__ __forceinline__ uint32_t scale_norm(uint32_t b) {
    return b >= 4 ? b + 8 : (0x0A080400u >> (b * 8)) & 0xFFu;
}
// Exponent key of an E5M2 scale byte, 0 for a zero scale.
__device__ __forceinline__ int scale_key(uint32_t b) { return (int)(scale_norm(b) >> 2); }
// Per-row word of a prepared FP4-GEMM operand: bits 15..0 the row's power-of-two offset (largest exponent key
// - 25; 0 for an all-zero row) as a signed 16-bit number, bit 16 set when some group of the row has a nonzero
// positive-side scale, bit 17 the same for the negative side.  A tile whose rows all lack a side has an
// all-zero plane for it, and the GEMM does not issue that plane's products.  Bits 31..18: how many nonzero
// scales of the row did not fit the UE4M3 range under the row's offset and were flushed to zero (see
// to_ue4m3), saturating at kRowFlushedMax.
constexpr int kRowHasPos = 1 << 16, kRowHasNeg = 1 << 17;
constexpr int kRowFlushedShift = 18, kRowFlushedMax = 0x3FFF;
__host__ __device__ __forceinline__ int row_word(int kmax, int side_bits, int flushed = 0) {
    const int f = flushed > kRowFlushedMax ? kRowFlushedMax : flushed;
    return ((kmax ? kmax - 25 : 0) & 0xFFFF) | side_bits | (int)((unsigned)f << kRowFlushedShift);
}
__host__ __device__ __forceinline__ int row_word_exp(int w) { return (int)(short)(w & 0xFFFF); }
__host__ __device__ __forceinline__ int row_word_flushed(int w) { return (int)((unsigned)w >> kRowFlushedShift); }
// side bits of a group's scale bytes {neg : pos}
__device__ __forceinline__ int side_bits_of(uint32_t sc) {
    return ((sc & 0xFFu) ? kRowHasPos : 0) | ((sc >> 8) ? kRowHasNeg : 0);
}

// Scale factors of a prepared operand: chunks of 512 bytes per [128 rows x 64 elements], the chunks of one block
// of 128 rows consecutive along K; inside a chunk byte (r % 32) * 16 + (r / 32) * 4 + (k16 % 4), one scale per 16
// elements.  Offset of row `row`'s bytes of its first chunk, and of 32-group g's two bytes relative to that.
constexpr int kSfChunkBytes = 512;
__host__ __device__ __forceinline__ int64_t sf_row_offset(int64_t row, int nk64) {
    const int rr = (int)(row & 127);
    return (row >> 7) * nk64 * (int64_t)kSfChunkBytes + (rr & 31) * 16 + (rr >> 5) * 4;
}
__host__ __device__ __forceinline__ int64_t sf_group_offset(int g) { return (int64_t)(g >> 1) * kSfChunkBytes + (g & 1) * 2; }

// UE4M3 bytes of a pair of E5M2 scale bytes (bits 15..0 of sc; what lies above is ignored) for a row whose scales are multiplied by
// `up` = sf_factor(the row's largest key): exponent field key - kmax + 15, the two mantissa bits in bits 2..1; zero where the
// exponent field would be below 1.  `lost` counts, in steps of 128, the nonzero scales this flushes.  (By way of the hardware's
// converts, both bytes at once: on integers, normal and subnormal scales apart, the preparation spent 60 instructions per group here.)
__device__ __forceinline__ float sf_factor(int kmax) { return __uint_as_float((uint32_t)(25 - kmax + 127) << 23); }
__device__ __forceinline__ uint32_t to_ue4m3x2(uint32_t sc, float up, uint32_t& lost) {
    unsigned short both;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(both) : "f"(scale_value((sc >> 8) & 0xFFu) * up), "f"(scale_value(sc & 0xFFu) * up));
    const uint32_t t = both + 0x7878u;                          // bit 7 of a byte: it is a normal number
    lost = __dp4a((sc + 0x7F7Fu) & ~t & 0x8080u, 0x0101u, lost);
    uint32_t normal;                                            // selectors 8 and 9 replicate bit 7 (not with __byte_perm)
    asm("prmt.b32 %0, %1, 0, 0x4498;" : "=r"(normal) : "r"(t));
    return both & normal;
}

}  // namespace amx
