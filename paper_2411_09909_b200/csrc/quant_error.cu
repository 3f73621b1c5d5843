// Squared error of a quantized tensor against its bf16 source, split into the max-clamping and the rounding
// part (arXiv 2411.09909, appendix "Determining PoT Shared Scale: Floor vs. Round": the output error of a shared
// scale decomposes into the error of elements beyond the largest representable magnitude and the rounding error
// of all others).  An element is clamped when |x| > 6 * (the scale of its side).
//
// A reduction: 2 bytes of source, half a byte of codes and the scale bytes per element are read once.  A thread takes 16
// consecutive elements at a time (two 16-byte loads of the source, one 8-byte load of codes), two chunks ahead of the one it works
// on; three blocks per SM have the registers for that.  What bounds the kernel is instruction issue (25 warp instructions per pair of
// elements, 69 % of the issue slots; the bytes alone take 18 of its 27 us on 4096 x 11008), so the arithmetic is packed: two
// codes are decoded by one convert and three f16 instructions (decode_math.cuh), the decoded f16 and the clamped bf16 values go into
// fp32 multiply-adds as they are (converted first: 30 instructions, 30 us), the sums are packed fp32 multiply-adds, and the
// clamping error needs no selection at all - with y = x clamped to the group's range, x - y is the error of a clamped element
// and zero for every other one.  (Copies through a ring in shared memory: no faster, the addresses cost what the waits did.)
// The 16 squares of a chunk are added in fp32 (relative error below 2^-20 of the chunk's sum: all terms are
// non-negative), everything above a chunk in fp64 - fp64 arithmetic per element would bound the kernel (the
// conversions alone cost more than the memory traffic).  The clamped count is an integer.  The summation order is fixed
// (grid-stride per thread, shuffles in a warp, warps in order, then one block over the per-block partial sums), so the
// result is the same bits on every run.
// F16S instantiation: binary16 shared scales ([rows, K/gs, 2] uint16); xhat then has up to 13 significant bits and
// x - xhat is still exact in fp32, element by element.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "cast_math.cuh"
#include "decode_math.cuh"

namespace amx {
namespace {

constexpr int kThreads = 256, kMaxBlocks = 2048, kBlocksPerSm = 3, kGrid = 148 * kBlocksPerSm;

struct Sums {
    double x2, e2, clamp2, clamped;
};
struct ThreadSums {
    double x2, e2, clamp2;
    uint32_t clamped;
};

__device__ __forceinline__ void add16(ThreadSums& s, const uint4 (&xw)[2], uint2 cw, float sp, float sn) {
    const uint32_t xs[8] = {xw[0].x, xw[0].y, xw[0].z, xw[0].w, xw[1].x, xw[1].y, xw[1].z, xw[1].w};
    const uint32_t cs[2] = {cw.x, cw.y};
    float x2 = 0.f, e2 = 0.f, c2 = 0.f;
    int clamped = 0;
    // A 3-bit E2M1 code at bits 24..22 of an fp32 pattern reads as (its value) x 2^-126 (code 1 is the subnormal
    // 2^-127); the side scales carry the 2^126 in two exact halves.
    const float up = 9223372036854775808.f;                      // 2^63
    const float sp_up = sp * up, sn_up = -sn * up, sp6 = 6.0f * sp, sn6 = 6.0f * sn;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float x = __uint_as_float((i & 1) ? (xs[i >> 1] & 0xFFFF0000u) : (xs[i >> 1] << 16));
        const uint32_t w = cs[i >> 3] >> ((i & 7) * 4);
        const bool neg = w & 8u;
        const float mag_dn = __uint_as_float((w & 7u) << 22) * up;   // value x 2^-63, exact
        const float e = fmaf(-mag_dn, neg ? sn_up : sp_up, x), ee = e * e;
        x2 = fmaf(x, x, x2);
        e2 += ee;
        if (fabsf(x) > (neg ? sn6 : sp6)) {
            c2 += ee;
            ++clamped;
        }
    }
    s.x2 += (double)x2; s.e2 += (double)e2; s.clamp2 += (double)c2; s.clamped += clamped;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Sum over the block; valid in thread 0.
__device__ __forceinline__ Sums block_sum(Sums s, double (*sh)[4]) {
    s.x2 = warp_sum(s.x2); s.e2 = warp_sum(s.e2); s.clamp2 = warp_sum(s.clamp2); s.clamped = warp_sum(s.clamped);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sh[warp][0] = s.x2; sh[warp][1] = s.e2; sh[warp][2] = s.clamp2; sh[warp][3] = s.clamped; }
    __syncthreads();
    Sums t = {0, 0, 0, 0};
    if (threadIdx.x == 0)
        for (int w = 0; w < kThreads / 32; ++w) { t.x2 += sh[w][0]; t.e2 += sh[w][1]; t.clamp2 += sh[w][2]; t.clamped += sh[w][3]; }
    return t;
}

// x - 16 h and x - y with element H of an f16 or bf16 pair straight in an fp32 multiply-add.
template <int H>
__device__ __forceinline__ uint32_t minus_16_times(uint32_t pair, uint32_t x) {
    uint32_t r;
    if (H == 0) asm("{.reg .b16 lo, hi, m; mov.b16 m, 0xCC00; mov.b32 {lo, hi}, %1; fma.rn.f32.f16 %0, lo, m, %2;}" : "=r"(r) : "r"(pair), "r"(x));
    else asm("{.reg .b16 lo, hi, m; mov.b16 m, 0xCC00; mov.b32 {lo, hi}, %1; fma.rn.f32.f16 %0, hi, m, %2;}" : "=r"(r) : "r"(pair), "r"(x));
    return r;
}
template <int H>
__device__ __forceinline__ uint32_t minus_bf16(uint32_t pair, uint32_t x) {
    uint32_t r;
    if (H == 0) asm("{.reg .b16 lo, hi, m; mov.b16 m, 0xBF80; mov.b32 {lo, hi}, %1; fma.rn.f32.bf16 %0, lo, m, %2;}" : "=r"(r) : "r"(pair), "r"(x));
    else asm("{.reg .b16 lo, hi, m; mov.b16 m, 0xBF80; mov.b32 {lo, hi}, %1; fma.rn.f32.bf16 %0, hi, m, %2;}" : "=r"(r) : "r"(pair), "r"(x));
    return r;
}

// The same for E5M2 scales (bytes {neg : pos}), two elements at a time.
__device__ __forceinline__ void add16_e5m2(ThreadSums& s, const uint4 (&xw)[2], uint2 cw, uint32_t sc) {
    const uint32_t xs[8] = {xw[0].x, xw[0].y, xw[0].z, xw[0].w, xw[1].x, xw[1].y, xw[1].z, xw[1].w};
    const decode_f16::Scales scl = decode_f16::make_scales(sc);
    // the largest values the two sides represent, 6 x scale: exact in bf16
    const uint32_t tp = __float_as_uint(6.0f * e5m2_to_float(sc & 0xFFu)), tn = __float_as_uint(-6.0f * e5m2_to_float((sc >> 8) & 0xFFu)),
                   top = __byte_perm(tp, tp, 0x3232), bottom = __byte_perm(tn, tn, 0x3232);
    uint64_t x2 = 0, e2 = 0, c2 = 0;
    uint32_t counts = 0;
    const uint4 v[2] = {decode_f16::decode_word(cw.x, scl), decode_f16::decode_word(cw.y, scl)};
    const uint32_t xh[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint64_t x = cast::pack_f32x2(xs[i] << 16, xs[i] & 0xFFFF0000u);
        const uint64_t e = cast::pack_f32x2(minus_16_times<0>(xh[i], xs[i] << 16), minus_16_times<1>(xh[i], xs[i] & 0xFFFF0000u));
        // clamped on the bit patterns: signed 16-bit order for the positive values (the negative ones are below), unsigned
        // order for the negative ones (larger magnitude, larger pattern; the positive ones are below)
        const uint32_t y = __vminu2(__vmins2(xs[i], top), bottom);
        const uint64_t d = cast::pack_f32x2(minus_bf16<0>(y, xs[i] << 16), minus_bf16<1>(y, xs[i] & 0xFFFF0000u));
        x2 = cast::fma_f32x2(x, x, x2);
        e2 = cast::fma_f32x2(e, e, e2);
        c2 = cast::fma_f32x2(d, d, c2);
        counts += __vminu2(xs[i] - y, 0x00010001u);              // x is never below y in its half: no borrow
    }
    float a, b;
    cast::unpack_f32x2(x2, a, b);
    s.x2 += (double)(a + b);
    cast::unpack_f32x2(e2, a, b);
    s.e2 += (double)(a + b);
    cast::unpack_f32x2(c2, a, b);
    s.clamp2 += (double)(a + b);
    s.clamped += (counts & 0xFFFFu) + (counts >> 16);
}

// CONTIG: rows without gaps, everything is indexed by the chunk number (a row holds whole groups).
template <bool F16S, bool CONTIG>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm) quant_error_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t K,
                                                                  int64_t ld_x, const uint8_t* __restrict__ codes,
                                                                  const uint8_t* __restrict__ scales, int gs_log2,
                                                                  double* __restrict__ partial) {
    begin_kernel();
    __shared__ double sh[kThreads / 32][4];
    const int64_t per_row = K / 16, chunks = rows * per_row, stride = (int64_t)gridDim.x * kThreads;
    int64_t v = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    ThreadSums s = {0, 0, 0, 0};
    struct Chunk {
        uint4 x[2];
        uint2 codes;
        uint32_t sc;
    };
    auto load = [&](Chunk& c, int64_t u) {
        if (u >= chunks) return;
        const uint4* xp = reinterpret_cast<const uint4*>(x) + u * 2;
        if (!CONTIG) xp = reinterpret_cast<const uint4*>(x + (u / per_row) * ld_x) + (u % per_row) * 2;
        c.x[0] = __ldg(xp);
        c.x[1] = __ldg(xp + 1);
        c.codes = __ldg(reinterpret_cast<const uint2*>(codes) + u);
        const int64_t g = u >> (gs_log2 - 4);
        c.sc = F16S ? __ldg(reinterpret_cast<const uint32_t*>(scales) + g) : __ldg(reinterpret_cast<const unsigned short*>(scales) + g);
    };
    auto add = [&](const Chunk& c) {
        if (F16S)
            add16(s, c.x, c.codes, __half2float(__ushort_as_half((unsigned short)(c.sc & 0xFFFFu))),
                  __half2float(__ushort_as_half((unsigned short)(c.sc >> 16))));
        else add16_e5m2(s, c.x, c.codes, c.sc);
    };
    Chunk c0, c1, c2;                                            // two chunks in flight while one is worked on
    load(c0, v);
    load(c1, v + stride);
    while (v < chunks) {
        load(c2, v + 2 * stride);
        add(c0);
        if ((v += stride) >= chunks) break;
        load(c0, v + 2 * stride);
        add(c1);
        if ((v += stride) >= chunks) break;
        load(c1, v + 2 * stride);
        add(c2);
        v += stride;
    }
    const Sums t = block_sum({s.x2, s.e2, s.clamp2, (double)s.clamped}, sh);
    if (threadIdx.x == 0) {
        double* p = partial + (int64_t)blockIdx.x * 4;
        p[0] = t.x2; p[1] = t.e2; p[2] = t.clamp2; p[3] = t.clamped;
    }
}

__global__ void __launch_bounds__(kThreads) quant_error_final_kernel(const double* __restrict__ partial, int blocks,
                                                                     double* __restrict__ out) {
    begin_kernel();
    __shared__ double sh[kThreads / 32][4];
    Sums s = {0, 0, 0, 0};
    for (int b = threadIdx.x; b < blocks; b += kThreads) {
        s.x2 += partial[b * 4]; s.e2 += partial[b * 4 + 1]; s.clamp2 += partial[b * 4 + 2]; s.clamped += partial[b * 4 + 3];
    }
    const Sums t = block_sum(s, sh);
    if (threadIdx.x == 0) { out[0] = t.x2; out[1] = t.e2; out[2] = t.clamp2; out[3] = t.clamped; }
}

}  // namespace
}  // namespace amx

using namespace amx;

extern "C" size_t amx_quant_error_workspace_bytes(void) { return (size_t)kMaxBlocks * 4 * sizeof(double); }

namespace {
int quant_error(const void* x, int64_t rows, int64_t K, int64_t ld_x, const uint8_t* codes, const void* scales,
                bool f16s, int group_size, double* out, void* workspace, size_t workspace_bytes, void* stream) {
    if (!fixed_group_size(group_size) || rows < 0 || K <= 0 || K % group_size || ld_x < K) return AMX_ERR_SHAPE;
    if (!out) return AMX_ERR_NULL;
    if (rows > 0 && (!x || !codes || !scales)) return AMX_ERR_NULL;
    if (!workspace || workspace_bytes < amx_quant_error_workspace_bytes()) return AMX_ERR_WORKSPACE;
    if (!aligned(x, 16) || ld_x % 8 || !aligned(codes, 8) || !aligned(scales, f16s ? 4 : 2) || !aligned(out, 8) ||
        !aligned(workspace, 8))
        return AMX_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t chunks = rows * (K / 16);
    const int64_t blocks = chunks <= kThreads ? 1 : chunks >= (int64_t)kGrid * kThreads ? kGrid : (chunks + kThreads - 1) / kThreads;
    static_assert(kGrid <= kMaxBlocks, "the workspace holds one set of sums per block");
    double* partial = static_cast<double*>(workspace);
    const int gs_log2 = group_size == 16 ? 4 : group_size == 32 ? 5 : group_size == 64 ? 6 : 7;
    const dim3 grid((unsigned)blocks);
    auto* kernel = f16s ? (ld_x == K ? quant_error_kernel<true, true> : quant_error_kernel<true, false>)
                        : (ld_x == K ? quant_error_kernel<false, true> : quant_error_kernel<false, false>);
    const int rc = launch(kernel, grid, kThreads, 0, st, static_cast<const uint16_t*>(x), rows, K, ld_x, codes,
                          static_cast<const uint8_t*>(scales), gs_log2, partial);
    if (rc != AMX_OK) return rc;
    return launch(quant_error_final_kernel, 1, kThreads, 0, st, partial, (int)blocks, out);
}
}  // namespace

extern "C" int amx_quant_error(const void* x, int64_t rows, int64_t K, int64_t ld_x, const uint8_t* codes,
                               const uint8_t* scales, int group_size, double* out, void* workspace,
                               size_t workspace_bytes, void* stream) {
    return quant_error(x, rows, K, ld_x, codes, scales, false, group_size, out, workspace, workspace_bytes, stream);
}

extern "C" int amx_quant_error_f16s(const void* x, int64_t rows, int64_t K, int64_t ld_x, const uint8_t* codes,
                                    const uint16_t* scales, int group_size, double* out, void* workspace,
                                    size_t workspace_bytes, void* stream) {
    return quant_error(x, rows, K, ld_x, codes, scales, true, group_size, out, workspace, workspace_bytes, stream);
}
