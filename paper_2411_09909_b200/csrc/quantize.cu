// bf16 -> AMXFP4 direct cast (arXiv 2411.09909, Sections 4.2-4.3; Algorithm 1 applied per sign
// with the FP8 E5M2 shared scale).  HBM-bound: 2 B read + 0.5625 B written per element.  The per-group
// arithmetic, with the argument for its exactness, is in cast_math.cuh.
#include <cuda_bf16.h>

#include "cast_math.cuh"
#include "cp_async.cuh"
#include "gemm.cuh"
#include "softmax_math.cuh"

namespace amx {
namespace {

using namespace cast;

constexpr int kThreads = 256;

// Quantizes 8 consecutive elements held as 4 bf16x2 words.  TPG threads (8*TPG = group size) hold
// one group and sit in consecutive lanes.  Returns the 8 nibbles; `sc` receives the scale bytes.
template <int TPG>
__device__ __forceinline__ uint32_t quantize8(const uint4 q, uint32_t& sc) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t c = side_maxima<4>(w);
#pragma unroll
    for (int d = 1; d < TPG; d <<= 1) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, d));
    float inv_p, inv_n;
    sc = group_scales(c, inv_p, inv_n);
    return encode8(w, inv_p, inv_n);
}

// Groups along the contiguous axis.  Each thread owns EPT = min(gs, 32) consecutive elements
// (EPT/8 16-byte loads, one EPT/2-byte store); a group is TPG = gs / EPT consecutive lanes, so a
// 16- or 32-group needs no shuffle and its scales are computed once.  n_items = rows * K / EPT.
template <int EPT, int TPG, bool CONTIG, int FMT = 0>
__global__ void __launch_bounds__(kThreads)
quantize_rows_kernel(const uint4* __restrict__ x, int64_t n_items, int64_t items_per_row,
                     int64_t ld_vec, uint4* __restrict__ codes, uint16_t* __restrict__ scales) {
    begin_kernel();
    constexpr int NV = EPT / 8;
    const int64_t v = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    uint32_t w[NV * 4];
    const bool live = v < n_items;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        uint4 q = make_uint4(0, 0, 0, 0);
        if (live) {
            int64_t off = v * NV + j;
            if (!CONTIG) off = (v / items_per_row) * ld_vec + (v % items_per_row) * NV + j;
            q = __ldg(x + off);
        }
        w[4 * j] = q.x; w[4 * j + 1] = q.y; w[4 * j + 2] = q.z; w[4 * j + 3] = q.w;
    }
    uint32_t c = side_maxima<NV * 4>(w);
#pragma unroll
    for (int d = 1; d < TPG; d <<= 1) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, d));
    float inv_p, inv_n;
    const uint32_t sc = group_scales_fmt<FMT>(c, inv_p, inv_n);
    uint32_t nib[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) nib[j] = encode8(w + 4 * j, inv_p, inv_n);
    if (live) {
        if (NV == 4) codes[v] = make_uint4(nib[0], nib[1], nib[2], nib[NV - 1]);
        else *reinterpret_cast<uint2*>(reinterpret_cast<uint8_t*>(codes) + v * 8) = make_uint2(nib[0], nib[NV - 1]);
        if ((threadIdx.x & (TPG - 1)) == 0) scales[v / TPG] = (uint16_t)sc;
    }
}

// Groups of 16, two of them per thread: four 16-byte loads in flight and a 16-byte store, as with groups of 32 (one group
// per thread streamed 4096 x 11008 at 4.7 TB/s).
template <bool CONTIG, int FMT>
__global__ void __launch_bounds__(kThreads)
quantize_rows16_kernel(const uint4* __restrict__ x, int64_t n_items, int64_t items_per_row, int64_t ld_vec,
                       uint4* __restrict__ codes, uint32_t* __restrict__ scales) {
    begin_kernel();
    const int64_t v = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (v >= n_items) return;
    const uint4* src = x + (CONTIG ? v * 4 : (v / items_per_row) * ld_vec + (v % items_per_row) * 4);
    uint32_t w[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint4 q = __ldg(src + j);
        w[4 * j] = q.x; w[4 * j + 1] = q.y; w[4 * j + 2] = q.z; w[4 * j + 3] = q.w;
    }
    uint32_t nib[4], sc[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        uint32_t wg[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) wg[i] = w[8 * g + i];
        float inv_p, inv_n;
        sc[g] = group_scales_fmt<FMT>(side_maxima<8>(wg), inv_p, inv_n);
        nib[2 * g] = encode8(wg, inv_p, inv_n);
        nib[2 * g + 1] = encode8(wg + 4, inv_p, inv_n);
    }
    codes[v] = make_uint4(nib[0], nib[1], nib[2], nib[3]);
    scales[v] = sc[0] | (sc[1] << 16);
}

// The whole row as one group (group_size == K; the grouping of the worked example in Appendix B.3): one block per
// row, two sweeps - the row's side maxima (block reduction), then the codes.  The second sweep re-reads the row
// from the caches.  Generic path, any K that is a multiple of 8.
template <int FMT>
__global__ void __launch_bounds__(kThreads)
quantize_whole_rows_kernel(const uint4* __restrict__ x, int64_t vec_per_row, int64_t ld_vec, uint32_t* __restrict__ codes,
                           uint16_t* __restrict__ scales) {
    begin_kernel();
    __shared__ uint32_t red[kThreads / 32];
    const int64_t row = blockIdx.x;
    const uint4* xr = x + row * ld_vec;
    uint32_t c = 0;
    for (int64_t i = threadIdx.x; i < vec_per_row; i += kThreads) {
        const uint4 q = __ldg(xr + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        c = __vmaxs2(c, side_maxima<4>(w));
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, d));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) c = __vmaxs2(c, red[i]);
    float inv_p, inv_n;
    const uint32_t sc = group_scales_fmt<FMT>(c, inv_p, inv_n);
    for (int64_t i = threadIdx.x; i < vec_per_row; i += kThreads) {
        const uint4 q = __ldg(xr + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        codes[row * vec_per_row + i] = encode8(w, inv_p, inv_n);
    }
    if (threadIdx.x == 0) scales[row] = (uint16_t)sc;
}

// Groups DOWN the rows (strided axis): x is [R, C]; output is the canonical layout of x^T.
// A block stages a [64 rows x 64 columns] tile in shared memory and re-reads it column-wise.
constexpr int kTR = 64, kTC = 64;

template <int TPG>
__global__ void __launch_bounds__(kThreads)
quantize_cols_kernel(const __nv_bfloat16* __restrict__ x, int64_t R, int64_t C, int64_t ld,
                     uint32_t* __restrict__ codes, uint16_t* __restrict__ scales, int gs) {
    begin_kernel();
    // blockIdx.z: one of several [R, C] matrices stored one after another (R * ld elements apart); their
    // transposed outputs follow one another as well
    __shared__ uint16_t tile[kTC][kTR + 2];  // [column][row], padded
    const int64_t r0 = (int64_t)blockIdx.y * kTR, c0 = (int64_t)blockIdx.x * kTC;
    const uint16_t* xs = reinterpret_cast<const uint16_t*>(x) + (int64_t)blockIdx.z * R * ld;
    codes += (int64_t)blockIdx.z * (C * R / 8);
    scales += (int64_t)blockIdx.z * (C * R / gs);
    for (int i = threadIdx.x; i < kTR * kTC; i += kThreads) {
        const int rr = i / kTC, cc = i % kTC;
        uint16_t v = 0;
        if (r0 + rr < R && c0 + cc < C) v = xs[(r0 + rr) * ld + c0 + cc];
        tile[cc][rr] = v;
    }
    __syncthreads();
    // kTR/8 = 8 threads cover one column's 64 rows; 256 threads -> 32 columns per pass
    for (int pass = 0; pass < kTC / (kThreads / (kTR / 8)); ++pass) {
        const int cc = pass * (kThreads / (kTR / 8)) + threadIdx.x / (kTR / 8);
        const int seg = threadIdx.x % (kTR / 8);
        const uint16_t* t = &tile[cc][seg * 8];
        uint4 q;
        q.x = t[0] | ((uint32_t)t[1] << 16);
        q.y = t[2] | ((uint32_t)t[3] << 16);
        q.z = t[4] | ((uint32_t)t[5] << 16);
        q.w = t[6] | ((uint32_t)t[7] << 16);
        uint32_t sc;
        const uint32_t nib = quantize8<TPG>(q, sc);
        const int64_t col = c0 + cc, row = r0 + seg * 8;
        if (col < C && row < R) {  // R % 8 == 0, so the 8 rows are all valid or all invalid
            codes[(col * R + row) / 8] = nib;
            if ((seg & (TPG - 1)) == 0) scales[(col * R + row) / gs] = (uint16_t)sc;
        }
    }
}

// The cast for an operand of the FP4 GEMM (32-groups, contiguous rows).  Besides the canonical codes and scales
// it writes, in the same pass, everything the GEMM reads: the two sign planes (every nibble in the plane of its
// sign bit, zero in the other), the UE4M3 scale factors of both planes - byte (r%32)*16 + (r/32)*4 + k16%4 of
// the 512-byte chunk of [128 rows x 64 elements]; one scale per 16 elements, so a 32-group's scale is stored
// twice - and per row the power of two by which those scale factors understate the true scales
// (row_exp = largest exponent key of the row - 25).  The scale factors depend on the row's largest scale, so
// whole rows belong to one warp (prepare_operands_kernel) or, in the softmax variant, to one block
// (finish_prepared_row).  Rows past the last row, and groups past the last group, get zero scale factors, so that
// padded tile rows and columns multiply zero codes by a finite scale.

// Second half of a prepared cast, for the GX threads (a multiple of 32) that own row `row` (`top`: the largest
// positive-side scale byte the thread has seen in bits 7..0, the largest negative-side one in bits 15..8;
// slot: the row's four shared-memory words, zero on entry): row maximum of the exponent keys and which sides
// occur, the row's scale factors in the tensor cores' layout, padding included, and the row word (with the
// number of scales that did not fit the UE4M3 range and were flushed: the last warp of the row to finish
// writes it, so no third block barrier is needed).
__device__ __forceinline__ void finish_prepared_row(int64_t row, bool row_live, int G, int gx, int GX, uint32_t top,
                                                    uint32_t sc_first, const uint16_t* __restrict__ scales,
                                                    int* slot, uint8_t* __restrict__ sf_pos,
                                                    uint8_t* __restrict__ sf_neg, int* __restrict__ row_exp, int nk64,
                                                    int* __restrict__ flushed_total = nullptr) {
    // Two shared-memory atomics per warp.  The key of an E5M2 byte grows with the byte (scales carry no sign
    // bit), so the largest byte has the largest key.
    const uint32_t top_p = __reduce_max_sync(0xFFFFFFFFu, top & 0xFFu), top_n = __reduce_max_sync(0xFFFFFFFFu, top >> 8);
    __syncthreads();                               // the slot was zeroed at the top of the kernel
    if ((gx & 31) == 0 && (top_p | top_n)) {
        atomicMax(&slot[0], scale_key(max(top_p, top_n)));
        atomicOr(&slot[1], side_bits_of(top_p | (top_n << 8)));
    }
    __syncthreads();
    const int kmax = slot[0];
    // offset of this row's bytes inside a chunk; the chunks of one block of 128 rows are consecutive along K
    const int64_t sf_row = sf_row_offset(row, nk64);
    const int64_t v_row = row * G;
    const float factor = sf_factor(kmax);
    uint32_t lost = 0;
    for (int g = gx; g < nk64 * 2; g += GX) {      // groups past G: padding to whole 256-element blocks
        uint32_t u = 0;
        // a later group of a striding thread: re-read the scale bytes this thread stored before
        if (row_live && g < G) u = to_ue4m3x2((g == gx) ? sc_first : scales[v_row + g], factor, lost);
        const int64_t off = sf_row + sf_group_offset(g);
        *reinterpret_cast<uint16_t*>(sf_pos + off) = (uint16_t)__byte_perm(u, 0, 0x4400);
        *reinterpret_cast<uint16_t*>(sf_neg + off) = (uint16_t)__byte_perm(u, 0, 0x4411);
    }
    if (!row_live) return;                         // uniform over the row's warps
    const int flushed = __reduce_add_sync(0xFFFFFFFFu, (int)(lost >> 7));
    if ((gx & 31) == 0) {
        if (flushed) atomicAdd(&slot[2], flushed);
        __threadfence_block();
        if (atomicAdd(&slot[3], 1) == GX / 32 - 1) {
            const int total = atomicAdd(&slot[2], 0);
            row_exp[row] = row_word(kmax, slot[1], total);
            if (total && flushed_total) atomicAdd(flushed_total, total);
        }
    }
}

// Operands of the FP4 GEMM, up to two of them in one launch (a small cast beside the preparation of a large weight, or
// both casts of a layer).  Per operand either the cast of a bf16 matrix (any fixed group size) or the preparation of a
// canonical one.  A row (or, when rows are short, several rows) belongs to one warp: LPR = 2^lpr_log2 lanes per row, lane lr
// of them owns the 32-element pieces lr, lr + LPR, ...  A lane streams its pieces through a private ring in shared memory
// with asynchronous copies (kCastDepth pieces ahead; the loads hold no registers).  First sweep: per piece the cast (or the
// split of its codes), the stores of the planes, the scale bytes and (when asked for) the canonical codes; the scale bytes
// stay in registers (GPL of them per lane; GPL = 0: any number, re-read from memory).  Then the row's largest exponent key
// by a warp reduction, and the second sweep turns the scale bytes into the row's scale factors, padding included, and
// writes the row word.
// Scale factors leave the block in whole 32-byte sectors: the tensor cores' layout interleaves eight rows (r, r+1,
// r+32, r+33, r+64, r+65, r+96, r+97, r even) in every sector, so a block of eight warps owns exactly such sets of
// rows - warp (q, h) has the rows 32 q + 2 k + h of a 128-row block, for the block's RPW = 32 / LPR values of k -
// collects the converted bytes in shared memory and stores them 16 bytes per thread.  (Written 2 bytes at a
// time straight from the owning lanes, the scale factors were 4 % of the bytes and doubled the kernel's L2
// write requests.)  Rows past the last row get zero scale factors.
constexpr int kCastDepth = 2;                              // pieces in flight per lane
constexpr int kCastWarps = 8;
constexpr int kCastRingBytes = kCastWarps * kCastDepth * 32 * 64;
constexpr int kCastMaxExchangeBytes = 96 * 1024;           // above this (K > 49152 at LPR = 32) the lanes store their bytes themselves

struct PrepParams {
    PrepOperand op[2];
    VtOperand vt;                                          // kAttention: blocks before those of the two operands
    unsigned vt_blocks;
    unsigned blocks0;                                      // blocks of the first operand; the others are the second's
    int G, lpr_log2, exchange, nk64, gs, gs_log2;
    int* flushed_total;
};

// The two scale bytes {neg : pos} as 16-bit halves, for packed maxima (byte-wise ones are eight instructions).
__device__ __forceinline__ uint32_t halves(uint32_t sc) { return __byte_perm(sc, 0, 0x4140); }

// Scale pairs {neg : pos} of one 32-element piece: of its first 16 elements in bits 15..0, of the others in bits 31..16
// (equal unless the group size is 16), from a row's canonical scales.
__device__ __forceinline__ uint32_t piece_scales(const uint16_t* __restrict__ row, int g, int gs) {
    if (gs == 16) return (uint32_t)row[2 * g] | ((uint32_t)row[2 * g + 1] << 16);
    const uint32_t v = row[gs == 32 ? g : gs == 64 ? g >> 1 : g >> 2];
    return v | (v << 16);
}

// A piece of a group of 16, 64 or 128 elements (AMXFP4): 64- and 128-groups are two or four consecutive lanes, which agree
// on the maxima.  Every lane of the warp takes part; `own`: the lane has a piece, number g of the row.
__device__ __forceinline__ uint32_t cast_piece_gs(const uint32_t (&w)[16], bool own, int gs, int64_t v, int g, uint16_t* __restrict__ row_scales,
                                                  uint4* __restrict__ codes, uint4* __restrict__ pos, uint4* __restrict__ neg) {
    uint32_t half[2], sc[2];
    uint64_t ip2[2], in2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t wh[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) wh[i] = w[8 * h + i];
        half[h] = side_maxima<8>(wh);
    }
    if (gs != 16) {
        uint32_t c = __vmaxs2(half[0], half[1]);
        if (gs >= 64) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, 1));
        if (gs == 128) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, 2));
        half[0] = half[1] = c;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float ip, in;
        sc[h] = group_scales(half[h], ip, in);
        ip2[h] = pack_f32x2(__float_as_uint(ip), __float_as_uint(ip));
        in2[h] = pack_f32x2(__float_as_uint(in), __float_as_uint(in));
    }
    uint32_t nib[4], pp[4], nn[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t cp, cn;
        encode8_both(w + 4 * j, ip2[j >> 1], in2[j >> 1], cp, cn);
        const uint32_t m = negative_nibbles(cp);
        pp[j] = cp & ~m;
        nn[j] = cn & m;
        nib[j] = pp[j] | nn[j];
    }
    if (!own) return 0;
    if (codes) codes[v] = make_uint4(nib[0], nib[1], nib[2], nib[3]);
    pos[v] = make_uint4(pp[0], pp[1], pp[2], pp[3]);
    neg[v] = make_uint4(nn[0], nn[1], nn[2], nn[3]);
    if (gs == 16) {
        row_scales[2 * g] = (uint16_t)sc[0];
        row_scales[2 * g + 1] = (uint16_t)sc[1];
    } else if (gs == 64) {
        if (!(g & 1)) row_scales[g >> 1] = (uint16_t)sc[0];
    } else if (!(g & 3)) row_scales[g >> 2] = (uint16_t)sc[0];
    return sc[0] | (sc[1] << 16);
}

// V^T of an attention call: V cast down its keys, with everything the FP4 kernel reads, beside the casts of Q and K.  A block owns
// eight columns of one head (eight operand rows) over all keys, so that the rows' largest scales are known inside the block and
// the scale factors follow without another launch.  Keys come in passes of 64 groups through shared memory; a group's rows
// are 528 bytes apart from the next group's, and lanes are eight groups x four column pairs: no bank conflicts on the way out,
// and a column's codes leave in pieces of 128 bytes.  What bounds it is latency (one load, one cast, one exchange): as two
// launches of its own, cast and scale factors, it cost 10 us for 8 heads x 1056 keys; here it runs beside Q and K (the call with
// 32 query heads, causal: 62.2 -> 55.4 us; 32 heads x 8192 1872 -> 1845).
constexpr int kVtCols = 8, kVtGroups = 64, kVtPitch = 528, kVtRows = 128, kVtKept = 256;   // kVtKept: groups whose scales stay in shared memory
size_t vt_smem_bytes(int64_t G) { return (size_t)std::min<int64_t>(G, kVtGroups) * kVtPitch + (G <= kVtKept ? G * kVtCols * 2 : 0); }

__device__ __forceinline__ void cast_vt_block(const VtOperand& o, unsigned block, uint8_t* smem, int* flushed_total) {
    __shared__ int top_s[kVtCols][2], flushed_s[kVtCols];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t head = block / (kVtRows / kVtCols), G = o.L / 32;
    const int c0 = (int)(block % (kVtRows / kVtCols)) * kVtCols;
    const bool in_use = c0 < o.d;                   // head dimension 64: the other rows have zero scale factors
    const int64_t row0 = head * kVtRows + c0;
    const bool kept = G <= kVtKept;
    uint16_t* sc_s = reinterpret_cast<uint16_t*>(smem + min(G, (int64_t)kVtGroups) * kVtPitch);   // [column][group]
    if (tid < kVtCols) top_s[tid][0] = top_s[tid][1] = flushed_s[tid] = 0;
    uint32_t top[2] = {0, 0};
    if (in_use) {
        const uint4* src = o.x + (head * o.L * o.d + c0) / 8;
        const int vec = o.d / 8, cw = tid & 3, g = tid >> 2;
        for (int64_t g0 = 0; g0 < G; g0 += kVtGroups) {
            const int n = (int)min(G - g0, (int64_t)kVtGroups);
            if (g0) __syncthreads();                // the pass before has been read
            for (int i = tid; i < n * 32; i += 256) cp_async16(smem + (i >> 5) * kVtPitch + (i & 31) * 16, src + (g0 * 32 + i) * vec);
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
            if (g >= n) continue;
            const uint32_t* tile = reinterpret_cast<const uint32_t*>(smem + g * kVtPitch) + cw;
            uint32_t lo[16], hi[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint32_t a = tile[8 * i], b = tile[8 * i + 4];
                lo[i] = __byte_perm(a, b, 0x5410);
                hi[i] = __byte_perm(a, b, 0x7632);
            }
            const int64_t v = (row0 + 2 * cw) * G + g0 + g;
            const uint32_t s0 = emit_group(lo, v, nullptr, o.scales, o.pos, o.neg), s1 = emit_group(hi, v + G, nullptr, o.scales, o.pos, o.neg);
            if (kept) {
                sc_s[2 * cw * G + g0 + g] = (uint16_t)s0;
                sc_s[(2 * cw + 1) * G + g0 + g] = (uint16_t)s1;
            }
            top[0] = __vmaxu2(top[0], halves(s0));
            top[1] = __vmaxu2(top[1], halves(s1));
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int d = 4; d < 32; d <<= 1) top[j] = __vmaxu2(top[j], __shfl_xor_sync(0xFFFFFFFFu, top[j], d));
    }
    __syncthreads();
    if (lane < 4)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            atomicMax(&top_s[2 * lane + j][0], (int)(top[j] & 0xFFFFu));
            atomicMax(&top_s[2 * lane + j][1], (int)(top[j] >> 16));
        }
    __syncthreads();
    const int r = tid & (kVtCols - 1);              // of all of this thread's items
    const int kmax = scale_key(max(top_s[r][0], top_s[r][1]));
    const int64_t row = row0 + r, sf_row = sf_row_offset(row, o.nk64);
    const uint16_t* sc = kept ? sc_s + r * G : o.scales + row * G;   // (written by this block)
    const float factor = sf_factor(kmax);
    uint32_t lost = 0;
    for (int c = tid / kVtCols; c < o.nk64; c += 256 / kVtCols) {
        const int g = 2 * c;
        const uint32_t u = to_ue4m3x2(in_use && g < G ? sc[g] : 0u, factor, lost) | to_ue4m3x2(in_use && g + 1 < G ? sc[g + 1] : 0u, factor, lost) << 16;
        const int64_t off = sf_row + (int64_t)c * kSfChunkBytes;
        *reinterpret_cast<uint32_t*>(o.sf_pos + off) = __byte_perm(u, 0, 0x2200);
        *reinterpret_cast<uint32_t*>(o.sf_neg + off) = __byte_perm(u, 0, 0x3311);
    }
    if (!in_use) return;                            // (nor are those rows' words read)
    int flushed = (int)(lost >> 7);
#pragma unroll
    for (int d = kVtCols; d < 32; d <<= 1) flushed += __shfl_xor_sync(0xFFFFFFFFu, flushed, d);
    if (lane < kVtCols && flushed) atomicAdd(&flushed_s[r], flushed);
    __syncthreads();
    if (tid < kVtCols) {
        o.row_exp[row] = row_word(kmax, side_bits_of((uint32_t)top_s[r][0] | ((uint32_t)top_s[r][1] << 8)), flushed_s[r]);
        if (flushed_s[r] && flushed_total) atomicAdd(flushed_total, flushed_s[r]);
    }
}

// MODE: one cast, two casts, operands that may be canonical, any of these with a group size other than 32, or the three casts
// of an attention call.  (The plain cast is kept lean - its pointers are compile-time places in constant memory: it is bound by
// instruction issue, and four blocks have to share an SM.  Five fit where little work per block leaves latency to hide, in the
// attention's casts: 54.3 -> 53.4 us for 32 over 8 heads x 1056 causal; elsewhere they are no faster, and the canonical operand's
// batch of loads spills: 1000 x 11008 x 4096 89.5 -> 94.7.)
enum PrepMode { kOneCast, kTwoCasts, kAnyKind, kAnyGroup, kAttention };
template <int FMT, int GPL, int MODE>
__global__ void __launch_bounds__(kCastWarps * 32, MODE == kAttention ? 5 : 4)
prepare_operands_kernel(const __grid_constant__ PrepParams p) {
    begin_kernel();
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr bool SPLIT = MODE == kAnyKind || MODE == kAnyGroup, ANY_GS = MODE == kAnyGroup;
    if (MODE == kAttention && blockIdx.x < p.vt_blocks) {
        cast_vt_block(p.vt, blockIdx.x, smem_raw, p.flushed_total);
        return;
    }
    const unsigned bid = blockIdx.x - (MODE == kAttention ? p.vt_blocks : 0u);
    const bool second = MODE != kOneCast && bid >= p.blocks0;
    const PrepOperand& o = p.op[second];
    const unsigned block = bid - (second ? p.blocks0 : 0u);
    const int G = p.G, lpr_log2 = p.lpr_log2, nk64 = p.nk64, gs = ANY_GS ? p.gs : 32;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, LPR = 1 << lpr_log2, lr = lane & (LPR - 1);
    const int RPW = 32 >> lpr_log2, sg = lane >> lpr_log2;      // rows per warp; which of them this lane works on
    // the block's rows: 128-row block rb, sector sets k0 .. k0 + RPW - 1 (16 / RPW blocks share a 128-row block)
    const unsigned rb = block >> (lpr_log2 - 1);
    const int k0 = ((int)block & ((16 >> (5 - lpr_log2)) - 1)) << (5 - lpr_log2);
    const int r_in = 32 * (wi >> 1) + 2 * (k0 + sg) + (wi & 1);  // row inside the 128-row block
    const int64_t row = (int64_t)rb * 128 + r_in;
    // Segments (the heads of an attention call): seg_rows source rows each, padded to seg_blocks blocks of 128 operand rows.
    int64_t src_row = row;
    bool live = row < o.R;
    if (MODE == kAttention && o.seg_blocks) {
        const unsigned seg = rb / o.seg_blocks, in_seg = (rb - seg * o.seg_blocks) * 128 + r_in;
        live = live && in_seg < o.seg_rows;
        src_row = seg * o.seg_rows + in_seg;
    }
    const unsigned seg_mask = LPR == 32 ? 0xFFFFFFFFu : ((1u << LPR) - 1u) << (lane & ~(LPR - 1));
    const int64_t v_row = row * G;
    // this lane's ring: kCastDepth slots of 64 bytes (one piece).  Part j of a piece sits at 16-byte position
    // j ^ ((lane >> 1) & 3) of the slot, so that the lanes of a quarter warp read eight different bank groups.
    uint8_t* ring = smem_raw + ((wi * kCastDepth * 32) + lane) * 64;
    uint8_t* xchg = smem_raw + kCastRingBytes;        // [plane][chunk][sector set][h][q] words of 4 scale-factor bytes
    const int swz = (lane >> 1) & 3;
    const int n_own = (live && lr < G) ? ((G - lr + LPR - 1) >> lpr_log2) : 0;   // pieces this lane owns
    const int n_max = (G + LPR - 1) >> lpr_log2;      // of any lane
    const int64_t scale_row = row * (ANY_GS ? G * 32 >> p.gs_log2 : G);
    uint16_t* const row_scales = o.scales + scale_row;                           // canonical scales: written by a cast, read otherwise
    const uint16_t* const in_scales = !SPLIT || o.x ? row_scales : o.in_scales + scale_row;
    auto issue = [&](int i) {                        // copies of the lane's i-th piece, one commit group per call
        if (i < n_own) {
            const uint4* src = o.x + src_row * o.ld_vec + (lr + ((int64_t)i << lpr_log2)) * 4;
            uint8_t* slot = ring + (i % kCastDepth) * (32 * 64);
#pragma unroll
            for (int j = 0; j < 4; ++j) cp_async16(slot + ((j ^ swz) << 4), src + j);
        }
        cp_async_commit();
    };
    auto cast_piece = [&](int i) -> uint32_t {       // the i-th piece has landed: read it back, cast, store
        const uint8_t* slot = ring + (i % kCastDepth) * (32 * 64);
        const bool own = i < n_own;
        if (gs == 32 && !own) return 0;
        uint32_t w[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint4 q = make_uint4(0, 0, 0, 0);
            if (own) q = *reinterpret_cast<const uint4*>(slot + ((j ^ swz) << 4));
            w[4 * j] = q.x; w[4 * j + 1] = q.y; w[4 * j + 2] = q.z; w[4 * j + 3] = q.w;
        }
        const int g = lr + (i << lpr_log2);
        if (ANY_GS && gs != 32) return cast_piece_gs(w, own, gs, v_row + g, g, row_scales, o.codes, o.pos, o.neg);
        const uint32_t sc = emit_group<FMT>(w, v_row + g, o.codes, reinterpret_cast<uint16_t*>(o.scales), o.pos, o.neg);
        return sc | (sc << 16);
    };
    uint32_t sc_reg[GPL > 0 ? GPL : 1];
    uint32_t top = 0;                               // largest scale bytes seen by this lane, {neg : pos} as halves
    auto see = [&](uint32_t sc) {
        top = __vmaxu2(top, halves(sc));
        if (ANY_GS && gs == 16) top = __vmaxu2(top, halves(sc >> 16));
    };
    if (!SPLIT || o.x) {
#pragma unroll
        for (int i = 0; i < kCastDepth - 1; ++i) issue(i);
        if (GPL > 0) {
#pragma unroll
            for (int i = 0; i < GPL; ++i) {
                issue(i + kCastDepth - 1);
                cp_async_wait<kCastDepth - 1>();
                sc_reg[i] = cast_piece(i);
                see(sc_reg[i]);
            }
        } else {
            for (int i = 0; i < n_max; ++i) {
                issue(i + kCastDepth - 1);
                cp_async_wait<kCastDepth - 1>();
                see(cast_piece(i));
            }
        }
        cp_async_wait<0>();
    } else {
        // canonical operand: the first codes are on their way while the scales are read - whether the row needs a split at
        // all is known only from all of them
        constexpr int kBatch = 4;                   // 16-byte loads in flight per lane
        uint4 q[kBatch];
        auto load_codes = [&](int i0) {
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (i0 + i < n_own) q[i] = __ldg(o.in_codes + v_row + lr + ((int64_t)(i0 + i) << lpr_log2));
        };
        load_codes(0);
        uint32_t differ = 0;
        if (GPL > 0) {
#pragma unroll
            for (int i = 0; i < GPL; ++i) {
                sc_reg[i] = i < n_own ? piece_scales(in_scales, lr + (i << lpr_log2), gs) : 0u;
                see(sc_reg[i]);
                differ |= sc_reg[i] ^ __byte_perm(sc_reg[i], 0, 0x2301);
            }
        } else {
            for (int i = 0; i < n_own; ++i) {
                const uint32_t sc = piece_scales(in_scales, lr + (i << lpr_log2), gs);
                see(sc);
                differ |= sc ^ __byte_perm(sc, 0, 0x2301);
            }
        }
        // A row whose two scales agree in every group (a symmetric format) needs no split: sum over both signs of
        // code x scale_side = code x scale.  Its signed codes go to the positive plane as they are.
        const bool unsplit = __reduce_or_sync(seg_mask, differ) == 0;
        const uint32_t keep_sc = unsplit ? 0x00FF00FFu : 0xFFFFFFFFu, keep = unsplit ? 0u : 0xFFFFFFFFu;
        if (unsplit) top &= 0xFFFFu;
        if (GPL > 0) {
#pragma unroll
            for (int i = 0; i < GPL; ++i) sc_reg[i] &= keep_sc;
        }
        for (int i0 = 0; i0 < n_own; i0 += kBatch) {
            if (i0) load_codes(i0);
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                if (i0 + i >= n_own) break;
                const uint32_t c[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
                uint32_t pp[4], nn[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t m = negative_nibbles(c[j]) & keep;
                    nn[j] = c[j] & m;
                    pp[j] = c[j] & ~m;
                }
                const int64_t v = v_row + lr + ((int64_t)(i0 + i) << lpr_log2);
                o.pos[v] = make_uint4(pp[0], pp[1], pp[2], pp[3]);
                o.neg[v] = make_uint4(nn[0], nn[1], nn[2], nn[3]);
            }
        }
        if (GPL == 0) sc_reg[0] = keep_sc;          // for the second sweep
    }
    // The key of an E5M2 byte grows with the byte (scales carry no sign bit): the largest byte has the largest key.
    const uint32_t top_p = __reduce_max_sync(seg_mask, top & 0xFFFFu), top_n = __reduce_max_sync(seg_mask, top >> 16);
    const int kmax = scale_key(max(top_p, top_n));
    const int64_t sf_row = sf_row_offset(row, nk64);
    // word of the exchange buffer that holds this row's bytes of chunk c: ((c * RPW + sg) * 2 + h) * 4 + q
    const int x_row = (sg * 2 + (wi & 1)) * 4 + (wi >> 1), x_plane = nk64 * RPW * 8;   // in words
    const float factor = sf_factor(kmax);
    uint32_t lost = 0;
    auto put = [&](int g, uint32_t sc) {            // scale factors of piece g (zero past the row's last one)
        const uint32_t before = lost, u0 = to_ue4m3x2(sc, factor, lost);
        if (ANY_GS && gs > 32 && (g & ((gs >> 5) - 1))) lost = before;   // groups, not pieces, are counted
        const uint32_t u1 = ANY_GS && gs == 16 ? to_ue4m3x2(sc >> 16, factor, lost) : u0;   // the second half has its own scales
        const uint32_t up = __byte_perm(u0, u1, 0x0040), un = __byte_perm(u0, u1, 0x0051);
        if (p.exchange) {
            uint16_t* w16 = reinterpret_cast<uint16_t*>(xchg) + (((g >> 1) * RPW * 8 + x_row) << 1) + (g & 1);
            w16[0] = (uint16_t)up;
            w16[x_plane << 1] = (uint16_t)un;
        } else {
            const int64_t off = sf_row + sf_group_offset(g);
            *reinterpret_cast<uint16_t*>(o.sf_pos + off) = (uint16_t)up;
            *reinterpret_cast<uint16_t*>(o.sf_neg + off) = (uint16_t)un;
        }
    };
    const int g_end = nk64 * 2;                     // pieces past G: padding to whole 256-element blocks
    if (GPL > 0) {
#pragma unroll
        for (int i = 0; i < GPL; ++i) {
            const int g = lr + (i << lpr_log2);
            if (g < g_end) put(g, sc_reg[i]);       // zero for a piece past G and for a padding row
        }
        for (int g = lr + (GPL << lpr_log2); g < g_end; g += LPR) put(g, 0u);
    } else {
        // (a cast in a symmetric format wrote its one scale to both bytes; only the positive side's counts)
        const uint32_t keep_sc = !SPLIT || o.x ? (FMT ? 0x00FF00FFu : 0xFFFFFFFFu) : sc_reg[0];
        if (ANY_GS) __syncwarp();                   // scales of larger groups were written by neighbouring lanes
        for (int g = lr; g < g_end; g += LPR) put(g, (live && g < G) ? piece_scales(in_scales, g, gs) & keep_sc : 0u);
    }
    const int flushed = __reduce_add_sync(seg_mask, (int)(lost >> 7));
    if (lr == 0 && live) {
        o.row_exp[row] = row_word(kmax, side_bits_of(top_p | (top_n << 8)), flushed);
        if (flushed && p.flushed_total) atomicAdd(p.flushed_total, flushed);
    }
    if (lr == 0 && !live && row < o.R) o.row_exp[row] = 0;       // padding rows of a segment
    if (!p.exchange) return;                        // uniform over the block
    __syncthreads();
    // 16 bytes per thread: the words of rows q = 0..3 (32 rows apart) for one (plane, chunk, sector set, h);
    // two neighbouring threads (h = 0, 1) fill one sector
    const int per_plane = nk64 * RPW * 2, set_log2 = 6 - lpr_log2;   // RPW * 2 = 1 << set_log2
    for (int item = threadIdx.x; item < 2 * per_plane; item += kCastWarps * 32) {
        const int plane = item >= per_plane, rest = item - plane * per_plane;
        const int c = rest >> set_log2, sh = rest & ((1 << set_log2) - 1);   // sh = sector set * 2 + h
        const uint4 v = reinterpret_cast<const uint4*>(xchg)[item];
        uint8_t* dst = (plane ? o.sf_neg : o.sf_pos) + ((int64_t)rb * nk64 + c) * kSfChunkBytes + (2 * k0 + sh) * 16;
        *reinterpret_cast<uint4*>(dst) = v;
    }
}

// Attention glue in one pass (Appendix C): row softmax of the fp32 logits (times alpha), rounding of the
// normalised map to bf16 - the cast's input type - and the cast of that row to AMXFP4, without the map ever
// reaching global memory as fp32 or bf16.  One block of softmax::kT threads per row (grid = padded rows when the
// prepared form is written, blocks past the last row only zero scale-factor padding).  Same bits as the
// stand-alone softmax kernel followed by the cast: both use softmax_math.cuh and cast_math.cuh.
// CACHED: the row has at most kT groups, so each thread keeps its one group in registers between the passes.
template <bool CACHED>
__global__ void __launch_bounds__(softmax::kT)
softmax_cast_kernel(const float* __restrict__ S, int64_t R, int G, int64_t ld_s, float alpha, int vec, int64_t causal,
                    uint4* __restrict__ codes, uint16_t* __restrict__ scales, uint4* __restrict__ pos,
                    uint4* __restrict__ neg, uint8_t* __restrict__ sf_pos, uint8_t* __restrict__ sf_neg,
                    int* __restrict__ row_exp, int nk64) {
    begin_kernel();
    __shared__ float sh[softmax::kT / 32];
    __shared__ int slot_s[4];
    const int gx = threadIdx.x;
    const int64_t row = blockIdx.x;
    const bool row_live = row < R;                  // uniform over the block
    if (gx < 4) slot_s[gx] = 0;
    uint32_t sc_first = 0, top = 0;
    if (row_live) {
        const float* s = S + row * ld_s;
        const int64_t cols = (int64_t)G * 32, v_row = row * G;
        const int64_t seen = causal ? min(cols, row % causal + 1) : cols;    // causal: query i of its matrix sees keys 0 .. i
        if (CACHED) {
            float e[32];
            const float sum = softmax::cached_row_exp(s, G, vec != 0, alpha, sh, e, seen);
            if (gx < G) {
                uint32_t w[16];
                softmax::normalised_group_e(e, sum, w);
                sc_first = emit_group(w, v_row + gx, codes, scales, pos, neg);
                top = sc_first;
            }
        } else {
            float mx, sum;
            softmax::row_stats(s, cols, vec != 0, alpha, sh, mx, sum, seen);
            for (int g = gx; g < G; g += softmax::kT) {
                float t[32];
                uint32_t w[16];
                softmax::load_group(s, g, cols, vec != 0, alpha, t, seen);
                softmax::normalised_group(t, mx, sum, w);
                const uint32_t sc = emit_group(w, v_row + g, codes, scales, pos, neg);
                if (g == gx) sc_first = sc;
                top = __vmaxu4(top, sc);
            }
        }
    }
    if (!pos) return;                               // canonical output only
    finish_prepared_row(row, row_live, G, gx, softmax::kT, top, sc_first, scales, slot_s, sf_pos, sf_neg, row_exp, nk64);
}

// The same for rows of at most 32 groups, canonical output only: a warp per row, a lane per group.  The block kernel's
// reductions over one warp's lanes and then over seven idle warps come to the same maximum and the same sum, so the
// bits are the same; a row of 320 columns leaves that kernel's block with ten busy threads.
__global__ void __launch_bounds__(256)
softmax_cast_warp_kernel(const float* __restrict__ S, int64_t R, int G, int64_t ld_s, float alpha, int vec, int64_t causal,
                         uint4* __restrict__ codes, uint16_t* __restrict__ scales) {
    begin_kernel();
    const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= R) return;
    const int64_t cols = (int64_t)G * 32, seen = causal ? min(cols, row % causal + 1) : cols;
    float e[32];
    if (lane < G) softmax::load_group(S + row * ld_s, lane, cols, vec != 0, alpha, e, seen);
    else {
#pragma unroll
        for (int i = 0; i < 32; ++i) e[i] = -INFINITY;
    }
    float mx = -INFINITY, sum = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) mx = fmaxf(mx, e[i]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, d));
    const float nm = softmax::neg_max_log2e(mx);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        e[i] = softmax::exp_rel(e[i], nm);
        sum += e[i];
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum = sum + __shfl_xor_sync(0xFFFFFFFFu, sum, d);
    if (lane >= G) return;
    uint32_t w[16];
    softmax::normalised_group_e(e, sum, w);
    emit_group(w, row * G + lane, codes, scales, nullptr, nullptr);
}

template <int EPT, int TPG, int FMT = 0>
int launch_rows(const void* x, int64_t rows, int64_t K, int64_t ld, uint8_t* codes,
                uint8_t* scales, cudaStream_t st) {
    const int64_t n_items = rows * (K / EPT);
    const int64_t blocks = (n_items + kThreads - 1) / kThreads;
    if (blocks > 0x7FFFFFFF) return AMX_ERR_SHAPE;
    auto* xv = reinterpret_cast<const uint4*>(x);
    auto* cv = reinterpret_cast<uint4*>(codes);
    auto* sv = reinterpret_cast<uint16_t*>(scales);
    if (ld == K)
        return launch(quantize_rows_kernel<EPT, TPG, true, FMT>, (unsigned)blocks, kThreads, 0, st, xv, n_items, K / EPT, ld / 8, cv, sv);
    return launch(quantize_rows_kernel<EPT, TPG, false, FMT>, (unsigned)blocks, kThreads, 0, st, xv, n_items, K / EPT, ld / 8, cv, sv);
}

}  // namespace

// One launch for one or two operands of the FP4 GEMM (K and group size in common): canonical scales (and codes, when asked
// for) of a cast, the two sign planes, the UE4M3 scale factors of both planes in the tensor cores' layout (nk64 chunks of
// 512 B per block of 128 rows, rows padded to padded_rows) and the row words.  format: of a cast (group size 32 unless
// AMXFP4).  flushed_total (optional): incremented by the number of scales flushed.
namespace {
// Everything but the columns of V; `blocks`: of all operands, `smem`: of a block; returns the pieces per lane.
int fill_prepare(PrepParams& p, const PrepOperand* op, int n, int64_t K, int gs, int nk64, int* flushed_total, int64_t& blocks, int& smem) {
    p.G = (int)(K / 32);
    p.lpr_log2 = 1;
    while (p.lpr_log2 < 5 && (1 << p.lpr_log2) < p.G) ++p.lpr_log2;  // lanes per row: a power of two, 2 .. 32
    const int rpw = 32 >> p.lpr_log2;                                // rows per warp
    blocks = 0;
    for (int i = 0; i < n; ++i) {
        p.op[i] = op[i];
        blocks += (op[i].padded_rows / 128) * (16 / rpw);            // a block has 8 * rpw rows of one 128-row block
        if (i == 0) p.blocks0 = (unsigned)blocks;
    }
    p.nk64 = nk64;
    p.gs = gs;
    p.gs_log2 = gs == 16 ? 4 : gs == 32 ? 5 : gs == 64 ? 6 : 7;
    p.flushed_total = flushed_total;
    const size_t exchange_bytes = (size_t)64 * rpw * nk64;           // both planes, 4 bytes per row and 64 elements
    p.exchange = exchange_bytes <= (size_t)kCastMaxExchangeBytes;
    smem = kCastRingBytes + (p.exchange ? (int)exchange_bytes : 0);
    return (p.G + (1 << p.lpr_log2) - 1) >> p.lpr_log2;
}

template <int FMT, int MODE>
int launch_prepare(const PrepOperand* op, int n, int64_t K, int gs, int nk64, cudaStream_t st, int* flushed_total) {
    PrepParams p{};
    int64_t blocks;
    int smem;
    const int gpl = fill_prepare(p, op, n, K, gs, nk64, flushed_total, blocks, smem);
    if (blocks > 0x7FFFFFFF) return AMX_ERR_SHAPE;
    auto* kernel = gpl <= 1 ? prepare_operands_kernel<FMT, 1, MODE> : gpl <= 2 ? prepare_operands_kernel<FMT, 2, MODE>
                 : gpl <= 4 ? prepare_operands_kernel<FMT, 4, MODE> : gpl <= 8 ? prepare_operands_kernel<FMT, 8, MODE>
                 : prepare_operands_kernel<FMT, 0, MODE>;   // longer rows: the scale bytes are re-read, not kept in registers
    static bool configured[64][5] = {};                 // the opt-in to > 48 KB of dynamic shared memory: per device, kernel
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return AMX_ERR_CUDA;
    const int slot = gpl <= 1 ? 0 : gpl <= 2 ? 1 : gpl <= 4 ? 2 : gpl <= 8 ? 3 : 4;
    if (!configured[dev][slot]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCastRingBytes + kCastMaxExchangeBytes) !=
            cudaSuccess) {
            cudaGetLastError();
            return AMX_ERR_CUDA;
        }
        configured[dev][slot] = true;
    }
    return launch(kernel, (unsigned)blocks, kCastWarps * 32, smem, st, p);
}
}  // namespace

int prepare_operands(const PrepOperand* op, int n, int64_t K, int gs, int nk64, cudaStream_t st, int format, int* flushed_total) {
    if (format == AMX_FMT_SYM_FP8) return launch_prepare<1, kOneCast>(op, n, K, gs, nk64, st, flushed_total);
    if (format == AMX_FMT_MXFP4) return launch_prepare<2, kOneCast>(op, n, K, gs, nk64, st, flushed_total);
    if (gs != 32) return launch_prepare<0, kAnyGroup>(op, n, K, gs, nk64, st, flushed_total);
    if (!op[0].x || (n > 1 && !op[1].x)) return launch_prepare<0, kAnyKind>(op, n, K, gs, nk64, st, flushed_total);
    return n == 1 ? launch_prepare<0, kOneCast>(op, n, K, gs, nk64, st, flushed_total)
                  : launch_prepare<0, kTwoCasts>(op, n, K, gs, nk64, st, flushed_total);
}

// The casts of an attention call in one launch: Q and K (head dimension 64 or 128, so one piece per lane) and V^T of `kv_heads` heads.
int prepare_attention(const PrepOperand (&qk)[2], int64_t d, int nk64, const VtOperand& vt, int64_t kv_heads, cudaStream_t st, int* flushed_total) {
    if (d != 64 && d != 128) return AMX_ERR_SHAPE;
    PrepParams p{};
    int64_t blocks;
    int smem;
    fill_prepare(p, qk, 2, d, 32, nk64, flushed_total, blocks, smem);
    p.vt = vt;
    p.vt_blocks = (unsigned)(kv_heads * (kVtRows / kVtCols));
    blocks += p.vt_blocks;
    if (blocks > 0x7FFFFFFF) return AMX_ERR_SHAPE;
    return launch(prepare_operands_kernel<0, 1, kAttention>, (unsigned)blocks, kCastWarps * 32, std::max<size_t>(smem, vt_smem_bytes(vt.L / 32)), st, p);
}

// Softmax of the rows of S (fp32 [rows, ld_s], cols % 32 == 0), rounded to bf16 and cast, in one launch.  With
// pos == nullptr only the canonical codes and scales are written.
int softmax_cast_rows(const float* S, int64_t rows, int64_t cols, int64_t ld_s, float alpha, uint8_t* codes,
                      uint8_t* scales, void* pos, void* neg, uint8_t* sf_pos, uint8_t* sf_neg, int* row_exp, int nk64,
                      int64_t padded_rows, cudaStream_t st, int64_t causal) {
    const int64_t G = cols / 32, blocks = pos ? padded_rows : rows;
    if (blocks > 0x7FFFFFFF || G > 0x7FFFFFFF / 32) return AMX_ERR_SHAPE;
    const int vec = aligned(S, 16) && ld_s % 4 == 0;
    if (!pos && G <= 32) {
        return launch(softmax_cast_warp_kernel, (unsigned)((rows + 7) / 8), 256, 0, st, S, rows, (int)G, ld_s, alpha, vec, causal,
                                                                            reinterpret_cast<uint4*>(codes), reinterpret_cast<uint16_t*>(scales));
    }
    auto* kernel = G <= softmax::kT ? softmax_cast_kernel<true> : softmax_cast_kernel<false>;
    return launch(kernel, (unsigned)blocks, softmax::kT, 0, st, S, rows, (int)G, ld_s, alpha, vec, causal, reinterpret_cast<uint4*>(codes),
                                                     reinterpret_cast<uint16_t*>(scales), reinterpret_cast<uint4*>(pos),
                                                     reinterpret_cast<uint4*>(neg), sf_pos, sf_neg, row_exp, nk64);
}

namespace {

template <int TPG>
int launch_cols(const void* x, int64_t R, int64_t C, int64_t ld, int gs, uint8_t* codes,
                uint8_t* scales, cudaStream_t st, int64_t batch = 1) {
    dim3 grid((unsigned)((C + kTC - 1) / kTC), (unsigned)((R + kTR - 1) / kTR), (unsigned)batch);
    if (grid.y > 65535 || batch > 65535) return AMX_ERR_SHAPE;
    return launch(quantize_cols_kernel<TPG>, grid, kThreads, 0, st, reinterpret_cast<const __nv_bfloat16*>(x), R, C, ld, reinterpret_cast<uint32_t*>(codes),
        reinterpret_cast<uint16_t*>(scales), gs);
}

}  // namespace

// amx_quantize_t with group size 32 on `batch` matrices [R, C] stored one after another (contiguous rows); the
// canonical outputs of their transposes follow one another too.
int quantize_cols_batched(const void* x, int64_t batch, int64_t R, int64_t C, uint8_t* codes, uint8_t* scales,
                          cudaStream_t st) {
    return launch_cols<4>(x, R, C, C, 32, codes, scales, st, batch);
}

}  // namespace amx

namespace amx {
namespace {
template <int FMT>
int launch_rows_gs(const void* x, int64_t rows, int64_t K, int64_t ld_x, int group_size, uint8_t* codes, uint8_t* scales,
                   cudaStream_t st) {
    if (group_size == K && !fixed_group_size(group_size)) {          // whole-row grouping
        if (rows > 0x7FFFFFFF) return AMX_ERR_SHAPE;
        return launch(quantize_whole_rows_kernel<FMT>, (unsigned)rows, kThreads, 0, st, reinterpret_cast<const uint4*>(x), K / 8, ld_x / 8, reinterpret_cast<uint32_t*>(codes),
            reinterpret_cast<uint16_t*>(scales));
    }
    switch (group_size) {
        case 16:
            // pairs of groups where a row holds whole pairs and the wider stores are aligned
            if (K % 32 == 0 && aligned(codes, 16) && aligned(scales, 4)) {
                const int64_t n_items = rows * (K / 32), blocks = (n_items + kThreads - 1) / kThreads;
                if (blocks > 0x7FFFFFFF) return AMX_ERR_SHAPE;
                auto* kernel = ld_x == K ? quantize_rows16_kernel<true, FMT> : quantize_rows16_kernel<false, FMT>;
                return launch(kernel, (unsigned)blocks, kThreads, 0, st, reinterpret_cast<const uint4*>(x), n_items, K / 32, ld_x / 8,
                              reinterpret_cast<uint4*>(codes), reinterpret_cast<uint32_t*>(scales));
            }
            return launch_rows<16, 1, FMT>(x, rows, K, ld_x, codes, scales, st);
        case 32: return launch_rows<32, 1, FMT>(x, rows, K, ld_x, codes, scales, st);
        case 64: return launch_rows<32, 2, FMT>(x, rows, K, ld_x, codes, scales, st);
        default: return launch_rows<32, 4, FMT>(x, rows, K, ld_x, codes, scales, st);
    }
}
}  // namespace
}  // namespace amx

extern "C" int amx_quantize(const void* x, int64_t rows, int64_t K, int64_t ld_x, int group_size,
                            uint8_t* codes, uint8_t* scales, void* stream) {
    return amx_quantize_fmt(x, rows, K, ld_x, group_size, AMX_FMT_AMXFP4, codes, scales, stream);
}

extern "C" int amx_quantize_fmt(const void* x, int64_t rows, int64_t K, int64_t ld_x, int group_size, int format,
                                uint8_t* codes, uint8_t* scales, void* stream) {
    using namespace amx;
    if (format < AMX_FMT_AMXFP4 || format > AMX_FMT_AMXFP4_POT_ROUND) return AMX_ERR_FLAGS;
    if (!valid_group_size(group_size, K) || rows < 0 || K <= 0 || K % group_size || K % 8 || ld_x < K)
        return AMX_ERR_SHAPE;
    if (rows == 0) return AMX_OK;
    if (!x || !codes || !scales) return AMX_ERR_NULL;
    const int code_align = fixed_group_size(group_size) ? (group_size == 16 ? 8 : 16) : 4;
    if (!aligned(x, 16) || ld_x % 8 || !aligned(codes, code_align) || !aligned(scales, 2)) return AMX_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (format == AMX_FMT_SYM_FP8) return launch_rows_gs<1>(x, rows, K, ld_x, group_size, codes, scales, st);
    if (format == AMX_FMT_MXFP4) return launch_rows_gs<2>(x, rows, K, ld_x, group_size, codes, scales, st);
    if (format == AMX_FMT_AMXFP4_POT) return launch_rows_gs<3>(x, rows, K, ld_x, group_size, codes, scales, st);
    if (format == AMX_FMT_MXFP4_POT_ROUND) return launch_rows_gs<4>(x, rows, K, ld_x, group_size, codes, scales, st);
    if (format == AMX_FMT_AMXFP4_POT_ROUND) return launch_rows_gs<5>(x, rows, K, ld_x, group_size, codes, scales, st);
    return launch_rows_gs<0>(x, rows, K, ld_x, group_size, codes, scales, st);
}

extern "C" int amx_quantize_t(const void* x, int64_t R, int64_t C, int64_t ld_x, int group_size,
                              uint8_t* codes, uint8_t* scales, void* stream) {
    using namespace amx;
    if (!fixed_group_size(group_size) || R < 0 || C < 0 || R % group_size || ld_x < C) return AMX_ERR_SHAPE;
    if (R == 0 || C == 0) return AMX_OK;
    if (!x || !codes || !scales) return AMX_ERR_NULL;
    if (!aligned(x, 2) || !aligned(codes, 4) || !aligned(scales, 2)) return AMX_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (group_size) {  // a 64-row tile holds whole groups only for gs <= 64
        case 16: return launch_cols<2>(x, R, C, ld_x, group_size, codes, scales, st);
        case 32: return launch_cols<4>(x, R, C, ld_x, group_size, codes, scales, st);
        case 64: return launch_cols<8>(x, R, C, ld_x, group_size, codes, scales, st);
        default: return AMX_ERR_SHAPE;
    }
}
