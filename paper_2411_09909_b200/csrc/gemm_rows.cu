// AMXFP4 x AMXFP4 -> fp32 for few rows of A against a large weight (the decode phase of inference, small layers):
// C[m,n] = sum_k Ahat[m,k] * What[n,k] (arXiv 2411.09909, Section 4.3), bound by streaming the 4.5-bit weight
// from HBM once.
//
// The weight is read in its canonical layout (codes [N, K/2], scales [N, K/gs, 2]); nothing is prepared ahead.
// Warp-level mma.sync m16n8k16 (f16 in, fp32 accumulate) with 16 weight rows as the M side and 8 token rows as the
// N side, so that a single token wastes 7 of 8 columns and not 15 of 16 rows.  The contraction index may be permuted
// freely as long as both operands use the same permutation: lane (g, t) (g = lane / 4, t = lane % 4) owns, per step
// of 128 elements of K, the 32-element piece t of weight rows g and g + 8 of each of its warp's two 16-row blocks.
//
// Exactness.  Operands are decoded to f16: E2M1 x E5M2 has at most 5 significant bits and magnitudes between 2^-17 and
// 6 * 57344; times 2^-4 every value is a (possibly subnormal) f16 number, on both sides, and the result is multiplied
// by 2^8.  Products are exact in fp32; only the fp32 additions round.
//
// Decode.  cvt.rn.f16x2.e2m1x2 turns a code byte into two signed values; the positive ones take the positive side's
// scale, the negative ones the other: v = relu(w * s_p) + min(w, 0) * s_n (one of the two terms is zero).  This is what
// bounds the kernel where the memory does not: 6.6 cycles of a warp per pair of elements, the MMAs included, with four
// warps on a scheduler.  Measured in the same loop: max/min, multiply, multiply-add 7.8; two clamped multiply-adds
// and a subtraction 7.4; the scale chosen by a sign mask 7.7; code bits shifted into bf16 fields and the scale chosen
// by a mask (the earlier form) 8.7; the signs kept apart through two MMAs 7.1.
//
// Two kernels share this: gemm_rows_stream_kernel for up to 32 tokens (a CTA covers 8 to 112 weight rows, its eight warps split K;
// plan_stream) and gemm_rows_kernel for 33 and more, in blocks of 32, 48 or 64: a CTA of eight warps covers 128 weight rows and one
// range of K, warp = (row group of 32) + 4 * (parity of its steps).
// In both the codes come through a ring in shared memory by asynchronous copies, a slot per warp and step (a lane reads back
// only its own copies; no registers are held by loads in flight): the copies alone stream at 5.4-5.8 TB/s.  Scales are
// copied along the rows, many steps at a time.  (Copied per step beside the codes, 8 bytes per row at 32 different rows per
// instruction, they took more of the load path than the codes themselves: streaming alone 7.5-9 instead of 4.7 us for
// 12288 x 4096.)  The K ranges of the same rows are the CTAs of one thread-block cluster (up to 8), which add their partial
// products over distributed shared memory in rank order - deterministic, no scratch in global memory and no second launch.
//
// What bounds it (times inside a chain of calls, weights from HBM).  One row of 12288 x 4096, 12.8 us: 1.9 from the end of the call
// before to the first block (the fragments kernel and a launch), 2.4 to the first step's data, 5 for the steps - decode at 6
// cycles of a warp per pair, six warps to a scheduler - 0.5 for the sums; the other 3 lie between these points and have not
// been traced.  From two token tiles on mma.sync: an m16n8k16 takes a scheduler about 16 cycles, for 24 rows 12 per pair of the 13
// that a pair takes (14336 x 4096: 20.5 us).  Fragments are re-read by every CTA, which is why few CTAs of many rows are better
// from 17 tokens on.  (Decoded to shared memory for tcgen05.mma instead, whatever the number of tokens: 23 us - the way from the
// decoding warps through the MMA and back takes a microsecond, and four steps of 32 KB are all that fits.)
//
// The token rows are cast (or decoded) once by a small kernel into the fragment order.  (Cast inside the main kernel by
// every CTA, one launch less, measured the same for one row and slower for more.)
// The fragments kernel waits for its predecessors before it lets the main kernel start, so the main kernel may fill its
// rings at once - whoever wrote the weight has completed - and waits only for the fragments.  (Prefetching the weight into
// the L2 across the boundary between two calls measured slower: the memory is not what this kernel waits for.)
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "cast_math.cuh"
#include "cp_async.cuh"
#include "decode_math.cuh"
#include "gemm.cuh"
#include "scale_words.cuh"

namespace cg = cooperative_groups;

namespace amx {
namespace {

using namespace decode_f16;

constexpr int kWarps = 8, kThreads = kWarps * 32;
constexpr int kRowGroups = 4, kStepGroups = 2;     // warps: 4 groups of 32 weight rows x 2 step parities
constexpr int kCtaRows = kRowGroups * 32;
constexpr int kStepK = 128;
constexpr int kTok = 8;                            // token rows of one tile (the N side of one MMA)
constexpr int kFragBytes = kTok * kStepK * 2;      // fragments of one tile and step
constexpr int kCodeBytes = 4 * 512;                // codes of 32 rows and one step: 4 pieces of 16 bytes per lane
constexpr int kMaxSlices = 8;                      // portable cluster size
constexpr int kPartPitch = kCtaRows + 4;           // floats per token row of the partial-product tile (bank spread)
constexpr int kMaxTiles = 8;                       // token tiles per CTA
// Steps whose scales are held at a time: those of 32 steps in groups of 16 (67 KB) do not fit beside the rings of eight token
// tiles (192 KB).
__host__ __device__ constexpr int scale_steps(int gs) { return gs == 16 ? 16 : 32; }
constexpr size_t kMaxSmem = 227 * 1024, kSmSmem = 228 * 1024, kCtaSmem = 1024;   // of a block; of an SM, which keeps some per block

// Fragment order of the token rows, per step and tile of 8 rows: pieces of 16 bytes [j = 0..3][lane 0..31]; the piece
// of (j, lane (g, t)) holds elements 32 t + 8 j .. + 7 of the step, row g of the tile.  Piece (j, l) sits at position
// l ^ (2 j): the casting lanes (same row, consecutive pieces of 8 elements) then hit eight bank groups.
__device__ __forceinline__ int frag_pos(int j, int l) { return j * 32 + (l ^ (2 * j)); }

// 8 consecutive elements of a row cast and decoded; TPG lanes hold one group.
template <int TPG>
__device__ __forceinline__ uint4 cast_piece(const uint4 q) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t c = cast::side_maxima<4>(w);
#pragma unroll
    for (int d = 1; d < TPG; d <<= 1) c = __vmaxs2(c, __shfl_xor_sync(0xFFFFFFFFu, c, d));
    float inv_p, inv_n;
    const uint32_t sc = cast::group_scales(c, inv_p, inv_n);
    return decode_word(cast::encode8(w, inv_p, inv_n), make_scales(sc));
}

// One thread per piece of 8 elements (grid y: the row).  Rows past M are zeros.  The kernel is a few thousand threads of
// pure latency, so a group's work is spread over lanes.
template <bool CAST, int GS>
__global__ void __launch_bounds__(128) rows_fragments_kernel(const uint8_t* __restrict__ codes,
                                                             const uint8_t* __restrict__ scales,
                                                             const uint16_t* __restrict__ x, int64_t ld_x, int M,
                                                             int tiles, int64_t K, uint4* __restrict__ frag,
                                                             int* __restrict__ status) {
    const int64_t per_row = K / 8;
    const int64_t k8 = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int row = blockIdx.y;
    grid_dependency_wait();                    // the previous call on this stream may still read the workspace
    grid_launch_dependents();                  // the main kernel may start filling its rings
    if (k8 == 0 && row == 0) status[0] = status[1] = 0;   // no device-side wait that can expire, no scale is flushed
    const bool live = k8 < per_row, seen = live && row < M;
    uint4 out = make_uint4(0, 0, 0, 0);
    if (CAST) {
        uint4 q = make_uint4(0, 0, 0, 0);
        if (seen) q = __ldg(reinterpret_cast<const uint4*>(x + row * ld_x + k8 * 8));
        out = cast_piece<GS / 8>(q);           // zeros cast to zeros
    } else if (seen) {
        const uint32_t word = __ldg(reinterpret_cast<const uint32_t*>(codes + row * (K / 2) + k8 * 4));
        const uint32_t sc = __ldg(reinterpret_cast<const unsigned short*>(scales + (row * (K / GS) + k8 * 8 / GS) * 2));
        out = decode_word(word, make_scales(sc));
    }
    if (!live) return;
    const int64_t step = k8 >> 4;
    const int j = (int)k8 & 3, t = (int)(k8 >> 2) & 3;
    frag[(step * tiles + (row >> 3)) * 128 + frag_pos(j, (row & 7) * 4 + t)] = out;
}

__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct RowsParams {
    const uint4* frag;           // [step][tiles of all rows]
    const uint8_t *w_codes, *w_scales;
    int M;
    int64_t N, K;
    float* C;
    int64_t ld_c;
    int steps_max;               // steps of the longest range
    int rows;                    // weight rows per CTA (streaming kernel)
};

// Shared-memory geometry.  kDepth ring slots per warp (kDepth - 1 steps in flight); with up to four token tiles two
// CTAs share an SM, which is what keeps enough of the weight in flight.
template <int NT, int GS>
struct Ring {
    static constexpr int kDepth = NT == 3 || NT == 4 ? 3 : 4;
    static constexpr int kFragSlot = NT * kFragBytes;
    static constexpr int kBytes = kWarps * kDepth * kCodeBytes;
    static constexpr int kFragRing = kStepGroups * kDepth * kFragSlot;
    static constexpr int kPart = NT * kTok * kPartPitch * 4;
    static_assert(kPart <= kBytes, "the partial-product tile reuses the rings");
};
// Groups of 128, an odd number of scale pairs in the tensor: its last half word, which the copies of words leave out, for a run of n steps
// that ends with the weight's last row.  row: where that row's words lie.  (Copies of a variable number of bytes instead cost calls with
// such groups 3 to 5 %: 73 x 4096 x 8576 33.9 us, so 32.5.)
__device__ __forceinline__ void load_last_pair(uint32_t* row, const uint8_t* scales, int64_t pairs, int n) {
    const int64_t word = pairs >> 1;
    row[word - ((pairs - n) >> 1)] = __ldg(reinterpret_cast<const uint16_t*>(scales + word * 4));
}

// Scales of one weight row over `n` steps: the most 4-byte words copied (groups of 128: two bytes per step, copied as the aligned
// words around them, scale_words.cuh), and the pitch of the rows in shared memory - twice an odd number of words, so that the words
// of eight rows that a warp reads together lie in different banks (groups of 16: four words per step, four times an odd number).
__host__ __device__ constexpr int scale_words(int n, int gs) { return gs == 128 ? n / 2 + 1 : n * (64 / gs); }
__host__ __device__ constexpr int scale_pitch(int n, int gs) {
    return gs == 16 ? (n | 1) * 4 : gs == 32 ? (n | 1) * 2 : gs == 64 ? (n | 1) : (n / 2 + 1) | 1;
}
__host__ __device__ constexpr int scale_bytes(int n, int gs) { return (kCtaRows * scale_pitch(n, gs) * 4 + 15) / 16 * 16; }

// NT: tiles of 8 token rows per CTA.
template <int NT, int GS>
__global__ void __launch_bounds__(kThreads, NT <= 4 ? 2 : 1) gemm_rows_kernel(const RowsParams p) {
    using R = Ring<NT, GS>;
    constexpr int kDepth = R::kDepth, kFragSlot = R::kFragSlot, kScaleSteps = scale_steps(GS);
    static_assert(R::kBytes + R::kFragRing + scale_bytes(kScaleSteps, GS) <= kMaxSmem, "shared memory of the longest range");
    extern __shared__ __align__(16) uint8_t smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int slices = (int)gridDim.y, slice = (int)blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int wr = warp & 3, wk = warp >> 2;
    const int64_t steps = p.K / kStepK;
    const int64_t s_begin = steps * slice / slices;
    const int n_total = (int)(steps * (slice + 1) / slices - s_begin);
    const int64_t row0 = (int64_t)blockIdx.x * kCtaRows;
    const int m0 = (int)blockIdx.z * (NT * kTok);

    uint8_t* ring = smem + warp * (kDepth * kCodeBytes);
    const int held = min(p.steps_max, kScaleSteps), pitch = scale_pitch(held, GS);
    uint32_t* scale_s = reinterpret_cast<uint32_t*>(smem + R::kBytes);
    uint8_t* frag_s = smem + R::kBytes + scale_bytes(held, GS);      // a ring of fragments per step parity

    // this lane's streams: piece t of rows g, g + 8 (block 0), g + 16, g + 24 (block 1) of the warp's 32 rows
    const uint8_t* pc[4];
    int odd[4];                                // groups of 128: which half of its word a row's first scale is
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int64_t r = row0 + wr * 32 + q * 8 + g;
        r = r < p.N ? r : p.N - 1;             // rows past the weight read its last row; their sums are not stored
        pc[q] = p.w_codes + r * (p.K / 2) + s_begin * 64 + t * 16;
        odd[q] = GS == 128 ? (int)((r * steps + s_begin) & 1) : 0;
    }
    const int n_mine = (n_total - wk + 1) / kStepGroups;             // this warp's steps: wk, wk + 2, ...
    auto issue_codes = [&](int i) {
        if (i < n_mine) {
            uint8_t* slot = ring + (i % kDepth) * kCodeBytes + lane * 16;
            const int64_t off = (int64_t)(wk + i * kStepGroups) * 64;
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async16(slot + q * 512, pc[q] + off);
        }
    };
    // scales of steps [first, first + n) of the range, all 128 rows: consecutive threads copy consecutive words of a row
    auto issue_scales = [&](int first, int n) {
        const int words = scale_words(n, GS);
        const int64_t pairs = p.N * steps;
        for (int i = threadIdx.x; i < kCtaRows * words; i += kThreads) {
            const int r_in = i / words, w = i - r_in * words;
            int64_t r = row0 + r_in;
            r = r < p.N ? r : p.N - 1;
            if (GS == 128) {
                const int64_t pair = r * steps + s_begin + first, word = (pair >> 1) + w;
                if (w < pair_words(pair, n) && pair_word_whole(word, pairs)) cp_async4(scale_s + r_in * pitch + w, p.w_scales + word * 4);
            } else {
                cp_async4(scale_s + r_in * pitch + w, p.w_scales + (r * (p.K / GS) + (s_begin + first) * (kStepK / GS)) * 2 + w * 4);
            }
        }
        if (GS == 128 && threadIdx.x == 0 && (pairs & 1) && row0 + kCtaRows >= p.N && s_begin + first + n == steps)
            load_last_pair(scale_s + (p.N - 1 - row0) * pitch, p.w_scales, pairs, n);
    };
    auto issue_frags = [&](int i) {            // the four warps of a step parity share the copies
        if (i < n_mine) {
            uint8_t* slot = frag_s + (wk * kDepth + i % kDepth) * kFragSlot;
            const int tiles_all = (int)gridDim.z * NT;
            const uint4* src = p.frag + ((s_begin + wk + i * kStepGroups) * tiles_all + (int)blockIdx.z * NT) * 128;
#pragma unroll
            for (int q = 0; q < NT; ++q) cp_async16(slot + (q * 128 + wr * 32 + lane) * 16, src + q * 128 + wr * 32 + lane);
        }
    };
    issue_scales(0, min(n_total, kScaleSteps));    // part of the first copy group
#pragma unroll
    for (int d = 0; d < kDepth - 1; ++d) {
        issue_codes(d);
        cp_async_commit();
    }
    grid_launch_dependents();                  // whatever follows waits for this grid's completion by itself
    grid_dependency_wait();                    // the rows (and the previous user of C) are complete from here on
#pragma unroll
    for (int d = 0; d < kDepth - 1; ++d) {
        issue_frags(d);
        cp_async_commit();
    }
    cp_async_wait<2 * kDepth - 3>();           // the first group: the scales
    __syncthreads();

    float acc[2][NT][4];
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[b][n][j] = 0.f;

    int scale_first = 0;                       // first step whose scales are held
    for (int i = 0; i < (n_total + 1) / kStepGroups; ++i) {
        const int ls = wk + i * kStepGroups;
        if (i * kStepGroups - scale_first == kScaleSteps) {      // a long range: the next steps' scales (all warps together)
            scale_first += kScaleSteps;
            __syncthreads();
            issue_scales(scale_first, min(n_total - scale_first, kScaleSteps));
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
        }
        if (i >= n_mine) break;                // an odd range: one step less for the second parity
        cp_async_wait<kDepth - 2>();           // this step's copies have landed
        // the fragments are visible to the parity's four warps, last step's slots free
        if (wk == 0) asm volatile("bar.sync 1, %0;" ::"n"(kRowGroups * 32) : "memory");
        else asm volatile("bar.sync 2, %0;" ::"n"(kRowGroups * 32) : "memory");
        issue_codes(i + kDepth - 1);
        issue_frags(i + kDepth - 1);
        cp_async_commit();
        const uint8_t* slot = ring + (i % kDepth) * kCodeBytes;
        const uint8_t* fs = frag_s + (wk * kDepth + i % kDepth) * kFragSlot;
        uint4 cw[4];
        uint32_t sc[4];                        // the scale bytes of the lane's group (groups of 16: of both)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            cw[q] = *reinterpret_cast<const uint4*>(slot + q * 512 + lane * 16);
            const uint32_t* w = scale_s + (wr * 32 + q * 8 + g) * pitch;
            const int s_in = ls - scale_first;
            if (GS == 16) sc[q] = w[s_in * 4 + t];
            else if (GS == 32) sc[q] = w[s_in * 2 + (t >> 1)] >> (16 * (t & 1));
            else if (GS == 64) sc[q] = w[s_in] >> (16 * (t >> 1));
            else {                             // the first held step may start in the upper half of its word
                const int h = odd[q] + s_in;
                sc[q] = w[h >> 1] >> (16 * (h & 1));
            }
        }
        Scales s[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {          // pieces of 8 elements of the lane's 32
            if (j == 0 || (GS == 16 && j == 2)) {
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = make_scales(j ? sc[q] >> 16 : sc[q]);
            }
            uint4 b[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) b[n] = *reinterpret_cast<const uint4*>(fs + n * kFragBytes + frag_pos(j, lane) * 16);
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
                const uint32_t w0 = j == 0 ? cw[2 * blk].x : j == 1 ? cw[2 * blk].y : j == 2 ? cw[2 * blk].z : cw[2 * blk].w;
                const uint32_t w1 = j == 0 ? cw[2 * blk + 1].x : j == 1 ? cw[2 * blk + 1].y : j == 2 ? cw[2 * blk + 1].z : cw[2 * blk + 1].w;
                const uint4 a0 = decode_word(w0, s[2 * blk]), a1 = decode_word(w1, s[2 * blk + 1]);
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    mma_f16(acc[blk][n], a0.x, a1.x, a0.y, a1.y, b[n].x, b[n].y);
                    mma_f16(acc[blk][n], a0.z, a1.z, a0.w, a1.w, b[n].z, b[n].w);
                }
            }
        }
    }
    cp_async_wait<0>();

    // Partial products [token][128 weight rows] in shared memory (over the rings, which are drained): odd steps first,
    // even steps added on top, then every CTA of the cluster adds its share of the outputs over all ranks, in rank order.
    __syncthreads();
    float* part = reinterpret_cast<float*>(smem);
    auto at = [&](int blk, int n, int j) -> float& {
        return part[(n * kTok + 2 * t + (j & 1)) * kPartPitch + wr * 32 + blk * 16 + (j >> 1) * 8 + g];
    };
    if (wk == 1)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) at(b, n, j) = acc[b][n][j];
    __syncthreads();
    if (wk == 0)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) at(b, n, j) += acc[b][n][j];
    if (slices > 1) cluster.sync();
    else __syncthreads();
    const int outputs = min(NT * kTok, p.M - m0) * kCtaRows;
    for (int o = slice * kThreads + threadIdx.x; o < outputs; o += slices * kThreads) {
        const int m = o / kCtaRows, col = o % kCtaRows;
        float sum = 0.f;
        if (slices > 1) {
            float v[kMaxSlices];
#pragma unroll
            for (int r = 0; r < kMaxSlices; ++r)                     // all remote reads in flight together
                v[r] = r < slices ? cluster.map_shared_rank(part, r)[m * kPartPitch + col] : 0.f;
#pragma unroll
            for (int r = 0; r < kMaxSlices; ++r) sum += v[r];
        } else sum = part[m * kPartPitch + col];
        const int64_t n = row0 + col;
        if (n < p.N) p.C[(int64_t)(m0 + m) * p.ld_c + n] = sum * 256.0f;
    }
    if (slices > 1) cluster.sync();                                  // no CTA leaves while its tile is still read
}

// ---- few rows (up to four token tiles): a CTA of eight warps covers p.rows weight rows (a multiple of 8, at most 16 x MB), its
// warps split the K range.  A warp's steps are consecutive, so its scales come along the rows, four steps (32 bytes per row
// with groups of 32) at a time.  Blocks of few rows share an SM (stream_ctas), so that a chain of calls keeps the weight stream going:
// the CTAs of the next call move in one by one as this call's leave.
constexpr int kScaleSlotSteps = 4;

template <int GS>
struct StreamRing {
    static constexpr int kDepth = 3;
    static constexpr int kWords = GS == 128 ? 3 : kScaleSlotSteps * 64 / GS;      // scale words per row and slot (128: aligned around)
    // Words of eight rows in different banks: an odd pitch (in units of the words a quad reads together), or rows of 8
    // words whose halves are exchanged on every other four rows.
    static constexpr int kPitch = GS == 16 ? 20 : GS == 32 ? 8 : GS == 64 ? 5 : 3;
    __host__ __device__ static constexpr int at(int r, int w) { return r * kPitch + (GS == 32 ? w ^ (r & 4) : w); }
    // of one warp: code slots, then two slots of scales
    __host__ __device__ static constexpr int warp_bytes(int rows) { return rows * (kDepth * 64 + 2 * kPitch * 4); }
};
__host__ __device__ constexpr int stream_part_bytes(int nt, int rows) { return kWarps * nt * kTok * (rows + 4) * 4; }
__host__ __device__ constexpr int stream_ctas(int nt, int mb) { return mb <= 2 ? (nt == 1 ? 3 : 2) : mb <= 4 && nt <= 2 ? 2 : 1; }

template <int NT, int MB, int GS>
__global__ void __launch_bounds__(kThreads, stream_ctas(NT, MB)) gemm_rows_stream_kernel(const RowsParams p) {
    using R = StreamRing<GS>;
    constexpr int kDepth = R::kDepth;
    extern __shared__ __align__(16) uint8_t smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int slices = (int)gridDim.y, slice = (int)blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int rows = p.rows, steps = (int)(p.K / kStepK);
    const int cta_begin = (int)((int64_t)steps * slice / slices), cta_steps = (int)((int64_t)steps * (slice + 1) / slices) - cta_begin;
    const int w_first = cta_steps * warp / kWarps;                   // this warp's steps inside the CTA's range
    const int n = cta_steps * (warp + 1) / kWarps - w_first;
    const int s_begin = cta_begin + w_first;
    const int64_t row0 = (int64_t)blockIdx.x * rows;
    const int rows_left = (int)min((int64_t)rows, p.N - row0);

    uint8_t* ring = smem + warp * R::warp_bytes(rows);
    const int slot_bytes = rows * 64;
    uint32_t* scale_ring = reinterpret_cast<uint32_t*>(ring + kDepth * slot_bytes);

    // piece t of rows g, g + 8, ...  Rows past the weight are not copied: what their slots hold only reaches sums that are not stored.
    const uint8_t* pc = p.w_codes + (row0 + g) * (p.K / 2) + (int64_t)s_begin * 64 + t * 16;
    const int64_t rows8 = p.K * 4;             // bytes between rows 8 apart
    auto issue = [&](int i) {
        if (i < n) {
            uint8_t* slot = ring + (i % kDepth) * slot_bytes + lane * 16;
            const uint8_t* src = pc + (int64_t)i * 64;
#pragma unroll
            for (int q = 0; q < 2 * MB; ++q, src += rows8)
                if (q * 8 + g < rows_left) cp_async16(slot + q * 512, src);
        }
    };
    const int64_t scale_pitch = p.K / GS * 2;
    auto issue_scales = [&](int slot) {
        const int first = slot * kScaleSlotSteps;
        if (first >= n) return;
        uint32_t* dst = scale_ring + (slot & 1) * rows * R::kPitch;
        const uint8_t* src0 = p.w_scales + row0 * scale_pitch + (int64_t)(s_begin + first) * (2 * kStepK / GS);
        if (GS == 32 && first + kScaleSlotSteps <= n && ((reinterpret_cast<uintptr_t>(src0) | scale_pitch) & 15) == 0) {
#pragma unroll
            for (int i = 0; i < MB; ++i) {     // two pieces of 16 bytes per row
                const int r = i * 16 + (lane >> 1), w = (lane & 1) * 4;
                if (r < rows_left) cp_async16(dst + R::at(r, w), src0 + r * scale_pitch + w * 4);
            }
            return;
        }
        // words past the warp's last step may lie past the end of the tensor
        if constexpr (GS == 128) {
            const int held = min(n - first, kScaleSlotSteps);
            const int64_t pairs = p.N * steps;
            for (int item = lane; item < rows_left * R::kWords; item += 32) {
                const int r = item / R::kWords, w = item - r * R::kWords;
                const int64_t pair = (row0 + r) * steps + s_begin + first, word = (pair >> 1) + w;
                if (w < pair_words(pair, held) && pair_word_whole(word, pairs)) cp_async4(dst + R::at(r, w), p.w_scales + word * 4);
            }
            if (lane == 0 && (pairs & 1) && row0 + rows_left == p.N && s_begin + first + held == steps)
                load_last_pair(dst + R::at(rows_left - 1, 0), p.w_scales, pairs, held);
        } else {
            const int words = min(R::kWords, (n - first) * (64 / GS));
            for (int item = lane; item < rows_left * R::kWords; item += 32) {
                const int r = item / R::kWords, w = item - r * R::kWords;
                const uint8_t* src = src0 + r * scale_pitch;
                if (w < words) cp_async4(dst + R::at(r, w), src + w * 4);
            }
        }
    };
    issue(0);
    issue_scales(0);
    cp_async_commit();
#pragma unroll
    for (int d = 1; d < kDepth - 1; ++d) {
        issue(d);
        cp_async_commit();
    }
    grid_launch_dependents();                  // whatever follows waits for this grid's completion by itself
    grid_dependency_wait();                    // the fragments (and the previous user of C) are complete from here on
    const int m0 = (int)blockIdx.z * (NT * kTok), live_tok = min(NT * kTok, p.M - m0);

    float acc[MB][NT][4];
#pragma unroll
    for (int b = 0; b < MB; ++b)
#pragma unroll
        for (int m = 0; m < NT; ++m)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[b][m][j] = 0.f;

    uint4 bf[4][NT];                           // the step's fragments
    const uint4* fg = p.frag + ((int64_t)s_begin * gridDim.z + blockIdx.z) * (NT * 128);
    const int64_t fg_step = (int64_t)gridDim.z * (NT * 128);
    for (int i = 0; i < n; ++i, fg += fg_step) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int m = 0; m < NT; ++m) bf[j][m] = __ldg(fg + m * 128 + frag_pos(j, lane));
        cp_async_wait<kDepth - 2>();           // this step's copies have landed
        __syncwarp();                          // the scales are read across lanes
        if ((i & (kScaleSlotSteps - 1)) == 0) issue_scales(i / kScaleSlotSteps + 1);
        issue(i + kDepth - 1);
        cp_async_commit();
        const uint8_t* slot = ring + (i % kDepth) * slot_bytes + lane * 16;
        const uint32_t* sw = scale_ring + ((i / kScaleSlotSteps) & 1) * rows * R::kPitch;
        const int s_in = i & (kScaleSlotSteps - 1);
#pragma unroll
        for (int blk = 0; blk < MB; ++blk) {
            if (blk * 16 >= rows) break;
            uint4 cw[2];
            uint32_t sc[2];                    // the scale bytes of the lane's group (groups of 16: of both)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int oct = min(blk * 2 + q, rows / 8 - 1);      // (an odd number of octets: the last one twice)
                cw[q] = *reinterpret_cast<const uint4*>(slot + oct * 512);
                const int r_in = oct * 8 + g;
                if (GS == 16) sc[q] = sw[R::at(r_in, s_in * 4 + t)];
                else if (GS == 32) sc[q] = sw[R::at(r_in, s_in * 2 + (t >> 1))] >> (16 * (t & 1));
                else if (GS == 64) sc[q] = sw[R::at(r_in, s_in)] >> (16 * (t >> 1));
                else {                         // the slot's first step may start in the upper half of its word
                    const int h = (int)(((row0 + r_in) * steps + s_begin + (i - s_in)) & 1) + s_in;
                    sc[q] = sw[R::at(r_in, h >> 1)] >> (16 * (h & 1));
                }
            }
            Scales s[2];
#pragma unroll
            for (int j = 0; j < 4; ++j) {      // pieces of 8 elements of the lane's 32
                if (j == 0 || (GS == 16 && j == 2)) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) s[q] = make_scales(j ? sc[q] >> 16 : sc[q]);
                }
                const uint32_t w0 = j == 0 ? cw[0].x : j == 1 ? cw[0].y : j == 2 ? cw[0].z : cw[0].w;
                const uint32_t w1 = j == 0 ? cw[1].x : j == 1 ? cw[1].y : j == 2 ? cw[1].z : cw[1].w;
                const uint4 a0 = decode_word(w0, s[0]), a1 = decode_word(w1, s[1]);
#pragma unroll
                for (int m = 0; m < NT; ++m) {
                    mma_f16(acc[blk][m], a0.x, a1.x, a0.y, a1.y, bf[j][m].x, bf[j][m].y);
                    mma_f16(acc[blk][m], a0.z, a1.z, a0.w, a1.w, bf[j][m].z, bf[j][m].w);
                }
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();                           // the rings become the partial products [warp][token][row]
    constexpr int kTokens = NT * kTok;
    const int pitch = rows + 4;
    float* part = reinterpret_cast<float*>(smem);
#pragma unroll
    for (int b = 0; b < MB; ++b)
#pragma unroll
        for (int m = 0; m < NT; ++m)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (b * 16 + (j >> 1) * 8 < rows)
                    part[(warp * kTokens + m * kTok + 2 * t + (j & 1)) * pitch + b * 16 + (j >> 1) * 8 + g] = acc[b][m][j];
    __syncthreads();
    // outputs: a warp takes tokens, its lanes rows
    const auto cta_sum = [&](int m, int col) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += part[(w * kTokens + m) * pitch + col];
        return sum;
    };
    if (slices == 1) {
        for (int m = warp; m < live_tok; m += kWarps)
            for (int col = lane; col < rows_left; col += 32) p.C[(int64_t)(m0 + m) * p.ld_c + row0 + col] = cta_sum(m, col) * 256.0f;
        return;
    }
    for (int m = warp; m < live_tok; m += kWarps)                    // the CTA's sum over its warps, on top of warp 0's part
        for (int col = lane; col < rows; col += 32) part[m * pitch + col] = cta_sum(m, col);
    cluster.sync();
    for (int m = slice * kWarps + warp; m < live_tok; m += slices * kWarps)
        for (int col = lane; col < rows_left; col += 32) {
            float sum = 0.f;
            for (int r = 0; r < slices; ++r) sum += cluster.map_shared_rank(part, r)[m * pitch + col];
            p.C[(int64_t)(m0 + m) * p.ld_c + row0 + col] = sum * 256.0f;
        }
    cluster.sync();                            // no CTA leaves while its sums are still read
}

// How a call is laid out: which kernel, token tiles per CTA, blocks of tokens, K ranges (= cluster size).
struct RowsPlan {
    bool stream;
    int nt, m_blocks, slices, steps_max;
    int mb, rows;                    // streaming kernel: 16-row blocks a CTA has accumulators for, weight rows it covers
    double us;                       // estimated time of both launches
    int tiles() const { return nt * m_blocks; }
};

constexpr int kSmCount = 148;

int stream_warp_bytes(int gs, int rows) {
    return gs == 16 ? StreamRing<16>::warp_bytes(rows) : gs == 32 ? StreamRing<32>::warp_bytes(rows)
         : gs == 64 ? StreamRing<64>::warp_bytes(rows) : StreamRing<128>::warp_bytes(rows);
}

// The streaming kernel's layout: weight rows per CTA and K ranges, by a time model fitted to 2700 calls with given layouts (22
// weights of N 512 to 14336, K 512 to 14336, from HBM; 1, 16, 24 and 32 rows).  Per wave of CTAs: the start, per step of a warp
// either the latency of its own 16-row blocks or the throughput of all blocks on the SM, the sums over the warps, and the meeting of a
// cluster.  The layout it picks is within 1.1, 1.2, 2.4 and 4.3 % of the best on average for one to four token tiles.  (CTAs
// of 32 rows with one and a half of them per SM by K ranges, as before: 24 rows of 6144 x 4096 18.3 us against 11.6, 16 rows of
// 5120 x 2560 13.1 / 8.0, one row of 4096 x 4096 8.9 / 7.2.)
RowsPlan plan_stream_uncached(int nt, int64_t N, int64_t K, int gs) {
    struct Fit { double call, start, latency, block, rate, row, meeting, full; };
    static constexpr Fit kFit[4] = {{0.92, 1.73, 0.36, 0.28, 0.38, 0.019, 1.63, 0.84}, {0.89, 2.26, 0.44, 0.25, 0.46, 0.019, 1.89, 0.86},
                                    {1.48, 2.00, 0.39, 0.40, 0.50, 0.021, 2.25, 0.92}, {1.36, 2.49, 0.33, 0.50, 0.50, 0.023, 2.29, 0.93}};
    const Fit& f = kFit[nt - 1];
    const int steps = (int)(K / kStepK);
    RowsPlan best{};
    for (int s = 1; s <= kMaxSlices && (s == 1 || steps >= 8 * s); s *= 2)
        for (int rows = 8; rows <= 112; rows += 8) {
            const int mb = rows <= 32 ? 2 : rows <= 64 ? 4 : 7;
            const size_t smem = (size_t)kWarps * stream_warp_bytes(gs, rows);
            if (smem > kMaxSmem) break;
            const int64_t sms = s <= 2 ? kSmCount : s == 4 ? 132 : 120, fit = (int64_t)(kSmSmem / (smem + kCtaSmem));
            const int64_t per_sm = fit < stream_ctas(nt, mb) ? fit : stream_ctas(nt, mb);
            const int64_t ctas = (N + rows - 1) / rows * s, waves = (ctas + per_sm * sms - 1) / (per_sm * sms);
            const int64_t last = (ctas - (waves - 1) * per_sm * sms + sms - 1) / sms;
            const int blocks = (rows + 15) / 16, n = ((steps + s - 1) / s + kWarps - 1) / kWarps;
            auto wave = [&](double resident) {
                const double alone = f.latency + blocks * f.block, shared = resident * blocks * f.rate;
                return f.start + n * (alone > shared ? alone : shared) + f.row * rows + (s > 1 ? f.meeting : 0.0);
            };
            const double us = f.call + (double)(waves - 1) * f.full * wave((double)per_sm) + wave((double)(last < per_sm ? last : per_sm));
            if (!best.nt || us < best.us) best = {true, nt, 1, s, (steps + s - 1) / s, mb, rows, us};
        }
    return best;
}

// A program decodes with the same few layers over and over: a thread keeps the layouts of the last ones, by their sizes.  (14
// to 56 estimates take 0.4 to 1.5 us, a call of a small layer 6.5.)
RowsPlan plan_stream(int nt, int64_t N, int64_t K, int gs) {
    struct Kept {
        int64_t N, K;
        int nt, gs;
        RowsPlan plan;
    };
    static thread_local Kept kept[32] = {};
    Kept& k = kept[((uint64_t)N * 31 + (uint64_t)K / kStepK * 7 + (uint64_t)nt * 5 + (uint64_t)gs / 16) & 31];
    if (k.N != N || k.K != K || k.nt != nt || k.gs != gs) k = {N, K, nt, gs, plan_stream_uncached(nt, N, K, gs)};
    return k.plan;
}

RowsPlan plan_rows(int64_t M, int64_t N, int64_t K, int gs) {
    const int64_t steps = K / kStepK;
    const int tiles = (int)((M + kTok - 1) / kTok);
    // Up to 32 tokens, or blocks of 32 tokens while all of them together are resident at once (a small layer: 6-9 us).
    const int64_t stream_blocks = (N + 31) / 32;
    const int m_blocks32 = (tiles + 3) / 4;
    if (tiles > 4 && stream_blocks * m_blocks32 <= 2 * kSmCount && N * K <= (1ll << 21)) {
        const int rows = (N + 15) / 16 * m_blocks32 <= 2 * kSmCount ? 16 : 32;
        return {true, 4, m_blocks32, 1, (int)steps, 2, rows, 9.0};
    }
    if (tiles <= 4) return plan_stream(tiles, N, K, gs);
    // Time in us, fitted to 2100 calls with given layouts (39 weights of N 256 to 28672, K 512 to 16384, from HBM; 33 to 256
    // rows): 3 for the fragments and the start, then per wave of CTAs its steps' decode and MMAs, its own start and, with a
    // cluster, the meeting at the end.  Within 4 % on average for blocks of 48 and 64 rows, 9 % for 32; the layout it picks
    // is within 1.2 % of the best on average.  (At most 64 rows: one block, the weight is read and decoded once.)  How many
    // SMs a wave fills is what cudaOccupancyMaxActiveClusters answers for the cluster sizes: clusters of three and more leave
    // SMs of a GPC empty.  64 rows of 5120 x 2560: three ranges 14.5 us, two 17.9, four (two waves) 21.6.  Blocks of 32 rows:
    // two CTAs share an SM and take turns.
    static constexpr int kSms[kMaxSlices] = {148, 148, 135, 132, 130, 132, 105, 120}, kSms32[kMaxSlices] = {148, 148, 139, 142, 140, 135, 129, 132};
    const int64_t row_blocks = (N + kCtaRows - 1) / kCtaRows;
    RowsPlan best{};
    for (int nt = 8; nt >= 4; nt -= 2) {
        if (tiles <= kMaxTiles && nt != (tiles <= 6 ? 6 : 8)) continue;
        const int m_blocks = (tiles + nt - 1) / nt;
        const double step = nt == 8 ? 0.93 : nt == 6 ? 0.78 : 0.72, start = nt == 4 ? 0.5 : 2.6, meeting = nt == 4 ? 3.5 : 4.3;
        for (int s = 1; s <= kMaxSlices && s <= steps; ++s) {
            const int64_t ctas = row_blocks * s * m_blocks, n = (steps + s - 1) / s, sms = (nt == 4 ? kSms32 : kSms)[s - 1];
            const double us = 3.0 + (double)((ctas + sms - 1) / sms) * ((double)n * step + (s > 1 ? meeting : start));
            if (!best.nt || us < best.us) best = {false, nt, m_blocks, s, (int)n, 0, 0, us};
        }
    }
    return best;
}

struct RowsKernel {
    void (*fn)(const RowsParams);
    size_t ring_bytes, frag_ring_bytes;
};

template <int GS>
RowsKernel kernel_for(const RowsPlan& pl) {
    if (pl.stream) {
        const size_t ring = (size_t)kWarps * StreamRing<GS>::warp_bytes(pl.rows), part = (size_t)stream_part_bytes(pl.nt, pl.rows);
        const size_t bytes = ring > part ? ring : part;
        auto pick = [&](auto two, auto four, auto seven) { return pl.mb <= 2 ? two : pl.mb <= 4 ? four : seven; };
        switch (pl.nt) {
            case 1: return {pick(gemm_rows_stream_kernel<1, 2, GS>, gemm_rows_stream_kernel<1, 4, GS>, gemm_rows_stream_kernel<1, 7, GS>), bytes, 0};
            case 2: return {pick(gemm_rows_stream_kernel<2, 2, GS>, gemm_rows_stream_kernel<2, 4, GS>, gemm_rows_stream_kernel<2, 7, GS>), bytes, 0};
            case 3: return {pick(gemm_rows_stream_kernel<3, 2, GS>, gemm_rows_stream_kernel<3, 4, GS>, gemm_rows_stream_kernel<3, 7, GS>), bytes, 0};
            default: return {pick(gemm_rows_stream_kernel<4, 2, GS>, gemm_rows_stream_kernel<4, 4, GS>, gemm_rows_stream_kernel<4, 7, GS>), bytes, 0};
        }
    }
    switch (pl.nt) {
        case 4: return {gemm_rows_kernel<4, GS>, Ring<4, GS>::kBytes, Ring<4, GS>::kFragRing};
        case 6: return {gemm_rows_kernel<6, GS>, Ring<6, GS>::kBytes, Ring<6, GS>::kFragRing};
        default: return {gemm_rows_kernel<8, GS>, Ring<8, GS>::kBytes, Ring<8, GS>::kFragRing};
    }
}

int launch_rows(RowsParams p, const RowsPlan& pl, int gs, bool programmatic, cudaStream_t st) {
    const RowsKernel kernel = gs == 16 ? kernel_for<16>(pl) : gs == 32 ? kernel_for<32>(pl) : gs == 64 ? kernel_for<64>(pl) : kernel_for<128>(pl);
    static bool configured[64][4][4][kMaxTiles + 1] = {};   // the opt-in to > 48 KB of shared memory: per device and kernel
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return AMX_ERR_CUDA;
    bool& done = configured[dev][pl.stream ? (pl.mb <= 2 ? 1 : pl.mb <= 4 ? 2 : 3) : 0][gs == 16 ? 0 : gs == 32 ? 1 : gs == 64 ? 2 : 3][pl.nt];
    if (!done) {
        if (cudaFuncSetAttribute(kernel.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess) {
            cudaGetLastError();
            return AMX_ERR_CUDA;
        }
        done = true;
    }
    const int held = pl.steps_max < scale_steps(gs) ? pl.steps_max : scale_steps(gs);
    p.steps_max = pl.steps_max;
    p.rows = pl.rows;
    const int cta_rows = pl.stream ? pl.rows : kCtaRows;
    const dim3 grid((unsigned)((p.N + cta_rows - 1) / cta_rows), (unsigned)pl.slices, (unsigned)pl.m_blocks);
    size_t smem = kernel.ring_bytes + (pl.stream ? 0 : (size_t)scale_bytes(held, gs) + kernel.frag_ring_bytes);
    if (pl.stream) {
        // Blocks crowd on the SMs that the launch before leaves first: shared memory is asked for such that an SM takes no more of
        // them than its share.
        const size_t share = (grid.x * grid.y * grid.z + kSmCount - 1) / kSmCount, crowded = kSmSmem / (share + 1) - kCtaSmem + 128;
        if (share < 4 && smem < crowded) smem = crowded;
    }
    return launch_with(dim3(1, (unsigned)pl.slices), programmatic, kernel.fn, grid, kThreads, smem, st, p);
}

// Workspace: 256 bytes whose first word is the status word amx_gemm_status reads, then the fragments of the rows.
constexpr size_t kHeaderBytes = 256;

template <bool CAST, int GS>
int launch_fragments_gs(const uint8_t* codes, const uint8_t* scales, const uint16_t* x, int64_t ld_x, int64_t M, int64_t K, int tiles,
                        void* workspace, bool programmatic, cudaStream_t st) {
    return launch_with(1, programmatic, rows_fragments_kernel<CAST, GS>, dim3((unsigned)((K / 8 + 127) / 128), (unsigned)(tiles * kTok)), 128, 0,
                       st, codes, scales, x, ld_x, (int)M, tiles, K, reinterpret_cast<uint4*>(static_cast<uint8_t*>(workspace) + kHeaderBytes),
                       static_cast<int*>(workspace));
}
template <bool CAST>
int launch_fragments(const uint8_t* codes, const uint8_t* scales, const uint16_t* x, int64_t ld_x, int64_t M, int64_t K, int gs,
                     int tiles, void* workspace, bool programmatic, cudaStream_t st) {
    auto* fn = gs == 16 ? launch_fragments_gs<CAST, 16> : gs == 32 ? launch_fragments_gs<CAST, 32>
             : gs == 64 ? launch_fragments_gs<CAST, 64> : launch_fragments_gs<CAST, 128>;
    return fn(codes, scales, x, ld_x, M, K, tiles, workspace, programmatic, st);
}

// x != nullptr: bf16 rows, cast here; otherwise quantized rows.
int run_rows(const uint8_t* a_codes, const uint8_t* a_scales, const void* x, int64_t ld_x, const uint8_t* w_codes,
             const uint8_t* w_scales, int64_t M, int64_t N, int64_t K, int gs, float* C, int64_t ld_c, void* workspace,
             cudaStream_t st) {
    const RowsPlan pl = plan_rows(M, N, K, gs);
    const bool programmatic = programmatic_launch_ok(st);      // asked once for both launches
    RowsParams p{};
    p.frag = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(workspace) + kHeaderBytes);
    p.w_codes = w_codes; p.w_scales = w_scales;
    p.M = (int)M; p.N = N; p.K = K; p.C = C; p.ld_c = ld_c;
    const int rc = x ? launch_fragments<true>(nullptr, nullptr, static_cast<const uint16_t*>(x), ld_x, M, K, gs, pl.tiles(), workspace,
                                              programmatic, st)
                     : launch_fragments<false>(a_codes, a_scales, nullptr, 0, M, K, gs, pl.tiles(), workspace, programmatic, st);
    if (rc != AMX_OK) return rc;
    return launch_rows(p, pl, gs, programmatic, st);
}

}  // namespace

bool gemm_rows_supported(int64_t M, int64_t N, int64_t K, int gs) {
    return fixed_group_size(gs) && M >= 1 && M <= kRowsMaxM && N >= 1 && K >= kStepK && K % kStepK == 0 &&
           N <= 0x7FFFFFFFll * 8;
}

size_t gemm_rows_workspace_bytes(int64_t M, int64_t N, int64_t K) {
    constexpr int gs = 32;                     // (the tokens' tiles do not depend on it)
    // (blocks of 32, 48 or 64 rows round M up differently: what suffices for M rows on this kernel also suffices for fewer)
    const int64_t tiles = (M + kTok - 1) / kTok;
    const int64_t rows = (tiles <= 4 ? tiles : (int64_t)plan_rows(M, N, K, gs).tiles()) * kTok, whole = M > 64 ? (M + 63) / 64 * 64 : 0;
    return kHeaderBytes + (size_t)(rows > whole ? rows : whole) * (size_t)K * 2;
}

double gemm_rows_estimated_us(int64_t M, int64_t N, int64_t K) { return plan_rows(M, N, K, 32).us; }

int gemm_rows(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes, const uint8_t* w_scales,
              int64_t M, int64_t N, int64_t K, int gs, float* C, int64_t ld_c, void* workspace, cudaStream_t st) {
    return run_rows(a_codes, a_scales, nullptr, 0, w_codes, w_scales, M, N, K, gs, C, ld_c, workspace, st);
}

int gemm_rows_cast(const void* x, int64_t ld_x, const uint8_t* w_codes, const uint8_t* w_scales, int64_t M, int64_t N,
                   int64_t K, int gs, float* C, int64_t ld_c, void* workspace, cudaStream_t st) {
    return run_rows(nullptr, nullptr, x, ld_x, w_codes, w_scales, M, N, K, gs, C, ld_c, workspace, st);
}

}  // namespace amx

// For tests: the layout a call on these kernels takes - {streaming kernel, token tiles of a block, blocks of tokens, weight rows of a
// CTA, K ranges} -, so that they can say which they cover.
extern "C" int amx_diag_rows_layout(int64_t M, int64_t N, int64_t K, int gs, int* layout) {
    if (!amx::gemm_rows_supported(M, N, K, gs) || !layout) return AMX_ERR_SHAPE;
    const amx::RowsPlan pl = amx::plan_rows(M, N, K, gs);
    layout[0] = pl.stream;
    layout[1] = pl.nt;
    layout[2] = pl.m_blocks;
    layout[3] = pl.stream ? pl.rows : amx::kCtaRows;
    layout[4] = pl.slices;
    return AMX_OK;
}
