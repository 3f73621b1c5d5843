// AMXFP4 x AMXFP4 -> fp32 on the FP4 tensor-core pipe (tcgen05 block-scaled MMA, sm_100a).
//
// The format picks one of two group scales per ELEMENT (by the element's sign; arXiv 2411.09909,
// Section 4.3), while a block-scaled MMA operand has one scale per (row, K block).  So each decoded
// operand is written as the sum of two single-scale operands,
//     Ahat = S_p o A+  +  S_n o A-      (A+ / A- = the codes with the other sign's nibbles zeroed),
// and the product becomes four block-scaled FP4 MMAs accumulating into one TMEM tile:
//     Ahat What^T = A+ W+^T + A+ W-^T + A- W+^T + A- W-^T.
//
// Scales: the MMA takes UE4M3 scales, one per 16 elements.  An E5M2 scale has the same four
// significands but a wider exponent range, so every operand row gets a power-of-two offset that
// maps its largest scale to the top UE4M3 binade; scale * 2^-offset is written as UE4M3 (each
// 32-group's scale twice) and the fp32 accumulator is multiplied by 2^(offset_A[m] + offset_W[n])
// in the epilogue (exact).  Scales more than 14 binades below their row's largest scale do not fit
// and are flushed to zero: their groups contribute less than 2^-14 of the row's largest group.
//
// Persistent CTAs (one per SM) walk over 128 x 256 tiles of C - pairs of CTAs over 256 x 256 tiles (PAIR below) -; the tiles
// that would leave most of a last wave idle are cut into halves or quarters of their columns.  K blocks cycle through four
// shared-memory stages (five in a pair):
//   warp 0   TMA producer: per stage one 3-D tile {A+, A-} and one {W+, W-} (swizzled rows) and the scale factors of either,
//            completion on the stage's `full` mbarrier
//   warp 1   allocates TMEM; one lane issues, per stage, the copies of the scale factors from shared to tensor memory
//            (tcgen05.cp, in order with the MMAs, either right before the first MMA that reads it) and the MMAs (4 sign
//            pairs x K steps of 64), then commits to the stage's `empty` mbarrier
//   warps 2-9 epilogue: TMEM -> registers (double-buffered loads), power-of-two rescale, 32-byte fp32
//            stores.  While a tile's accumulator is read out the producer already prefetches the next
//            tile's stages, and the MMA issuer starts the next tile as soon as the columns the two tiles
//            share have been read (see "Tensor memory" below).
// What bounds the K loop is shared memory: per K block of a pair's CTA the copies write 38 KB and the MMAs read 32 (one plane) or 64
// (two).  Eight more warps that carried the scale factors through registers read another 24 KB (each quarter of tensor
// memory wants a copy): MXFP4 8192 x 14336 x 4096 249 us against 233, 1000 x 11008 x 4096 93.5 against 89.2, 16384 x 10240 x 8192
// 1897 against 1871.  (All copies of a stage ahead of its MMAs: 90.0 for the second.)
// A preparation kernel per operand derives the planes, the UE4M3 scale-factor
// blocks in the 128 x 4 interleaved layout the MMA reads, and the row offsets from the canonical
// codes and scales.  Every device-side wait is bounded.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "cast_math.cuh"
#include "fp4_operand.cuh"
#include "gemm.cuh"
#include "tcgen05.cuh"

namespace amx {
namespace {

using namespace tc;
using namespace fp4;

constexpr int BM = 128, BN = 256;
constexpr int kEpilogueWarps = 8;
constexpr int kThreads = (2 + kEpilogueWarps) * 32;
constexpr int kTmemCols = 512;
// Tensor memory.  Two fp32 accumulators of 256 columns are all 512 columns, and the block-scaled MMA reads its
// scale factors from tensor memory too.  So consecutive tiles of a CTA alternate between two accumulator windows
// that overlap: columns [0, 256) for its even tiles, [160, 416) for the odd ones; the scale factors of the K blocks
// in flight take the 96 columns from 416.  The epilogue reads the 96 shared columns of a finished tile first and
// releases them (`ovl_free`); the next tile's MMAs start then, while the other 160 columns are still being read
// and stored (`rest_free` guards their reuse by the tile after next).  Only the read of 96 of 256 columns stays
// between two tiles, instead of the whole drain.  (Tiles of 128 columns use [0, 128) and [160, 288): no overlap.)
constexpr int kAccWindow = 160;        // first column of the odd tiles' accumulator
constexpr uint32_t kTmemSf = 416;      // scale-factor columns
constexpr int kTmemSfCols = 96;

// Shared-memory stage geometry: four stages of a K block each, five in a pair (four there: MXFP4 8192 x 14336 x 4096 240 us for
// the call, five 223).  Two planes per operand: BK = 128 elements (64-byte rows), 48 KB
// (K blocks of 256 elements in two stages measured slower).  ONE_PLANE (both operands in a symmetric format, one product per K
// step): BK = 256 (128-byte rows); with 128 the tensor cores waited on copies of 1 KB and on a barrier round per two MMAs
// (MXFP4 8192 x 14336 x 4096: 347 us against 219).  PAIR: the stage of one CTA of the pair, half of the W rows.
template <int BK_, bool ONE_PLANE = false, bool PAIR = false>
struct Cfg {
    static constexpr int BK = BK_;
    static constexpr int kPlanes = ONE_PLANE ? 1 : 2;
    static constexpr int kRowBytes = BK / 2;
    static constexpr int kSteps = BK / 64;                            // MMAs (K = 64) per K block and sign pair
    static constexpr int kStages = PAIR ? 5 : 4;
    static constexpr int kTileA = BM * kRowBytes, kTileB = BN / (PAIR ? 2 : 1) * kRowBytes;   // one plane
    static constexpr int kOffAp = 0, kOffAn = ONE_PLANE ? 0 : kTileA, kOffWp = kPlanes * kTileA,
                         kOffWn = kOffWp + (ONE_PLANE ? 0 : kTileB);
    static constexpr int kStageBytes = kPlanes * (kTileA + kTileB);   // {A+, A-} and {W+, W-}: one TMA each
    // scale factors of a stage: per plane one run of kSteps chunks for the A rows and for either half of the W rows
    static constexpr int kSfRun = kSteps * kSfChunk, kSfStage = kPlanes * 3 * kSfRun;
    static constexpr int kSmemBytes = kStages * (kStageBytes + kSfStage) + 1024 + 2048 + 512;   // + alignment slack + Control
    // TMEM columns of one stage's scale factors: A planes (4 columns per K step), then W planes (8)
    static constexpr int kSfColsA = kPlanes * kSteps * 4, kSfCols = kSfColsA + kPlanes * kSteps * 8;
    // The scale factors of kSfSlots K blocks are in tensor memory at a time, so that a block's copies do not touch what the MMAs
    // just ahead of them read.  They do overwrite what the MMAs of block b - kSfSlots read, with no barrier between: that a
    // tcgen05.cp does not overtake the tcgen05.mma issued before it by the same thread is an ASSUMPTION.  PTX names the order of
    // a copy and a later MMA only; the other one is taken from the hardware, which works both off in the order of issue (CUTLASS's
    // block-scaled main loop relies on it as well: one place for the factors of all K blocks).  A wait for those MMAs costs products
    // of one plane 2 to 8 % (1000 x 11008 x 4096 26.0 -> 26.6 us, 500 x 4096 x 4096 12.7 -> 13.6), with three slots and the poll
    // moved between the MMAs still 3 % (8192 x 14336 x 4096 209 -> 215).
    static constexpr int kSfSlots = kTmemSfCols / kSfCols;
    static_assert(kSfSlots >= 2 && kSfSlots <= kStages, "scale-factor ring");
    static_assert(kAccWindow + BN <= (int)kTmemSf && kTmemSf + kSfSlots * kSfCols <= kTmemCols, "tensor memory map");
    static_assert(BK == 128 || BK == 256, "rows of 64 or 128 bytes, swizzled over their length");
};
constexpr int kMaxStages = 5;

struct __align__(16) Control {
    uint64_t full[kMaxStages], empty[kMaxStages], accum_full;
    uint64_t ovl_free;              // the columns a finished tile shares with the next tile's accumulator have been read
    uint64_t rest_free[2];          // its other columns have been read ([i]: tiles with number % 2 == i)
    uint64_t sides_ready[2];        // the epilogue warps have written sides[i] for the CTA's tile number 2 k + i
    uint32_t tmem_base;
    volatile int abort;
    volatile int sides[2][8];       // per epilogue warp: which sign planes its share of the tile's rows uses
    alignas(16) float w_fac[2][BN];   // 2^(row offset of W): read four at a time in the epilogue
};
static_assert(sizeof(Control) <= 2048 + 512, "Control must fit its reserved space");

// K-major operand rows of 64 bytes with the 64-byte swizzle: groups of 8 rows are 512 B apart.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Instruction descriptor, kind::mxf4nvf4 block-scaled: A and B E2M1 (format code 1), K-major,
// UE4M3 scale factors (bit 23 = 0), N >> 3 at bit 17, M >> 4 at bit 24, K = 64 (bit 31 = 0).
__host__ __device__ constexpr uint32_t instr_desc(int n) { return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24); }

// -------------------------------------------------------------------------------- GEMM --
struct Params {
    const int *a_exp, *w_exp;
    int64_t M, N, K, ld_c;
    int64_t a_row0, w_row0;      // first rows of this product's operands inside the (stacked) prepared operands

    float* C;
    int vec_store;
    int out_bf16;                // C holds bf16 (each fp32 result rounded to nearest even) instead of fp32
    int band;                    // tile order: row blocks of A per band, see blk_m / blk_n
    int whole, split_log2;       // tail: work items below `whole` are tiles, the others 1 / 2^split_log2 of a tile's columns
    int slices;                  // SLICED instantiation: K is cut into this many ranges, each (tile, range) a work item
    int64_t slice_stride;        //   whose partial product goes to C + range * slice_stride
    int* status;
    const float *scale_a, *scale_w;   // not NULL: one fp32 factor per operand (the tensor scales of NVFP4 operands);
                                 // the store epilogue multiplies every result by their product
    const int* gate;             // not NULL: the kernel returns at once when this word is nonzero (the caller then
                                 // runs the exact bf16-decode kernel on the same operands, gated the other way)
};
// 16 consecutive fp32 results of one row -> global memory, as two 32-byte stores when allowed.
__device__ __forceinline__ void store_row16(float* out, const float (&f)[16], bool vec, int64_t n_left) {
    if (vec && n_left >= 16) {
#pragma unroll
        for (int j = 0; j < 16; j += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + j), "f"(f[j]), "f"(f[j + 1]),
                         "f"(f[j + 2]), "f"(f[j + 3]), "f"(f[j + 4]), "f"(f[j + 5]), "f"(f[j + 6]), "f"(f[j + 7]) : "memory");
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < n_left) out[j] = f[j];
    }
}

// The same 16 results rounded to bf16 (nearest even): one 32-byte store.
__device__ __forceinline__ void store_row16_bf16(__nv_bfloat16* out, const float (&f)[16], bool vec, int64_t n_left) {
    if (vec && n_left >= 16) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
            w[j] = *reinterpret_cast<const uint32_t*>(&h);
        }
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                     "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < n_left) out[j] = __float2bfloat16_rn(f[j]);
    }
}

// NHALF: tiles of 128 x 128 for products with at most 128 columns: the W box, the MMA and the epilogue are half as
// wide, the stage layout keeps its size.
// PAIR: two CTAs (a cluster) compute a tile of 256 x 256, each the accumulator of 128 of its rows and the load of its A rows and
// of half of the W rows; their tensor cores read both halves.  The first CTA's warp 1 issues for both: all copies of a stage are
// counted on its `full` barrier, the other CTA's epilogue warps arrive on its barriers too, and its commits
// arrive on the barriers of both.
// ONE_PLANE: the caller states that neither operand has a second sign plane (Cfg above): only the first planes and
// their scale factors are read, one product per K step.  A tile whose row words show a second plane after all puts
// AMX_ERR_FLAGS into the status word (the kernel runs to its end; C is then not the product).
template <int BK_, bool SLICED = false, bool NHALF = false, bool ONE_PLANE = false, bool PAIR = false>
__global__ void __launch_bounds__(kThreads, 1)
gemm_fp4_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w,
                const __grid_constant__ CUtensorMap tm_a1, const __grid_constant__ CUtensorMap tm_w1,
                const __grid_constant__ CUtensorMap tm_wt, const __grid_constant__ CUtensorMap tm_wt1,
                const __grid_constant__ CUtensorMap tm_sfa, const __grid_constant__ CUtensorMap tm_sfw, const Params p) {
    using C_ = Cfg<BK_, ONE_PLANE, PAIR>;
    constexpr int kPlanes = C_::kPlanes;
    constexpr int BNT = NHALF ? BN / 2 : BN;                     // tile width
    constexpr uint32_t kOffWnT = NHALF ? C_::kOffWp + C_::kTileB / 2 : C_::kOffWn;   // the box packs its two planes
    constexpr int kTileWT = NHALF ? C_::kTileB / 2 : C_::kTileB;   // one plane of the W tile as loaded (PAIR: of this CTA's half)
    constexpr uint32_t kIdescT = PAIR ? instr_desc(BNT) + ((uint32_t)(BM >> 4) << 24) : instr_desc(BNT);   // PAIR: M = 256
    constexpr int BMT = PAIR ? 2 * BM : BM;                      // tile height: of the pair
    const int rank = PAIR ? (int)(blockIdx.x & 1) : 0, worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x,
              workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    constexpr int BK = C_::BK, kRowBytes = C_::kRowBytes, kSteps = C_::kSteps, kStages = C_::kStages;
    constexpr int kStageBytes = C_::kStageBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sf_stages = tiles + kStages * kStageBytes;
    Control* ctl = reinterpret_cast<Control*>(sf_stages + kStages * C_::kSfStage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Work items: tile x K range (one range unless SLICED); an item index is tile * S + range, num_kb the K blocks
    // of one item when there is one range.
    const int S = SLICED ? p.slices : 1;
    const int kb_total = (int)((p.K + BK - 1) / BK);
    const int num_kb = kb_total / S;                             // per item; SLICED: ranges differ by at most one block
    auto kb_begin = [&](int64_t tile) -> int { return SLICED ? (int)((int)(tile % S) * kb_total / S) : 0; };
    // Persistent CTA: tiles blockIdx.x, blockIdx.x + gridDim.x, ...; neighbouring tiles share their A rows.
    const int64_t n_tiles = (p.N + BNT - 1) / BNT, m_tiles = (p.M + BMT - 1) / BMT;
    const int64_t total_tiles = m_tiles * n_tiles * S;
    // Work items: the first `whole` tiles, then the parts of the tiles that are left after the last whole wave (each
    // 1 / 2^split_log2 of a tile's columns, at most one for a CTA: its last item).
    constexpr bool kSplits = !SLICED && !NHALF;
    const int64_t whole = kSplits ? p.whole : total_tiles;
    auto part_log2 = [&](int64_t item) -> int { return kSplits && item >= whole ? p.split_log2 : 0; };
    auto tile_of = [&](int64_t item) { return kSplits && item >= whole ? whole + ((item - whole) >> p.split_log2) : item; };
    auto part_col = [&](int64_t item) -> int {                   // first column of an item inside its tile
        return kSplits && item >= whole ? (int)((item - whole) & ((1 << p.split_log2) - 1)) * (BNT >> p.split_log2) : 0;
    };
    // Tile order.  The CTAs work on ~148 consecutive tiles at a time and advance through K roughly together, so what
    // they read from DRAM per wave is the operand rows the wave touches, once.  Tiles are ordered in bands of
    // p.band row blocks of A: inside a band the tile index walks down the band's row blocks first, then along N.
    // A wave then touches band x 128 rows of A and (148 / band) x 256 rows of W (with 16: 2048 + 2368 rows, near
    // the minimum), and consecutive waves of a band share its rows of A in L2.  Walking along N first, a wave of a
    // tall product touched a few row blocks of A and ALL of W: 3.6 GB of DRAM reads for 0.23 GB of operands at
    // 16384 x 10240 x 8192.  A band as tall as the matrix is the plain "down M first" order (small M).
    // (two 32-bit divisions per call: the host rejects products with 2^31 tiles or more)
    const uint32_t band = (uint32_t)p.band, per_band = band * (uint32_t)n_tiles;
    auto banded = [&](int64_t item, uint32_t& m, uint32_t& n) {
        const uint32_t t = (uint32_t)tile_of(item) / (uint32_t)S, b = t / per_band, r = t - b * per_band;
        const uint32_t rows_here = min(band, (uint32_t)m_tiles - b * band);      // the last band may be shorter
        n = r / rows_here;
        m = b * band + (r - n * rows_here);
    };
    auto blk_m = [&](int64_t tile) -> int64_t {                  // this CTA's block of 128 rows
        uint32_t m, n;
        banded(tile, m, n);
        return PAIR ? 2 * (int64_t)m + rank : (int64_t)m;
    };
    auto blk_n = [&](int64_t tile) -> int64_t {
        uint32_t m, n;
        banded(tile, m, n);
        return n;
    };
    // K blocks of a tile (of an item)
    auto nkb_of = [&](int64_t tile) -> int {
        if (SLICED) return (int)(((int)(tile % S) + 1) * kb_total / S) - kb_begin(tile);
        return num_kb;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ctl->full[s], 1);                         // the byte count; a pair's stages are all reported to its first CTA
            mbar_init(&ctl->empty[s], 1);
        }
        mbar_init(&ctl->accum_full, 1);
        constexpr int kReaders = kEpilogueWarps * (PAIR ? 2 : 1);      // of an accumulator (PAIR: both CTAs' halves)
        mbar_init(&ctl->ovl_free, kReaders);
        mbar_init(&ctl->rest_free[0], kReaders);
        mbar_init(&ctl->rest_free[1], kReaders);
        mbar_init(&ctl->sides_ready[0], kEpilogueWarps);
        mbar_init(&ctl->sides_ready[1], kEpilogueWarps);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if (PAIR) tmem_alloc_pair(&ctl->tmem_base, kTmemCols);
        else tmem_alloc(&ctl->tmem_base, kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();                                    // the other CTA's barriers are there before they are used
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    // Everything above overlaps the end of the launches before (1024 x 4096 x 4096: 0.8 us from the wait to here).
    grid_dependency_wait();
    // a gated launch that has nothing to do has no items (uniform over the grid)
    const int64_t total_items = p.gate && *p.gate != 0 ? 0 : whole < total_tiles ? whole + ((total_tiles - whole) << p.split_log2) : total_tiles;

    // Which sign planes a tile's rows use at all (bits of the row words, OR-ed over the tile's 128 + 256 rows; each
    // lane its share, to be OR-ed over the warp): bit 0/1: A has +/-, bit 2/3: W has +/-.  The products with a plane
    // that is zero for the whole tile are not issued, and that plane is not even loaded: an operand in a symmetric
    // format, or the all-positive attention map, moves half the bytes.
    auto tile_sides = [&](int64_t tile) {
        int bits = 0;
        if (tile < total_items) {
            const int64_t m0 = blk_m(tile) * BM, n0 = blk_n(tile) * BNT;  // (PAIR: only the first CTA asks)
#pragma unroll
            for (int i = 0; i < BMT / 32; ++i)
                if (m0 + i * 32 + lane < p.M) bits |= (__ldg(p.a_exp + m0 + i * 32 + lane) >> 16) & 3;
#pragma unroll
            for (int i = 0; i < BNT / 32; ++i)
                if (n0 + i * 32 + lane < p.N) bits |= ((__ldg(p.w_exp + n0 + i * 32 + lane) >> 16) & 3) << 2;
        }
        return bits;
    };
    auto whole_sides = [&](int lane_bits) {                         // over the warp; an all-zero operand keeps one plane
        int sides = __reduce_or_sync(0xFFFFFFFFu, lane_bits);
        if (!(sides & 3)) sides |= 1;
        if (!(sides & 12)) sides |= 4;
        return sides;
    };

    if (warp == 0) {
        // -------------------------------------------------------------- TMA producer
        // The whole warp runs the loop, one elected lane issues, and the scale factors of an operand are one copy: with eight
        // copies per stage issued under a test of the lane index this warp was what the kernel waited for (a K block took 730 ns
        // whatever the tile's width, 690 with the four copies below).
        // Which planes of a tile are not zero comes from the epilogue warps, which read the tile's row words a tile
        // ahead anyway (sides[] in the control block): nothing on this warp's path but a barrier that has long
        // completed and eight shared-memory words.  (For the first tile it has not: 1 us.)
        int it = 0, j = 0;                                       // K blocks issued so far over all tiles; tiles so far
        bool ok = true;
        auto wait = [&](uint64_t* b, uint32_t parity) { return __all_sync(0xFFFFFFFFu, mbar_wait(b, parity, &ctl->abort, p.status)) != 0; };
        for (int64_t tile = worker; tile < total_items && ok; tile += workers, ++j) {
            // ONE_PLANE: the first plane of each operand, always.  Otherwise the CTA's first stages take both planes without
            // waiting to hear which occur.
            const int ahead = j == 0 ? kStages : 0, part = part_log2(tile), tile_w = kTileWT >> part;
            int a_planes = ONE_PLANE ? 1 : 3, w_planes = a_planes;
            const int64_t m_blk = blk_m(tile), n_blk = blk_n(tile);
            const int kb0 = kb_begin(tile), nkb = nkb_of(tile);
            const int ya = (int)(p.a_row0 + m_blk * BM), yw = (int)(p.w_row0 + n_blk * BNT + part_col(tile) + (PAIR ? rank * (BNT / 2) >> part : 0));
            const int ysa = (int)(p.a_row0 / 128 + m_blk), ysw = (int)(p.w_row0 / 128 + n_blk * (BNT / 128));
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int s = it % kStages;
                if (!ONE_PLANE && kb == ahead) {
                    ok = wait(&ctl->sides_ready[j & 1], (j >> 1) & 1);
                    if (!ok) break;
                    int sides = 0;
#pragma unroll
                    for (int i = 0; i < 8; ++i) sides |= ctl->sides[j & 1][i];
                    a_planes = sides & 3 ? sides & 3 : 1;        // as the MMA warp: an all-zero operand keeps one plane
                    w_planes = sides & 12 ? sides >> 2 : 1;
                }
                if (it >= kStages) {
                    ok = wait(&ctl->empty[s], ((it / kStages) - 1) & 1);
                    if (!ok) break;
                }
                if (elect_one()) {
                    uint8_t *st = tiles + s * kStageBytes, *sf = sf_stages + s * C_::kSfStage;
                    const int x = (kb0 + kb) * kRowBytes, xs = (kb0 + kb) * (C_::kSfRun / 8);
                    const uint32_t bytes = (a_planes == 3 ? 2 : 1) * C_::kTileA + (w_planes == 3 ? 2 : 1) * tile_w + kPlanes * (NHALF ? 2 : 3) * C_::kSfRun;
                    if (!PAIR) mbar_expect_tx(&ctl->full[s], bytes);
                    else if (rank == 0) mbar_expect_tx(&ctl->full[s], 2 * bytes);   // (the other CTA's bytes may be counted first)
                    const uint32_t full = PAIR ? cluster_addr(&ctl->full[s], 0) : 0;
                    auto load_at = [&](uint8_t* dst, const CUtensorMap* map, int x0, int y, int z) {
                        if (PAIR) tma_load_3d_pair(dst, map, x0, y, z, full);
                        else tma_load_3d(dst, map, x0, y, z, &ctl->full[s]);
                    };
                    auto load = [&](uint8_t* dst, const CUtensorMap* map, int y, int z) { load_at(dst, map, x, y, z); };
                    // the scale factors of an operand: {K steps, row blocks, planes}
                    load_at(sf, &tm_sfa, xs, ysa, 0);
                    load_at(sf + kPlanes * C_::kSfRun, &tm_sfw, xs, ysw, 0);
                    // one 3-D tile per operand: {row bytes, rows, both sign planes} - or the one plane that is not zero
                    if (a_planes == 3) load(st + C_::kOffAp, &tm_a, ya, 0);
                    else load(st + (a_planes == 2 ? C_::kOffAn : C_::kOffAp), &tm_a1, ya, a_planes == 2 ? 1 : 0);
                    uint8_t *wp = st + C_::kOffWp, *w1 = wp + (w_planes == 2 ? tile_w : 0);   // the box packs its two planes
                    const int z1 = w_planes == 2 ? 1 : 0;
                    if (part == 0) {
                        if (w_planes == 3) load(wp, &tm_w, yw, 0);
                        else load(w1, &tm_w1, yw, z1);
                    } else {
                        if (w_planes == 3) load(wp, &tm_wt, yw, 0);
                        else load(w1, &tm_wt1, yw, z1);
                    }
                }
                __syncwarp();
            }
        }
        // after an abort: let the copies already in flight land before shared memory is released
        if (ctl->abort && lane == 0)
            // (PAIR: the first CTA waits for both, the other one for the first at the end of the kernel)
            for (int i = max(0, it - kStages); i < it && rank == 0; ++i)
                for (uint32_t n = 0; n < kSpinLimit && !mbar_try_wait(&ctl->full[i % kStages], (i / kStages) & 1); ++n) {}
    } else if (PAIR && warp == 1 && rank == 1) {
        // the pair's MMAs are issued by its first CTA
    } else if (warp == 1) {
        // -------------------------------------------------------------- MMA issuer
        // The whole warp runs the loop (so that addresses and descriptors stay warp-uniform); one elected
        // lane issues.  All operand descriptors differ from the first stage's only in their 14-bit address
        // field (bytes >> 4); the per-plane and per-K-step offsets are compile-time constants.
        const uint64_t desc0 = kRowBytes == 128 ? smem_desc_sw128(smem_u32(tiles)) : smem_desc_sw64(smem_u32(tiles));
        const uint64_t desc_sf0 = smem_desc_rows16(smem_u32(sf_stages));
        int it = 0, t = 0;
        bool ok = true, ready = false;                           // ready: the next K block's barrier was seen complete
        // (the planes of a tile: tile_sides above; the words of the next tile are fetched while the current one runs)
        int sides_next = ONE_PLANE ? 0 : tile_sides(worker);
        for (int64_t tile = worker; tile < total_items && ok; tile += workers) {
            const int part = part_log2(tile);
            const uint32_t idesc = kIdescT - ((uint32_t)((BNT - (BNT >> part)) >> 3) << 17);          // N of the item
            const uint32_t w_minus = (uint32_t)(C_::kOffWp + (ONE_PLANE ? 0 : kTileWT >> part)) >> 4;   // the second plane of W
            const uint32_t sf_col = (uint32_t)part_col(tile) / 32;                                      // 32 rows of W to a column
            const int sides = ONE_PLANE ? 5 : whole_sides(sides_next);   // an all-zero operand: one product, which zeroes the tile
            if (!ONE_PLANE) sides_next = tile_sides(tile + workers);
            const int nkb = nkb_of(tile);
            const int n_mma = ((sides & 1) + ((sides >> 1) & 1)) * (((sides >> 2) & 1) + ((sides >> 3) & 1)) * kSteps;
            // this tile's accumulator window: the columns it shares with the previous tile's must have been read, and
            // so must the rest of the window's last use (tile t - 2).  Neither barrier can run a phase ahead of this
            // wait: its next completion needs this tile's own MMAs.
            const uint32_t acc = tmem + ((t & 1) ? kAccWindow : 0);
            if (t > 0) ok = mbar_wait(&ctl->ovl_free, (t - 1) & 1, &ctl->abort, p.status);
            if (t > 1 && ok) ok = mbar_wait(&ctl->rest_free[t & 1], ((t >> 1) - 1) & 1, &ctl->abort, p.status);
            tc_fence_after();
            uint32_t accumulate = 0;
            // The item's K blocks.  ALL: all planes are in use; PLAIN: and it is a whole tile - everything but the stage is a
            // constant then.  A test per MMA in the issuing thread shows: half tiles took 19.2 us with, 16.5 without those of
            // the planes.
            auto blocks = [&](auto all, auto plain) {
                constexpr bool ALL = decltype(all)::value, PLAIN = decltype(plain)::value;
                for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
                    const int s = it % kStages;
                    // the stage has landed; usually already seen by the poll that was slipped between the previous block's MMAs
                    if (!ready) ok = mbar_wait(&ctl->full[s], (it / kStages) & 1, &ctl->abort, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dstage = desc0 + (uint64_t)((s * kStageBytes) >> 4);
                    const uint32_t sfa = tmem + kTmemSf + (it % C_::kSfSlots) * C_::kSfCols, sfb = sfa + C_::kSfColsA + (PLAIN ? 0u : sf_col);
                    const int s_next = (it + 1) % kStages;
                    const uint32_t parity_next = ((it + 1) / kStages) & 1;
                    uint32_t seen = 0;
                    if (elect_one()) {
                        // the stage's scale factors, 32 rows x 16 bytes to four columns
                        const uint64_t dsf = desc_sf0 + (uint64_t)((s * C_::kSfStage) >> 4);
                        auto copy = [&](uint32_t col, int run, int kk) {
                            if (PAIR) tmem_cp_32x128b_warpx4_pair(col, dsf + ((run * C_::kSfRun + kk * kSfChunk) >> 4));
                            else tmem_cp_32x128b_warpx4(col, dsf + ((run * C_::kSfRun + kk * kSfChunk) >> 4));
                        };
                        const uint32_t sfw = sfa + C_::kSfColsA;
                        auto copy_a = [&](int pl, int kk) { copy(sfa + (pl * kSteps + kk) * 4, pl, kk); };
                        auto copy_w = [&](int pl, int kk) {
                            copy(sfw + (pl * kSteps + kk) * 8, kPlanes + pl * (NHALF ? 1 : 2), kk);
                            if (!NHALF) copy(sfw + (pl * kSteps + kk) * 8 + 4, kPlanes + pl * 2 + 1, kk);
                        };
                        int idx = 0;                                 // MMAs issued so far in this K block
#pragma unroll
                        for (int pa = 0; pa < kPlanes; ++pa)
#pragma unroll
                            for (int pw = 0; pw < kPlanes; ++pw)
#pragma unroll
                                for (int kk = 0; kk < kSteps; ++kk) {   // 64 elements = 32 bytes along the swizzled row
                                    if (pw == 0) copy_a(pa, kk);
                                    if (pa == 0) copy_w(pw, kk);
                                    if (ALL || (((sides >> pa) & 1) && ((sides >> (2 + pw)) & 1))) {
                                        const uint64_t da = dstage + (((pa ? C_::kOffAn : C_::kOffAp) + kk * 32) >> 4),
                                                       dw = dstage + (!pw ? (uint32_t)C_::kOffWp >> 4 : PLAIN ? kOffWnT >> 4 : w_minus) + (kk * 32 >> 4);
                                        const uint32_t sa = sfa + (pa * kSteps + kk) * 4, sw = sfb + (pw * kSteps + kk) * 8;
                                        const uint32_t id = PLAIN ? kIdescT : idesc;
                                        if (PAIR) mma_fp4_block16_pair(acc, da, dw, id, sa, sw, idx ? 1u : accumulate);
                                        else mma_fp4_block16(acc, da, dw, id, sa, sw, idx ? 1u : accumulate);
                                        // with two MMAs still to go (they keep the pipe busy meanwhile), look whether the
                                        // next K block is complete, so that its MMAs can follow without a wait
                                        if (idx == max((ALL ? kPlanes * kPlanes * kSteps : n_mma) - 3, 0)) seen = mbar_try_wait(&ctl->full[s_next], parity_next);
                                        ++idx;
                                    }
                                }
                        if (PAIR) mma_commit_pair(&ctl->empty[s]);
                        else mma_commit(&ctl->empty[s]);
                    }
                    ready = __any_sync(0xFFFFFFFFu, seen) != 0;
                    accumulate = 1;
                }
            };
            if (!ONE_PLANE && sides != 15) blocks(std::false_type{}, std::false_type{});
            else if (part) blocks(std::true_type{}, std::false_type{});
            else blocks(std::true_type{}, std::true_type{});
            if (ok && elect_one()) {
                if (PAIR) mma_commit_pair(&ctl->accum_full);
                else mma_commit(&ctl->accum_full);
            }
            __syncwarp();
            ++t;
        }
    } else {
        // -------------------------------------------------------------- epilogue
        // Eight warps: quarter q = warp % 4 of the lanes (= rows), one half of the columns each.
        const int e = warp - 2;                     // 0..7
        const int q = warp & 3;
        constexpr int kOvl = BNT > kAccWindow ? BNT - kAccWindow : 0;        // columns two consecutive tiles share
        constexpr int kC1 = kOvl / 2 / 16, kC2 = (BNT - kOvl) / 2 / 16;       // this warp's chunks of either part
        static_assert(kOvl % 32 == 0 && (BNT - kOvl) % 32 == 0, "both parts split into two halves of 16-column chunks");
        const int tid_e = threadIdx.x - 64;
        int t = 0;
        static_assert(kEpilogueWarps * 32 == BN, "one column offset per epilogue thread");   // BNT <= BN
        // The per-tile constants (this thread's column offset and row offset) are fetched one tile ahead, so that
        // their latency is off the path between two tiles.
        struct TileConsts {
            float w_fac, a_fac;         // 2^(row offset)
            int planes;                 // planes: bit 0/1 this thread's row of A has +/-, bit 2/3 its row of W has
        };
        // (row offsets lie between -24 and 7, so neither a factor nor the product of two leaves the normal range: the scaled
        // results are exact, as before the optional tensor scales' one rounding)
        auto pow2 = [](int e) { return __uint_as_float((uint32_t)(e + 127) << 23); };
        auto load_consts = [&](int64_t tl) {
            TileConsts c = {1.f, 1.f, 0};
            if (tl < total_items) {
                const int64_t n = blk_n(tl) * BNT + tid_e, mm = blk_m(tl) * BM + q * 32 + lane;
                if (tid_e < BNT && n < p.N) {
                    const int w = __ldg(p.w_exp + n);
                    c.w_fac = pow2(row_word_exp(w));
                    c.planes |= ((w >> 16) & 3) << 2;
                }
                if (mm < p.M) {
                    const int w = __ldg(p.a_exp + mm);
                    c.a_fac = pow2(row_word_exp(w));
                    c.planes |= (w >> 16) & 3;
                }
                const int64_t mo = mm + (rank ? -BM : BM);       // the pair's other row block: its planes are loaded here too
                if (PAIR && mo < p.M) c.planes |= (__ldg(p.a_exp + mo) >> 16) & 3;
            }
            return c;
        };
        // The eight warps' row words cover the tile's 128 + 256 rows: each tells the producer which planes its rows
        // use (tile number j of this CTA); the producer reads them before the tile's first load.
        auto publish = [&](const TileConsts& c, int64_t tl, int j) {
            if (tl >= total_items) return;
            const int bits = __reduce_or_sync(0xFFFFFFFFu, c.planes);
            if (ONE_PLANE) {                                     // nobody waits for the planes; a second one is an error
                if (lane == 0 && (bits & 10)) atomicExch(p.status, (int)AMX_ERR_FLAGS);
                return;
            }
            if (lane == 0) {
                ctl->sides[j & 1][e] = bits;
                mbar_arrive(&ctl->sides_ready[j & 1]);
            }
        };
        auto released = [&](uint64_t* b) {                       // this warp's columns have been read: tells the issuer
            __syncwarp();
            if (lane == 0) {
                if (PAIR && rank) mbar_arrive_remote(b, 0);
                else mbar_arrive(b);
            }
        };
        const float out_scale = p.scale_a ? __ldg(p.scale_a) * __ldg(p.scale_w) : 1.0f;
        int64_t tile = worker;
        TileConsts nxt = load_consts(tile);
        publish(nxt, tile, 0);
        while (tile < total_items) {
            const TileConsts cur = nxt;
            const int64_t tile_after = tile + workers;
            nxt = load_consts(tile_after);                       // in flight while this tile is worked on
            publish(nxt, tile_after, t + 1);
            const int64_t m0 = blk_m(tile) * BM, n0 = blk_n(tile) * BNT;
            float* const C_item = p.C + (SLICED ? (tile % S) * p.slice_stride : 0);
            float* w_fac = ctl->w_fac[t & 1];
            w_fac[tid_e] = cur.w_fac;
            const int64_t m = m0 + q * 32 + lane;
            const float a_fac = cur.a_fac * out_scale;
            const uint64_t a_fac2 = cast::pack_f32x2(__float_as_uint(a_fac), __float_as_uint(a_fac));
            // every epilogue warp has written its part of w_fac (named barrier: the other roles do not join), and has done with the
            // tile two before, whose factors were there
            asm volatile("bar.sync 1, %0;" ::"n"(kEpilogueWarps * 32) : "memory");
            const bool ok = mbar_wait(&ctl->accum_full, t & 1, &ctl->abort, p.status);
            // After a timeout one warp may see the barrier complete where another saw the abort flag, and every tile's named barrier
            // wants all eight.  (Here, out of the way: with the outcome carried through the loop 1000 x 11008 x 4096 took 1.8 us longer.)
            if (__builtin_expect(!ok, 0)) {
#pragma unroll 1
                for (tile = tile_after; tile < total_items; tile += workers) asm volatile("bar.sync 1, %0;" ::"n"(kEpilogueWarps * 32) : "memory");
                break;
            }
            tc_fence_after();
            // 16 columns of the tile: scaled and stored
            auto put = [&](const uint32_t (&v)[16], int col) {
                float f[16];
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const ulonglong2 w2 = *reinterpret_cast<const ulonglong2*>(&w_fac[col + j]);
                    cast::unpack_f32x2(cast::mul_f32x2(cast::pack_f32x2(v[j], v[j + 1]), cast::mul_f32x2(w2.x, a_fac2)), f[j], f[j + 1]);
                    cast::unpack_f32x2(cast::mul_f32x2(cast::pack_f32x2(v[j + 2], v[j + 3]), cast::mul_f32x2(w2.y, a_fac2)), f[j + 2], f[j + 3]);
                }
                if (m < p.M) {
                    if (p.out_bf16)
                        store_row16_bf16(reinterpret_cast<__nv_bfloat16*>(C_item) + m * p.ld_c + n0 + col, f, p.vec_store != 0,
                                         p.N - (n0 + col));
                    else
                        store_row16(C_item + m * p.ld_c + n0 + col, f, p.vec_store != 0, p.N - (n0 + col));
                }
            };
            const int h = e >> 2, odd = t & 1;
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(odd ? kAccWindow : 0);
            const int part = part_log2(tile);
            if (part) {                                    // the CTA's last item: no accumulator follows
                const int cols = (BNT / 2) >> part, col0 = part_col(tile);   // of this warp: half h of the item's
                uint32_t v[2][16];
                tmem_ld16(taddr + h * cols, v[0]);
                for (int i = 0; i < cols; i += 32) {             // (32 or 64 columns)
                    tmem_ld_wait();
                    tmem_ld16(taddr + h * cols + i + 16, v[1]);
                    put(v[0], col0 + h * cols + i);
                    tmem_ld_wait();
                    if (i + 32 < cols) tmem_ld16(taddr + h * cols + i + 32, v[0]);
                    put(v[1], col0 + h * cols + i + 16);
                }
            } else {
                // The tile's window starts at column 0 (even t) or kAccWindow (odd t).  The kOvl columns it shares with
                // the next tile's window - its last ones when even, its first ones when odd - are read first; this warp
                // takes its half h of both parts, kC1 + kC2 chunks of 16 columns.
                const int o1 = odd ? 0 : BNT - kOvl, o2 = odd ? kOvl : 0;
                auto chunk_col = [&](int i) {                    // first column (inside the tile) of this warp's chunk i
                    return i < kC1 ? o1 + h * (kOvl / 2) + 16 * i : o2 + h * ((BNT - kOvl) / 2) + 16 * (i - kC1);
                };
                // (All of them before anything is scaled or stored: the tensor cores wait for this.)
                if (kC1 == 0) released(&ctl->ovl_free);          // nothing shared: the next tile may start at once
                uint32_t first[kC1 ? kC1 : 1][16], v[2][16];
                if (kC1) {
#pragma unroll
                    for (int i = 0; i < kC1; ++i) tmem_ld16(taddr + chunk_col(i), first[i]);
                    tmem_ld_wait();
                    tc_fence_before();
                    released(&ctl->ovl_free);
                }
                tmem_ld16(taddr + chunk_col(kC1), v[0]);
#pragma unroll
                for (int i = 0; i < kC1; ++i) put(first[i], chunk_col(i));
#pragma unroll
                for (int i = 0; i < kC2; ++i) {
                    tmem_ld_wait();
                    if (i + 1 == kC2) {                          // the rest is in registers: tile t + 2 may overwrite the window
                        tc_fence_before();
                        released(&ctl->rest_free[odd]);
                    } else tmem_ld16(taddr + chunk_col(kC1 + i + 1), v[(i & 1) ^ 1]);   // loads while this chunk is stored
                    put(v[i & 1], chunk_col(kC1 + i));
                }
            }
            ++t;
            tile = tile_after;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();                                    // no CTA leaves while the other still uses its memory
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem, kTmemCols);
        else tmem_dealloc(tmem, kTmemCols);
    }
    // As the last thing: the next launch's blocks then find all SMs free, instead of crowding on those that ended first.
    grid_launch_dependents();
}

// ---------------------------------------------------------------------------------- host --
}  // namespace

bool gemm_fp4_supported(int64_t M, int64_t N, int64_t K, int gs) {
    return gs == 32 && M > 0 && N > 0 && K > 0 && K % 32 == 0 && (M + BM - 1) / BM <= 65535 &&
           M < (1ll << 31) && N < (1ll << 31) && K < (1ll << 31);
}

size_t gemm_fp4_workspace_bytes(int64_t M, int64_t N, int64_t K) {
    return 256 + operand_layout(M, K, BM).total + operand_layout(N, K, BN).total;
}

namespace {

int sm_count(int dev) {                                              // 0: the device cannot be asked
    static int count[64] = {};
    if (!count[dev] && cudaDeviceGetAttribute(&count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return count[dev];
}

// Into how many parts (log2) the tiles of a wave that has places for more are cut.
int parts_log2(int64_t tiles, int64_t places) { return tiles * 4 <= places ? 2 : tiles * 2 <= places ? 1 : 0; }

template <int BK_, bool SLICED = false, bool NHALF = false, bool ONE_PLANE = false, bool PAIR = false>
int launch_fp4(const uint8_t* pa, const uint8_t* pw, const OperandLayout& oa, const OperandLayout& ow, int64_t a_rows,
               int64_t w_rows, Params p, int dev, cudaStream_t st) {
    using C_ = Cfg<BK_, ONE_PLANE, PAIR>;
    constexpr int kBoxW = PAIR ? BN / 2 : NHALF ? BN / 2 : BN;
    constexpr int BNT = NHALF ? BN / 2 : BN;
    static bool configured[64] = {};
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(gemm_fp4_kernel<BK_, SLICED, NHALF, ONE_PLANE, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::kSmemBytes) != cudaSuccess)
            return AMX_ERR_CUDA;
        configured[dev] = true;
    }
    if (!sm_count(dev)) return AMX_ERR_CUDA;
    constexpr int kCtas = PAIR ? 2 : 1, BMT = BM * kCtas;
    const int64_t tiles = ((p.N + BNT - 1) / BNT) * ((p.M + BMT - 1) / BMT) * (SLICED ? p.slices : 1);
    const int64_t places = sm_count(dev) / kCtas;                // one persistent CTA (or pair) per SM
    int64_t items = tiles;
    if (!SLICED && !NHALF) {
        // The last, partly filled wave takes as long as a whole one: its tiles are cut into halves or quarters of their
        // columns, as many as there are places for.  An MMA of 128 columns takes 0.7, of 64 columns half the time of one of 256,
        // so more parts are always faster as long as each has a place of its own (1000 x 11008 x 4096, 172 tiles on 74 pairs: the
        // third wave 16.5 us instead of 23.5).
        const int64_t left = tiles % places;
        p.whole = (int)(tiles - left);
        p.split_log2 = parts_log2(left, places);
        items = p.whole + (left << p.split_log2);
    }
    const int64_t workers = std::min<int64_t>(items, places);
    CUtensorMap tm_a, tm_w, tm_a1, tm_w1, tm_wt, tm_wt1, tm_sfa, tm_sfw;   // both planes of a tile in one box, and one plane alone; of a part
    const int box_part = kBoxW >> p.split_log2;
    if (!make_map(&tm_a, pa, a_rows, p.K, oa.plane, BM, C_::kRowBytes) || !make_map(&tm_w, pw, w_rows, p.K, ow.plane, kBoxW, C_::kRowBytes) ||
        !make_map(&tm_a1, pa, a_rows, p.K, oa.plane, BM, C_::kRowBytes, 1) ||
        !make_map(&tm_w1, pw, w_rows, p.K, ow.plane, kBoxW, C_::kRowBytes, 1) ||
        !make_map(&tm_wt, pw, w_rows, p.K, ow.plane, box_part, C_::kRowBytes) ||
        !make_map(&tm_wt1, pw, w_rows, p.K, ow.plane, box_part, C_::kRowBytes, 1) ||
        !make_sf_map(&tm_sfa, pa, oa, C_::kSteps, 1, C_::kPlanes) || !make_sf_map(&tm_sfw, pw, ow, C_::kSteps, NHALF ? 1 : 2, C_::kPlanes))
        return AMX_ERR_CUDA;
    if (PAIR) p.band = (p.band + 1) / 2;
    const unsigned grid = (unsigned)workers * kCtas;
    // Chained up to 8e11 issued products, 5.5e11 of one plane (260 and 200 us with the cast).  Cast and product, ordinary / chained:
    // 4096 x 11008 x 4096 265.5 / 258.5, MXFP4 8192 x 14336 x 4096 200.3 / 197.1, 9000 x 4096 x 14336 263.6 / 259; from there on no
    // difference beyond the runs' own (MXFP4 12000 x 12288 x 4096 316 / 319, 16384 x 14336 x 4096 416 / 415).
    const double products = (double)p.M * (double)p.N * (double)p.K * (ONE_PLANE ? 1.0 : 4.0);
    return launch_clusters(kCtas, products <= (ONE_PLANE ? 5.5e11 : 8e11), gemm_fp4_kernel<BK_, SLICED, NHALF, ONE_PLANE, PAIR>, grid, kThreads, C_::kSmemBytes, st, tm_a, tm_w,
                           tm_a1, tm_w1, tm_wt, tm_wt1, tm_sfa, tm_sfw, p);
}

}  // namespace

namespace {
// Kernel parameters for the product of row ranges of two prepared operands.
int fill_params(const Fp4Operand& a, const Fp4Operand& w, int64_t M, int64_t N, int64_t K, float* C, int64_t ld_c,
                void* workspace, cudaStream_t st, Params& p, OperandLayout& oa, OperandLayout& ow, int& dev) {
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return AMX_ERR_CUDA;
    if (a.row0 % 128 || w.row0 % 128) return AMX_ERR_SHAPE;
    if (((M + BM - 1) / BM) * ((N + BN - 1) / BN) >= (1ll << 27)) return AMX_ERR_SHAPE;   // tile indices are 32-bit
    oa = operand_layout(a.layout_rows, K, BM);
    ow = operand_layout(w.layout_rows, K, BN);
    const uint8_t* pa = static_cast<const uint8_t*>(a.prepared);
    const uint8_t* pw = static_cast<const uint8_t*>(w.prepared);
    int* status = static_cast<int*>(workspace);
    p = Params{};
    p.a_exp = reinterpret_cast<const int*>(pa + 2 * oa.plane + 2 * oa.sf) + a.row0;
    p.w_exp = reinterpret_cast<const int*>(pw + 2 * ow.plane + 2 * ow.sf) + w.row0;
    p.M = M; p.N = N; p.K = K; p.ld_c = ld_c; p.C = C;
    p.a_row0 = a.row0; p.w_row0 = w.row0;
    p.vec_store = C && aligned(C, 32) && ld_c % 8 == 0;     // 32-byte stores in the epilogue
    p.status = status;
    {
        const char* e = getenv("AMX_FP4_BAND");              // row blocks of A per band of the tile order (default 16)
        const int64_t want = e && atoi(e) > 0 ? atoi(e) : 16, m_tiles = (M + BM - 1) / BM;
        p.band = (int)(want < m_tiles ? want : m_tiles);
    }
    return AMX_OK;
}

}  // namespace

// Few output tiles and a long K (a few token rows against a big weight): K ranges as separate work items, so
// that more SMs stream the operands; their partial products go to the workspace and are added in range order.
// Returns the number of ranges (1: none) a workspace is sized for; ranges hold the same number of 128-element K blocks up to
// one.  Whether a call takes them: slices_pay.
int gemm_fp4_slices(int64_t M, int64_t N, int64_t K) {
    const int64_t tiles = ((N + BN - 1) / BN) * ((M + BM - 1) / BM);
    const int num_kb = (int)((K + 127) / 128);
    int s = (int)(148 / tiles);
    if (s > num_kb / 6) s = num_kb / 6;                  // at least six K blocks per range
    if (s > 8) s = 8;
    return s < 2 ? 1 : s;
}
// K ranges or parts of tiles (launch_fp4) for a call of so few tiles, by estimates in us: the launches and a K block of a range's
// tile, the partial products written and read, against the launches and a K block of a half or a quarter.  Fitted to 222 products
// of M 64 to 500, N 512 to 14336, K 2048 to 28672.  Ranges / parts of two planes: 128 x 4096 x 14336 30 / 52, 256 x 4096 x 14336 40 / 52,
// 500 x 4096 x 11008 54 / 46, 256 x 4096 x 4096 27 / 19; of one: 128 x 512 x 14336 17 / 22, 128 x 1024 x 28672 23 / 44,
// 128 x 8192 x 28672 53 / 47, 500 x 4096 x 4096 34 / 13.  (Tiles of 128 columns have no parts and take a quarter's time; both
// planes' figures, which a product of one plane is 3 to 20 % below.)  Rows of results that are no multiple of 32 bytes are stored one
// by one, which a range's whole tile takes 0.11 us a row for, a half 0.07, a quarter 0.025: 92 x 412 x 8192 of one plane 23 / 16,
// 121 x 315 x 2304 of two 26 / 15.  The choice costs 0.2 % on average over these and 420 others, M from 8, N from 64, a third of them ragged.
namespace {
bool slices_pay(int64_t M, int64_t N, int64_t K, int slices, int sms, bool one_plane, bool half, bool vec_store) {
    if (slices < 2) return false;
    struct Fit { double ranges, block, parts, of_half, of_quarter; };
    static constexpr Fit kFit[2] = {{8.0, 0.73, 5.4, 0.50, 0.41}, {8.4, 0.48, 5.2, 0.224, 0.166}};
    const Fit& f = kFit[one_plane && !half];
    const int64_t blocks = (K + 127) / 128;
    const bool quarters = half || parts_log2(((N + BN - 1) / BN) * ((M + BM - 1) / BM), sms) == 2;
    const double rows = half ? 0.0 : (double)std::min<int64_t>(M, BM);
    const double ranges = f.ranges + f.block * (double)((blocks + slices - 1) / slices) + 3.0e-6 * slices * (double)M * (double)N;
    const double parts = f.parts + (quarters ? f.of_quarter : f.of_half) * (double)blocks;
    return ranges + (N % 8 ? 0.11 * rows : 0.0) < parts + (vec_store ? 0.0 : (quarters ? 0.025 : 0.07) * rows);
}
}  // namespace
size_t gemm_fp4_prepared_workspace_bytes(int64_t M, int64_t N, int64_t K) {
    const int s = gemm_fp4_slices(M, N, K);
    return 256 + (s > 1 ? (size_t)s * M * N * 4 : 0);
}

// The GEMM proper on two prepared operands (each laid out by operand_layout()), or on row ranges of them.
// workspace_bytes >= gemm_fp4_prepared_workspace_bytes() enables the K ranges; 256 bytes always suffice.
int gemm_fp4_prepared_at(const Fp4Operand& a, const Fp4Operand& w, int64_t M, int64_t N, int64_t K, float* C,
                         int64_t ld_c, void* workspace, cudaStream_t st, size_t workspace_bytes, const int* gate,
                         const float* scale_a, const float* scale_w, bool one_plane, bool out_bf16) {
    Params p;
    OperandLayout oa, ow;
    int dev;
    const int rc = fill_params(a, w, M, N, K, C, ld_c, workspace, st, p, oa, ow, dev);
    if (rc != AMX_OK) return rc;
    // the status word; a caller that hands over a gate has cleared it (the gate is the word behind it)
    if (!gate && clear_words(workspace, st, 1) != AMX_OK) return AMX_ERR_CUDA;
    p.gate = gate;
    p.scale_a = scale_a;
    p.scale_w = scale_w;
    if (out_bf16) {                                         // 32-byte stores hold 16 results
        p.out_bf16 = 1;
        p.vec_store = aligned(C, 32) && ld_c % 16 == 0;
    }
    const uint8_t* pa = static_cast<const uint8_t*>(a.prepared);
    const uint8_t* pw = static_cast<const uint8_t*>(w.prepared);
    const int slices = gemm_fp4_slices(M, N, K);
    // at most 128 columns: tiles of 128 x 128, so that no half of a W tile is padding
    const bool half = N <= BN / 2 && !getenv("AMX_FP4_NO_HALF_TILE");
    if (!gate && !scale_a && !out_bf16 && slices_pay(M, N, K, slices, sm_count(dev), one_plane, half, p.vec_store != 0) &&
        workspace_bytes >= gemm_fp4_prepared_workspace_bytes(M, N, K)) {
        float* part = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + 256);
        p.C = part;
        p.ld_c = N;
        p.vec_store = N % 8 == 0;
        p.slices = slices;
        p.slice_stride = M * N;
        const int r2 = launch_fp4<128, true>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st);
        return r2 != AMX_OK ? r2 : reduce_slices(part, slices, M, N, C, ld_c, st);
    }
    // A pair of SMs per tile (256 x 256) where there is more than a tile for every SM: either SM loads half of the W rows.
    // 2048 x 12288 x 4096: 159 -> 154 us; 16384 x 10240 x 8192: 1.4 % fewer cycles, the call 2 % shorter under the power cap.
    // With at most one tile per SM there is nothing to overlap the pair's longer start and end with (1024 x 4096 x 4096: 36 us
    // alone, 39 in pairs); an odd row block leaves half a pair idle, which a sixteenth of the rows may cost.
    const int64_t m_blocks = (M + BM - 1) / BM;
    const bool pair = !half && m_blocks * ((N + BN - 1) / BN) > sm_count(dev) && (m_blocks % 2 == 0 || m_blocks >= 15);
    if (pair)
        return one_plane ? launch_fp4<256, false, false, true, true>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st)
                         : launch_fp4<128, false, false, false, true>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st);
    // both operands stated to be single planes (full-width tiles; the half-width ones are short products and run the general
    // kernel, which skips absent planes by itself)
    if (one_plane && !half) return launch_fp4<256, false, false, true>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st);
    return half ? launch_fp4<128, false, true>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st)
                : launch_fp4<128>(pa, pw, oa, ow, a.rows_total, w.rows_total, p, dev, st);
}

int gemm_fp4_prepared(const void* a_prepared, const void* w_prepared, int64_t M, int64_t N, int64_t K, float* C,
                      int64_t ld_c, void* workspace, cudaStream_t st, size_t workspace_bytes, const int* gate) {
    return gemm_fp4_prepared_at({a_prepared, M, M, 0}, {w_prepared, N, N, 0}, M, N, K, C, ld_c, workspace, st,
                                workspace_bytes, gate);
}

// Size of a prepared operand: as the A operand (rows padded to 128) or the W operand (rows padded to 256).
size_t gemm_fp4_prepared_bytes(int64_t rows, int64_t K, bool is_weight) {
    return operand_layout(rows, K, is_weight ? BN : BM).total;
}

// Parts of a prepared operand, for the launch that fills them.
namespace {
PrepOperand describe(int64_t rows, int64_t K, bool is_weight, void* prepared, int64_t layout_rows) {
    const OperandLayout o = operand_layout(layout_rows ? layout_rows : rows, K, is_weight ? BN : BM);
    uint8_t* base = static_cast<uint8_t*>(prepared);
    PrepOperand p{};
    p.R = rows;
    p.pos = reinterpret_cast<uint4*>(base);
    p.neg = reinterpret_cast<uint4*>(base + o.plane);
    p.sf_pos = base + 2 * o.plane;
    p.sf_neg = p.sf_pos + o.sf;
    p.row_exp = reinterpret_cast<int*>(p.sf_neg + o.sf);
    p.padded_rows = o.row_blocks * 128;
    return p;
}
}  // namespace

PrepOperand gemm_fp4_cast_operand(const void* x, int64_t ld, int64_t rows, int64_t K, bool is_weight, uint8_t* codes, uint8_t* scales,
                                  void* prepared, int64_t layout_rows, int64_t seg_rows, int64_t seg_pad) {
    PrepOperand p = describe(rows, K, is_weight, prepared, layout_rows);
    p.x = static_cast<const uint4*>(x);
    p.ld_vec = ld / 8;
    p.codes = reinterpret_cast<uint4*>(codes);
    p.scales = reinterpret_cast<uint16_t*>(scales);
    p.seg_rows = (unsigned)seg_rows;
    p.seg_blocks = (unsigned)(seg_pad / 128);
    if (seg_pad) p.padded_rows = (rows + 127) / 128 * 128;
    return p;
}

PrepOperand gemm_fp4_split_operand(const uint8_t* codes, const uint8_t* scales, int64_t rows, int64_t K, bool is_weight,
                                   void* prepared, int64_t layout_rows) {
    PrepOperand p = describe(rows, K, is_weight, prepared, layout_rows);
    p.in_codes = reinterpret_cast<const uint4*>(codes);
    p.in_scales = reinterpret_cast<const uint16_t*>(scales);
    return p;
}

int gemm_fp4_prepare_operands(const PrepOperand* op, int n, int64_t K, int gs, cudaStream_t st, int format, int* flushed_total) {
    return prepare_operands(op, n, K, gs, operand_layout(128, K, BM).nk64, st, format, flushed_total);
}

// (The rows of V^T past d of a head, and their words, are whatever they were: not read.)
int gemm_fp4_prepare_attention(const PrepOperand (&qk)[2], const void* v, int64_t kv_heads, int64_t L, int64_t d, int64_t layout_rows,
                               uint8_t* v_scales, void* v_prepared, cudaStream_t st, int* flushed_total) {
    const OperandLayout o = operand_layout(layout_rows, L, BN);
    uint8_t* base = static_cast<uint8_t*>(v_prepared);
    const VtOperand vt = {static_cast<const uint4*>(v), L, (int)d, o.nk64, reinterpret_cast<uint4*>(base), reinterpret_cast<uint4*>(base + o.plane),
                          reinterpret_cast<uint16_t*>(v_scales), base + 2 * o.plane, base + 2 * o.plane + o.sf,
                          reinterpret_cast<int*>(base + 2 * o.plane + 2 * o.sf)};
    return prepare_attention(qk, d, operand_layout(128, d, BM).nk64, vt, kv_heads, st, flushed_total);
}

// Bytes from the first to the second sign plane of a prepared operand.
size_t gemm_fp4_plane_bytes(int64_t rows, int64_t K) { return operand_layout(rows, K, BM).plane; }

// Row words of a prepared operand (rows of them, device memory).
const int* gemm_fp4_row_words(const void* prepared, int64_t rows, int64_t K, bool is_weight) {
    const OperandLayout o = operand_layout(rows, K, is_weight ? BN : BM);
    return reinterpret_cast<const int*>(static_cast<const uint8_t*>(prepared) + 2 * o.plane + 2 * o.sf);
}

int gemm_fp4_softmax_prepared(const float* S, int64_t rows, int64_t cols, int64_t ld_s, float alpha, bool is_weight,
                              uint8_t* codes, uint8_t* scales, void* prepared, cudaStream_t st, int64_t causal) {
    const OperandLayout o = operand_layout(rows, cols, is_weight ? BN : BM);
    uint8_t* base = static_cast<uint8_t*>(prepared);
    return softmax_cast_rows(S, rows, cols, ld_s, alpha, codes, scales, base, base + o.plane, base + 2 * o.plane,
                             base + 2 * o.plane + o.sf, reinterpret_cast<int*>(base + 2 * o.plane + 2 * o.sf), o.nk64,
                             o.row_blocks * 128, st, causal);
}

// Workspace: word 0 the status, word 1 the number of scales flushed while preparing the two operands (see
// to_ue4m3), then the prepared operands.  gate_on_flushed: the GEMM kernel returns at once when that count is
// not zero (the caller follows with the exact kernel, gated the other way).
int gemm_fp4(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes, const uint8_t* w_scales,
             int64_t M, int64_t N, int64_t K, float* C, int64_t ld_c, void* workspace, cudaStream_t st,
             bool gate_on_flushed, int gs) {
    const OperandLayout oa = operand_layout(M, K, BM);
    uint8_t* base = static_cast<uint8_t*>(workspace);
    uint8_t* pa = base + 256;
    uint8_t* pw = pa + oa.total;
    int* flushed = reinterpret_cast<int*>(base) + 1;
    if (clear_words(base, st) != AMX_OK) return AMX_ERR_CUDA;
    const PrepOperand op[2] = {gemm_fp4_split_operand(a_codes, a_scales, M, K, false, pa), gemm_fp4_split_operand(w_codes, w_scales, N, K, true, pw)};
    const int rc = gemm_fp4_prepare_operands(op, 2, K, gs, st, AMX_FMT_AMXFP4, flushed);
    if (rc != AMX_OK) return rc;
    return gemm_fp4_prepared(pa, pw, M, N, K, C, ld_c, base, st, 256, gate_on_flushed ? flushed : nullptr);
}

}  // namespace amx
