// Fully quantized attention on the FP4 tensor-core pipe for head dimensions 128 and 64 (arXiv 2411.09909, Appendix C:
// Query, Key, the self-attention map and Value are all cast to AMXFP4; Section 1: at long context these products
// are a large share of the prefill work).  Neither the logits nor the attention map ever reach global memory.
//
// What is quantized is the NORMALISED map P = softmax(Q K^T / sqrt(d)), rounded to bf16, with groups of 32 along
// the keys.  Its scales depend on the final row maximum and sum, so the product Q K^T is computed for the statistics
// before it is computed for the map:
//   map    S tiles -> P tile = 2^(s - max) / sum, rounded to bf16 and cast to AMXFP4 in registers (P has no negative
//          element: one sign plane), written to shared memory in the layout the MMA reads, its scale factors copied to
//          tensor memory, and O += P V on the tensor cores in the same kernel.
// The statistics come in two forms.  One rounding of a row's sum or of an exponent decides now and then which bf16 value a
// probability takes, that value which step of E5M2 its group's scale takes, and that a quarter of the group's magnitude:
//   ordered  (ragged lengths, head dimension 64, short sequences: wherever these products also exist with the logits in
//            global memory) first the maxima, then the sums: same argument t log2(e) - max log2(e) with
//            t = alpha s rounded, same order of additions as softmax_math.cuh, hence the bits of the stored path.  The
//            logits are the same numbers too: a sum of head-dimension-many products of E2M1 codes under E5M2 scales a few
//            binades apart needs fewer than 24 bits.  (Online sums moved up to 3 rows of 33792 at 32 over 8 heads x 1056, now and
//            then an element by half of the result's rms.)  Maxima, sums and map of an item - a block of 128 queries - are three
//            phases of one launch: a row's statistics stay in shared memory and a short item pays for one start and one end.
//            (Three launches with the statistics in global memory: 32 over 8 heads x 1056 causal 73.7 us for the call, 62.7 now;
//            16 heads x 4000 causal 233 / 217.)
//   online   (long whole blocks at head dimension 128) one launch keeps a running maximum and a rescaled sum, log2(e) folded
//            into the column factors, a second one computes the map.
// Both products use the sign split of the GEMM (gemm_fp4.cu): S = Q+K+ + Q+K- + Q-K+ + Q-K- (8 block-scaled MMAs
// per 128 x 128 tile at K = 128, 4 at K = 64), O += P V+ + P V- (4 MMAs per tile of 128 keys).
// Any sequence length: every head's Q and K rows are padded to whole 128-row blocks (zero scale factors, zero row
// words), V^T to 128 rows; keys past the sequence are masked in the last key tile, queries past it are not stored.
// At head dimension 64 the K tile's rows are half as long (the TMA box fills the rest with zeros and one K step is
// issued) and O is 64 columns wide.
//
// One persistent CTA per SM walks over (head, block of 128 queries) items; per item it loops over the key tiles:
//   warp 0      TMA: the item's Q tile; per key tile the K tile and (for the map) the V^T tile, {+, -} planes and scale
//               factors each, into rings of stages
//   warp 1      issues the MMAs of the logits as far ahead as there are accumulators (three in the launch for online
//               statistics, where the third takes O's columns, else two)
//   warp 2      the per-key column factors alpha * 2^(K row offset) of the tile (online: times log2(e))
//   warp 3      (map) issues the MMAs of P V.  A warp of its own: issued by warp 1 in turn with the logits, every wait
//               for P held up the next logits (32 heads x 8192 x 128: 2198 us against 1994)
//   warps 4-    epilogue, groups of eight warps (as many as accumulators): group g takes the key tiles with
//               (tile count) % groups == g, so the groups are in different phases of their tiles (tensor-memory loads
//               and maxima in one, exponentials in the other) and keep both the issue slots and the special-function
//               unit busy; a thread owns one query row and 64 keys of its tiles: tensor memory -> registers, softmax
//               arithmetic, the cast, stores to shared memory.  (A third group for the map has no accumulator of its own
//               to work on: 2023 us against 1994.)  The probabilities of both 32-key groups come before either is cast, so that
//               the exponentials of one (special-function unit) and the cast of the other (ALU, FMA) overlap in a warp (1888 us
//               for the call -> 1850).  In the ordered form all sixteen warps share every tile, 32 keys each: an item
//               of few tiles is as long as its last tile takes (32 over 8 heads x 1056 causal 64.6 us with tiles in turn, 62.7
//               shared; 16 heads x 4000 causal 221 / 217; not causal 16 x 1280 79.6 / 80.8).
//   after the last key tile of an item the epilogue warps read out O, rescale by the rows' powers of two and store.
// Scale factors go from global to shared memory with the tiles and on to tensor memory by the issuing warps
// (tcgen05.cp, ordered with the MMAs): four warps that carried them through registers were a sixth of all instructions.
// What bounds it (32 heads x 8192): per key tile the tensor cores need 600 cycles for the statistics and 900 for the map; of
// the epilogue's units the special-function unit is busy for 1024 cycles in either, the FMA pipe for 480 and 1030, the ALU for
// 330 and 1010; a tile takes 1450 and 2200.  No unit is within 1.4 times of its limit: the rest is waiting of one unit's
// instructions for another's with four (six) warps to a scheduler.
// Tensor memory: S0, S1, O (128 columns each), scale factors of Q (16), of three K and V^T stages or six of K (96), of the
// two P tiles (8 each): 512 columns.  Every wait is bounded; on a timeout all roles run their loops out without
// work, tensor memory is released and the status word reports AMX_ERR_TIMEOUT.
#include <cuda_bf16.h>

#include <type_traits>

#include "cast_math.cuh"
#include "fp4_operand.cuh"
#include "gemm.cuh"
#include "softmax_math.cuh"
#include "tcgen05.cuh"

namespace amx {
namespace {

using namespace tc;
using namespace fp4;

constexpr int BM = 128, BNK = 128;                   // queries per item, keys per tile
constexpr int kVRows = 128;                           // rows of one head of V^T (padded at head dimension 64)
// What a launch does, and what is done with a tile of logits.
enum Pass { kPassStats, kPassMapOnline, kPassOrdered };
enum Phase { kStats, kMapOnline, kMax, kSum, kMapOrdered };
__host__ __device__ constexpr bool has_map(int pass) { return pass != kPassStats; }
__host__ __device__ constexpr int phases(int pass) { return pass == kPassOrdered ? 3 : 1; }
__host__ __device__ constexpr bool is_map(int phase) { return phase == kMapOnline || phase == kMapOrdered; }
// Stages of the K and V^T rings.  Without V^T its place holds three more of K: a statistics pass
// waits for loads (32 heads x 8192: 1946 -> 1897 us).
constexpr int kStages = 3, kStagesMax = 6;
__host__ __device__ constexpr int k_stages(int pass) { return pass == kPassStats ? kStagesMax : pass == kPassOrdered ? 5 : kStages; }
// ... and of the scale factors of K in tensor memory (the copies there and the MMAs run in the order of their issue)
__host__ __device__ constexpr int sf_slots(int pass) { return has_map(pass) ? 3 : 6; }
// Ring of the per-tile column factors.  A group may still read those of tile j when it has released j's accumulator and the
// other groups theirs, so the MMAs may be done up to tile j + 5 and the writer (warp 2), kStagesMax ahead of those, at tile
// j + 11: 16 slots never collide and need no barrier of their own.
constexpr int kKcRing = 16;
constexpr int kFirstEpi = 4;                          // warps 0-3: TMA, logits MMAs, column factors, P V MMAs
constexpr int kOWarps = 16;                           // of the epilogue warps, those that read out O
// Epilogue groups, each with an accumulator (the third in O's columns).  The ordered sums take two: a thread then meets the key
// tiles of one parity, four of every eight, in the order in which the stored path's tree adds them.
__host__ __device__ constexpr int epi_groups(int pass) { return pass == kPassStats ? 3 : 2; }
// Whether all groups share every tile, a warp 32 of its keys, instead of taking the tiles in turn.
__host__ __device__ constexpr bool share_tiles(int pass) { return pass == kPassOrdered; }
__host__ __device__ constexpr int tile_warps(int pass) { return share_tiles(pass) ? 16 : 8; }
__host__ __device__ constexpr int s_buffers(int pass) { return epi_groups(pass); }   // (a group meets every phase of its s_full barrier)
__host__ __device__ constexpr int threads(int pass) { return (kFirstEpi + 8 * epi_groups(pass)) * 32; }
constexpr int kParts = 2 * epi_groups(kPassStats);    // partial row statistics: a thread's columns of its group's tiles
// Ordered sums: per 8 key tiles {even, odd tiles} x 4 groups of a tile.  Past 8192 keys (64 tiles) the stored path adds in another
// order anyway: then once per row, so that they fit in shared memory at any length.
constexpr int kSumParts = 8, kSumBlocks = 8;
__host__ __device__ constexpr int sum_shift(int64_t tiles) { return tiles <= 8 * kSumBlocks ? 3 : 30; }
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kPlane = 128 * 64;                      // one sign plane of a 128 x 128 tile: 64-byte rows
constexpr int kTileBytes = 2 * kPlane;                // {+, -}
constexpr int kSfBytes = 4 * kSfChunk;                // a tile's scale factors: {+, -} x two K steps of 64
// tensor-memory columns
constexpr uint32_t kColS = 0, kColO = 256, kColSfQ = 384, kColSfKV = 400, kColSfP = 496, kTmemCols = 512;
static_assert(kStagesMax * 16 == kStages * 32 && kColSfKV + kStages * 32 == kColSfP && kColSfP + 2 * 8 == kTmemCols, "tensor-memory budget");

struct __align__(16) Control {
    uint64_t q_full, q_empty, k_full[kStagesMax], k_empty[kStagesMax], v_full[kStages], v_empty[kStages], s_full[3], s_empty[3], p_full[2], p_empty[2], o_full, o_empty;
    uint32_t tmem_base;
    volatile int abort;
};

// shared-memory layout (offsets from the 1024-aligned base)
template <int PASS>
struct Smem {
    static constexpr int kOffQ = 0;
    // K and V^T tiles, each with its scale factors, in rings of their own: a K stage is free as soon as its logits are
    // computed, two tiles before the V^T tile of the same keys is used
    static constexpr int kOffK = kTileBytes, kOffV = kOffK + k_stages(PASS) * kTileBytes;
    static constexpr int kOffP = kOffV + (has_map(PASS) ? kStages * kTileBytes : 0);  // two P planes (map pass)
    static constexpr int kOffSfP = kOffP + (has_map(PASS) ? 2 * kPlane : 0);          // two buffers x two 512-byte chunks
    static constexpr int kOffSfQ = kOffSfP + (has_map(PASS) ? 2 * 2 * 512 : 0);
    static constexpr int kOffSfK = kOffSfQ + kSfBytes, kOffSfV = kOffSfK + k_stages(PASS) * kSfBytes;
    static constexpr int kOffKc = kOffSfV + (has_map(PASS) ? kStages * kSfBytes : 0); // 128 column factors per slot
    static constexpr int kOffTab = kOffKc + kKcRing * 512;                        // per scale byte: see cast_group
    static constexpr int kOffMax = kOffTab + (has_map(PASS) ? 128 * 8 : 0);       // ordered: maxima of {groups x halves} of the rows
    static constexpr int kOffSums = kOffMax + (PASS == kPassOrdered ? 4 * 128 * 4 : 0);   // and sums of key groups
    static constexpr int kOffCtl = kOffSums + (PASS == kPassOrdered ? kSumBlocks * kSumParts * 128 * 4 : 0);
    static constexpr int kBytes = kOffCtl + 512 + 1024;                           // + Control + alignment slack
};
static_assert(sizeof(Control) <= 512, "Control must fit its reserved space");
static_assert(Smem<kPassOrdered>::kBytes <= 227 * 1024 && Smem<kPassMapOnline>::kBytes <= 227 * 1024, "shared memory");

// K-major operand rows of 64 bytes with the 64-byte swizzle: groups of 8 rows are 512 B apart.  lo: the address in units of
// 16 bytes (the descriptor's low word); the rest is constant, so that a tile's descriptors differ by constants in one word.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint64_t desc_sw64(uint32_t lo) {
    return ((uint64_t)((512u >> 4) | (1u << 14) | (4u << 29)) << 32) | lo;
}
// 32 rows x 16 bytes without swizzle (the source of tcgen05.cp), likewise
__device__ __forceinline__ uint32_t sf_lo(uint32_t addr) { return (addr >> 4) & 0x3FFFu; }
__device__ __forceinline__ uint64_t desc_sf(uint32_t lo) { return ((uint64_t)((128u >> 4) | (1u << 14)) << 32) | lo; }
// kind::mxf4nvf4 block-scaled, A and B E2M1, K-major, UE4M3 scale factors, M = 128, K = 64 per instruction
__host__ __device__ constexpr uint32_t idesc(int n) { return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24); }

// cast::cast_nonneg_group with what follows from the group's scale byte looked up in shared memory, {1 / scale, the UE4M3
// byte under a row offset of zero (far below zero for a zero scale)} (32 heads x 8192: 1978 -> 1948 us).
__device__ __forceinline__ uint2 scale_entry(uint32_t b) {
    return make_uint2(__float_as_uint(cast::inv_scale(b)), b ? scale_norm(b) << 1 : 0x80000000u);
}
__device__ __forceinline__ uint32_t cast_group(const uint32_t (&w)[16], const uint2* tab, int key_ofs, uint32_t (&nib)[4], uint32_t& up) {
    const uint32_t sc = cast::nonneg_group_scale(w);
    const uint2 e = tab[sc];
    const int t = (int)e.y + key_ofs;
    up = t >= 8 ? (uint32_t)t : 0u;
    cast::nonneg_group_codes(w, e.x, nib);
    return sc;
}

struct Maps {
    CUtensorMap q, k, v, sfq, sfk, sfv;              // planes and scale factors of the operands
};

struct Params {
    // prepared operands (fp4_operand.cuh); row ranges of stacked heads: head h of the launch has its queries at
    // rows q_row0 + h * Lp of Q, its keys at k_row0 + (h / kv_group) * Lp of K, its V^T rows at
    // v_row0 + (h / kv_group) * 128 (kv_group query heads share one head of keys and values: grouped-query attention)
    const int *q_words, *k_words, *v_words;          // row words, from the operand's first row
    int64_t q_row0, k_row0, v_row0;
    int vec_o;               // O is 16-byte aligned
    int heads, m_tiles, kv_group;
    int64_t L, Lp;           // sequence length, and padded to whole blocks of 128
    float alpha;
    const int* gate;         // not NULL: nothing is done when this word is nonzero (the caller runs the exact kernel then)
    float2* part;            // online: [heads * Lp][kParts]: per row {max, sum of 2^(t - max)}, base-2 units
    int sum_shift;           // ordered: tiles of a block, log2
    float* O;                // map pass out: [heads][L][head dimension]
    int* status;
    // optional outputs of the online map pass for head 0 of the launch (verification): the bf16 map the cast started from
    // [L][L/2 words], canonical codes [L][L/32] x 16 bytes, scale bytes, and the prepared form of P (plane, scale
    // factors, row words)
    uint4 *p_bits, *p_codes, *p_plane;
    uint16_t* p_scales;
    uint8_t* p_sf;
    int* p_words;
    int p_nk64;
};

// Which keys a tile masks: none (whole tiles, no causal mask), the causal diagonal, or those past a ragged sequence.
enum Mask { kMaskNone, kMaskCausal, kMaskTail };

template <int PASS, int MASK, int HD>
__global__ void __launch_bounds__(threads(PASS), 1)
attention_fp4_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_sfq,
                     const __grid_constant__ CUtensorMap tm_sfk, const __grid_constant__ CUtensorMap tm_sfv, const Params p) {
    using S_ = Smem<PASS>;
    constexpr bool CAUSAL = MASK == kMaskCausal;
    constexpr int kGroups = epi_groups(PASS), kSBufs = s_buffers(PASS), kKStages = k_stages(PASS);
    constexpr int kSfSlots = sf_slots(PASS), kPhases = phases(PASS);
    constexpr uint32_t kSfStage = 96 / kSfSlots;          // tensor-memory columns of a slot's scale factors: K, then V^T
    constexpr int kQkSteps = HD / 64;                     // MMAs along the head dimension per sign pair
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Control* ctl = reinterpret_cast<Control*>(sm + S_::kOffCtl);
    float* kc_all = reinterpret_cast<float*>(sm + S_::kOffKc);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // The CTA's item number ii: a boustrophedon over the CTAs, so that under a causal mask - long items (late query blocks)
    // first - a CTA that starts with a long item goes on with a short one.
    auto item_id = [&](int ii) { return ii * (int)gridDim.x + ((ii & 1) ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x); };
    // item -> (head, query block)
    auto item_head = [&](int id) { return id % p.heads; };
    auto item_m = [&](int id) { const int mi = id / p.heads; return CAUSAL ? p.m_tiles - 1 - mi : mi; };
    auto tiles_of = [&](int m_blk) { return CAUSAL ? m_blk + 1 : p.m_tiles; };

    if (threadIdx.x == 0) {
        mbar_init(&ctl->q_full, 1);
        mbar_init(&ctl->q_empty, 1);
        for (int s = 0; s < kKStages; ++s) {
            mbar_init(&ctl->k_full[s], 2);                       // the copies and the column factors
            mbar_init(&ctl->k_empty[s], 1);
        }
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ctl->v_full[s], 1);
            mbar_init(&ctl->v_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl->p_full[b], tile_warps(PASS));
        }
        for (int b = 0; b < kSBufs; ++b) mbar_init(&ctl->s_empty[b], tile_warps(PASS));
        for (int g = 0; g < kGroups; ++g) mbar_init(&ctl->s_full[g], 1);
        for (int b = 0; b < 2; ++b) mbar_init(&ctl->p_empty[b], 1);
        mbar_init(&ctl->o_full, 1);
        mbar_init(&ctl->o_empty, kOWarps);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    uint2* scale_tab = reinterpret_cast<uint2*>(sm + S_::kOffTab);
    if (has_map(PASS) && threadIdx.x >= 128 && threadIdx.x < 256) scale_tab[threadIdx.x - 128] = scale_entry(threadIdx.x - 128);
    if (warp == 1) tmem_alloc(&ctl->tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    grid_dependency_wait();
    const int n_items = p.gate && *p.gate != 0 ? 0 : p.heads * p.m_tiles;        // (uniform over the grid)

    if (warp == 0) {
        // ---------------------------------------------------------------------------------- TMA producer
        // (The whole warp runs the loop, an elected lane issues, a tile's scale factors are one copy: three copies per tile issued
        // under a lane test, 32 heads x 8192 1898 us, 1056 keys 75.4; as it is 1872 and 73.7.)
        int ii = 0, n_k = 0, n_v = 0;                               // items, copies of K and of V^T issued
        bool ok = true;
        auto wait = [&](uint64_t* b, uint32_t parity) { return __all_sync(0xFFFFFFFFu, mbar_wait(b, parity, &ctl->abort, p.status)) != 0; };
        // a tile and its scale factors: {+, -} of 128 rows from row y, columns from byte x, the two K steps from step k64
        auto load = [&](int off, int sf_off, const CUtensorMap* map, const CUtensorMap* sf_map, int x, int y, int k64, uint64_t* full) {
            if (elect_one()) {
                mbar_expect_tx(full, kTileBytes + kSfBytes);
                tma_load_3d(sm + sf_off, sf_map, k64 * (kSfChunk / 8), y >> 7, 0, full);
                tma_load_3d(sm + off, map, x, y, 0, full);
            }
            __syncwarp();
        };
        for (int id = item_id(ii); id < n_items && ok; id = item_id(++ii)) {
            const int h = item_head(id), m_blk = item_m(id);
            // the previous item's logits MMAs have read the Q tile
            if (ii > 0 && !wait(&ctl->q_empty, (ii - 1) & 1)) break;
            const int k_row0 = (int)(p.k_row0 + (int64_t)(h / p.kv_group) * p.Lp), v_row = (int)(p.v_row0 + (int64_t)(h / p.kv_group) * kVRows);
            load(S_::kOffQ, S_::kOffSfQ, &tm_q, &tm_sfq, 0, (int)(p.q_row0 + (int64_t)h * p.Lp) + m_blk * BM, 0, &ctl->q_full);
            const int T = tiles_of(m_blk);
            for (int ph = 0; ph < kPhases && ok; ++ph)
                for (int j = 0; j < T; ++j) {
                    const int s = n_k % kKStages;
                    if (n_k >= kKStages) ok = wait(&ctl->k_empty[s], ((n_k / kKStages) - 1) & 1);
                    if (!ok) break;
                    load(S_::kOffK + s * kTileBytes, S_::kOffSfK + s * kSfBytes, &tm_k, &tm_sfk, 0, k_row0 + j * BNK, 0, &ctl->k_full[s]);
                    ++n_k;
                    if (has_map(PASS) && ph == kPhases - 1) {
                        const int sv = n_v % kStages;
                        if (n_v >= kStages) ok = wait(&ctl->v_empty[sv], ((n_v / kStages) - 1) & 1);
                        if (!ok) break;
                        load(S_::kOffV + sv * kTileBytes, S_::kOffSfV + sv * kSfBytes, &tm_v, &tm_sfv, j * 64, v_row, j * 2, &ctl->v_full[sv]);
                        ++n_v;
                    }
                }
        }
        // after a timeout: let the copies already in flight land before shared memory is released
        if (ctl->abort && lane == 0) {
            for (int i = max(0, n_k - kKStages); i < n_k; ++i)
                for (uint32_t n = 0; n < kSpinLimit && !mbar_try_wait(&ctl->k_full[i % kKStages], (i / kKStages) & 1); ++n) {}
            for (int i = max(0, n_v - kStages); i < n_v; ++i)
                for (uint32_t n = 0; n < kSpinLimit && !mbar_try_wait(&ctl->v_full[i % kStages], (i / kStages) & 1); ++n) {}
            if (ii > 0)
                for (uint32_t n = 0; n < kSpinLimit && !mbar_try_wait(&ctl->q_full, (ii - 1) & 1); ++n) {}
        }
    } else if (warp == 1 || (has_map(PASS) && warp == 3)) {
        // ---------------------------------------------------------------------------------- MMA issuers
        // The whole warp runs the loops (addresses stay warp-uniform); one elected lane issues.
        const uint32_t base = smem_u32(sm);
        // scale factors of a tile, {+, -} x k_steps chunks, shared memory -> tensor memory (ordered with the MMAs of this thread)
        auto copy_sf = [&](uint32_t col, uint32_t lo, int k_steps) {
#pragma unroll
            for (int pl = 0; pl < 2; ++pl)
#pragma unroll
                for (int kk = 0; kk < k_steps; ++kk)
                    tmem_cp_32x128b_warpx4(col + (pl * 2 + kk) * 4, desc_sf(lo + (uint32_t)((pl * 2 + kk) * kSfChunk >> 4)));
        };
        int s = 0, b = 0;                                            // stage, and accumulator (logits) or P buffer of the next tile
        uint32_t full = 0, freed = 1;                                 // their barriers' parities
        bool ok = true;
        if (warp == 1) {
            const uint32_t q_lo = desc_lo(base + S_::kOffQ), k_lo = desc_lo(base + S_::kOffK);
            const uint32_t sfq_lo = sf_lo(base + S_::kOffSfQ), sfk_lo = sf_lo(base + S_::kOffSfK);
            int slot = 0, ii = 0;                                    // scale factors in tensor memory
            for (int id = item_id(ii); id < n_items; id = item_id(++ii)) {
                const int T = tiles_of(item_m(id)) * kPhases;        // the tiles of all phases
                if (ok) ok = mbar_wait(&ctl->q_full, ii & 1, &ctl->abort, p.status);
                for (int j = 0; j < T; ++j) {
                    // S[b] = Q K^T of a key tile, four sign pairs x K steps of 64; as far ahead of the epilogue as there are
                    // accumulators
                    if (ok) ok = mbar_wait(&ctl->k_full[s], full, &ctl->abort, p.status);
                    if (ok) ok = mbar_wait(&ctl->s_empty[b], freed, &ctl->abort, p.status);   // (passes at once the first time)
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t kt = k_lo + (uint32_t)s * (kTileBytes >> 4), sfk = tmem + kColSfKV + slot * kSfStage;
                        if (j == 0) copy_sf(tmem + kColSfQ, sfq_lo, kQkSteps);
                        copy_sf(sfk, sfk_lo + (uint32_t)s * (kSfBytes >> 4), kQkSteps);
                        uint32_t acc = 0;
#pragma unroll
                        for (int pa = 0; pa < 2; ++pa)
#pragma unroll
                            for (int pw = 0; pw < 2; ++pw)
#pragma unroll
                                for (int kk = 0; kk < kQkSteps; ++kk) {
                                    mma_fp4_block16(tmem + kColS + b * 128, desc_sw64(q_lo + ((pa * kPlane + kk * 32) >> 4)),
                                                    desc_sw64(kt + ((pw * kPlane + kk * 32) >> 4)), idesc(128),
                                                    tmem + kColSfQ + (pa * 2 + kk) * 4, sfk + (pw * 2 + kk) * 4, acc);
                                    acc = 1;
                                }
                        mma_commit(&ctl->s_full[b]);
                        mma_commit(&ctl->k_empty[s]);
                        if (j == T - 1) mma_commit(&ctl->q_empty);   // the Q tile is free for the next item
                    }
                    __syncwarp();
                    if (++s == kKStages) s = 0, full ^= 1;
                    if (++b == kSBufs) b = 0, freed ^= 1;
                    if (++slot == kSfSlots) slot = 0;
                }
            }
        } else if (has_map(PASS)) {
            // O (+)= P V: P from the epilogue warps (shared memory + scale-factor chunks)
            const uint32_t p_lo = desc_lo(base + S_::kOffP), v_lo = desc_lo(base + S_::kOffV);
            const uint32_t sfp_lo = sf_lo(base + S_::kOffSfP), sfv_lo = sf_lo(base + S_::kOffSfV);
            int ii = 0;
            uint32_t p_full = 0;
            for (int id = item_id(ii); id < n_items; id = item_id(++ii)) {
                const int T = tiles_of(item_m(id));
                for (int j = 0; j < T; ++j) {
                    if (ok) ok = mbar_wait(&ctl->v_full[s], full, &ctl->abort, p.status);
                    // the previous item's O has been read out before it is overwritten
                    if (ok && j == 0 && ii > 0) ok = mbar_wait(&ctl->o_empty, (ii - 1) & 1, &ctl->abort, p.status);
                    if (ok) ok = mbar_wait(&ctl->p_full[b], p_full, &ctl->abort, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t vt = v_lo + (uint32_t)s * (kTileBytes >> 4), pt = p_lo + (uint32_t)b * (kPlane >> 4);
                        const uint32_t sfp = tmem + kColSfP + b * 8, sfv = tmem + kColSfKV + s * kSfStage + 16;
                        copy_sf(sfv, sfv_lo + (uint32_t)s * (kSfBytes >> 4), 2);
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) tmem_cp_32x128b_warpx4(sfp + kk * 4, desc_sf(sfp_lo + (uint32_t)((b * 2 + kk) * 512 >> 4)));
                        uint32_t acc = j == 0 ? 0u : 1u;
#pragma unroll
                        for (int pv = 0; pv < 2; ++pv)
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                mma_fp4_block16(tmem + kColO, desc_sw64(pt + ((kk * 32) >> 4)), desc_sw64(vt + ((pv * kPlane + kk * 32) >> 4)),
                                                idesc(HD), sfp + kk * 4, sfv + (pv * 2 + kk) * 4, acc);
                                acc = 1;
                            }
                        mma_commit(&ctl->v_empty[s]);
                        mma_commit(&ctl->p_empty[b]);
                        if (j == T - 1) mma_commit(&ctl->o_full);
                    }
                    __syncwarp();
                    if (++s == kStages) s = 0, full ^= 1;
                    if (++b == 2) b = 0, p_full ^= 1;
                }
            }
        }
    } else if (warp == 2) {
        // ---------------------------------------------------------------------------------- column factors
        int it = 0, ii = 0;
        bool ok = true;
        const float unit = PASS == kPassOrdered ? p.alpha : p.alpha * kLog2e;
        for (int id = item_id(ii); id < n_items; id = item_id(++ii)) {
            const int T = tiles_of(item_m(id));
            const int4* words = reinterpret_cast<const int4*>(p.k_words + p.k_row0 + (int64_t)(item_head(id) / p.kv_group) * p.Lp) + lane;
            for (int j = 0, jt = 0; j < T * kPhases; ++j, ++it, jt = jt + 1 == T ? 0 : jt + 1) {
                const int4 w = __ldg(words + jt * 32);
                auto factor = [&](int word) { return unit * __uint_as_float((uint32_t)(row_word_exp(word) + 127) << 23); };
                if (ok && it >= kKStages) ok = mbar_wait(&ctl->k_empty[it % kKStages], ((it / kKStages) - 1) & 1, &ctl->abort, p.status);
                if (!ok) continue;
                reinterpret_cast<float4*>(kc_all + (it % kKcRing) * 128)[lane] = make_float4(factor(w.x), factor(w.y), factor(w.z), factor(w.w));
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->k_full[it % kKStages]);
            }
        }
    } else if (warp >= kFirstEpi) {
        // ---------------------------------------------------------------------------------- epilogue
        // Warp e: group g = e / 8 (the key tiles whose global count is g modulo the groups), lane quarter
        // q = warp % 4 (its rows), half = (e / 4) % 2 of the tile's 128 keys: a thread owns one query row and two
        // 32-key groups (64 columns) of each of its group's tiles.  For reading out O every warp takes 32 columns.
        const int e = warp - kFirstEpi, q = warp & 3, grp = e >> 3, half = (e >> 2) & 1, cg_o = e >> 2;
        const int r = q * 32 + lane;                                 // row inside the item = tensor-memory lane
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        constexpr bool kShare = share_tiles(PASS);
        constexpr int kStep = kShare ? 1 : kGroups;
        int it = kShare ? 0 : grp, n = 0, it0 = 0, ii = 0;            // this warp's next tile, its tiles so far, the phase's first tile
        int mt0 = 0;                                                 // tiles of the map so far
        bool ok = true;
        float *max_s = reinterpret_cast<float*>(sm + S_::kOffMax), *sums_s = reinterpret_cast<float*>(sm + S_::kOffSums);
        auto exp2_approx = [](float y) {
            float v;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(y));
            return v;
        };
        for (int id = item_id(ii); id < n_items; id = item_id(++ii)) {
            const int h = item_head(id), m_blk = item_m(id);
            const int64_t m = (int64_t)m_blk * BM + r;                // query index inside the head
            const int64_t grow = (int64_t)h * p.Lp + m;              // row of the launch's stacked heads
            const int a_exp = row_word_exp(__ldg(p.q_words + p.q_row0 + grow));
            const float ra = __uint_as_float((uint32_t)(a_exp + 127) << 23);
            const int T = tiles_of(m_blk);
            // the row's statistics, merged from the partial results of the passes before in a fixed order: the exponent of
            // an element is u x row_unit + neg_mx
            float row_unit = ra, neg_mx = 0.f, inv = 0.f;
            int kmax = 0;
            if (PASS == kPassMapOnline) {
                const float4* pp = reinterpret_cast<const float4*>(p.part + grow * kParts);
                float4 a[kParts / 2];                                 // {max, sum, max, sum}
                float mx = -INFINITY, sum = 0.f;
#pragma unroll
                for (int i = 0; i < kParts / 2; ++i) {
                    a[i] = __ldg(pp + i);
                    mx = fmaxf(mx, fmaxf(a[i].x, a[i].z));
                }
#pragma unroll
                for (int i = 0; i < kParts / 2; ++i) {
                    sum += a[i].y * exp2f(a[i].x - mx);
                    sum += a[i].w * exp2f(a[i].z - mx);
                }
                inv = 1.0f / sum;
                neg_mx = -mx;
                // the row's largest element is 2^0 / sum: its group has the row's largest scale
                float ip, in;
                const uint32_t sc = cast::group_scales((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(inv)), ip, in);
                kmax = scale_key(sc & 0xFFu);
                if (p.p_words && h == 0 && (e >> 2) == 0) p.p_words[m] = row_word(kmax, kRowHasPos);
            }
            float run_mx = -INFINITY, run_sum = 0.f;                  // statistics: over this thread's columns of its tiles
            float part0 = 0.f, part1 = 0.f, part2 = 0.f, part3 = 0.f;  // ordered sums: by tile number modulo 4
            auto tiles = [&](auto phase) {
            constexpr int PHASE = decltype(phase)::value;
            for (; it < it0 + T; it += kStep, ++n) {
                const int j = it - it0, mt = mt0 + j, b = mt & 1;                   // number and buffer of P
                const uint32_t s_col = tq + kColS + (it % kSBufs) * 128;
                if (ok) ok = kShare ? mbar_wait(&ctl->s_full[it & 1], (it >> 1) & 1, &ctl->abort, p.status) : mbar_wait(&ctl->s_full[grp], n & 1, &ctl->abort, p.status);
                if (!ok) continue;
                tc_fence_after();
                // (the tile's column factors were stored before warp 2 arrived on the stage's barrier,
                // which the MMA warp waited for before it issued what s_full reports as complete)
                // u = accumulator x column factor: the logit (online: in base-2 units) up to the query row's power of two
                // ra, by which multiplying is exact: t = u ra.  (Packed fp32 pairs: same roundings as the
                // scalar operations, half the instructions.)
                uint32_t acc[32];
                uint64_t u2[16];
                const int cg0 = kShare ? e >> 2 : half * 2;
                auto release = [&] {                                  // both halves are in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->s_empty[it % kSBufs]);
                };
                auto scale_columns = [&](int cg) {
                    const ulonglong2* kc2 = reinterpret_cast<const ulonglong2*>(kc_all + (it % kKcRing) * 128 + cg * 32);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const ulonglong2 k2 = kc2[c];                 // four column factors
                        u2[2 * c] = cast::mul_f32x2(cast::pack_f32x2(acc[4 * c], acc[4 * c + 1]), k2.x);
                        u2[2 * c + 1] = cast::mul_f32x2(cast::pack_f32x2(acc[4 * c + 2], acc[4 * c + 3]), k2.y);
                    }
                    // the diagonal tile: keys after the query are masked; the last tile of a ragged sequence: keys past it
                    if (MASK != kMaskNone && j == (CAUSAL ? m_blk : T - 1)) {
                        const int n_local = (int)((CAUSAL ? m : p.L - 1) - (int64_t)j * BNK) - cg * 32;   // last visible column of this group
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            float lo, hi;
                            cast::unpack_f32x2(u2[c], lo, hi);
                            if (2 * c > n_local) lo = -INFINITY;
                            if (2 * c + 1 > n_local) hi = -INFINITY;
                            u2[c] = cast::pack_f32x2(__float_as_uint(lo), __float_as_uint(hi));
                        }
                    }
                };
                const uint64_t ra2 = cast::pack_f32x2(__float_as_uint(row_unit), __float_as_uint(row_unit));
                auto work = [&](int cg) {                             // one 32-key group, from u2
                    if (PHASE == kSum) {
                        const uint64_t nm2 = cast::pack_f32x2(__float_as_uint(neg_mx), __float_as_uint(neg_mx));
                        float sum = 0.f;                              // in the order of the keys
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            float t0, t1;
                            cast::unpack_f32x2(cast::fma_f32x2(u2[c], ra2, nm2), t0, t1);
                            sum += exp2_approx(t0);
                            sum += exp2_approx(t1);
                        }
                        // of every eight tiles those of one parity are numbers 0 .. 3: 0 + 2 and 1 + 3 first
                        const int i = j & 3;
                        part0 += i == 0 ? sum : 0.f;                  // (sums are not negative: adding zero changes nothing)
                        part1 += i == 1 ? sum : 0.f;
                        part2 += i == 2 ? sum : 0.f;
                        part3 += i == 3 ? sum : 0.f;
                    } else if (!is_map(PHASE)) {
                        float u[32];
#pragma unroll
                        for (int c = 0; c < 16; ++c) cast::unpack_f32x2(u2[c], u[2 * c], u[2 * c + 1]);
                        float c4[4] = {u[0], u[1], u[2], u[3]};
#pragma unroll
                        for (int c = 4; c < 32; ++c) c4[c & 3] = fmaxf(c4[c & 3], u[c]);
                        const float cm = fmaxf(fmaxf(c4[0], c4[1]), fmaxf(c4[2], c4[3]));
                        const float nmx = fmaxf(run_mx, cm * ra);
                        if (PHASE == kMax) {
                            run_mx = nmx;
                            return;
                        }
                        // 2^(-inf) = 0 on the first tile; a maximum still at -inf (everything masked so far) must
                        // not meet itself in a difference
                        const float ref = nmx == -INFINITY ? 0.f : nmx;
                        run_sum *= exp2_approx(run_mx - ref);
                        run_mx = nmx;
                        const uint64_t nref2 = cast::pack_f32x2(__float_as_uint(-ref), __float_as_uint(-ref));
                        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            float t0, t1;
                            cast::unpack_f32x2(cast::fma_f32x2(u2[c], ra2, nref2), t0, t1);
                            s4[(2 * c) & 3] += exp2_approx(t0);
                            s4[(2 * c + 1) & 3] += exp2_approx(t1);
                        }
                        run_sum += (s4[0] + s4[1]) + (s4[2] + s4[3]);
                    }
                };
                // The map, from u2: normalised and rounded to bf16 ...
                auto probabilities = [&](uint32_t (&w)[16]) {
                    const uint64_t nm2 = cast::pack_f32x2(__float_as_uint(neg_mx), __float_as_uint(neg_mx));
                    const uint64_t inv2 = cast::pack_f32x2(__float_as_uint(inv), __float_as_uint(inv));
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        float t0, t1, p0, p1;
                        cast::unpack_f32x2(cast::fma_f32x2(u2[c], ra2, nm2), t0, t1);
                        cast::unpack_f32x2(cast::mul_f32x2(cast::pack_f32x2(__float_as_uint(exp2_approx(t0)),
                                                                            __float_as_uint(exp2_approx(t1))), inv2), p0, p1);
                        const __nv_bfloat162 pr = __floats2bfloat162_rn(p0, p1);
                        w[c] = *reinterpret_cast<const uint32_t*>(&pr);
                    }
                };
                // ... and a 32-key group of it cast (P has no negative element: one plane) and stored
                struct Codes { uint32_t nib[4], up, sc; };
                auto codes_of = [&](const uint32_t (&w)[16]) {
                    Codes c;
                    c.sc = cast_group(w, scale_tab, (15 - kmax) * 8, c.nib, c.up);
                    return c;
                };
                auto store = [&](int cg, const Codes& c, const uint32_t (&w)[16]) {
                    // plane: row r, 16-byte piece cg of its 64 bytes, 64-byte swizzle; scale factors: chunk of the
                    // K step cg / 2, byte (r % 32) * 16 + (r / 32) * 4 + (cg % 2) * 2, each scale twice (blocks of 16)
                    *reinterpret_cast<uint4*>(sm + S_::kOffP + b * kPlane + r * 64 + ((cg ^ ((r >> 1) & 3)) << 4)) =
                        make_uint4(c.nib[0], c.nib[1], c.nib[2], c.nib[3]);
                    *reinterpret_cast<uint16_t*>(sm + S_::kOffSfP + (b * 2 + (cg >> 1)) * 512 + (r & 31) * 16 + (r >> 5) * 4 +
                                                 (cg & 1) * 2) = (uint16_t)(c.up * 257u);
                    if (PHASE == kMapOnline && p.p_plane && h == 0) {                    // verification outputs (head 0 of the launch)
                        const int64_t g = (int64_t)j * 4 + cg, v = m * (p.L / 32) + g;
                        p.p_plane[v] = make_uint4(c.nib[0], c.nib[1], c.nib[2], c.nib[3]);
                        *reinterpret_cast<uint16_t*>(p.p_sf + sf_row_offset(m, p.p_nk64) + sf_group_offset((int)g)) = (uint16_t)(c.up * 257u);
                        if (p.p_codes) p.p_codes[v] = make_uint4(c.nib[0], c.nib[1], c.nib[2], c.nib[3]);
                        if (p.p_scales) p.p_scales[v] = (uint16_t)c.sc;
                        if (p.p_bits) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) p.p_bits[v * 4 + i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
                        }
                    }
                };
                auto p_free = [&] {                                   // the previous P in this buffer has been multiplied
                    if (ok && mt >= 2) ok = mbar_wait(&ctl->p_empty[b], ((mt >> 1) - 1) & 1, &ctl->abort, p.status);
                    return ok;
                };
                tmem_ld32(s_col + cg0 * 32, acc);
                tmem_ld_wait();
                if constexpr (kShare) {
                    release();
                    scale_columns(cg0);
                    if constexpr (is_map(PHASE)) {
                        uint32_t w[16];
                        probabilities(w);
                        const Codes c = codes_of(w);
                        if (p_free()) store(cg0, c, w);
                    } else work(cg0);
                } else {
                    // two epilogue groups have the registers to take the second key group before they work on the first, which
                    // frees the accumulator early (32 heads x 8192: 2001 -> 1981 us); three have not
                    scale_columns(cg0);
                    if (kGroups == 3) work(cg0);
                    if constexpr (is_map(PHASE)) {
                        uint32_t acc1[32], w0[16], w1[16];
                        tmem_ld32(s_col + (cg0 + 1) * 32, acc1);
                        tmem_ld_wait();
                        release();
                        probabilities(w0);
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[i] = acc1[i];
                        scale_columns(cg0 + 1);
                        probabilities(w1);
                        const Codes c0 = codes_of(w0), c1 = codes_of(w1);
                        if (p_free()) {
                            store(cg0, c0, w0);
                            store(cg0 + 1, c1, w1);
                        }
                    } else {
                        tmem_ld32(s_col + (cg0 + 1) * 32, acc);
                        tmem_ld_wait();
                        release();
                        if (kGroups == 2) work(cg0);
                        scale_columns(cg0 + 1);
                        work(cg0 + 1);
                    }
                }
                const int last = (1 << p.sum_shift) - 1;
                if (PHASE == kSum && ((j & last) == last || j + 1 == T)) {   // the last tile of the block
                    float* sp = sums_s + ((j >> p.sum_shift) * kSumParts + cg0) * 128 + r;
                    sp[0] = part0 + part2;
                    sp[4 * 128] = part1 + part3;
                    part0 = part1 = part2 = part3 = 0.f;
                }
                if (is_map(PHASE)) {
                    fence_proxy_async();                              // visible to the tensor core's reads
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->p_full[b]);
                }
            }
            it0 += T;
            if (is_map(PHASE)) mt0 += T;
            };
            if constexpr (PASS == kPassOrdered) {
                // What the threads of a row found goes through shared memory between the phases.  (What they write next they
                // write after the other barrier, when all have read.)
                auto meet = [] { asm volatile("bar.sync 1, %0;" ::"n"(8 * kGroups * 32) : "memory"); };
                tiles(std::integral_constant<int, kMax>{});
                max_s[cg_o * 128 + r] = run_mx;
                meet();
                float mx = max_s[r];
#pragma unroll
                for (int i = 1; i < 4; ++i) mx = fmaxf(mx, max_s[i * 128 + r]);
                row_unit = ra * kLog2e;
                neg_mx = softmax::neg_max_log2e(mx);
                tiles(std::integral_constant<int, kSum>{});
                meet();
                // the stored path's order: over 32 groups a tree by strides 16, 8, 4, 2, 1 (the first two inside `sums_s`), then
                // along the row
                float sum = 0.f;
                const float* sp = sums_s + r;
                for (int t0 = 0; t0 < T; t0 += 1 << p.sum_shift, sp += kSumParts * 128) {
                    float c[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        c[i] = sp[i * 128];
                        if (t0 + 1 < T) c[i] += sp[(4 + i) * 128];
                    }
                    sum += (c[0] + c[2]) + (c[1] + c[3]);
                }
                inv = 1.0f / sum;
                // the group of the row's largest element has the row's largest scale (one bf16 step above: the
                // approximate exponential is not promised to be monotonic)
                float ip, in;
                const uint32_t top = __bfloat16_as_ushort(__float2bfloat16_rn(softmax::exp_rel(mx, neg_mx) * inv));
                kmax = scale_key(cast::group_scales(top + 1, ip, in) & 0xFFu);
                tiles(std::integral_constant<int, kMapOrdered>{});
            } else if constexpr (PASS == kPassStats) {
                tiles(std::integral_constant<int, kStats>{});
                if (ok) p.part[grow * kParts + grp * 2 + half] = make_float2(run_mx, run_sum);
            } else tiles(std::integral_constant<int, kMapOnline>{});
            if (has_map(PASS) && e < kOWarps) {
                // O of the item: rows x (32 columns of the head dimension per thread), rescaled by 2^(row offset of P
                // + row offset of V^T) - exact - and stored
                if (ok) ok = mbar_wait(&ctl->o_full, ii & 1, &ctl->abort, p.status);
                if (!ok) continue;
                tc_fence_after();
                constexpr int kCols = HD / 4;                          // columns of O per warp
                uint32_t acc[kCols];
                if constexpr (HD == 128) tmem_ld32(tq + kColO + cg_o * kCols, acc);
                else tmem_ld16(tq + kColO + cg_o * kCols, acc);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->o_empty);
                const int4* vw = reinterpret_cast<const int4*>(p.v_words + p.v_row0 + (int64_t)(h / p.kv_group) * kVRows + cg_o * kCols);
                float* out = p.O + ((int64_t)h * p.L + m) * HD + cg_o * kCols;
                const int p_exp = kmax ? kmax - 25 : 0;
                if (MASK == kMaskNone || m < p.L) {
#pragma unroll
                    for (int c = 0; c < kCols / 4; ++c) {
                        const int4 w4 = __ldg(vw + c);
                        const int ex[4] = {row_word_exp(w4.x), row_word_exp(w4.y), row_word_exp(w4.z), row_word_exp(w4.w)};
                        float f[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int sh = min(127, max(-126, p_exp + ex[i]));
                            f[i] = __uint_as_float(acc[4 * c + i]) * __uint_as_float((uint32_t)(sh + 127) << 23);
                        }
                        if (p.vec_o) *reinterpret_cast<float4*>(out + 4 * c) = make_float4(f[0], f[1], f[2], f[3]);
                        else {
#pragma unroll
                            for (int i = 0; i < 4; ++i) out[4 * c + i] = f[i];
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
    // As the last thing: the next launch's blocks then find all SMs free, instead of crowding on those that ended first.
    grid_launch_dependents();
}

template <int PASS, int MASK, int HD>
int launch_pass(const Maps& maps, const Params& p, int dev, int sms,
                cudaStream_t st) {
    static bool configured[64] = {};
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(attention_fp4_kernel<PASS, MASK, HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<PASS>::kBytes) !=
            cudaSuccess) {
            cudaGetLastError();
            return AMX_ERR_CUDA;
        }
        configured[dev] = true;
    }
    const int items = p.heads * p.m_tiles;
    // Chained up to about 350 us.  The whole call, ordinary / chained: 32 heads of 128, 1536 keys 120.0 / 116.5 us, 2048 185.3 / 180.2,
    // 2560 262 / 260, 3072 353.7 / 354.4, 6144 1127 / 1132, causal 2048 130 / 125, 3072 225.6 / 221.7, 4096 351.5 / 346.2; of 64: 2560
    // 271.7 / 269.6, 4096 562.8 / 560.3.
    const double work = (double)p.heads * (double)p.L * (double)p.L * HD / (MASK == kMaskCausal ? 2.0 : 1.0);
    return launch_chained(work <= 3.6e10, attention_fp4_kernel<PASS, MASK, HD>, (unsigned)(items < sms ? items : sms), threads(PASS),
                          Smem<PASS>::kBytes, st, maps.q, maps.k, maps.v, maps.sfq, maps.sfk, maps.sfv, p);
}

}  // namespace

bool attn_fused_supported(int64_t L, int64_t d) {
    return (d == 128 || d == 64) && L > 0 && L % 32 == 0 && L / BNK <= 32766;
}

int64_t attn_fused_padded(int64_t L) { return (L + BM - 1) / BM * BM; }

// per-row partial softmax statistics of the heads of one launch
size_t attn_fused_scratch_bytes(int64_t heads, int64_t L, bool ordered) {
    return ordered ? 0 : up256((size_t)(heads * attn_fused_padded(L)) * kParts * sizeof(float2));
}

namespace {
template <int MASK, int HD>
int launch_ordered(const Maps& maps, const Params& p, int dev, int sms,
                   cudaStream_t st) {
    return launch_pass<kPassOrdered, MASK, HD>(maps, p, dev, sms, st);
}
template <int MASK>
int launch_online(const Maps& maps, const Params& p, int dev, int sms,
                  cudaStream_t st) {
    const int rc = launch_pass<kPassStats, MASK, 128>(maps, p, dev, sms, st);
    return rc != AMX_OK ? rc : launch_pass<kPassMapOnline, MASK, 128>(maps, p, dev, sms, st);
}
template <int HD>
int launch_mask(int mask, const Maps& maps, const Params& p, int dev,
                int sms, cudaStream_t st) {
    return mask == kMaskCausal ? launch_ordered<kMaskCausal, HD>(maps, p, dev, sms, st)
         : mask == kMaskTail   ? launch_ordered<kMaskTail, HD>(maps, p, dev, sms, st)
                               : launch_ordered<kMaskNone, HD>(maps, p, dev, sms, st);
}
}  // namespace

// Attention for `heads` stacked heads whose operands were prepared ahead, Lp = attn_fused_padded(L) rows per head: q
// (left-hand layout, K = d), k (right-hand layout), vt (right-hand layout, 128 rows of V^T per head, K = L).  O: fp32
// [heads][L][d].  workspace: 256 bytes (status word).  ordered: the form of the statistics (see above); the online form takes
// head dimension 128 and whole blocks only, and has the dbg_* outputs for head 0 (verification, see Params).
int attn_fused(const Fp4Operand& q, const Fp4Operand& k, const Fp4Operand& vt, int heads, int64_t L, int64_t d, float alpha,
               int causal, bool ordered, void* scratch, float* O, void* workspace, cudaStream_t st, void* dbg_bits, uint8_t* dbg_codes,
               uint8_t* dbg_scales, void* dbg_prepared, int kv_group, const int* gate) {
    if (!attn_fused_supported(L, d) || (!ordered && (d != 128 || L % BNK)) || heads <= 0 || q.row0 % 128 || k.row0 % 128 || vt.row0 % 128) return AMX_ERR_SHAPE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return AMX_ERR_CUDA;
    static int sm_count[64] = {};
    if (!sm_count[dev] && cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return AMX_ERR_CUDA;
    const OperandLayout oq = operand_layout(q.layout_rows, d, 128), ok_ = operand_layout(k.layout_rows, d, 256),
                        ov = operand_layout(vt.layout_rows, L, 256);
    const uint8_t* pq = static_cast<const uint8_t*>(q.prepared);
    const uint8_t* pk = static_cast<const uint8_t*>(k.prepared);
    const uint8_t* pv = static_cast<const uint8_t*>(vt.prepared);
    Maps maps;
    if (!make_map(&maps.q, pq, q.rows_total, d, oq.plane, 128, 64) || !make_map(&maps.k, pk, k.rows_total, d, ok_.plane, 128, 64) ||
        !make_map(&maps.v, pv, vt.rows_total, L, ov.plane, 128, 64) || !make_sf_map(&maps.sfq, pq, oq, 2, 1, 2) ||
        !make_sf_map(&maps.sfk, pk, ok_, 2, 1, 2) || !make_sf_map(&maps.sfv, pv, ov, 2, 1, 2))
        return AMX_ERR_CUDA;
    int* status = static_cast<int*>(workspace);              // cleared by the caller
    Params p{};
    p.q_words = reinterpret_cast<const int*>(pq + 2 * oq.plane + 2 * oq.sf);
    p.k_words = reinterpret_cast<const int*>(pk + 2 * ok_.plane + 2 * ok_.sf);
    p.v_words = reinterpret_cast<const int*>(pv + 2 * ov.plane + 2 * ov.sf);
    p.q_row0 = q.row0; p.k_row0 = k.row0; p.v_row0 = vt.row0;
    p.heads = heads; p.Lp = attn_fused_padded(L); p.m_tiles = (int)(p.Lp / BM); p.gate = gate;
    p.kv_group = kv_group > 0 ? kv_group : 1;
    p.L = L; p.alpha = alpha;
    p.part = static_cast<float2*>(scratch);
    p.sum_shift = sum_shift(p.m_tiles);
    p.O = O;
    p.vec_o = aligned(O, 16);
    p.status = status;
    if (dbg_prepared) {
        const OperandLayout op = operand_layout(L, L, 128);
        uint8_t* pp = static_cast<uint8_t*>(dbg_prepared);
        p.p_plane = reinterpret_cast<uint4*>(pp);
        p.p_sf = pp + 2 * op.plane;
        p.p_words = reinterpret_cast<int*>(pp + 2 * op.plane + 2 * op.sf);
        p.p_nk64 = op.nk64;
        p.p_bits = static_cast<uint4*>(dbg_bits);
        p.p_codes = reinterpret_cast<uint4*>(dbg_codes);
        p.p_scales = reinterpret_cast<uint16_t*>(dbg_scales);
    }
    if (!ordered) return causal ? launch_online<kMaskCausal>(maps, p, dev, sm_count[dev], st)
                                : launch_online<kMaskNone>(maps, p, dev, sm_count[dev], st);
    const int mask = causal ? kMaskCausal : L % BNK ? kMaskTail : kMaskNone;
    return d == 128 ? launch_mask<128>(mask, maps, p, dev, sm_count[dev], st)
                    : launch_mask<64>(mask, maps, p, dev, sm_count[dev], st);
}

}  // namespace amx
