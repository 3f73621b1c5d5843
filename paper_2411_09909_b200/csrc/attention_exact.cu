// Fully quantized attention on CUDA cores, exact for any scale range: what runs instead of the fused FP4 kernel when
// casting Q, K or V met a scale that kernel cannot represent (see to_ue4m3: 15 or more binades below its row's largest).
// The decision is taken on the device, from the count the casts leave in the workspace; without such a scale - every
// input but adversarial ones - the launch returns at once.  Same arithmetic as everywhere: products of exactly decoded
// values with fp32 accumulation, softmax in fp32 by softmax_math.cuh's expressions and order of additions, the normalised map
// rounded to bf16 and cast with groups of 32 keys.
//
// A block owns 16 query rows of one head: their logits stay in shared memory as fp32, are normalised, cast and decoded
// again in place, and multiplied with V.  Nothing is tuned: it runs where correctness needs it.  The launch has as many blocks as
// fit the GPU at once, which walk over the items: a block per item, 2112 of them for 32 heads x 1056, took 3 us longer to return.
#include <cuda_bf16.h>

#include <algorithm>

#include "cast_math.cuh"
#include "gemm.cuh"
#include "softmax_math.cuh"

namespace amx {
namespace {

constexpr int kRows = 16, kThreads = 256, kKeys = 64, kSmCount = 148;

__device__ __forceinline__ float code_value(uint32_t c, float sp, float sn) {
    const float mag = e2m1_mag_to_float(c & 7u);
    return (c & 8u) ? -(mag * sn) : mag * sp;
}
// Element k of operand row `row` (K elements per row).
__device__ __forceinline__ float element(const ExactOperand& o, int64_t row, int64_t K, int64_t k) {
    const int64_t byte = row * (K / 2) + k / 2;
    const uint32_t c = ((uint32_t)__ldg(o.pos + byte) | __ldg(o.neg + byte)) >> (4 * (k & 1));
    const uint8_t* s = o.scales + (row * (K / 32) + k / 32) * 2;
    return code_value(c & 15u, e5m2_to_float(__ldg(s)), e5m2_to_float(__ldg(s + 1)));
}

__global__ void __launch_bounds__(kThreads)
attention_exact_kernel(const ExactOperand q, const ExactOperand k, const ExactOperand v, int64_t L, int64_t Lp, int d, int kv_group,
                       float alpha, int causal, float* __restrict__ O, const int* __restrict__ run_if_nonzero, int heads) {
    begin_kernel();
    if (*run_if_nonzero == 0) return;
    extern __shared__ float sm[];
    float* S = sm;                                   // [16][L]
    float* Qs = S + kRows * L;                       // [16][d]
    float* Ts = Qs + kRows * d;                      // [64 keys][d + 1]
    const int64_t row_blocks = (L + kRows - 1) / kRows;
    for (int64_t item = blockIdx.x; item < row_blocks * heads; item += gridDim.x) {
        const int head = (int)(item / row_blocks), kv = head / kv_group;
        const int64_t m0 = item % row_blocks * kRows, seen = causal ? min(L, m0 + kRows) : L;
        for (int i = threadIdx.x; i < kRows * d; i += kThreads)
            Qs[i] = m0 + i / d < L ? element(q, head * Lp + m0 + i / d, d, i % d) : 0.f;
        for (int64_t k0 = 0; k0 < seen; k0 += kKeys) {
            __syncthreads();
            for (int i = threadIdx.x; i < kKeys * d; i += kThreads)
                Ts[i / d * (d + 1) + i % d] = k0 + i / d < L ? element(k, kv * Lp + k0 + i / d, d, i % d) : 0.f;
            __syncthreads();
            const int r = threadIdx.x / 16, c = threadIdx.x % 16;
            for (int j = c; j < kKeys && k0 + j < seen; j += 16) {
                float acc = 0.f;
                for (int x = 0; x < d; ++x) acc = fmaf(Qs[r * d + x], Ts[j * (d + 1) + x], acc);
                S[r * L + k0 + j] = alpha * acc;
            }
        }
        __syncthreads();
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int r = warp; r < kRows; r += kThreads / 32) {
            float* s = S + r * L;
            const int64_t vis = causal ? min(L, m0 + r + 1) : L;
            float mx = -INFINITY, sum = 0.f;
            for (int64_t i = lane; i < vis; i += 32) mx = fmaxf(mx, s[i]);
            for (int x = 16; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, x));
            const float nm = softmax::neg_max_log2e(mx);
            for (int64_t g0 = 0; g0 < L / 32; g0 += 32) {            // keys in order within a group, a tree over 32 groups
                float part = 0.f;
                for (int64_t a = (g0 + lane) * 32; a < min(vis, (g0 + lane + 1) * 32); ++a) part += softmax::exp_rel(s[a], nm);
                for (int x = 16; x > 0; x >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, x);
                sum += part;
            }
            const float inv = 1.0f / sum;
            for (int64_t g = lane; g < L / 32; g += 32) {            // a lane per group of 32 keys
                uint32_t w[16], nib[4];
                for (int i = 0; i < 16; ++i) {
                    const int64_t a = g * 32 + 2 * i;
                    const __nv_bfloat162 h = __floats2bfloat162_rn(a < vis ? softmax::exp_rel(s[a], nm) * inv : 0.f,
                                                                   a + 1 < vis ? softmax::exp_rel(s[a + 1], nm) * inv : 0.f);
                    w[i] = *reinterpret_cast<const uint32_t*>(&h);
                }
                const float sc = e5m2_to_float(cast::cast_nonneg_group(w, nib));
                for (int i = 0; i < 32; ++i) s[g * 32 + i] = code_value(nib[i >> 3] >> (4 * (i & 7)) & 15u, sc, sc);
            }
        }
        float acc[8] = {};                                           // dims c, c + 16, ...
        for (int64_t k0 = 0; k0 < (seen + 31) / 32 * 32; k0 += kKeys) {
            __syncthreads();
            for (int i = threadIdx.x; i < kKeys * d; i += kThreads) {
                const int key = i % kKeys, x = i / kKeys;
                Ts[key * (d + 1) + x] = k0 + key < L ? element(v, (int64_t)kv * 128 + x, L, k0 + key) : 0.f;
            }
            __syncthreads();
            const int r = threadIdx.x / 16, c = threadIdx.x % 16;
            for (int j = 0; j < kKeys && k0 + j < L; ++j) {
                const float pv = S[r * L + k0 + j];
                for (int x = 0; x < d / 16; ++x) acc[x] = fmaf(pv, Ts[j * (d + 1) + c + 16 * x], acc[x]);
            }
        }
        const int r = threadIdx.x / 16, c = threadIdx.x % 16;
        if (m0 + r < L)
            for (int x = 0; x < d / 16; ++x) O[((int64_t)head * L + m0 + r) * d + c + 16 * x] = acc[x];
        __syncthreads();                             // before the next item's rows
    }
}

size_t smem_bytes(int64_t L, int64_t d) { return ((size_t)kRows * L + (size_t)kRows * d + (size_t)kKeys * (d + 1)) * 4; }

}  // namespace

bool attn_exact_supported(int64_t L, int64_t d) { return (d == 64 || d == 128) && L % 32 == 0 && smem_bytes(L, d) <= 227 * 1024; }

int attn_exact(const ExactOperand& q, const ExactOperand& k, const ExactOperand& vt, int heads, int64_t L, int64_t d, int kv_group,
               float alpha, int causal, float* O, const int* run_if_nonzero, cudaStream_t st) {
    if (!attn_exact_supported(L, d) || heads > 65535) return AMX_ERR_SHAPE;
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return AMX_ERR_CUDA;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(attention_exact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) {
            cudaGetLastError();
            return AMX_ERR_CUDA;
        }
        configured[dev] = true;
    }
    const int64_t items = (L + kRows - 1) / kRows * heads, resident = std::min<int64_t>(4, (int64_t)(228 * 1024 / (smem_bytes(L, d) + 1024)));
    return launch(attention_exact_kernel, (unsigned)std::min(items, resident * kSmCount), kThreads, smem_bytes(L, d), st, q, k, vt, L,
                  attn_fused_padded(L), (int)d, kv_group, alpha, causal, O, run_if_nonzero, heads);
}

}  // namespace amx
