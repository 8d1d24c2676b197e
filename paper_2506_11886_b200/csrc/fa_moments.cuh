// What the kernels that work on block moments share (fa_compress_mom.cu: from tokens to coefficients; fa_select_mom.cu: back).
// Within a block of R tokens, t in [-1, 1] across it and phi_n = pi n R / T,
//   e^{i phi t} = sum_r (2 r + 1) i^r j_r(phi) P_r(t),  r < 32 for R <= 6 T / k.
#pragma once

#include "fa_umma.cuh"

namespace fa {
namespace mom {

using bf16 = __nv_bfloat16;
using namespace umma;

constexpr int kMF = 32;              // moments per block
constexpr int kChunk = 64;           // tokens per box and pipeline stage
constexpr int kMaxBlockTokens = 768;
__host__ __device__ inline int blocks_of(int n_mid, int R) { return (n_mid + R - 1) / R; }
// The longest block of a layout: a whole number of boxes, k R <= 6 T.
inline int block_tokens(const Dims& s) {
    const long long r = 6LL * s.T / s.k / kChunk * kChunk;
    return (int)(r > kMaxBlockTokens ? kMaxBlockTokens : r);
}

__device__ __forceinline__ void split_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// (2 r + 1) j_r(phi_n) for r = NR tq .. NR tq + NR - 1
template <int NR>
__device__ __forceinline__ void legendre_factors(unsigned n, int R, int T, int tq, float (&gb)[NR]) {
    // j_r by the recurrence downward from r = 10 + 2.4 phi (55 at most: far enough past phi that what is left out is
    // below 1e-9, near enough that the values stay in range), scaled by the closed form of j_0 or j_1, whichever is larger
    float keep[NR], sn, cs, jn = 0.f, jc = 0.f, j0 = 1.f, j1 = 0.f;
#pragma unroll
    for (int i = 0; i < NR; ++i) keep[i] = 0.f;
    const double invd = n ? (double)T / (3.14159265358979324 * (double)(n * (unsigned)R)) : 0.0;      // 1 / phi: fp32's rounding of it adds up
    const float x = (float)(n * (unsigned)R) / (float)T, inv = (float)invd;
    const int top = min(55, 10 + (int)(7.54f * x));
#pragma unroll 1
    for (int r8 = 48; r8 >= 0 && n; r8 -= 8) {
#pragma unroll
        for (int i = 7; i >= 0; --i) {         // jc = j_r, jn = j_{r + 1}
            const int r = r8 + i;
            if (r == top) jc = 1e-20f;
#pragma unroll
            for (int u = 0; u < NR; u += 8)
                if (r8 == NR * tq + u) keep[u + i] = (float)(2 * r + 1) * jc;
            if (i == 1) j1 = jc;
            if (i == 0) j0 = jc;
            const float jp = fmaf((float)((double)(2 * r + 1) * invd), jc, -jn);
            jn = jc;
            jc = jp;
        }
    }
    sincospif(x, &sn, &cs);
    const float t0 = sn * inv, t1 = (t0 - cs) * inv, sc = fabsf(t0) > fabsf(t1) ? t0 / j0 : t1 / j1;
#pragma unroll
    for (int i = 0; i < NR; ++i) gb[i] = n ? keep[i] * sc : (i == 0 && tq == 0 ? 1.f : 0.f);
}

// 4-D view (dim, head, token, batch) of a prefilled K or V with element strides (1, sh, st, sb); box = box_dims dims x 64 tokens.
inline bool prefill_map(CUtensorMap* tm, const void* base, const Dims& s, int64_t sb, int64_t st, int64_t sh, int L, int box_dims = 64,
                        CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)s.d, (cuuint64_t)s.Hkv, (cuuint64_t)L, (cuuint64_t)s.B};
    cuuint64_t strides[3] = {(cuuint64_t)sh * 2, (cuuint64_t)st * 2, (cuuint64_t)(s.B > 1 ? sb : st * (int64_t)L) * 2};
    cuuint32_t box[4] = {(cuuint32_t)box_dims, 1, (cuuint32_t)kChunk, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace mom
}  // namespace fa
