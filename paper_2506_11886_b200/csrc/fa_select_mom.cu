// fa_select_dims (Sec. 3.4) by block moments: the middle tokens rebuilt from the coefficients of every dimension over an axis R / 32
// times shorter than the coefficient axis, and the squared error against the prefill summed per dimension.
//
// The expansion of fa_moments.cuh read the other way: within a block of R tokens x~(t) = sum_{r < 32} P_r(t) y[r], with
//   y[r] = sum_n Re(F_n e^{i theta n d} i^r (2 r + 1) j_r(phi_n)),  F_n = w_n conj(C_n) e^{i theta n m} = a_n + i b_n,
// m the middle of the row and d the block's distance from it.  Blocks at +d and -d share the basis: with Pa = sum_n Re(e^{i theta n d} i^r g_r) a_n and
// Pb = sum_n Im(..) b_n,  y(+d) = Pa - Pb  and  y(-d) = (-1)^r (Pa + Pb).
//   1. rotate_kernel: a, b as two bf16 numbers each, laid out as the products want them; the factors g_r(n).
//   2. expand_kernel (tcgen05): 128 rows = 32 moments of four pairs of blocks, 2 d columns (K and V dims of a head), contraction over n.
//   3. residual_kernel (tcgen05): one pass over the prefill.  P times y per 64 tokens into tensor memory, lanes dims, columns tokens; the boxes of
//      the prefill come in by TMA beside it and a lane sums the squares of its dim's differences.
// All factors carry 2^-17 (two bf16 numbers, three products), where the direct reconstruction (fa_select_tc.cu) rounds basis and coefficients
// to bf16: the floor under the reported errors falls from 1e-6 to 1e-9 of a dimension's mean square.
// What bounds it: the third kernel HBM and the shared-memory reads of its differences (31 us for the 134 MB of 8 heads, 32 K tokens), the second its
// loads (every tile of four pairs reads all of a head's a and b: 92 MB through L2) beside 24.6 K cycles of products on 88 SMs (30 us).  The whole
// selection of that prompt, 1024 coefficients: 246 us with the reconstruction over coefficient rows (166 of them), 131 us here.
#include "fa_moments.cuh"

namespace fa {
namespace {

using namespace mom;

constexpr int kPairs = 4;              // pairs of blocks to a tile of the second kernel
constexpr int kKn = 16;                // frequencies per stage
constexpr int kBoxB = kKn * 128;       // [16 frequencies x 64 dims]
constexpr int kTileA = 128 * 128;      // [128 rows x (Re hi, Re lo, Im hi, Im lo of the 16)]
constexpr int kBoxY = 32 * 128;        // [32 moments x 64 dims]
constexpr int kGenWarpsE = 8;
constexpr int kThreadsE = 64 + 32 * kGenWarpsE;
constexpr int kStagesE = 4;
constexpr int kBoxX = 128 * kChunk * 2;        // [64 tokens x 64 dims] twice
constexpr int kTileP = kChunk * 128;           // [64 tokens x (32 hi, 32 lo)]
constexpr int kTileY = 16384;                  // hi, lo x two halves of 64 dims x [32 moments x 64 dims]
constexpr int kYStages = 2, kAccR = 8 /* (a multiple of the sets) */, kErrSets = 4, kErrWarps = 4 * kErrSets;
constexpr int kThreadsR = 64 + 32 * kErrWarps;

// Sizes of one call.
struct SelPlan {
    int R, n_blk, n_pair, nbx;         // tokens to a block, blocks of a row and pairs of them, 64-dim boxes of a head's K and V
    const float* coef_k;
    const float* coef_v;
    char* ab;                          // [B][Hkv][k / 16][a hi, a lo, b hi, b lo][nbx][16][128 bytes, 128-byte swizzle]
    float* g;                          // [32][k]
    char* y;                           // [B][n_blk][Hkv][nbx / 2][hi, lo][2][32][128 bytes, 128-byte swizzle]
};

// One thread per (frequency, eight dims) of a (batch row, head); the first blocks of the grid make the factors, a warp's worth each (their
// recurrence is one long chain).
__global__ void __launch_bounds__(256) rotate_kernel(Dims s, SelPlan p, int n_fac) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x < n_fac) {
        const int n = (int)blockIdx.x * 32 + threadIdx.x;
        if (threadIdx.x < 32 && n < s.k) {
            float g[kMF];
            legendre_factors<kMF>((unsigned)n, p.R, s.T, 0, g);
#pragma unroll
            for (int r = 0; r < kMF; ++r) p.g[(size_t)r * s.k + n] = g[r];
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int ch = p.nbx * 8;                              // pieces of eight dims of a head: 16 or 32
    const size_t i = (size_t)((int)blockIdx.x - n_fac) * 256 + threadIdx.x;
    const int c = (int)(i % ch), bx = c >> 3, q = c & 7;
    const size_t hn = i / ch;
    const int n = (int)(hn % s.k);
    const size_t bh = hn / s.k;
    asm volatile("griddepcontrol.wait;" ::: "memory");    // the coefficients
    if (bh >= (size_t)s.B * s.Hkv) return;
    const int side = bx >= p.nbx / 2, d0 = (bx - side * (p.nbx / 2)) * 64 + 8 * q;
    const float* src = (side ? p.coef_v : p.coef_k) + (bh * s.M + 2 * n) * (size_t)s.d + d0;
    const unsigned T2 = 2u * (unsigned)s.T;
    float sn, cs;
    sincospif((float)(((unsigned)n * (unsigned)(p.n_blk * p.R - 1)) % T2) / (float)s.T, &sn, &cs);
    const float w0 = recon_weight(s.norm, 2 * n, s.k, s.T), w1 = recon_weight(s.norm, 2 * n + 1, s.k, s.T);
    float re[8], im[8];
    *reinterpret_cast<float4*>(re) = *reinterpret_cast<const float4*>(src);
    *reinterpret_cast<float4*>(re + 4) = *reinterpret_cast<const float4*>(src + 4);
    *reinterpret_cast<float4*>(im) = *reinterpret_cast<const float4*>(src + s.d);
    *reinterpret_cast<float4*>(im + 4) = *reinterpret_cast<const float4*>(src + s.d + 4);
    uint32_t o[4][4];                                      // a hi, a lo, b hi, b lo
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float a[2], b[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const float x = w0 * re[2 * u + v], z = w1 * im[2 * u + v];
            a[v] = x * cs + z * sn;
            b[v] = x * sn - z * cs;
        }
        split_bf16(a[0], a[1], o[0][u], o[1][u]);
        split_bf16(b[0], b[1], o[2][u], o[3][u]);
    }
    char* dst = p.ab + (bh * (s.k / kKn) + n / kKn) * (size_t)(4 * p.nbx * kBoxB) + bx * kBoxB + (n % kKn) * 128 + ((q ^ (n & 7)) << 4);
#pragma unroll
    for (int m = 0; m < 4; ++m) *reinterpret_cast<uint4*>(dst + (size_t)m * p.nbx * kBoxB) = make_uint4(o[m][0], o[m][1], o[m][2], o[m][3]);
}

// grid (tiles of four pairs, Hkv, B).
template <int D>
__global__ void __launch_bounds__(kThreadsE, 1) expand_kernel(Dims s, SelPlan p, int32_t* status) {
    constexpr int N = 2 * D, kNbx = N / 64, kB = 4 * kNbx * kBoxB, kStage = kTileA + kB;
    // A K-major, B MN-major
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    extern __shared__ unsigned char smem_unaligned[];
    unsigned char* smem = smem_unaligned + ((1024u - (smem_u32(smem_unaligned) & 1023u)) & 1023u);
    unsigned char* stage0 = smem;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStagesE * kStage);
    uint64_t* empty = full + kStagesE;
    uint64_t* acc_ready = empty + kStagesE;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_ready + 1);
    volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int p0 = blockIdx.x * kPairs, h = blockIdx.y, b = blockIdx.z, n_k = s.k / kKn;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int i = 0; i < kStagesE; ++i) { mbar_init(full + i, kGenWarpsE / kStagesE + 1); mbar_init(empty + i, 1); }
        mbar_init(acc_ready, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(2 * N) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    asm volatile("griddepcontrol.wait;" ::: "memory");    // a, b and the factors
    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool live = true;
            const char* src = p.ab + (((size_t)b * s.Hkv + h) * n_k) * (size_t)kB;
            for (; it < n_k; ++it) {
                const int st = it % kStagesE;
                if (!mbar_wait(empty + st, ((it / kStagesE) & 1) ^ 1, fail, status)) { live = false; break; }
                mbar_expect_tx(full + st, (uint32_t)kB);
                bulk_load(stage0 + (size_t)st * kStage + kTileA, src + (size_t)it * kB, (uint32_t)kB, full + st);
            }
            if (!live)                                     // a wait ran out: the copies under way land, or the bound is reached, first
                for (int q = it < kStagesE ? 0 : it - kStagesE; q < it; ++q)
                    for (uint32_t n = 0; n < (1u << 16) && !mbar_try_wait(full + q % kStagesE, (uint32_t)(q / kStagesE) & 1u); ++n) { }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            for (int it = 0; it < n_k; ++it) {
                const int st = it % kStagesE;
                if (!mbar_wait(full + st, (it / kStagesE) & 1, fail, status)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a_addr = smem_u32(stage0 + (size_t)st * kStage), b_addr = a_addr + kTileA;
#pragma unroll
                for (int ty = 0; ty < 2; ++ty)             // Re against a, Im against b
#pragma unroll
                    for (int pr = 0; pr < 3; ++pr)         // hi hi, lo hi, hi lo
                        umma_bf16(tmem_base + ty * N, umma_desc(a_addr + 64 * ty + (pr == 1 ? 32 : 0), 1, 1024 >> 4),
                                  umma_desc(b_addr + (2 * ty + (pr == 2 ? 1 : 0)) * kNbx * kBoxB, kBoxB >> 4, 1024 >> 4), kIdesc, (it > 0 || pr > 0) ? 1u : 0u);
                umma_commit(empty + st);
            }
            umma_commit(acc_ready);
        }
    } else {
        // ---------------- generators: two warps to a stage, four stages in the making: a stage's chain (phases, products, the fence) is longer
        // than its products take on the tensor cores.  A warp has two pairs, a lane two frequencies and eight moments ----------------
        const int gw = warp - 2, np2 = lane & 7, sub = lane >> 3, q0 = 2 * (gw & 1);       // pairs q0, q0 + 1; moments 16 j + 4 sub + i
        const unsigned T2 = 2u * (unsigned)s.T;
        const float inv_T = 1.0f / (float)s.T;
        const uint32_t word = (uint32_t)(np2 & 3) * 4;
        const float* g0 = p.g + 2 * np2 + (size_t)(4 * sub) * s.k;
        float2 g[2][4];
        auto fetch = [&](int it) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) g[j][i] = *reinterpret_cast<const float2*>(g0 + (size_t)(16 * j + i) * s.k + it * kKn);
        };
        const int st = gw >> 1;
        uint32_t par = 1;
        if (st < n_k) fetch(st);
        for (int it = st; it < n_k; it += kStagesE, par ^= 1) {
            float C[2][2], S[2][2];                        // [pair][frequency]
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const unsigned dist = (unsigned)(max(0, p.n_blk - 1 - 2 * (p0 + q0 + q)) * p.R);
#pragma unroll
                for (int v = 0; v < 2; ++v) {              // pi n dist / T, exact in integers
                    const float f = (float)(((unsigned)(it * kKn + 2 * np2 + v) * dist) % T2) * inv_T;
                    const float an = 3.14159265358979f * (f - (f >= 1.0f ? 2.0f : 0.0f));
                    C[q][v] = __cosf(an);
                    S[q][v] = __sinf(an);
                }
            }
            if (!mbar_wait(empty + st, par, fail, status)) break;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    unsigned char* at = stage0 + (size_t)st * kStage + (((q0 + q) * 32 + 16 * j + 4 * sub) >> 3) * 1024 + word;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {          // (r & 3) = i: i^r = 1, i, -1, -i
                        const float x = (i & 2) ? -g[j][i].x : g[j][i].x, z = (i & 2) ? -g[j][i].y : g[j][i].y;
                        uint32_t w[4];                     // Re hi, Re lo, Im hi, Im lo
                        if (i & 1) {
                            split_bf16(-x * S[q][0], -z * S[q][1], w[0], w[1]);
                            split_bf16(x * C[q][0], z * C[q][1], w[2], w[3]);
                        } else {
                            split_bf16(x * C[q][0], z * C[q][1], w[0], w[1]);
                            split_bf16(x * S[q][0], z * S[q][1], w[2], w[3]);
                        }
                        const int r7 = (4 * sub + i) & 7;  // row & 7
                        unsigned char* row = at + r7 * 128;
#pragma unroll
                        for (int u = 0; u < 4; ++u) *reinterpret_cast<uint32_t*>(row + (((2 * u + (np2 >> 2)) ^ r7) << 4)) = w[u];
                    }
                }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(full + st);
            if (it + kStagesE < n_k) fetch(it + kStagesE);
        }
        // ---------------- epilogue: a warp has a pair (lanes its moments) and half of the columns.  A block's moments are put together in the idle
        // ring and leave with bulk copies (stored by the lanes, every 16 bytes went to a line of its own: 16 K cycles) ----------------
        const bool ok = mbar_wait(acc_ready, 0, fail, status);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int lg = warp & 3, pp = p0 + lg, half = (warp - 2) >> 2;
        if (ok && pp < p.n_pair) {
            constexpr int kHalfBoxes = D / 64, kPart = kHalfBoxes * kBoxY;       // a half's 64-dim boxes; its hi or lo values
            unsigned char* buf = stage0 + (warp - 2) * (2 * kPart);
            const int b_hi = p.n_blk - 1 - pp;
            for (int w = 0; w < (b_hi != pp ? 2 : 1); ++w) {                    // the block at +d, the one at -d
                const float sa = w && (lane & 1) ? -1.f : 1.f, sb = w ? 1.f : -1.f;
                if (w) {
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    __syncwarp();
                }
#pragma unroll 1
                for (int c0 = 0; c0 < D; c0 += 32) {
                    float u[32], v[32];
                    tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(half * D + c0), u);
                    tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(N + half * D + c0), v);
                    unsigned char* row = buf + (c0 >> 6) * kBoxY + lane * 128;
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int e = 8 * q4 + 2 * x;
                            split_bf16(sa * (u[e] + sb * v[e]), sa * (u[e + 1] + sb * v[e + 1]), hi[x], lo[x]);
                        }
                        const int at = ((((c0 & 63) >> 3) + q4) ^ (lane & 7)) << 4;
                        *reinterpret_cast<uint4*>(row + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *reinterpret_cast<uint4*>(row + kPart + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    char* y = p.y + (((size_t)b * p.n_blk + (w ? pp : b_hi)) * s.Hkv + h) * (size_t)(kNbx / 2) * kTileY;
#pragma unroll
                    for (int hl = 0; hl < 2; ++hl) {
                        char* dst = D == 128 ? y + half * kTileY + hl * kPart : y + (2 * hl + half) * kPart;
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)), "r"(smem_u32(buf + hl * kPart)),
                                     "r"(kPart)
                                     : "memory");
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
            if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(2 * N) : "memory");
    }
}

// Persistent; item = (block, KV head[, side]) as in the moment kernel.  sq [B][Hkv][2][D] is added to.
template <int D>
__global__ void __launch_bounds__(kThreadsR, 1) residual_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, Dims s,
                                                                SelPlan p, int n_init, int n_mid, int n_items, int n_stages, float* __restrict__ sq,
                                                                int32_t* status) {
    constexpr int kSides = D == 128 ? 2 : 1;
    // A: y, MN-major; B: P, K-major; M = 128 dims, N = 64 tokens
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(kChunk >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    extern __shared__ unsigned char smem_unaligned[];
    unsigned char* smem = smem_unaligned + ((1024u - (smem_u32(smem_unaligned) & 1023u)) & 1023u);
    const int n_chunk = p.R / kChunk;
    unsigned char* stage0 = smem;
    unsigned char* y_s = stage0 + (size_t)n_stages * kBoxX;
    unsigned char* Ps = y_s + kYStages * kTileY;
    uint64_t* full = reinterpret_cast<uint64_t*>(Ps + n_chunk * kTileP);
    uint64_t* empty = full + n_stages;
    uint64_t* y_full = empty + n_stages;
    uint64_t* y_empty = y_full + kYStages;
    uint64_t* acc_full = y_empty + kYStages;
    uint64_t* acc_empty = acc_full + kAccR;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kAccR);
    volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int i = 0; i < n_stages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 4); }
        for (int i = 0; i < kYStages; ++i) { mbar_init(y_full + i, 1); mbar_init(y_empty + i, 1); }
        for (int i = 0; i < kAccR; ++i) { mbar_init(acc_full + i, 1); mbar_init(acc_empty + i, 4); }
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the polynomials, a token per thread: 32 hi values, 32 lo values to a row
    for (int t = tid; t < p.R; t += kThreadsR) {
        const float x = (float)(2 * t + 1 - p.R) / (float)p.R;
        unsigned char* row = Ps + (t >> 6) * kTileP + (t & 63) * 128;
        float p0 = 1.f, p1 = x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = 8 * q + u;
                v[u] = p0;
                const float p2 = ((float)(2 * r + 3) * x * p1 - (float)(r + 1) * p0) * (1.0f / (float)(r + 2));
                p0 = p1;
                p1 = p2;
            }
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split_bf16(v[2 * u], v[2 * u + 1], hi[u], lo[u]);
            *reinterpret_cast<uint4*>(row + ((q ^ (t & 7)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(row + (((4 + q) ^ (t & 7)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    struct Item { int side, h, blk, b; };
    auto item = [&](int i) {
        Item w;
        w.side = kSides == 2 ? i & 1 : 0;
        const int t = kSides == 2 ? i >> 1 : i, gblk = t / s.Hkv;
        w.h = t - gblk * s.Hkv;
        w.b = gblk / p.n_blk;
        w.blk = gblk - w.b * p.n_blk;
        return w;
    };
    auto boxes = [&](const Item& w) { return min(n_chunk, (n_mid - w.blk * p.R + kChunk - 1) / kChunk); };
    asm volatile("griddepcontrol.wait;" ::: "memory");    // y (and, before that, the sums' zeros)
    if (warp == 0) {
        if (lane == 0) {
            int st = 0, issued = 0, yi = 0;
            uint32_t par = 1;
            bool live = true;
            for (int i = blockIdx.x; live && i < n_items; i += gridDim.x, ++yi) {
                const Item w = item(i);
                const int ys = yi % kYStages;
                if (!mbar_wait(y_empty + ys, ((yi / kYStages) & 1) ^ 1, fail, status)) { live = false; break; }
                mbar_expect_tx(y_full + ys, (uint32_t)kTileY);
                bulk_load(y_s + ys * kTileY, p.y + ((((size_t)w.b * p.n_blk + w.blk) * s.Hkv + w.h) * kSides + w.side) * (size_t)kTileY, (uint32_t)kTileY, y_full + ys);
                int tok = n_init + w.blk * p.R;
                const int n_ch = boxes(w);
                for (int q = 0; q < n_ch; ++q, tok += kChunk) {
                    if (!mbar_wait(empty + st, par, fail, status)) { live = false; break; }
                    unsigned char* dst = stage0 + (size_t)st * kBoxX;
                    mbar_expect_tx(full + st, (uint32_t)kBoxX);
                    const CUtensorMap* t0 = kSides == 2 && w.side ? &tmV : &tmK;
                    tma_load_4d(dst, t0, 0, w.h, tok, w.b, full + st);
                    tma_load_4d(dst + kBoxX / 2, kSides == 2 ? t0 : &tmV, kSides == 2 ? 64 : 0, w.h, tok, w.b, full + st);
                    ++issued;
                    if (++st == n_stages) { st = 0; par ^= 1; }
                }
            }
            if (!live) {                                   // a wait ran out: the copies under way land, or the bound is reached, first
                for (int q = issued < n_stages ? 0 : issued - n_stages; q < issued; ++q)
                    for (uint32_t n = 0; n < (1u << 16) && !mbar_try_wait(full + q % n_stages, (uint32_t)(q / n_stages) & 1u); ++n) { }
                for (int q = yi < kYStages ? 0 : yi - kYStages; q <= yi; ++q)
                    for (uint32_t n = 0; n < (1u << 16) && !mbar_try_wait(y_full + q % kYStages, (uint32_t)(q / kYStages) & 1u); ++n) { }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int a = 0, yi = 0;
            bool live = true;
            for (int i = blockIdx.x; live && i < n_items; i += gridDim.x, ++yi) {
                const Item w = item(i);
                const int ys = yi % kYStages, n_ch = boxes(w);
                if (!mbar_wait(y_full + ys, (yi / kYStages) & 1, fail, status)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t y_addr = smem_u32(y_s + ys * kTileY);
                for (int q = 0; q < n_ch; ++q, ++a) {
                    if (!mbar_wait(acc_empty + a % kAccR, ((a / kAccR) & 1) ^ 1, fail, status)) { live = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t p_addr = smem_u32(Ps + q * kTileP);
#pragma unroll
                    for (int pr = 0; pr < 3; ++pr)         // hi hi, lo hi, hi lo
#pragma unroll
                        for (int ks = 0; ks < kMF / 16; ++ks)
                            umma_bf16(tmem_base + (uint32_t)(a % kAccR) * kChunk, umma_desc(y_addr + (pr == 1 ? 2 * kBoxY : 0) + ks * 2048, kBoxY >> 4, 1024 >> 4),
                                      umma_desc(p_addr + (pr == 2 ? 64 : 0) + ks * 32, 1, 1024 >> 4), kIdesc, (pr > 0 || ks > 0) ? 1u : 0u);
                    umma_commit(acc_full + a % kAccR);
                }
                if (live && i + kYStages * (int)gridDim.x < n_items) umma_commit(y_empty + ys);      // (else nobody would wait for it: the CTA could end first)
            }
        }
    } else {
        // ---------------- differences: sets of four warps take the chunks in turn; a lane has a dim ----------------
        const int lg = warp & 3, set = (warp - 2) >> 2, e = lg * 32 + lane, col = e & 63;
        uint32_t off[8];                                   // of this dim in a row of a box, by row & 7
#pragma unroll
        for (int u = 0; u < 8; ++u) off[u] = (uint32_t)((e >> 6) * (kBoxX / 2) + u * 128 + (((col >> 3) ^ u) << 4) + (col & 7) * 2);
        int a = 0, st = 0;
        uint32_t par = 0;
        for (int i = blockIdx.x; i < n_items; i += gridDim.x) {
            const Item w = item(i);
            const int n_ch = boxes(w);
            int left = n_mid - w.blk * p.R;
            float e0 = 0.f, e1 = 0.f;
            for (int q = 0; q < n_ch; ++q, ++a, left -= kChunk) {
                if (a % kErrSets == set) {
                    // (after a time-out the walk goes on, on what is there)
                    mbar_wait(full + st, par, fail, status);
                    mbar_wait(acc_full + a % kAccR, (a / kAccR) & 1, fail, status);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t box = smem_u32(stage0) + (uint32_t)(st * kBoxX);
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        float v[32];
                        tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)((a % kAccR) * kChunk + 32 * hf), v);
                        auto add = [&](int t) {
                            uint16_t x;
                            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(box + off[t & 7] + (uint32_t)((32 * hf + (t & ~7)) * 128)) : "memory");
                            const float df = v[t] - __uint_as_float((uint32_t)x << 16);
                            if (t & 1) e1 = fmaf(df, df, e1);
                            else e0 = fmaf(df, df, e0);
                        };
                        if (left >= 32 * hf + 32) {
#pragma unroll
                            for (int t = 0; t < 32; ++t) add(t);
                        } else {
#pragma unroll
                            for (int t = 0; t < 32; ++t)
                                if (32 * hf + t < left) add(t);
                        }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) { mbar_arrive(empty + st); mbar_arrive(acc_empty + a % kAccR); }
                }
                if (++st == n_stages) { st = 0; par ^= 1; }
            }
            const int side = kSides == 2 ? w.side : e >> 6;
            atomicAdd(sq + (((size_t)w.b * s.Hkv + w.h) * 2 + side) * D + (kSides == 2 ? e : col), e0 + e1);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

size_t up256(size_t v) { return (v + 255) / 256 * 256; }
size_t ab_bytes(const Dims& s) { return up256((size_t)s.B * s.Hkv * s.k * 4 * 2 * s.d * 2); }
size_t g_bytes(const Dims& s) { return up256((size_t)kMF * s.k * 4); }
size_t residual_fixed(const Dims& s) { return (size_t)block_tokens(s) / kChunk * kTileP + kYStages * kTileY + 8 * (2 * 2 * kErrSets + 2 * kYStages + 2 * kAccR) + 64 + 1024; }
// Stages of the prefill's ring: a multiple of the sets of warps that take them in turn, so that a stage always falls to the same set.  (A set
// waits for the boxes that it takes only.  Were a stage's box before the one that it waits for another set's and late, the barrier's
// parity would still be that of two boxes ago and the wait would fall through.)
int residual_stages(const Dims& s) {
    const int n = (int)((227 * 1024 - residual_fixed(s)) / kBoxX);
    return n >= 2 * kErrSets ? 2 * kErrSets : n >= kErrSets ? kErrSets : 0;
}

template <typename... Params, typename... Args>
cudaError_t launch_behind(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaError_t err = smem > 48 * 1024 ? ensure_dynamic_smem(kernel, smem) : cudaSuccess;
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <int D>
cudaError_t launch_select_mom_t(const Dims& s, const SelPlan& p, const void* K, const void* V, int64_t sb, int64_t st, int64_t sh, int n_init, int n_mid,
                                int L, float* sq, int32_t* status, cudaStream_t stream) {
    CUtensorMap tmK, tmV;
    if (!prefill_map(&tmK, K, s, sb, st, sh, L) || !prefill_map(&tmV, V, s, sb, st, sh, L)) return cudaErrorInvalidValue;
    const long long pieces = (long long)s.B * s.Hkv * s.k * p.nbx * 8, n_rot = (pieces + 255) / 256;
    const long long items = (long long)s.B * p.n_blk * s.Hkv * (D == 128 ? 2 : 1);
    if (n_rot >= (1ll << 30) || items >= (1ll << 30)) return cudaErrorInvalidValue;
    cudaError_t err = launch_behind(rotate_kernel, dim3((unsigned)(n_rot + s.k / 32)), 256, 0, stream, s, p, s.k / 32);
    if (err != cudaSuccess) return err;
    constexpr size_t smem_e = (size_t)kStagesE * (kTileA + 4 * (2 * D / 64) * kBoxB) + 8 * (2 * kStagesE + 1) + 16 + 1024;
    err = launch_behind(expand_kernel<D>, dim3((p.n_pair + kPairs - 1) / kPairs, s.Hkv, s.B), kThreadsE, smem_e, stream, s, p, status);
    if (err != cudaSuccess) return err;
    const int n_stages = residual_stages(s);
    return launch_behind(residual_kernel<D>, dim3((unsigned)(items < sm_count() ? items : sm_count())), kThreadsR, residual_fixed(s) + (size_t)n_stages * kBoxX, stream,
                         tmK, tmV, s, p, n_init, n_mid, (int)items, n_stages, sq, status);
}

}  // namespace

// Bytes of scratch of the reconstruction by block moments (0: it does not serve this layout).
size_t select_mom_bytes(const Dims& s, int dtype) {
    if (dtype != FA_BF16 || (s.d != 64 && s.d != 128) || !compress_mom_supported(s) || residual_stages(s) == 0) return 0;
    const size_t n_blk = (size_t)blocks_of(s.max_mid, block_tokens(s));
    return ab_bytes(s) + g_bytes(s) + n_blk * s.B * s.Hkv * (2 * s.d / 128) * kTileY;
}

// sq [B][Hkv][2][d] += sum over the middle tokens of (x~ - x)^2, from the coefficients [B][Hkv][M][d] of all dims.  s: the layout with every dim
// compressed; K, V: 16-byte aligned, strides multiples of eight; scratch: select_mom_bytes, 256-byte aligned.
cudaError_t launch_select_mom(const Dims& s, const float* coef_k, const float* coef_v, const void* K, const void* V, int64_t sb, int64_t st, int64_t sh,
                              int n_init, int n_mid, int L, float* sq, int32_t* status, char* scratch, cudaStream_t stream) {
    SelPlan p = {};
    p.R = block_tokens(s);
    p.n_blk = blocks_of(n_mid, p.R);
    p.n_pair = (p.n_blk + 1) / 2;
    p.nbx = 2 * s.d / 64;
    p.coef_k = coef_k;
    p.coef_v = coef_v;
    p.ab = scratch;
    p.g = reinterpret_cast<float*>(scratch + ab_bytes(s));
    p.y = scratch + ab_bytes(s) + g_bytes(s);
    return s.d == 128 ? launch_select_mom_t<128>(s, p, K, V, sb, st, sh, n_init, n_mid, L, sq, status, stream)
                      : launch_select_mom_t<64>(s, p, K, V, sb, st, sh, n_init, n_mid, L, sq, status, stream);
}

}  // namespace fa
