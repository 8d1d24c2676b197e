// fa_compress, block-moment path (Eq.3-4; bf16 caches, sm_100a): the projection on the basis in two contractions, the
// second of them over an axis that is R / 32 times shorter than the token axis.
//
// Within a block of R tokens the basis functions of Eq.4 are band-limited: with t in [-1, 1] across the block and
// phi_n = theta n R / 2 (theta = 2 pi / T) the plane-wave expansion in Legendre polynomials,
//   e^{i phi t} = sum_r (2 r + 1) i^r j_r(phi) P_r(t)          (j_r: spherical Bessel functions),
// falls off faster than exponentially beyond r = phi.  R is at most 6 T / k, so phi <= 6 pi, and 32 terms leave at most
// 4e-5 at the very edge of band and block (1e-6 of the sums' norm).  Hence
//   C_n = sum_j x_j e^{i theta n j} = sum_blocks e^{i theta n center} sum_{r < 32} (2 r + 1) i^r j_r(phi_n) Y_{block, r}
//   Y_{block, r} = sum_{t in block} P_r(t) x_t                   (the block's moments).
//   1. moments_kernel: one pass over the prefill.  Boxes of 64 tokens come in by TMA; the tensor cores multiply them with
//      P (as bf16 hi + lo: exact to 2^-17; x is bf16 already), the gather warps write the kept-dim rows of the middle from
//      the same boxes, the epilogue warps write the moments of the compressed dims, again as bf16 hi + lo.
//   2. moment_project_kernel: C += G Y on CTA pairs (tcgen05.mma.cta_group::2), G generated from exact integer phases
//      and 32 Bessel factors per frequency; three products hi hi, lo hi, hi lo.
// Both factors carry 2^-17, where the contraction over tokens rounds its basis to bf16 (2^-9).
// Where the frequencies fill tiles of 256 the blocks are folded in pairs about the middle of the row, which halves the second contraction (see there).
//
// What bounds it: the first kernel HBM (per box of 64 tokens of one side 740 to 840 cycles against the 700 that 16 KB take at an SM's
// share of the measured rate; its write of the moments is 10 % of the traffic at k / T = 1 / 64 and 20 % at 1 / 32), the
// second the tensor cores (1152 cycles of products a position and pair) plus 20 K cycles a segment, at the rate at which L2 adds vectors of
// floats (four rows of 128 K tokens: 242 K cycles, 69 % of them on the tensor cores).
// Direct contraction against this path, in us: six layers of 32 K tokens, 1024 rows: 701 -> 374, with one projection for all 333, folded 292, the
// moments of all layers in one launch and the windows beside the projection 277; 128 K tokens, batch 4, 2048 rows: 3207 -> 777, folded 664; six ragged
// rows of 3 to 12 K tokens, 512 rows: 123 -> 85, folded 79, windows beside it 73; 4 K tokens of 256 heads, 256 rows (T / k = 32, blocks of 192
// tokens, too few frequencies to fold): 231 -> 221, windows beside it 199.  The projection of the four rows of 128 K tokens alone:
// 275 -> 162.  Relative error of the coefficients 4e-6 against 2.4e-4.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "fa_moments.cuh"

namespace fa {
namespace {

using namespace mom;

constexpr int kChunkBytes = 128 * kChunk * 2;      // [64 tokens x 64 dims] twice
constexpr int kHChunk = 2 * kMF * kChunk * 2;      // P of 64 tokens, hi and lo rows
constexpr int kAcc = 8;              // accumulators (64 columns each) in tensor memory
constexpr int kEpiWarps = 4, kGathWarps = 8;
constexpr int kThreadsMom = 32 * (2 + kEpiWarps + kGathWarps);


// two runs of 16 columns of tensor memory
__device__ __forceinline__ void tmem_ld16_two(uint32_t a0, uint32_t a1, float (&x)[16], float (&y)[16]) {
    uint32_t r[16], q[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
          "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]),
          "=r"(q[6]), "=r"(q[7]), "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
        : "r"(a0), "r"(a1)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) { x[i] = __uint_as_float(r[i]); y[i] = __uint_as_float(q[i]); }
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}

// Blocks of a launch: batch rows b0 .. b0 + nb of the call; row b owns blocks first[b] .. first[b + 1] of the launch
// (lens.n = 0: nblk each, and first is not used).  R tokens to a block.
// Folded (the tiles of frequencies are whole, k a multiple of 256): a position of the launch is a PAIR of blocks of a row, p and n - 1 - p of
// its n blocks (the middle one of an odd number by itself); nblk, first and total then count pairs.
struct MomRows {
    int R, nblk, b0, nb, total, n_blk;                     // (n_blk: blocks of a row, where all are alike)
    RowLens lens;
    uint32_t first[kMaxRagged + 1];
};

// Layers of a launch: its batch row b is row b % B of layer b / B (several layers, all of their rows; one, some of them).
struct MomIn {
    CUtensorMap k[kMomLayers], v[kMomLayers];
    CacheDev c[kMomLayers];
    int n;
};

// Item = (block, KV head[, side]): D = 128: one side's 128 dims, D = 64: K dims and V dims side by side.  A persistent CTA
// takes items blockIdx.x, blockIdx.x + gridDim.x, ...: CTAs that run together read the same tokens' heads.
template <int D, bool RAG, bool FOLD>
__global__ void __launch_bounds__(kThreadsMom, 1) moments_kernel(const __grid_constant__ MomIn in, Dims s, int Lall, const __grid_constant__ MomRows rows,
                                                                 bf16* __restrict__ Y, int n_stages, int n_items, int wait_first) {
    constexpr int kSides = D == 128 ? 2 : 1;               // items per (block, head)
    constexpr int kTypes = FOLD ? 2 : 1;                   // operands per position: real and imaginary rows want different sums of a pair
    // A: 64-dim rows of a token, MN-major; B: P, K-major; M = 128 dims, N = 64 (hi and lo rows of P)
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(2 * kMF >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    extern __shared__ unsigned char smem_unaligned[];
    unsigned char* smem = smem_unaligned + ((1024u - (smem_u32(smem_unaligned) & 1023u)) & 1023u);
    unsigned char* stage0 = smem;
    const int n_chunk = rows.R / kChunk;
    unsigned char* Hs = stage0 + (size_t)n_stages * kChunkBytes;
    unsigned char* y_s = Hs + (size_t)n_chunk * kHChunk;   // [128 columns][128 bytes] moments of an item on their way out
    uint64_t* full = reinterpret_cast<uint64_t*>(y_s + kTypes * 128 * 4 * kMF);
    uint64_t* empty = full + n_stages;
    uint64_t* acc_full = empty + n_stages;
    uint64_t* acc_empty = acc_full + kAcc;
    uint64_t* masked = acc_empty + kAcc;                   // per stage: rows past the end of a batch row's last box are zero
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(masked + n_stages);
    volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint8_t* inv_s = reinterpret_cast<uint8_t*>(tmem_slot + 2);      // [layer][Hkv][2][D] position of a dim among the compressed ones, 255: kept
    uint8_t* idf_s = inv_s + in.n * s.Hkv * 2 * D;                   // [layer][Hkv][nfk + nfv] the kept dims
    int32_t* status = in.c[0].status;
    const int nf = s.nfk + s.nfv;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int i = 0; i < n_stages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1 + kGathWarps); mbar_init(masked + i, kGathWarps); }
        for (int i = 0; i < kAcc; ++i) { mbar_init(acc_full + i, 1); mbar_init(acc_empty + i, kEpiWarps); }
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp > 0) {                                        // (the producer's boxes set off meanwhile)
        constexpr int kW = kThreadsMom / 32 - 1;
        const int u = tid - 32, wu = warp - 1;
        // where a dim is: a warp takes whole rows (head, side)
        for (int r = wu; r < 2 * in.n * s.Hkv; r += kW) {
            const int lh = r >> 1, sd = r & 1, nfr = sd ? s.nfv : s.nfk, ncr = D - nfr, layer = lh / s.Hkv, h = lh - layer * s.Hkv;
            const CacheDev& c = in.c[layer];
            const int32_t* idf = (sd ? c.idx_full_v : c.idx_full_k) + h * nfr;
            const int32_t* idc = (sd ? c.idx_comp_v : c.idx_comp_k) + h * ncr;
            uint8_t* inv = inv_s + r * D;
#pragma unroll
            for (int e0 = 0; e0 < D; e0 += 32) {
                const int e = e0 + lane;
                const int d = e < nfr ? idf[e] : idc[e - nfr];
                if (e < nfr) idf_s[lh * nf + (sd ? s.nfk : 0) + e] = (uint8_t)d;
                inv[d] = e < nfr ? 255 : (uint8_t)(e - nfr);
            }
        }
        // the polynomials, by their recurrence, one token per thread
        for (int t = u; t < rows.R; t += 32 * kW) {
            const float x = (float)(2 * t + 1 - rows.R) / (float)rows.R;
            unsigned char* hq = Hs + (t >> 6) * kHChunk;
            const int tok = t & 63;
            float p0 = 1.f, p1 = x;
#pragma unroll
            for (int r = 0; r < kMF; ++r) {
                const bf16 hi = __float2bfloat16_rn(p0), lo = __float2bfloat16_rn(p0 - __bfloat162float(hi));
                unsigned char* at = hq + (r >> 3) * 1024 + (r & 7) * 128 + (((tok >> 3) ^ (r & 7)) << 4) + (tok & 7) * 2;
                *reinterpret_cast<bf16*>(at) = hi;
                *reinterpret_cast<bf16*>(at + (kMF >> 3) * 1024) = lo;
                const float p2 = ((float)(2 * r + 3) * x * p1 - (float)(r + 1) * p0) * (1.0f / (float)(r + 2));
                p0 = p1;
                p1 = p2;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // P is read by the tensor cores
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kW) : "memory");
    }
    const uint32_t tmem_base = *tmem_slot;

    // A role's place in the CTA's items: the next item is gridDim.x further on, taken by additions with carries.
    const int n_mid_all = mid_of(s, Lall);
    struct Walk { int i, side, h, gblk, b, blk, nblk, n_mid, n_blk, layer; };      // (b: row of the layer)
    const int d_side = kSides == 2 ? (int)gridDim.x & 1 : 0, d_t = kSides == 2 ? (int)gridDim.x >> 1 : (int)gridDim.x;
    const int d_blk = d_t / s.Hkv, d_h = d_t - d_blk * s.Hkv;
    auto settle = [&](Walk& w) {                           // block number -> batch row and block of the row
        if (w.i >= n_items) return;
        while (w.blk >= w.nblk) {
            w.blk -= w.nblk;
            if (++w.b == s.B && w.layer + 1 < in.n) { w.b = 0; ++w.layer; }
            if (RAG) w.nblk = (int)(rows.first[w.b + 1] - rows.first[w.b]);
        }
        if (RAG) w.n_mid = mid_of(s, rows.lens.len[w.b]);
        if (RAG && FOLD) w.n_blk = blocks_of(w.n_mid, rows.R);
    };
    // the blocks of an item: one, or (folded) the pair p, n - 1 - p; a block's boxes
    auto halves = [&](const Walk& w) { return FOLD && w.n_blk - 1 - w.blk != w.blk ? 2 : 1; };
    auto block_of = [&](const Walk& w, int half) { return FOLD && half ? w.n_blk - 1 - w.blk : w.blk; };
    auto boxes_of = [&](const Walk& w, int blk) { return min(n_chunk, (w.n_mid - blk * rows.R + kChunk - 1) / kChunk); };
    auto walk_begin = [&]() {
        Walk w;
        w.i = blockIdx.x;
        const int t = kSides == 2 ? w.i >> 1 : w.i;
        w.side = kSides == 2 ? w.i & 1 : 0;
        w.gblk = t / s.Hkv;
        w.h = t - w.gblk * s.Hkv;
        w.blk = w.gblk;
        w.b = RAG ? 0 : rows.b0;
        w.layer = 0;
        w.nblk = RAG ? (int)rows.first[1] : rows.nblk;
        w.n_mid = n_mid_all;
        w.n_blk = FOLD ? blocks_of(n_mid_all, rows.R) : 0;
        settle(w);
        return w;
    };
    auto walk_next = [&](Walk& w) {
        w.i += gridDim.x;
        w.side += d_side;
        int c1 = 0;
        if (w.side >= 2) { w.side -= 2; c1 = 1; }
        w.h += d_h + c1;
        int c2 = 0;
        if (w.h >= s.Hkv) { w.h -= s.Hkv; c2 = 1; }
        w.gblk += d_blk + c2;
        w.blk += d_blk + c2;
        settle(w);
    };

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            int st = 0, issued = 0;
            uint32_t par = 1;
            bool live = true;
            for (Walk it = walk_begin(); live && it.i < n_items; walk_next(it))
            for (int half = 0; live && half < halves(it); ++half) {
                const int blk = block_of(it, half), n_ch = boxes_of(it, blk);
                int tok = s.l_init + blk * rows.R;
                for (int q = 0; q < n_ch; ++q, tok += kChunk) {
                    if (!mbar_wait(empty + st, par, fail, status)) { live = false; break; }
                    unsigned char* dst = stage0 + (size_t)st * kChunkBytes;
                    mbar_expect_tx(full + st, (uint32_t)kChunkBytes);
                    if (kSides == 2) {
                        const CUtensorMap* tm = it.side ? &in.v[it.layer] : &in.k[it.layer];
                        tma_load_4d(dst, tm, 0, it.h, tok, it.b, full + st);
                        tma_load_4d(dst + kChunkBytes / 2, tm, 64, it.h, tok, it.b, full + st);
                    } else {
                        tma_load_4d(dst, &in.k[it.layer], 0, it.h, tok, it.b, full + st);
                        tma_load_4d(dst + kChunkBytes / 2, &in.v[it.layer], 0, it.h, tok, it.b, full + st);
                    }
                    ++issued;
                    if (++st == n_stages) { st = 0; par ^= 1; }
                }
            }
            if (!live)                                     // a wait ran out: the boxes still under way land before the CTA ends
                for (int q = issued - n_stages < 0 ? 0 : issued - n_stages; q < issued; ++q)
                    for (uint32_t n = 0; n < (1u << 20) && !mbar_try_wait(full + q % n_stages, (uint32_t)(q / n_stages) & 1u); ++n) { }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: moments[dim][hi rows | lo rows] of a block ----------------
        if (lane == 0) {
            int st = 0, a = 0;
            uint32_t par = 0, mpar = 0;
            bool live = true;
            // descriptors with the addresses of stage 0 and box 0 of P (in units of 16 bytes; the sums stay below the field's end)
            const uint64_t xdesc0 = umma_desc(smem_u32(stage0), (kChunkBytes / 2) >> 4, 1024 >> 4), hdesc0 = umma_desc(smem_u32(Hs), 1, 1024 >> 4);
            for (Walk it = walk_begin(); live && it.i < n_items; walk_next(it))
            for (int half = 0; live && half < halves(it); ++half, ++a) {
                const int blk = block_of(it, half), n_ch = boxes_of(it, blk);
                const int ab = a % kAcc;
                if (a >= kAcc && !mbar_wait(acc_empty + ab, ((a / kAcc) - 1) & 1, fail, status)) { live = false; break; }
                const uint32_t acc = tmem_base + ab * (2 * kMF);
                uint64_t hdesc = hdesc0;
                int left = it.n_mid - blk * rows.R;
                for (int q = 0; q < n_ch; ++q, left -= kChunk, hdesc += kHChunk >> 4) {
                    if (!mbar_wait(full + st, par, fail, status)) { live = false; break; }
                    if (left < kChunk) {
                        if (!mbar_wait(masked + st, (mpar >> st) & 1u, fail, status)) { live = false; break; }
                        mpar ^= 1u << st;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t xdesc = xdesc0 + (uint64_t)(st * (kChunkBytes >> 4));
#pragma unroll
                    for (int ks = 0; ks < kChunk / 16; ++ks)
                        umma_bf16(acc, xdesc + ks * (2048 >> 4), hdesc + ks * 2, kIdesc, (q > 0 || ks > 0) ? 1u : 0u);
                    umma_commit(empty + st);
                    if (++st == n_stages) { st = 0; par ^= 1; }
                }
                if (live) umma_commit(acc_full + ab);
            }
        }
    } else if (warp < 2 + kEpiWarps) {
        // ---------------- epilogue: moments of the compressed dims, bf16 hi then lo, 128 bytes per (block, column) ----------------
        if (wait_first) asm volatile("griddepcontrol.wait;" ::: "memory");   // Y may still be read by the kernel before this one
        const int lg = warp & 3, e = lg * 32 + lane;       // tensor-memory lane: the dim, or (D = 64) K's dims then V's
        const int ncol = s.dck + s.dcv;
        // the projection adds to the coefficients: they are cleared here
        for (int lb = 0; lb < rows.nb; ++lb) {
            const int layer = lb / s.B, b = rows.b0 + lb - layer * s.B;
            if (RAG && rows.first[b] == rows.first[b + 1]) continue;       // (a short row: the direct contraction's)
            for (int sd = 0; sd < 2; ++sd) {
                const int nc = sd ? s.dcv : s.dck, n4 = s.Hkv * (s.M >> 2) * nc;
                float4* z = reinterpret_cast<float4*>(coef_rows(sd ? in.c[layer].coef_v : in.c[layer].coef_k, s, b, 0, nc));
                for (int i = blockIdx.x * (32 * kEpiWarps) + tid - 64; i < n4; i += gridDim.x * (32 * kEpiWarps)) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        int a = 0;
        for (Walk it = walk_begin(); it.i < n_items; walk_next(it)) {
            const int n_half = halves(it);
            // (after a time-out the walk goes on, on what is there: the four warps keep meeting)
            for (int half = 0; half < n_half; ++half) mbar_wait(acc_full + (a + half) % kAcc, ((a + half) / kAcc) & 1, fail, status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int side = kSides == 2 ? it.side : e >> 6, dim = kSides == 2 ? e : e & 63;
            const int pos = inv_s[((it.layer * s.Hkv + it.h) * 2 + side) * D + dim];
            // The columns of the item are one contiguous run of rows of Y: they are put together in shared memory and leave with one
            // bulk copy (stored by the lanes, every 16 bytes went to a line of its own).  The 16-byte pieces of a row are
            // permuted as the 128-byte swizzle of the products' operand wants them, so the second kernel copies rows as they are.
            if (warp == 2 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the copy before has read the buffer
            asm volatile("bar.sync 2, %0;" ::"n"(32 * kEpiWarps) : "memory");
            const uint32_t t0 = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)((a % kAcc) * 2 * kMF), t1 = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(((a + 1) % kAcc) * 2 * kMF);
            const int col = (kSides == 1 && side ? s.dck : 0) + pos;
            // 16 moments at a time (all 32 of two blocks do not fit the registers)
#pragma unroll
            for (int r0 = 0; r0 < kMF; r0 += 16) {
                auto put = [&](unsigned char* dst, const float (&v)[16]) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) split_bf16(v[8 * r + 2 * u], v[8 * r + 2 * u + 1], hi[u], lo[u]);
                        const int piece = r0 / 8 + r;
                        *reinterpret_cast<uint4*>(dst + ((piece ^ (col & 7)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *reinterpret_cast<uint4*>(dst + (((4 + piece) ^ (col & 7)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                };
                float y[16], t[16];                        // of the one block, or of block p
                tmem_ld16_two(t0 + r0, t0 + kMF + r0, y, t);
#pragma unroll
                for (int r = 0; r < 16; ++r) y[r] += t[r];
                if (FOLD) {
                    float z[16];                           // of block n - 1 - p
#pragma unroll
                    for (int r = 0; r < 16; ++r) z[r] = 0.f;
                    if (n_half == 2) {
                        tmem_ld16_two(t1 + r0, t1 + kMF + r0, z, t);
#pragma unroll
                        for (int r = 0; r < 16; ++r) z[r] += t[r];
                    }
                    // even orders: sum and difference, odd ones: difference and sum (the middle block by itself: itself and nothing)
#pragma unroll
                    for (int r = 0; r < 16; ++r) {
                        const float sum = z[r] + y[r], dif = n_half == 2 ? z[r] - y[r] : 0.f;
                        y[r] = (r & 1) ? dif : sum;
                        z[r] = (r & 1) ? sum : dif;
                    }
                    if (pos != 255) put(y_s + (128 + col) * (4 * kMF), z);
                }
                if (pos != 255) put(y_s + col * (4 * kMF), y);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                for (int half = 0; half < n_half; ++half) mbar_arrive(acc_empty + (a + half) % kAcc);
            a += n_half;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("bar.sync 2, %0;" ::"n"(32 * kEpiWarps) : "memory");
            if (warp == 2 && lane == 0) {
                const int c0 = kSides == 2 && it.side ? s.dck : 0, nc = kSides == 1 ? ncol : it.side ? s.dcv : s.dck;
#pragma unroll
                for (int ty = 0; ty < kTypes; ++ty) {
                    char* dst = reinterpret_cast<char*>(Y) + ((((size_t)it.gblk * kTypes + ty) * s.Hkv + it.h) * ncol + c0) * (size_t)(4 * kMF);
                    if (nc > 0)
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)),
                                     "r"(smem_u32(y_s + ty * 128 * 4 * kMF)), "r"(nc * (4 * kMF))
                                     : "memory");
                }
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        if (warp == 2 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory"); // the end of this grid implies the end of the one before
    } else {
        // ---------------- kept dims of the middle tokens: boxes -> K^mu, V^mu ----------------
        // A warp takes eight consecutive rows of a box, a lane eight kept dims (16 bytes of a kept-dim row) of one row.  The swizzle
        // puts the same dim of eight consecutive rows into eight different bank groups, so a fetch of 8 rows x 4 dims
        // meets about two dims to a bank.  Four lanes to a row where a row has at most 32 kept dims (all rows in one round), else
        // 8 or 16 (2 or 4 rounds); in round k the rows differ in the bits above the lanes', which moves a source by an xor.
        const int w = warp - 2 - kEpiWarps;
        const bool p2 = (s.P & (s.P - 1)) == 0;
        const int lgP = 31 - __clz(s.P);
        // chunk swizzle of V^mu rows as a shift and a mask of the slot (v_swz)
        const int nchv = s.nfv >> 3, vsh = nchv == 4 ? 1 : nchv == 8 ? 0 : 2, vmask = nchv == 4 ? 3 : nchv == 8 ? 7 : (nchv == 2 || nchv == 6) ? 1 : 0;
        int st = 0;
        uint32_t par = 0;
        bool live = true;
        for (Walk it = walk_begin(); live && it.i < n_items; walk_next(it)) {
            // 16-byte chunks of this item's kept-dim rows: one side's, or K's then V's
            const int nk8 = (kSides == 2 && it.side) ? 0 : s.nfk >> 3, np = kSides == 2 ? (it.side ? s.nfv : s.nfk) >> 3 : nf >> 3;
            const size_t bh = ((size_t)it.b * s.Hkv + it.h) * (size_t)s.P * (size_t)s.S_cap;
            auto gather = [&](auto lg_lp) {
                constexpr int LG = decltype(lg_lp)::value, RP = 32 >> LG, NI = 8 / RP;      // lanes to a row: 2^LG; rows at a time, rounds
                const int sub = lane >> LG, p = lane & ((1 << LG) - 1);
                const bool on = p < np, v = p >= nk8;
                uint32_t o[4];                             // source offsets of the eight dims, two to a register
                const int rowb = 2 * (v ? s.nfv : s.nfk);
#pragma unroll
                for (int u = 0; u < 4; ++u) o[u] = 0;
                if (on) {
                    const uint8_t* id = idf_s + (it.layer * s.Hkv + it.h) * nf + (v ? s.nfk : 0) + 8 * (v ? p - nk8 : p);
                    const int bx = kSides == 1 && v ? kChunkBytes / 2 : 0;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int d = id[u];
                        const uint32_t off = (uint32_t)(bx + (d >> 6) * (kChunkBytes / 2) + ((((d & 63) >> 3) ^ sub) << 4) + (d & 7) * 2);
                        o[u >> 1] |= off << (16 * (u & 1));
                    }
                }
                const uint32_t col = (uint32_t)(16 * (v ? p - nk8 : p));
                const int mask = v ? vmask : 0;
                char* dst0 = reinterpret_cast<char*>(v ? in.c[it.layer].v_mid : in.c[it.layer].k_mid) + bh * (size_t)rowb;
                for (int half = 0; live && half < halves(it); ++half) {
                const int blk = block_of(it, half), n_ch = boxes_of(it, blk);
                int j0 = blk * rows.R + 8 * w + sub, left = it.n_mid - blk * rows.R;
                for (int q = 0; q < n_ch; ++q, j0 += kChunk, left -= kChunk) {
                    if (!mbar_wait(full + st, par, fail, status)) { live = false; break; }
                    const uint32_t box = smem_u32(stage0) + (uint32_t)(st * kChunkBytes + w * 1024), src = box + (uint32_t)(sub * 128);
                    uint4 val[NI];
#pragma unroll
                    for (int k = 0; k < NI; ++k) {
                        uint32_t x[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint32_t oo = o[u] ^ (uint32_t)(((k * RP) << 4) * 0x10001);
                            x[u] = 0;
                            if (on) x[u] = __byte_perm(lds_u16(src + (uint32_t)(k * RP * 128) + (oo & 0xffffu)), lds_u16(src + (uint32_t)(k * RP * 128) + (oo >> 16)), 0x5410);
                        }
                        val[k] = make_uint4(x[0], x[1], x[2], x[3]);
                    }
                    if (left < kChunk) {
                        // rows past the middle would count as tokens: zero them in front of the products
                        __syncwarp();
                        const uint32_t z = box + (uint32_t)((lane >> 4) * 128 + ((lane >> 3) & 1) * (kChunkBytes / 2) + (lane & 7) * 16);
                        for (int k = 0; k < 8; k += 2)
                            if (8 * w + k + (lane >> 4) >= left)
                                asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(z + (uint32_t)k * 128u), "r"(0) : "memory");
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(masked + st);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty + st);    // the values are in registers: the stage goes back before the stores
                    if (++st == n_stages) { st = 0; par ^= 1; }
#pragma unroll
                    for (int k = 0; k < NI; ++k) {
                        if (on && 8 * w + sub + k * RP < left) {
                            const int j = j0 + k * RP;
                            const int cls = p2 ? (j & (s.P - 1)) : j % s.P, slot = p2 ? (j >> lgP) : j / s.P;
                            // logical chunk of a V^mu row is stored at chunk ^ swizzle
                            const uint32_t at = col ^ (uint32_t)(((slot >> vsh) & mask) << 4);
                            *reinterpret_cast<uint4*>(dst0 + (size_t)(uint32_t)(cls * s.S_cap + slot) * (uint32_t)rowb + at) = val[k];
                        }
                    }
                }
                }
            };
            using std::integral_constant;
            if (np <= 4) gather(integral_constant<int, 2>{});
            else if (np <= 8) gather(integral_constant<int, 3>{});
            else gather(integral_constant<int, 4>{});
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && *fail)                                 // (a wait that runs out tells the first layer)
        for (int l = 1; l < in.n; ++l) in.c[l].status[0] = status[0];
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- second contraction ------------------------------------------------------------------------------------------
constexpr int kBMp = 128;             // coefficient rows per CTA (256 per pair)
constexpr int kGenWarpsP = 8;
constexpr int kThreadsP = 64 + 32 * kGenWarpsP;
constexpr int kABytesP = kBMp * 128;  // rows of 32 hi and 32 lo values
constexpr int kStagesP = 4;             // stages at most

// Positions: the blocks of all (batch row, head group) units of the launch, laid end to end; a team of M / 256 pairs takes
// positions start[t] .. start[t + 1] (cut on the host so that every team has the same cost, as in fa_compress_tc2.cu).
constexpr int kMaxTeamsP = 96;
struct MomCuts { uint32_t start[kMaxTeamsP + 1]; };
// Coefficients of the layers of a launch: its batch row b is row b % B of layer b / B.
struct MomLayers { int n; float *k[kMomLayers], *v[kMomLayers]; int32_t* status[kMomLayers]; };

// npad: accumulator columns of a product (the compressed dims of both sides, up to a multiple of 32); each CTA of a CTA pair brings half of
// them.  A stage feeds two products:
//   as they are: one tile of 128 frequencies (rows Re and Im interleaved) against HP heads;
//   folded: with t_b = m + d_b about the middle m of the row, blocks at +d and -d enter as e^{i theta n d} Y+ + e^{-i theta n d} Y- =
//     cos E + i sin O with E, O = Y+ +- Y-.  By the parity of i^r, the real part of e^{-i theta n m} C_n takes E of even r and O of odd r only, the
//     imaginary part the others: two tiles (256 frequencies, Re; the same, Im) against one head's two operands, each 32 long for TWO
//     blocks.  Half the products of the plain form; the epilogue turns (Re, Im) by e^{i theta n m} in registers.
// (128 registers at most: three warps on one scheduler then leave room for those of the windows kernel's, or the partition kernel's, CTAs)
template <int HP, bool RAG, bool FOLD>
__global__ void __maxnreg__(128) moment_project_kernel(const bf16* __restrict__ Y, Dims s, const __grid_constant__ MomLayers layers,
                                                                      const __grid_constant__ MomRows rows, const __grid_constant__ MomCuts cuts, int npad, int n_stages) {
    constexpr int kTiles = FOLD ? 2 : 1, kOps = FOLD ? 2 : HP;     // A tiles and B operands of a stage
    const int nh = npad >> 1, b_op = nh * 128, n_stage = kTiles * kABytesP + kOps * b_op;     // rows of 128 bytes
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(npad >> 3) << 17) | ((uint32_t)((2 * kBMp) >> 4) << 24);
    extern __shared__ unsigned char smem_unaligned[];
    unsigned char* smem = smem_unaligned + ((1024u - (smem_u32(smem_unaligned) & 1023u)) & 1023u);
    unsigned char* stage0 = smem;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + n_stages * n_stage);
    uint64_t* peer = full + kStagesP;                      // even CTA: the odd CTA's stage is complete
    uint64_t* empty = peer + kStagesP;
    uint64_t* acc_ready = empty + kStagesP;
    uint64_t* epi_done = acc_ready + 1;                    // the epilogue has left the stage ring (its scratch)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(epi_done + 1);
    volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const int n_pairs = s.M / (kTiles * 2 * kBMp);
    const int cluster = (int)blockIdx.x >> 1, team = cluster / n_pairs, pair = cluster - team * n_pairs;
    const int mt = 2 * pair + (int)rank;
    const int n_hg = s.Hkv / HP, ncol = s.dck + s.dcv;
    const uint32_t pos_begin = cuts.start[team], pos_end = cuts.start[team + 1];
    int32_t* status = layers.status[0];
    // batch row, heads, positions, blocks of the row, whether these are all positions of the unit; first position of the row in the launch
    struct Seg { int b, h0, kb0, kb1, n_blk; bool whole; uint32_t g0; };
    auto seg_at = [&](uint32_t pos) {
        int b, nblk = rows.nblk;
        uint32_t g0, off;
        if (RAG) {
            b = 0;
            while (pos >= rows.first[b + 1] * (uint32_t)n_hg) ++b;
            g0 = rows.first[b];
            nblk = (int)(rows.first[b + 1] - g0);
            off = pos - g0 * (uint32_t)n_hg;
        } else {
            b = (int)(pos / (uint32_t)(n_hg * nblk));
            off = pos - (uint32_t)(b * n_hg * nblk);
            g0 = (uint32_t)(b * nblk);
            b += rows.b0;
        }
        const int hg = (int)(off / (uint32_t)nblk), kb0 = (int)off - hg * nblk;
        const int n_blk = !FOLD ? 0 : RAG ? blocks_of(mid_of(s, rows.lens.len[b]), rows.R) : rows.n_blk;
        const int kb1 = (int)min((uint32_t)nblk, (uint32_t)kb0 + (pos_end - pos));
        return Seg{b, hg * HP, kb0, kb1, n_blk, kb0 == 0 && kb1 == nblk, g0};
    };

    if (tid == 0) {
        for (int i = 0; i < n_stages; ++i) {
            mbar_init(full + i, kGenWarpsP + 1);
            mbar_init(peer + i, 1);
            mbar_init(empty + i, 1);
        }
        mbar_init(acc_ready, 1);
        mbar_init(epi_done, kGenWarpsP);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kOps * 256) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    if (pos_end > pos_begin) {
        if (warp == 0) {
            // ---------------- TMA producer: this CTA's half of the columns ----------------
            if (lane == 0) {
                asm volatile("griddepcontrol.wait;" ::: "memory");       // the moments
                // (only now: a kernel that this lets start may count the kernel before this one as finished)
                asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
                int it = 0, seg = 0, st = 0;
                uint32_t par = 1;
                bool live = true;
                // (the rows past the last column are whatever the stage held: their accumulator columns are not read)
                const uint32_t bytes = (uint32_t)min(nh, max(0, ncol - (int)rank * nh)) * (4 * kMF);
                for (uint32_t pos = pos_begin; live && pos < pos_end; ++seg) {
                    const Seg g = seg_at(pos);
                    if (seg > 0 && !mbar_wait(epi_done, (seg - 1) & 1, fail, status)) { live = false; break; }
                    for (int kb = g.kb0; kb < g.kb1; ++kb, ++it) {
                        if (!mbar_wait(empty + st, par, fail, status)) { live = false; break; }
                        unsigned char* bdst = stage0 + (size_t)st * n_stage + kTiles * kABytesP;
                        mbar_expect_tx(full + st, kOps * bytes);
                        const char* src = reinterpret_cast<const char*>(Y) +
                                          ((((size_t)g.g0 + kb) * kTiles * s.Hkv + g.h0) * ncol + (size_t)rank * nh) * (size_t)(4 * kMF);
                        if (bytes) {
#pragma unroll
                            for (int o = 0; o < kOps; ++o) bulk_load(bdst + o * b_op, src + (size_t)o * (FOLD ? s.Hkv : 1) * ncol * (4 * kMF), bytes, full + st);
                        }
                        if (++st == n_stages) { st = 0; par ^= 1; }
                    }
                    pos += (uint32_t)(g.kb1 - g.kb0);
                }
                if (!live)                                 // a wait ran out: this CTA's boxes under way land, or the bound is reached, before it ends
                    for (int q = it - n_stages < 0 ? 0 : it - n_stages; q < it; ++q)
                        for (uint32_t n = 0; n < (1u << 16) && !mbar_try_wait(full + q % n_stages, (uint32_t)(q / n_stages) & 1u); ++n) { }
            }
        } else if (warp == 1) {
            // ---------------- MMA issuer: the even CTA, for the pair ----------------
            if (lane == 0 && rank == 0) {
                int st = 0;
                uint32_t par = 0;
                bool live = true;
                for (uint32_t pos = pos_begin; live && pos < pos_end;) {
                    const Seg g = seg_at(pos);
                    for (int kb = g.kb0; kb < g.kb1; ++kb) {
                        if (!mbar_wait(full + st, par, fail, status) || !mbar_wait(peer + st, par, fail, status)) { live = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t a_addr = smem_u32(stage0 + (size_t)st * n_stage), b_addr = a_addr + kTiles * kABytesP;
                        // rows of 128 bytes, 32 hi and 32 lo values: hi hi, lo hi, hi lo, sixteen values at a time
#pragma unroll
                        for (int pr = 0; pr < 3; ++pr)
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks) {
#pragma unroll
                                for (int o = 0; o < kOps; ++o)
                                    umma_bf16_pair(tmem_base + o * 256, umma_desc(a_addr + (FOLD ? o * kABytesP : 0) + (pr == 1 ? 64 : 0) + ks * 32, 1, 1024 >> 4),
                                                   umma_desc(b_addr + o * b_op + (pr == 2 ? 64 : 0) + ks * 32, 1, 1024 >> 4), idesc,
                                                   (kb > g.kb0 || pr > 0 || ks > 0) ? 1u : 0u);
                            }
                        umma_commit_pair(empty + st);
                        if (++st == n_stages) { st = 0; par ^= 1; }
                    }
                    if (live) umma_commit_pair(acc_ready);
                    pos += (uint32_t)(g.kb1 - g.kb0);
                }
            } else if (lane == 0) {
                const int n_it = (int)(pos_end - pos_begin);
                int st = 0;
                uint32_t par = 0;
                for (int it = 0; it < n_it; ++it) {
                    if (!mbar_wait(full + st, par, fail, status)) break;
                    mbar_arrive_cluster(peer + st, 0);
                    if (++st == n_stages) { st = 0; par ^= 1; }
                }
            }
        } else {
            // ---------------- generators: rows Re and Im of e^{i theta n t_b} (2 r + 1) i^r j_r(phi_n), t_b the block's middle or (folded)
            // its distance from the row's middle; Re and Im rows of a frequency follow one another, or lie in tiles of their own ----------------
            constexpr int LT = FOLD ? 1 : 2, NR = kMF >> LT;       // 2^LT threads to a frequency, NR moments each
            const int t = tid - 64;
            const int fi = t >> LT, tq = t & ((1 << LT) - 1);      // frequency of the tile, this thread's share of the moments
            const unsigned n = (unsigned)(mt * (FOLD ? kBMp : kBMp / 2) + fi);
            float gb[NR];                                  // (2 r + 1) j_r(phi_n) for r = NR tq .. NR tq + NR - 1
            legendre_factors<NR>(n, rows.R, s.T, tq, gb);
            const int r0 = FOLD ? fi : 2 * fi, r1 = FOLD ? fi : 2 * fi + 1;
            const uint32_t off0 = (uint32_t)((r0 >> 3) * 1024 + (r0 & 7) * 128), off1 = (uint32_t)((r1 >> 3) * 1024 + (r1 & 7) * 128) + (FOLD ? kABytesP : 0);
            const unsigned T2 = 2u * (unsigned)s.T;
            const float inv_T = 1.0f / (float)s.T;
            int seg = 0, st = 0;
            uint32_t par = 1;
            bool live = true;
            for (uint32_t pos = pos_begin; live && pos < pos_end; ++seg) {
                const Seg g = seg_at(pos);
                for (int kb = g.kb0; kb < g.kb1; ++kb) {
                    // phase of the block's middle: pi n (2 kb R + R - 1) / T, or of its distance: pi n (n_blk - 1 - 2 kb) R / T; exact in integers
                    const unsigned ph = (n * (unsigned)(FOLD ? (g.n_blk - 1 - 2 * kb) * rows.R : 2 * kb * rows.R + rows.R - 1)) % T2;
                    const float f = (float)ph * inv_T;     // in half turns, [0, 2)
                    const float an = 3.14159265358979f * (f - (f >= 1.0f ? 2.0f : 0.0f));
                    const float C = __cosf(an), S = __sinf(an);
                    if (!mbar_wait(empty + st, par, fail, status)) { live = false; break; }
                    unsigned char* a_dst = stage0 + (size_t)st * n_stage;
#pragma unroll
                    for (int u = 0; u < NR / 8; ++u) {
                        const int cq = tq * (NR / 8) + u;  // 16-byte piece of a row: eight moments
                        uint32_t h0[4], l0[4], h1[4], l1[4];
#pragma unroll
                        for (int i2 = 0; i2 < 4; ++i2) {   // moments 2 i2 (i^r = +-1), 2 i2 + 1 (i^r = +-i)
                            const float sg = (i2 & 1) ? -1.f : 1.f;
                            const float ga = sg * gb[8 * u + 2 * i2], go = sg * gb[8 * u + 2 * i2 + 1];
                            split_bf16(ga * C, -go * S, h0[i2], l0[i2]);
                            split_bf16(ga * S, go * C, h1[i2], l1[i2]);
                        }
                        *reinterpret_cast<uint4*>(a_dst + off0 + ((cq ^ (r0 & 7)) << 4)) = make_uint4(h0[0], h0[1], h0[2], h0[3]);
                        *reinterpret_cast<uint4*>(a_dst + off0 + (((4 + cq) ^ (r0 & 7)) << 4)) = make_uint4(l0[0], l0[1], l0[2], l0[3]);
                        *reinterpret_cast<uint4*>(a_dst + off1 + ((cq ^ (r1 & 7)) << 4)) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
                        *reinterpret_cast<uint4*>(a_dst + off1 + (((4 + cq) ^ (r1 & 7)) << 4)) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full + st);
                    if (++st == n_stages) { st = 0; par ^= 1; }
                }
                if (!live) break;
                // ---------------- epilogue of the segment: accumulators are added to the coefficient rows ----------------
                const bool ok = mbar_wait(acc_ready, seg & 1, fail, status);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                asm volatile("griddepcontrol.wait;" ::: "memory");      // (the coefficients are cleared by a kernel before this one)
                if (!ok) break;
                {
                    const int lane_grp = warp & 3, part = (warp - 2) >> 2;
                    // 32 accumulator rows x 32 columns at a time (folded: of both products) through the idle ring: then eight lanes hold a row's 128 bytes
                    float* tile = reinterpret_cast<float*>(stage0) + (warp - 2) * (kTiles * 32 * 36);
                    const int npc = (ncol + 31) >> 5;      // pieces of 32 columns per head
                    const int layer = RAG ? 0 : g.b / s.B;
                    const int row0 = FOLD ? 2 * (mt * kBMp + lane_grp * 32) : mt * kBMp + lane_grp * 32;
                    float cm = 1.f, sm = 0.f;              // e^{i theta n m}, m the row's middle
                    if (FOLD) sincospif((float)(((unsigned)(mt * kBMp + lane_grp * 32 + lane) * (unsigned)(g.n_blk * rows.R - 1)) % T2) * inv_T, &sm, &cm);
#pragma unroll 1
                    for (int pc = part; pc < HP * npc; pc += 2) {
                        const int hh = pc / npc, c0 = (pc - hh * npc) * 32;
                        const uint32_t at = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + (uint32_t)(hh * 256 + c0);
                        if (FOLD) {                        // (16 columns at a time: registers, see below)
#pragma unroll
                            for (int x = 0; x < 32; x += 16) {
                                float v[16], w[16];
                                tmem_ld16_two(at + x, at + 256 + x, v, w);
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    const float re = cm * v[i] - sm * w[i];
                                    w[i] = sm * v[i] + cm * w[i];
                                    v[i] = re;
                                }
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    *reinterpret_cast<float4*>(tile + lane * 36 + x + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                                    *reinterpret_cast<float4*>(tile + (32 + lane) * 36 + x + 4 * i) = make_float4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
                                }
                            }
                        } else {
                            float v[32];
                            tmem_ld32(at, v);
#pragma unroll
                            for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(tile + lane * 36 + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        }
                        __syncwarp();
                        const int q = lane & 7, rr0 = lane >> 3, col = c0 + 4 * q;
                        if (col < ncol) {
                            const bool is_k = col < s.dck;
                            const int nc = is_k ? s.dck : s.dcv;
                            float* dst = coef_rows(is_k ? layers.k[layer] : layers.v[layer], s, g.b - layer * s.B, g.h0 + hh, nc) + (size_t)row0 * nc + (is_k ? col : col - s.dck);
#pragma unroll
                            for (int i = 0; i < 8 * kTiles; ++i) {
                                // row of the coefficients: the tile's, or (folded) Re in rows 0 - 31 and Im in 32 - 63 of the tile, taken in turn
                                const int m = rr0 + 4 * i, src = FOLD ? (m >> 1) + 32 * (m & 1) : m;
                                const float4 x = *reinterpret_cast<const float4*>(tile + src * 36 + 4 * q);
                                if (g.whole) *reinterpret_cast<float4*>(dst + (size_t)m * nc) = x;       // nobody else adds to these
                                else
                                    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + (size_t)m * nc), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w)
                                                 : "memory");
                            }
                        }
                        __syncwarp();
                    }
                }
                pos += (uint32_t)(g.kb1 - g.kb0);
                if (pos < pos_end) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(epi_done);
                    if (!mbar_wait(epi_done, seg & 1, fail, status)) break;
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();
    if (tid == 0 && *fail)                                 // (a wait that runs out tells the first layer)
        for (int l = 1; l < layers.n; ++l) layers.status[l][0] = status[0];
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kOps * 256) : "memory");
    }
}

// ---- windows and counters -------------------------------------------------------------------------------------------
// Behind the projection and beside it: that one leaves the memory idle, this one needs a warp and 49 KB.  A CTA takes a few boxes of 64 tokens of one head and
// side, which one lane moves: in by TMA, out by bulk copies (the window rows of a head are contiguous), two boxes on their way in all the time.
// 270 MB of 256 heads and a projection of 43 us: one after the other 101 us, the partition kernel (16-byte loads and stores, 24 warps of it beside the
// projection) 77 us, this one 63.
constexpr int kWinStages = 3, kWinBytes = 64 * 256;
struct WinIn {
    CUtensorMap k[kMomLayers], v[kMomLayers];
    CacheDev c[kMomLayers];
    int n;
};
__global__ void __launch_bounds__(32) windows_kernel(const __grid_constant__ WinIn in, Dims s, int Lall, const __grid_constant__ RowLens lens, int n_init_ch,
                                                     int n_ch, int per_cta, int n_items, int n_stages) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + n_stages * kWinBytes);
    volatile int* fail = reinterpret_cast<volatile int*>(full + n_stages);
    const int lane = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0)
        for (int i = lane; i < in.n * s.B; i += 32) {
            const int layer = i / s.B, b = i - layer * s.B, L = row_len(lens, Lall, b), n_init = min(L, s.l_init), n_local = min(L - n_init, s.l_local);
            int32_t* st = in.c[layer].state + kStateStride * b;
            st[0] = n_init;
            st[1] = n_local;
            st[2] = L - n_init - n_local;
            st[3] = 0;                                     // ring starts at physical row 0
            st[4] = 0;                                     // append ticket
        }
    if (lane == 0) {
        for (int i = 0; i < n_stages; ++i) mbar_init(full + i, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // box i: head fastest, then the chunk of the windows, side, batch row, layer
        struct Box { int layer, b, h, side, tok, rows; bf16* dst; };
        auto box = [&](int i) {
            Box x;
            int r = i / s.Hkv, ch;
            x.h = i - r * s.Hkv;
            ch = r % n_ch; r /= n_ch;
            x.side = r & 1; r >>= 1;
            x.layer = r / s.B;
            x.b = r - x.layer * s.B;
            const int L = row_len(lens, Lall, x.b), n_init = min(L, s.l_init), n_local = min(L - n_init, s.l_local);
            const CacheDev& c = in.c[x.layer];
            const int row = (ch < n_init_ch ? ch : ch - n_init_ch) * 64, n = ch < n_init_ch ? n_init : n_local;
            x.rows = min(64, n - row);
            x.tok = (ch < n_init_ch ? 0 : L - n_local) + row;
            x.dst = x.rows <= 0 ? nullptr : ch < n_init_ch ? win_row<bf16>(x.side ? c.v_init : c.k_init, s, x.b, x.h, s.l_init, row)
                                                           : win_row<bf16>(x.side ? c.v_local : c.k_local, s, x.b, x.h, s.l_local, row);
            return x;
        };
        const int i0 = blockIdx.x * per_cta, i1 = min(n_items, i0 + per_cta);
        const uint32_t bytes = (uint32_t)(64 * s.d * 2);
        auto load = [&](int i) {
            const Box x = box(i);
            const int st = (i - i0) % n_stages;
            if (x.rows <= 0) { mbar_arrive(full + st); return; }
            mbar_expect_tx(full + st, bytes);
            tma_load_4d(smem + st * kWinBytes, x.side ? &in.v[x.layer] : &in.k[x.layer], 0, x.h, x.tok, x.b, full + st);
        };
        for (int i = i0; i < i1 && i < i0 + n_stages - 1; ++i) load(i);
        int i = i0;
        for (; i < i1; ++i) {
            const int st = (i - i0) % n_stages;
            if (!mbar_wait(full + st, ((i - i0) / n_stages) & 1, fail, in.c[0].status)) break;
            const Box x = box(i);
            if (x.rows > 0)
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(x.dst)), "r"(smem_u32(smem + st * kWinBytes)),
                             "r"(x.rows * s.d * 2)
                             : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");       // the copy before has read its stage
            if (i + n_stages - 1 < i1) load(i + n_stages - 1);
        }
        if (i < i1)                                        // a wait ran out: the boxes under way land, or the bound is reached, first
            for (int q = i; q < i1 && q < i + n_stages - 1; ++q)
                for (uint32_t n = 0; n < (1u << 16) && !mbar_try_wait(full + (q - i0) % n_stages, ((q - i0) / n_stages) & 1); ++n) { }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if (*fail)
            for (int l = 1; l < in.n; ++l) in.c[l].status[0] = in.c[0].status[0];
        // (one CTA waits for the kernel in front, so that the end of this grid implies that one's)
        if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
}

int npad_of(const Dims& s) { return (s.dck + s.dcv + 31) / 32 * 32; }

// Whether the blocks may be taken in pairs about the middle of a row: the projection then takes 256 frequencies at a time.
bool can_fold(const Dims& s) { return s.k % 256 == 0; }
// Whether a launch does so: n_pairs pairs, n_blocks blocks of all rows and layers.  In us: 3 for coarser work (256 frequencies to a segment, SMs without a pair while the
// last of the moments are formed), less a 110th of the projection's positions for its halved products; what is longer at the moments' end, where the busiest
// CTA has two blocks more instead of one (a 320th of a us per token); a 190th per pair and head of blocks past 384 tokens, whose tables leave the
// moments' ring a stage less.  Fitted to 270 launches of 4 to 32 heads, 512 to 2048 coefficients, rows of one length and of several: 0.25 % behind the better form on average,
// 5 % at worst (2048 coefficients, 448 positions: 47.5/49.4).  us, plain / folded:
//   512 coefficients, 32 heads, blocks of 384: 352 positions 58.2/58.3, 384 61.9/63.0 (two blocks more), 416 64.8/64.1, 512 73.5/72.4, 1024 135/128
//   the same, blocks of 768: 416 positions 98.1/99.0, 448 103.9/109.3, 480 108.1/111.9 (both two blocks more), 576 129.6/130.1, 1088 216/213
//   1024 coefficients, 8 heads, blocks of 384: 368 positions 43.4/43.4, 400 46.1/44.5, 432 47.5/45.3, 688 62.1/58.3
//   2048 coefficients, 8 heads, blocks of 768: 416 positions 45.5/47.8 (two blocks more), 480 51.8/50.6, 1024 84.4/80.4, 11008 765/673
//   512 coefficients, 8 heads, six ragged rows: 424 positions 70.2/68.7, 544 82.6/80.8
bool folds(const Dims& s, long long n_pairs, long long n_blocks) {
    if (!can_fold(s)) return false;
    const long long items = s.Hkv * (s.d == 128 ? 2 : 1), sms = sm_count();
    auto turns = [&](long long n) { return (n * items + sms - 1) / sms; };
    const int R = block_tokens(s);
    const double more = 3.0 - (double)(n_pairs * s.Hkv * (s.k / 256)) / 110.0 + (double)(2 * turns(n_pairs) - turns(n_blocks)) * R / 320.0 +
                        (R > 384 ? (double)(n_pairs * s.Hkv) / 190.0 : 0.0);
    return more < 0.0;
}

// The projection's stages leave room for a CTA of the windows kernel beside it: one of three stages, or of two where the projection would otherwise
// have two itself (more than 192 columns, folded: 22 us instead of 16 for a head group of 256 columns, 512 coefficients and 3600 tokens).
constexpr size_t kProjectFixed = 8 * (3 * kStagesP + 2) + 16 + 1024;
size_t project_stage_bytes(const Dims& s, bool fold) {
    return fold ? 2 * kABytesP + (size_t)npad_of(s) * 128 : kABytesP + (size_t)(s.Hkv % 2 == 0 ? 2 : 1) * (npad_of(s) / 2) * 128;
}
int project_fit(const Dims& s, bool fold, int win_stages) {
    const int n = (int)((227 * 1024 - (win_stages * kWinBytes + 1280) - kProjectFixed) / project_stage_bytes(s, fold));
    return n < kStagesP ? n : kStagesP;
}
int windows_stages(const Dims& s) { return project_fit(s, can_fold(s), kWinStages) >= 3 ? kWinStages : kWinStages - 1; }
int project_stages(const Dims& s, bool fold) { return project_fit(s, fold, windows_stages(s)); }

size_t mom_tables(const Dims& s) { return (size_t)s.Hkv * (2 * s.d + s.nfk + s.nfv); }
size_t mom_smem_fixed(const Dims& s, bool fold, int n_layers) {      // everything but the stages, the slack of the alignment among it
    return (size_t)block_tokens(s) / kChunk * kHChunk + (fold ? 2 : 1) * 128 * 4 * kMF + 8 * (3 * 16 + 2 * kAcc) + 16 + (size_t)n_layers * mom_tables(s) + 64 + 1024;
}
int mom_stages(const Dims& s, bool fold, int n_layers) {
    const long long left = 227 * 1024 - (long long)mom_smem_fixed(s, fold, n_layers);
    const int n = (int)(left / kChunkBytes);
    return n > 16 ? 16 : n;
}

// chained: behind a kernel of the same call (else all work in front of it on the stream has ended when it starts, so that it may write anything)
template <int D, bool RAG, bool FOLD>
cudaError_t launch_moments(const MomIn& in, const Dims& s, int L, const MomRows& rows, void* Y, bool wait_first, bool chained, cudaStream_t stream) {
    const int n_stages = mom_stages(s, FOLD, in.n);
    const size_t smem = mom_smem_fixed(s, FOLD, in.n) + (size_t)n_stages * kChunkBytes;
    cudaError_t err = ensure_dynamic_smem(moments_kernel<D, RAG, FOLD>, smem);
    if (err != cudaSuccess) return err;
    const long long items = (long long)rows.total * s.Hkv * (D == 128 ? 2 : 1);
    if (items <= 0 || items >= (1ll << 31)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items < sm_count() ? items : sm_count()));
    cfg.blockDim = dim3(kThreadsMom);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, moments_kernel<D, RAG, FOLD>, in, s, L, rows, static_cast<bf16*>(Y), n_stages, (int)items, wait_first ? 1 : 0);
}

template <int HP, bool RAG, bool FOLD>
cudaError_t launch_project(const void* Y, const Dims& s, const CacheDev* c, int n_layers, const MomRows& rows, cudaStream_t stream) {
    MomLayers layers = {};
    layers.n = n_layers;
    for (int i = 0; i < n_layers; ++i) { layers.k[i] = c[i].coef_k; layers.v[i] = c[i].coef_v; layers.status[i] = c[i].status; }
    const int n_stages = project_stages(s, FOLD);
    // (more than half of an SM's: each CTA takes all of its tensor memory, a second one could only wait for that)
    const size_t smem = std::max(n_stages * project_stage_bytes(s, FOLD) + kProjectFixed, (size_t)116 * 1024);
    cudaError_t err = ensure_dynamic_smem(moment_project_kernel<HP, RAG, FOLD>, smem);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreadsP);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    // all of the SM's memory as shared memory, whatever this kernel takes of it: CTAs of the windows kernel start beside it
    attr[2].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[2].val.sharedMemCarveout = 100;
    cfg.attrs = attr;
    cfg.numAttrs = 3;
    const int n_pairs = s.M / ((FOLD ? 4 : 2) * kBMp), n_hg = s.Hkv / HP;
    const long long total = (long long)rows.total * n_hg;
    if (total <= 0 || total >= (1ll << 31)) return cudaErrorInvalidValue;
    int n_teams;
    {
        // pairs resident at once (cached per device): the teams fill them, no second wave
        static int resident[16] = {};
        static std::mutex mu;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) return cudaErrorInvalidValue;
        std::lock_guard<std::mutex> lock(mu);
        if (resident[dev] == 0) {
            cfg.gridDim = dim3(2 * sm_count());
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, moment_project_kernel<HP, RAG, FOLD>, &cfg) != cudaSuccess || n < 1) {
                cudaGetLastError();
                n = sm_count() / 2 - 2;
            }
            cfg.numAttrs = 3;
            resident[dev] = n;
        }
        n_teams = resident[dev] / n_pairs;
    }
    if (n_teams < 1) n_teams = 1;
    if (n_teams > kMaxTeamsP) n_teams = kMaxTeamsP;
    if (n_teams > total) n_teams = (int)total;
    // Equal cost per team: a segment costs its positions plus its epilogue and refill, kEpi where its sums are added to others', kWhole where a unit is
    // taken whole and they are stored; the smallest budget with which the walk covers all positions in n_teams teams, by bisection.
    // (Folded units of fewer than 16 positions were taken whole at a kWhole of 9, by as many teams as there are units, where the others had nothing to
    // do.  us at 9 / 12, the same at 16: 32 heads of 512 coefficients, 13 positions each 69.3/64.1, 15 each 75.6/70.2; 8 heads of 2048, 14 each 52.2/49.4;
    // four rows of 86 positions and 2048 coefficients 690/673; six layers of 32 K tokens 273/273 (277 at 16).  Rows of different length, whose longest
    // units alone are shared, at 9 / 10 / 12: six rows of 2 to 15 positions and 8 heads, 104 and 88 columns, windows of 1024 tokens 72.0/72.0/72.9;
    // 96 columns 69.6/68.0/68.1, windows of 64 tokens 66.2/65.1/62.8; five rows of 4 to 13 120.7/115.4/121.9.)
    MomCuts cuts = {};
    constexpr long long kEpi = FOLD ? 16 : 6, kWhole = FOLD ? (RAG ? 10 : 12) : 4, kMinSeg = 2;
    auto unit_of = [&](long long pos, long long* begin) {  // returns its end
        long long first = 0, nblk = rows.nblk;
        if (RAG) {
            int b = 0;
            while (pos >= (long long)rows.first[b + 1] * n_hg) ++b;
            first = (long long)rows.first[b] * n_hg;
            nblk = (long long)rows.first[b + 1] - rows.first[b];
        }
        *begin = first + (pos - first) / nblk * nblk;
        return *begin + nblk;
    };
    auto walk = [&](long long budget, uint32_t* start) {
        long long pos = 0;
        int t = 0;
        for (; t < n_teams && pos < total; ++t) {
            if (start) start[t] = (uint32_t)pos;
            long long left = budget;
            while (pos < total && left >= kWhole + kMinSeg) {
                long long unit_begin;
                const long long unit_end = unit_of(pos, &unit_begin);
                if (pos == unit_begin && unit_end - pos + kWhole <= left) {
                    pos = unit_end;
                    left -= unit_end - unit_begin + kWhole;
                    continue;
                }
                if (left < kEpi + kMinSeg) break;
                long long take = unit_end - pos < left - kEpi ? unit_end - pos : left - kEpi;
                if (unit_end - pos - take > 0 && unit_end - pos - take < kMinSeg) take = unit_end - pos - kMinSeg;
                if (take <= 0) break;
                pos += take;
                left -= take + kEpi;
            }
        }
        if (start)
            for (int u = t; u <= n_teams; ++u) start[u] = (uint32_t)(u == n_teams ? total : pos);
        return pos >= total;
    };
    long long lo = kEpi + kMinSeg, hi = total + kEpi * (total + 1) + kMinSeg;
    while (lo < hi) {
        const long long mid = (lo + hi) / 2;
        if (walk(mid, nullptr)) hi = mid; else lo = mid + 1;
    }
    while (!walk(lo, cuts.start)) ++lo;
    cuts.start[n_teams] = (uint32_t)total;
    cfg.gridDim = dim3(2 * n_teams * n_pairs);
    return cudaLaunchKernelEx(&cfg, moment_project_kernel<HP, RAG, FOLD>, static_cast<const bf16*>(Y), s, layers, rows, cuts, npad_of(s), n_stages);
}

}  // namespace

// True if the two-step contraction serves this layout: what the pair kernel of the direct contraction needs, tables that
// fit beside the ring, and blocks of at least three boxes (T / k >= 32: the axis is then six times shorter, which three products
// and the round trip of the moments still leave 5 % ahead of the direct contraction; half of that would lose).
bool compress_mom_supported(const Dims& s) {
    if (s.M % (2 * kBMp) != 0 || s.d > 128 || s.dck + s.dcv == 0) return false;
    if (block_tokens(s) < 3 * kChunk) return false;
    if (mom_stages(s, can_fold(s), 1) < 5) return false;
    // phases n (2 j + R - 1) stay in 32 bits
    return (unsigned long long)(s.M / 2) * (2ull * (unsigned long long)s.T + 2ull * kMaxBlockTokens) < (1ull << 32);
}

// Bytes of moments that a batch row of n_mid middle tokens needs (of a layout that is supported).
size_t compress_mom_row_bytes(const Dims& s, int n_mid) {
    const int R = block_tokens(s);
    const int n = blocks_of(n_mid, R);
    return (size_t)(can_fold(s) ? (n + 1) / 2 * 2 : n) * s.Hkv * (s.dck + s.dcv) * (4 * kMF);
}

static cudaError_t launch_rows(const Dims& s, const CacheDev* c, const void* const* K, const void* const* V, int n_layers, int64_t sb, int64_t st,
                               int64_t sh, int L, MomRows rows, bool fold, char* Y, bool wait_first, bool chained, cudaStream_t stream) {
    const bool rag = rows.lens.n != 0;
    cudaError_t err;
    // Layers to a launch: as many as a sixth of the ring's room holds the tables of.  A launch of its own for each pays its start, its first loads
    // and its last items every time.
    int per = (int)(32 * 1024 / (mom_tables(s) + 1));
    if (per < 1) per = 1;
    per = (n_layers + (n_layers + per - 1) / per - 1) / ((n_layers + per - 1) / per);
    for (int i = 0; i < n_layers; i += per) {
        MomIn in = {};
        in.n = n_layers - i < per ? n_layers - i : per;
        for (int l = 0; l < in.n; ++l) {
            in.c[l] = c[i + l];
            if (!prefill_map(&in.k[l], K[i + l], s, sb, st, sh, L) || !prefill_map(&in.v[l], V[i + l], s, sb, st, sh, L)) return cudaErrorInvalidValue;
        }
        MomRows part = rows;
        part.nb *= in.n;
        part.total *= in.n;
        char* y = Y + (size_t)i * rows.total * (fold ? 2 : 1) * s.Hkv * (s.dck + s.dcv) * (4 * kMF);
        auto launch = [&](auto d, auto r, auto f) { return launch_moments<decltype(d)::value, decltype(r)::value, decltype(f)::value>(in, s, L, part, y, wait_first, chained || i > 0, stream); };
        auto by_fold = [&](auto d, auto r) { return fold ? launch(d, r, std::true_type{}) : launch(d, r, std::false_type{}); };
        auto by_rows = [&](auto d) { return rag ? by_fold(d, std::true_type{}) : by_fold(d, std::false_type{}); };
        err = s.d == 128 ? by_rows(std::integral_constant<int, 128>{}) : by_rows(std::integral_constant<int, 64>{});
        if (err != cudaSuccess) return err;
    }
    rows.nb *= n_layers;
    rows.total *= n_layers;
    if (fold) return rag ? launch_project<1, true, true>(Y, s, c, n_layers, rows, stream) : launch_project<1, false, true>(Y, s, c, n_layers, rows, stream);
    if (s.Hkv % 2 == 0) return rag ? launch_project<2, true, false>(Y, s, c, n_layers, rows, stream) : launch_project<2, false, false>(Y, s, c, n_layers, rows, stream);
    return rag ? launch_project<1, true, false>(Y, s, c, n_layers, rows, stream) : launch_project<1, false, false>(Y, s, c, n_layers, rows, stream);
}

// Coefficients and the kept-dim rows of the middle tokens of batch rows b0 .. b0 + nb; the windows and the counters are left to launch_windows
// or the partition kernel, launched behind.  lens: prompt lengths of all batch rows (at most L; rows
// with fewer than tc_min middle tokens are left out), or none.  Y: room for these rows' moments, 128-byte aligned;
// wait_first: a kernel of this call that may still run reads Y; chained: there is a kernel of this call in front.
cudaError_t launch_compress_mom(const Dims& s, const CacheDev& c, const void* K, const void* V, int64_t sb, int64_t st, int64_t sh, int L, int b0,
                                int nb, void* Y, bool wait_first, bool chained, cudaStream_t stream, const RowLens* lens, int tc_min) {
    MomRows rows = {};
    rows.R = block_tokens(s);
    rows.b0 = b0;
    rows.nb = nb;
    auto pairs = [&](int n_mid) { return (blocks_of(n_mid, rows.R) + 1) / 2; };
    long long n_pairs = 0, n_blocks = 0;
    for (int b = b0; b < b0 + nb; ++b) {
        const int m = lens && lens->n == s.B ? mid_of(s, lens->len[b]) : mid_of(s, L);
        if (!lens || !lens->n || m >= tc_min) { n_pairs += pairs(m); n_blocks += blocks_of(m, rows.R); }
    }
    const bool fold = folds(s, n_pairs, n_blocks);
    auto positions = [&](int n_mid) { return fold ? pairs(n_mid) : blocks_of(n_mid, rows.R); };
    if (lens && lens->n) {
        if (lens->n != s.B) return cudaErrorInvalidValue;
        rows.lens = *lens;
        long long at = 0;
        for (int b = 0; b < s.B; ++b) {
            const int m = mid_of(s, lens->len[b]);
            if (b >= b0 && b < b0 + nb && m >= tc_min) at += positions(m);
            if (at >= (1ll << 24)) return cudaErrorInvalidValue;
            rows.first[b + 1] = (uint32_t)at;
        }
        rows.total = (int)at;
    } else {
        rows.n_blk = blocks_of(mid_of(s, L), rows.R);
        rows.nblk = positions(mid_of(s, L));
        if ((long long)rows.nblk * nb >= (1ll << 24)) return cudaErrorInvalidValue;
        rows.total = rows.nblk * nb;
    }
    if (rows.total == 0) return cudaSuccess;
    return launch_rows(s, &c, &K, &V, 1, sb, st, sh, L, rows, fold, static_cast<char*>(Y), wait_first, chained, stream);
}

// The same for all batch rows of up to kMomLayers layers of one shape: moment kernels of several layers each, then one projection.  A projection
// takes 31 us (plain form) for a layer of 8 heads, 32K tokens and 1024 coefficients, a third of it its start and the segments that teams
// share, which six layers together pay once: 6 x 31 -> 115 us, folded 72.  Y: room for the moments of all of them.
cudaError_t launch_compress_mom_layers(const Dims& s, const CacheDev* c, const void* const* K, const void* const* V, int n_layers, int64_t sb, int64_t st,
                                       int64_t sh, int L, void* Y, bool wait_first, bool chained, cudaStream_t stream) {
    if (n_layers < 1 || n_layers > kMomLayers) return cudaErrorInvalidValue;
    MomRows rows = {};
    rows.R = block_tokens(s);
    rows.nb = s.B;
    rows.n_blk = blocks_of(mid_of(s, L), rows.R);
    const long long n_rows = (long long)s.B * n_layers;
    const bool fold = folds(s, (long long)(rows.n_blk + 1) / 2 * n_rows, rows.n_blk * n_rows);
    rows.nblk = fold ? (rows.n_blk + 1) / 2 : rows.n_blk;
    rows.total = rows.nblk * s.B;
    if (rows.total == 0) return cudaSuccess;
    if ((long long)rows.nblk * s.B * n_layers >= (1ll << 24)) return cudaErrorInvalidValue;
    return launch_rows(s, c, K, V, n_layers, sb, st, sh, L, rows, fold, static_cast<char*>(Y), wait_first, chained, stream);
}

// The windows and counters of layers whose middles launch_compress_mom(_layers) has enqueued in front, on the same stream.
cudaError_t launch_windows(const Dims& s, const CacheDev* c, const void* const* K, const void* const* V, int n_layers, int64_t sb, int64_t st, int64_t sh, int L,
                           cudaStream_t stream, const RowLens* lens) {
    RowLens rl = {};
    if (lens) rl = *lens;
    // chunks of the longest windows of any row (a row's own may be fewer)
    const int n_init = L < s.l_init ? L : s.l_init, n_local = L - n_init < s.l_local ? L - n_init : s.l_local;
    const int n_init_ch = (n_init + 63) / 64, n_ch = n_init_ch + (n_local + 63) / 64;
    const int n_stages = windows_stages(s);
    const size_t smem = n_stages * kWinBytes + 8 * n_stages + 16;
    cudaError_t err = ensure_dynamic_smem(windows_kernel, smem);
    if (err != cudaSuccess) return err;
    for (int i = 0; i < n_layers; i += kMomLayers) {
        WinIn in = {};
        in.n = n_layers - i < kMomLayers ? n_layers - i : kMomLayers;
        for (int l = 0; l < in.n; ++l) {
            in.c[l] = c[i + l];
            if (!prefill_map(&in.k[l], K[i + l], s, sb, st, sh, L, s.d, CU_TENSOR_MAP_SWIZZLE_NONE) || !prefill_map(&in.v[l], V[i + l], s, sb, st, sh, L, s.d, CU_TENSOR_MAP_SWIZZLE_NONE))
                return cudaErrorInvalidValue;
        }
        const long long items = (long long)in.n * s.B * 2 * n_ch * s.Hkv;
        if (items >= (1ll << 30)) return cudaErrorInvalidValue;
        // (a few boxes to a CTA: short enough for an even end, long enough for the ring to pay)
        long long per = items / (2 * sm_count());
        per = per < 3 ? 3 : per > 8 ? 8 : per;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(items > 0 ? (items + per - 1) / per : 1));
        cfg.blockDim = dim3(32);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        err = cudaLaunchKernelEx(&cfg, windows_kernel, in, s, L, rl, n_init_ch, n_ch > 0 ? n_ch : 1, (int)per, (int)items, n_stages);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

}  // namespace fa
