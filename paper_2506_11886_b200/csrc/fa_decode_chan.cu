// fa_decode_attention and fa_decode_step (Eq.5-6) for bf16 caches: the compressed dims by Legendre channels over the residue
// classes.
//
// A middle token j = c + P a (class c, slot a) sees the basis at phases theta n j = theta n c0 + phi_n t_c + 2 pi n a / S with
// c0 = (P - 1) / 2, t_c = (2 c + 1 - P) / P in [-1, 1], S = T / P slots and phi_n = pi n / S <= pi (n < k <= S), so
//   e^{i theta n j} = e^{i theta n c0} e^{2 pi i n a / S} sum_{r < 16} (2 r + 1) i^r j_r(phi_n) P_r(t_c)      (left out: 5e-10).
// The scores of the compressed dims are then  sum_r P_r(t_c) Z[a][r]  with one transform of length S per CHANNEL r
// and head, Z[.][r] = Re DFT_n((2 r + 1) i^r j_r u~_n e^{i theta n c0}), instead of one per class (16 instead of P = 32 to 256),
// and the way back is  W[a][r] = sum_c P_r(t_c) p[c][a],  z_n = e^{i theta n c0} sum_r (2 r + 1) i^r j_r DFT_a(W[a][r]).
// Expanding channels to tokens and back are small matrix products, so the kernel that streams the tokens is an ordinary
// attention kernel with three more mma per 32 tokens each way.
//
// Three launches, a push of Eq.5 included:
//   chan_in_kernel    u = scale log2(e) W C^K q, then Z; a cluster of up to eight CTAs per (batch row, KV head)
//   chan_main_kernel  tokens: parts of the slots, and parts of the window tokens; per part (m, l, o), W per slot
//   chan_out_kernel   parts merged, z, its product with C^V, the output rows; clusters as in front
// No CTA waits for another one outside its cluster; the kernels are chained with programmatic dependent launch.  P and Z, and the
// probabilities of the way back, are held as two bf16 numbers each (2^-17), three products; the kept dims as everywhere
// (q . K exact, p rounded to bf16 for p . V).
// A launch takes up to four layers whose memory is apart: the outer kernels are chains of round trips that leave the SMs half idle, and the middle
// one's parts end evenly.  A step, transform kernel -> a layer by itself -> layers together: 8 rows of 32 KV heads, 4K tokens 118 -> 100 -> 78 us (14 + 50 + 14
// by kernel, four layers; 56 us of bytes), 4 rows of 8 KV heads, 128K tokens 242 -> 190 -> 162 us (28 + 103 + 30, two layers; 101 us of bytes).
#include <type_traits>

#include "fa_decode_fft.cuh"

namespace fa {
namespace {

constexpr int kMR = 16;              // channels
constexpr int kMainWarps = 4;
constexpr int kMainCtas = 3;         // CTAs of the main kernel to an SM
constexpr int kWinStage = 4096;      // window parts of the main kernel: 16 rows of K or of V
// CTAs of the outer kernels to an SM: three where 80 registers do without spills, which several layers in a launch fill (the instances of 64 and 512
// slots, whose last pass is of eight points, spill 400 bytes there).
// Threads of an outer kernel's CTA.  Where the longest transforms leave room for one CTA to an SM, it has sixteen warps instead of eight (wide, see plan_channels).
__host__ __device__ constexpr int outer_threads(bool wide) { return wide ? 512 : 256; }
__host__ __device__ constexpr int outer_ctas(int ls, bool wide) { return wide ? 1 : ls == 5 || ls == 7 || ls == 8 ? 3 : 2; }
// Stages of rows that a turn of an outer kernel's loops takes: two of the kernel in front's (eight lanes to a row), and the threads' share; one with the longest transforms
// in eight warps, whose CTAs have few rows or little room for stages.
__host__ __device__ constexpr int in_turn(int ls, bool wide) { return ls == 10 && !wide ? 1 : 2; }
__host__ __device__ constexpr int out_stages(int ls, bool wide) { return ls == 10 && !wide ? 1 : outer_threads(wide) / 128; }
constexpr double kPartCost = 64 * 1024;          // what a part of the main kernel costs beside its bytes, in bytes

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
// x, y as bf16 pairs: rounded, and what the rounding left
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
    hi = pack2(x, y);
    lo = pack2(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}

// (2 r + 1) j_r(pi n / S) of channels 2 q0 .. 2 q0 + 2 nq for n < k, into g_s[2 nq][k].
template <int NT>
__device__ __forceinline__ void channel_factors(float* g_s, int q0, int nq, int k, int S, int tid) {
    for (int n = tid; n < k; n += NT) {
        float keep[kMR];
#pragma unroll
        for (int r = 0; r < kMR; ++r) keep[r] = 0.f;
        if (n == 0) {
            keep[0] = 1.f;
        } else {
            // recurrence downward from r = 24 (phi <= pi), scaled by the closed form of the larger of j_0 and j_1; the start is
            // lower for small phi, whose values would leave fp32's range
            const float x = (float)n / (float)S, phi = 3.14159265358979f * x, inv = 1.0f / phi;
            const int top = min(24, 8 + (int)(24.0f * x));
            float jn = 0.f, jc = 0.f;
#pragma unroll
            for (int r = 24; r >= 0; --r) {
                if (r == top) jc = 1e-18f;
                if (r < kMR) keep[r] = jc;
                const float jp = fmaf((float)(2 * r + 1) * inv, jc, -jn);
                jn = jc;
                jc = jp;
            }
            float sn, cs;
            sincospif(x, &sn, &cs);
            const float t0 = sn * inv, t1 = (t0 - cs) * inv, sc = fabsf(t0) > fabsf(t1) ? t0 / keep[0] : t1 / keep[1];
#pragma unroll
            for (int r = 0; r < kMR; ++r) keep[r] *= sc * (float)(2 * r + 1);
        }
#pragma unroll
        for (int r = 0; r < kMR; ++r)
            if (r >= 2 * q0 && r < 2 * (q0 + nq)) g_s[(r - 2 * q0) * k + n] = keep[r];
    }
}

// Over how many threads (as a power of two) the nq channel pairs (a power of two) of a bin are split so that `items` bins fill the CTA.
__device__ __forceinline__ int split_pairs(int items, int nq, int threads) {
    int lg = 0;
    while ((items << lg) < threads && (2 << lg) <= nq) ++lg;
    return lg;
}
template <int LS, int NT>
__device__ __forceinline__ void pass_twiddles(float* twf, int tid) {
    for (int l = LS; l > 0;) {
        const int rl = radix_log2(l), R = 1 << rl, st = 1 << (l - rl);
        if (l > rl) {
            const int off = tw_offset(LS, l);
            for (int i = tid; i < (R - 1) * st; i += NT) {
                const int qm1 = i >> (l - rl), j = i & (st - 1);
                reinterpret_cast<float2*>(twf)[off + i] = cis_frac((float)(((qm1 + 1) * j) & ((1 << l) - 1)) * (1.0f / (float)(1 << l)));
            }
        }
        l -= rl;
    }
}
// e^{i theta n c0}, c0 = (P - 1) / 2
__device__ __forceinline__ float2 mid_phase(int n, const Dims& s) {
    return cis_frac((float)(((unsigned)n * (unsigned)(s.P - 1)) & (unsigned)(2 * s.T - 1)) * (0.5f / (float)s.T));
}

// ---- clusters: the CTAs of one (batch row, KV head, pass of query heads) ----
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_meet(int n) {
    if (n > 1) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_peer(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void st_peer4(uint32_t a, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ float2 ld_peer2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float ld_peer(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
// the sum of the CTAs' values at one place of their shared memory, in rank order
__device__ __forceinline__ float sum_peers(uint32_t a, int n) {
    float y[8], v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) y[w] = w < n ? ld_peer(peer_addr(a, (uint32_t)w)) : 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += y[w];
    return v;
}

__device__ __forceinline__ float2 sum_peers2(uint32_t a, int n) {
    float2 y[8], v = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < 8; ++w) y[w] = w < n ? ld_peer2(peer_addr(a, (uint32_t)w)) : make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < 8; ++w) { v.x += y[w].x; v.y += y[w].y; }
    return v;
}

// Eq.5's decision for one batch row: the state before it, where the new token goes, the basis column (or -1).
struct Push { int n_init, n_local, n_mid, head, j, buf, row; bool full; };
__device__ __forceinline__ Push push_of(const int32_t* st, const Dims& s) {
    Push x;
    const int4 v = *reinterpret_cast<const int4*>(st);
    x.n_init = v.x; x.n_local = v.y; x.n_mid = v.z; x.head = v.w;
    const bool to_init = x.n_init < s.l_init, evict = !to_init && x.n_local == s.l_local;
    x.full = evict && (x.n_mid >= s.max_mid || x.n_mid >= s.T);
    x.j = evict && !x.full ? x.n_mid : -1;
    x.buf = to_init ? 0 : evict && s.l_local == 0 ? -1 : 1;
    x.row = to_init ? x.n_init : evict ? x.head : (x.head + x.n_local >= s.l_local ? x.head + x.n_local - s.l_local : x.head + x.n_local);
    return x;
}
// The row that leaves the local window on a push (the new token itself without a local window), one side.
__device__ __forceinline__ const bf16* leaving_row(const CacheDev& c, const Dims& s, int b, int h, int side, int head, const bf16* tok) {
    if (s.l_local == 0) return tok + ((size_t)b * s.Hkv + h) * s.d;
    return win_row<bf16>(side == 0 ? c.k_local : c.v_local, s, b, h, s.l_local, head);
}

// Rows of coefficients of a CTA come in by bulk copies, kStageRows rows to a stage; as many as the stages hold set off at once, the
// rest is asked for in L2.  All threads use a stage (wait), then one refills it (done).  Stages and their phases are carried along: as remainders and
// quotients of the stage's number they were a third of the time of the loops over the rows.
constexpr int kStageRows = 32, kMaxRowStages = 8;
struct RowStream {
    uint64_t* bar;                                         // [stages]
    float* buf;
    const float* src;
    int rows, nc, n_st, n_chunk;
    int st = 0, ist = 0;                                   // next stage to use; to refill (one thread)
    uint32_t ph = 0;
    __device__ __forceinline__ void issue(int i) {         // (one thread) chunk i into the stage after the one before
        const uint32_t bytes = (uint32_t)(min(kStageRows, rows - i * kStageRows) * nc * 4), bb = smem_addr(bar + ist);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bb), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(buf + ist * kStageRows * nc)),
                     "l"(__cvta_generic_to_global(src + (size_t)i * kStageRows * nc)), "r"(bytes), "r"(bb)
                     : "memory");
        if (++ist == n_st) ist = 0;
    }
    __device__ __forceinline__ void begin() {              // (one thread; the barriers are initialised)
        for (int i = 0; i < n_st && i < n_chunk; ++i) issue(i);
        const int left = rows - n_st * kStageRows;
        if (left > 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(src + (size_t)n_st * kStageRows * nc)), "r"(left * nc * 4) : "memory");
    }
    __device__ __forceinline__ const float* wait(int k, volatile int* fail, int32_t* status) const {      // the k-th stage from the next one on
        int x = st + k;
        uint32_t p = ph;
        if (x >= n_st) { x -= n_st; p ^= 1; }
        mbar_wait(bar + x, p, fail, status);
        return buf + x * kStageRows * nc;
    }
    __device__ __forceinline__ void next(int n) {          // past n stages (at most as many as there are)
        st += n;
        if (st >= n_st) { st -= n_st; ph ^= 1; }
    }
    __device__ __forceinline__ void done(int i, int n, int tid) {                // chunks i .. i + n (all threads)
        if (i + n_st < n_chunk) {
            __syncthreads();
            if (tid == 0)
                for (int x = i; x < i + n && x + n_st < n_chunk; ++x) issue(x + n_st);
        }
    }
};

// The main kernel's class parts of batch row b: n_cx CTAs per (KV head, pass), shared out over the rows by their filled slots, at
// least one each (a row with three times the mean's tokens gets three times the CTAs).
struct RowParts { int b, x0, cnt; };
__device__ __forceinline__ int supersteps(const int32_t* state, const Dims& s, int b) {
    return (min(state[kStateStride * b + 2], s.max_mid) + 4 * s.P - 1) / (4 * s.P);
}
// the row whose parts hold CTA x (x < 0: the parts of row b); b = s.B: what the shares' rounding left over
__device__ __forceinline__ RowParts row_parts(const int32_t* state, const Dims& s, int n_cx, int x, int b) {
    if (s.B == 1) return RowParts{0, 0, n_cx};
    int total = 0;
#pragma unroll 8
    for (int i = 0; i < s.B; ++i) total += supersteps(state, s, i);
    RowParts r = {0, 0, 0};
#pragma unroll 4
    for (; r.b < s.B; ++r.b) {
        r.x0 += r.cnt;
        r.cnt = 1 + (total > 0 ? (int)((long long)(n_cx - s.B) * supersteps(state, s, r.b) / total) : 0);
        if (x >= 0 ? x < r.x0 + r.cnt : r.b == b) break;
    }
    return r;
}

// The layers of a call (each a fa_decode_step or fa_decode_attention of its own; k_new null: the latter).  Layers of one layout that do not touch
// one another's memory share the three launches: the kernels in front and behind are chains of short phases, which CTAs at different places in theirs fill
// for one another, and a launch's start and end are paid once.
struct ChanLayer {
    CacheDev c;
    const bf16 *q, *k_new, *v_new;
    bf16* out;
    char* ws;
};
struct ChanCall {
    int n;
    ChanLayer l[kChanLayers];
};
struct LayerMaps { CUtensorMap km, vm, ki, vi, kl, vl; };
struct ChanMaps { LayerMaps l[kChanLayers]; };

// Cluster per job.  u = scale log2(e) W C^K q, a slice of the rows per CTA, exchanged through distributed shared
// memory; then Z of nq channel pairs per CTA (a transform carries channels 2 q and 2 q + 1 of one head).  With k_new (a step, one
// pass) also the push: C^K's rows are updated on their way, the leaving row's kept dims and the new token are written.
template <int LS, int NH, bool WIDE>
__global__ void __launch_bounds__(outer_threads(WIDE), NH == 4 && outer_ctas(LS, WIDE) == 3 ? 2 : outer_ctas(LS, WIDE)) chan_in_kernel(Dims s, ChanPlan mp, const __grid_constant__ ChanCall call) {
    constexpr int S = 1 << LS, NT = outer_threads(WIDE);
    extern __shared__ __align__(16) float smz[];
    const int tid = threadIdx.x, CL = mp.nz, rank = CL > 1 ? (int)cluster_rank() : 0, h = blockIdx.y / mp.n_pass, pass = blockIdx.y - h * mp.n_pass;
    const int layer = blockIdx.z / s.B, b = blockIdx.z - layer * s.B;
    const CacheDev& c = call.l[layer].c;
    const bf16 *q = call.l[layer].q, *k_new = call.l[layer].k_new, *v_new = call.l[layer].v_new;
    char* wsp = call.l[layer].ws;
    const int g_first = h * s.G + pass * mp.nh, ng = min(mp.nh, s.G - pass * mp.nh), nh = mp.nh, nq = mp.nq, q0 = rank * nq;
    constexpr int fb = pf_size(S * 2);
    const int m0 = 2 * ((rank * s.k) / CL), m1 = 2 * (((rank + 1) * s.k) / CL), nv = s.dck >> 2;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smz);     // [8]
    volatile int* fail = reinterpret_cast<volatile int*>(smz + 16);
    float* twf = smz + 20;
    float* u_s = twf + ((2 * (tw_total(LS) + 1) + 3) & ~3);            // [nh][M]
    float* g_s = u_s + nh * s.M;                           // [2 nq][k]
    float* qc = g_s + ((2 * nq * s.k + 3) & ~3);           // [4][dck]
    float* xc = qc + 4 * s.dck;                            // [dck] compressed dims of the leaving row
    float* f_s = xc + s.dck;                               // [rows] basis column of the push
    float2* ph_s = reinterpret_cast<float2*>(f_s + (((s.M + CL - 1) / CL + 5) & ~3));          // [k] e^{i theta n c0}
    bf16* qs = reinterpret_cast<bf16*>(ph_s + ((s.k + 1) & ~1));       // [4][d] query rows, [2][d] the leaving row, [2][d] the new one
    bf16* xr = qs + 4 * s.d;
    bf16* nr = xr + 2 * s.d;
    float* fbuf = reinterpret_cast<float*>(nr + 2 * s.d);  // [nq nh][fb]; before the transforms: staged rows of C^K
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float* ckg = coef_rows(c.coef_k, s, b, h, s.dck);
    RowStream rs = {bars, fbuf, ckg + (size_t)m0 * s.dck, m1 - m0, s.dck, mp.st_in, (m1 - m0 + kStageRows - 1) / kStageRows};
    if (tid == 0) {
        for (int i = 0; i < mp.st_in; ++i) mbar_init(bars + i, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pass_twiddles<LS, NT>(twf, tid);
    channel_factors<NT>(g_s, q0, nq, s.k, S, tid);
    for (int n = tid; n < s.k; n += NT) ph_s[n] = mid_phase(n, s);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid == 0) rs.begin();
    // everything that a CTA needs of memory, each read once and all at the same time as far as addresses are known
    const bool step = k_new != nullptr;
    const int per_row = s.d >> 3;
    Push pu;
    pu.j = -1;
    pu.full = false;
    if (step) pu = push_of(c.state + kStateStride * b, s);
    if (tid < 8 * per_row) {
        const int g = tid / per_row, ch = tid - g * per_row;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (g < ng) v = *reinterpret_cast<const uint4*>(q + ((size_t)b * s.Hq + g_first + g) * s.d + 8 * ch);
        else if (step && g >= 6) v = *reinterpret_cast<const uint4*>((g == 6 ? k_new : v_new) + ((size_t)b * s.Hkv + h) * s.d + 8 * ch);
        if (g < 4 || g >= 6) *reinterpret_cast<uint4*>(qs + g * s.d + 8 * ch) = v;
    }
    int my_idx = 0;                                        // compressed dim of this thread's column
    if (tid < s.dck) my_idx = c.idx_comp_k[(size_t)h * s.dck + tid];
    if (pu.j >= 0) {
        if (tid < 2 * per_row) {
            const int side = tid >= per_row, ch = tid - side * per_row;
            *reinterpret_cast<uint4*>(xr + side * s.d + 8 * ch) =
                *reinterpret_cast<const uint4*>(leaving_row(c, s, b, h, side, pu.head, side == 0 ? k_new : v_new) + 8 * ch);
        }
        for (int r = tid; r < m1 - m0; r += NT) f_s[r] = basis_value(m0 + r, pu.j, s.T);
    }
    __syncthreads();
    if (tid < s.dck) {
#pragma unroll
        for (int g = 0; g < 4; ++g) qc[g * s.dck + tid] = __bfloat162float(qs[g * s.d + my_idx]);
        if (pu.j >= 0) xc[tid] = __bfloat162float(xr[my_idx]);
    }
    const int l8 = tid & 7, rgi = tid >> 3;
    const float sl2 = s.scale * kLog2e, inv_T = __int_as_float((127 << 23) - ((31 - __clz(s.T)) << 23));      // T is a power of two
    const float w_gen = sl2 * (s.norm == FA_NORM_PAPER ? 1.0f / (float)s.k : 2.f * inv_T), w_0 = s.norm == FA_NORM_PAPER ? w_gen : 0.5f * w_gen, w_1 = s.norm == FA_NORM_PAPER ? w_gen : 0.f;
    // A thread has the same columns of every row, up to four vectors: the query's and the leaving row's are in registers.  (Read for every row
    // they were most of what kept the shared-memory pipe busy, and that, not memory, set this loop's pace: 2.6 K cycles per 64 rows of four heads; sums sent to every
    // CTA of the cluster one by one were the rest.)
    float4 qr[NH][4], xr4[4];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool on = l8 + 8 * i < nv;
#pragma unroll
        for (int g = 0; g < NH; ++g) qr[g][i] = on && g < nh ? *reinterpret_cast<const float4*>(qc + g * s.dck + 4 * (l8 + 8 * i)) : make_float4(0.f, 0.f, 0.f, 0.f);
        xr4[i] = on && pu.j >= 0 ? *reinterpret_cast<const float4*>(xc + 4 * (l8 + 8 * i)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // two stages at a time: eight lanes take a row of each, so that a turn's chain (row, sums over lanes, barrier) is paid half as
    // often (a step of 8 rows of 32 heads, 4K tokens 101.8 -> 100.3 us, of 4 rows of 128K tokens 192.8 -> 190.5, with the same in the last kernel)
    constexpr int RP = NT / 8, SP = RP / kStageRows, U = in_turn(LS, WIDE);       // rows at a time, their stages; U of these to a turn
    for (int i = 0; i < rs.n_chunk; i += U * SP) {
        const int r0 = i * kStageRows + rgi;               // rows r0 and r0 + RP (a warp's are in one stage each)
        bool on[U];
        const float* xs[U];
        float f[U], a[U][NH];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            on[u] = r0 + u * RP < rs.rows;
            xs[u] = on[u] ? rs.wait(u * SP + rgi / kStageRows, fail, c.status) + (rgi % kStageRows) * s.dck : nullptr;
            f[u] = pu.j >= 0 && on[u] ? f_s[r0 + u * RP] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int g = 0; g < NH; ++g) a[u][g] = 0.f;
#pragma unroll
        for (int x4 = 0; x4 < 4; ++x4) {
            const int v = l8 + 8 * x4;
            if (v < nv) {
                float4 x[U];
#pragma unroll
                for (int u = 0; u < U; ++u) x[u] = on[u] ? *reinterpret_cast<const float4*>(xs[u] + 4 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (pu.j >= 0) {
                    const float4 y = xr4[x4];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        x[u].x = fmaf(f[u], y.x, x[u].x); x[u].y = fmaf(f[u], y.y, x[u].y); x[u].z = fmaf(f[u], y.z, x[u].z); x[u].w = fmaf(f[u], y.w, x[u].w);
                        if (on[u]) *reinterpret_cast<float4*>(ckg + (size_t)(m0 + r0 + u * RP) * s.dck + 4 * v) = x[u];
                    }
                }
#pragma unroll
                for (int g = 0; g < NH; ++g) {
                    const float4 z = qr[g][x4];
#pragma unroll
                    for (int u = 0; u < U; ++u) a[u][g] = fmaf(x[u].x, z.x, fmaf(x[u].y, z.y, fmaf(x[u].z, z.z, fmaf(x[u].w, z.w, a[u][g]))));
                }
            }
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int g = 0; g < NH; ++g)
#pragma unroll
                for (int u = 0; u < U; ++u) a[u][g] += __shfl_xor_sync(0xffffffffu, a[u][g], o);
        // lane x of a row keeps head x's
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = m0 + r0 + u * RP;
            float mine = a[u][0];
#pragma unroll
            for (int g = 1; g < NH; ++g) if (l8 == g) mine = a[u][g];
            if (on[u] && l8 < nh) u_s[l8 * s.M + m] = (m == 0 ? w_0 : m == 1 ? w_1 : w_gen) * mine;
        }
        rs.next(U * SP);
        rs.done(i, U * SP, tid);
    }
    if (CL > 1) {                                          // this CTA's rows to the others
        cluster_meet(CL);                                  // every CTA of the cluster has started: its shared memory can be written; all rows are there
        const int n = m1 - m0;
        if (((m0 | n) & 3) == 0) {
            for (int i = tid; i < nh * (n >> 2); i += NT) {
                const int g = i / (n >> 2), at = g * s.M + m0 + 4 * (i - g * (n >> 2));
                const float4 v = *reinterpret_cast<const float4*>(u_s + at);
                for (int w = 0; w < CL; ++w)
                    if (w != rank) st_peer4(peer_addr(smem_addr(u_s + at), (uint32_t)w), v);
            }
        } else {
            for (int i = tid; i < nh * n; i += NT) {
                const int g = i / n, at = g * s.M + m0 + i - g * n;
                const float v = u_s[at];
                for (int w = 0; w < CL; ++w)
                    if (w != rank) st_peer(peer_addr(smem_addr(u_s + at), (uint32_t)w), v);
            }
        }
    }
    cluster_meet(CL);
    if (blockIdx.y == 0 && b == 0) {                       // the channels' factors, for the last kernel of the chain
        float* gg = reinterpret_cast<float*>(wsp + mp.off_g) + (size_t)2 * q0 * s.k;
        for (int i = tid; i < 2 * nq * s.k; i += NT) gg[i] = g_s[i];
    }
    // packed Hermitian spectra: X_m = V^A_m + i V^B_m, V_m = v_m + conj(v_{S-m}), v_n = (1/2) (2 r + 1) i^r j_r u~_n e^{i theta n c0}
    // (with few bins the channel pairs of a bin go to neighbouring runs of threads)
    const int lg_q = split_pairs(S / 2 * nh, nq, NT), nq_t = nq >> lg_q;
    for (int i = tid; i < ((S / 2) * nh) << lg_q; i += NT) {
        const int pr = i & (S / 2 - 1), gq = i >> (LS - 1), qs0 = (gq & ((1 << lg_q) - 1)) * nq_t, g = gq >> lg_q, m = pr, mc = pr == 0 ? S / 2 : S - pr;
        float2 bm = make_float2(0.f, 0.f), bc = bm;
        const float* ug = u_s + g * s.M;
        if (m < s.k) { const float2 x = *reinterpret_cast<const float2*>(ug + 2 * m); bm = cmulf(make_float2(0.5f * x.x, -0.5f * x.y), ph_s[m]); }
        if (mc < s.k) { const float2 x = *reinterpret_cast<const float2*>(ug + 2 * mc); bc = cmulf(make_float2(0.5f * x.x, -0.5f * x.y), ph_s[mc]); }
#pragma unroll 2
        for (int qi = qs0; qi < qs0 + nq_t; ++qi) {
            const float sg = ((q0 + qi) & 1) ? -1.f : 1.f;
            const float am = m < s.k ? sg * g_s[2 * qi * s.k + m] : 0.f, om = m < s.k ? sg * g_s[(2 * qi + 1) * s.k + m] : 0.f;
            const float ac = mc < s.k ? sg * g_s[2 * qi * s.k + mc] : 0.f, oc = mc < s.k ? sg * g_s[(2 * qi + 1) * s.k + mc] : 0.f;
            const float2 vA = make_float2(am * bm.x, am * bm.y), vB = make_float2(-om * bm.y, om * bm.x);
            const float2 wA = make_float2(ac * bc.x, ac * bc.y), wB = make_float2(-oc * bc.y, oc * bc.x);
            float* base = fbuf + (qi * nh + g) * fb;
            if (pr != 0) {
                const float2 VA = make_float2(vA.x + wA.x, vA.y - wA.y), VB = make_float2(vB.x + wB.x, vB.y - wB.y);
                *reinterpret_cast<float2*>(base + pf(m * 2)) = make_float2(VA.x - VB.y, VA.y + VB.x);
                *reinterpret_cast<float2*>(base + pf(mc * 2)) = make_float2(VA.x + VB.y, VB.x - VA.y);
            } else {
                *reinterpret_cast<float2*>(base + pf(0)) = make_float2(2.f * vA.x, 2.f * vB.x);
                *reinterpret_cast<float2*>(base + pf(S)) = make_float2(2.f * wA.x, 2.f * wB.x);
            }
        }
    }
    __syncthreads();
    fft_run<2, LS, LS, false, 1, NT>(fbuf, fb, nq * nh, twf, tid);
    // last pass, and Z as [channel pair][slot][HP heads][hi, lo]: a thread has all heads of its slots
    constexpr int RL = last_radix_log2(LS), R = 1 << RL, JL = LS - RL;
    const int job = (b * s.Hkv + h) * mp.n_pass + pass;
    uint32_t* Z = reinterpret_cast<uint32_t*>(wsp + mp.off_z) + ((size_t)job * (kMR / 2) + q0) * S * 2 * mp.hp;
    const int lg_h = mp.hp == 4 && (nq << JL) < NT ? 1 : 0;            // a slot's two pairs of heads by two neighbouring threads where there are threads for it
    for (int i = tid; i < (nq << JL) << lg_h; i += NT) {
        const int it = i >> lg_h, qi = it >> JL, j = it & ((1 << JL) - 1);
        for (int hv = i & lg_h; hv < (mp.hp >> 1); hv += 1 + lg_h) {
            uint32_t hl[R][2][2];
#pragma unroll
            for (int g2 = 0; g2 < 2; ++g2) {
                const int g = 2 * hv + g2;
                PC<1> v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = PC<1>{PR<1>{0.f}, PR<1>{0.f}};
                if (g < nh) {
                    const float* base = fbuf + (qi * nh + g) * fb + pf(dif_pos<LS>(j) * 2);
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = ld_pt<1>(base + pf(r * 2));
                    dft<R, 1>(v);
                }
#pragma unroll
                for (int r = 0; r < R; ++r) split2(v[r].re.v, v[r].im.v, hl[r][g2][0], hl[r][g2][1]);
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                reinterpret_cast<uint4*>(Z + ((size_t)qi * S + j + (r << JL)) * 2 * mp.hp)[hv] = make_uint4(hl[r][0][0], hl[r][0][1], hl[r][1][0], hl[r][1][1]);
        }
    }
    // The push's rows and counters.  What the cluster reads of the old ones it has read before its meeting (one cluster per KV
    // head: a step has one pass); V's leaving row goes to the workspace for the last kernel of the chain.
    if (step && rank == CL - 1) {
        if (!pu.full) {
            if (pu.j >= 0) {
                const int cls = pu.j & (s.P - 1), slot = pu.j >> (31 - __clz(s.P));
                bf16* dk = mid_row<bf16>(c.k_mid, s, b, h, cls, slot, s.nfk);
                bf16* dv = mid_row<bf16>(c.v_mid, s, b, h, cls, slot, s.nfv);
                bf16* xg = reinterpret_cast<bf16*>(wsp + mp.off_x) + ((size_t)b * s.Hkv + h) * s.d;
                if (tid < s.nfk) dk[tid] = xr[c.idx_full_k[(size_t)h * s.nfk + tid]];
                else if (tid >= 64 && tid < 64 + s.nfv) dv[v_mid_col(slot, tid - 64, s.nfv, FA_BF16)] = xr[s.d + c.idx_full_v[(size_t)h * s.nfv + tid - 64]];
                else if (tid >= 128 && tid < 128 + s.d) xg[tid - 128] = xr[s.d + tid - 128];
            }
            if (pu.buf >= 0 && tid < 2 * per_row) {
                const int side = tid >= per_row, ch = tid - side * per_row;
                bf16* dst = pu.buf == 0 ? win_row<bf16>(side == 0 ? c.k_init : c.v_init, s, b, h, s.l_init, pu.row)
                                        : win_row<bf16>(side == 0 ? c.k_local : c.v_local, s, b, h, s.l_local, pu.row);
                *reinterpret_cast<uint4*>(dst + 8 * ch) = *reinterpret_cast<const uint4*>(nr + side * s.d + 8 * ch);
            }
        }
        if (tid == 0) {
            // the last KV head of the batch row publishes the counters: all have read the old ones
            int32_t* st = c.state + kStateStride * b;
            if (pu.full && h == 0) atomicExch(c.status, (int)FA_ERR_CAPACITY);
            if (atomicAdd(st + 4, 1) == s.Hkv - 1) {
                reinterpret_cast<int32_t*>(wsp + mp.off_j)[b] = pu.j;       // for the last kernel of the chain
                if (!pu.full) {
                    if (pu.n_init < s.l_init) st[0] = pu.n_init + 1;
                    else if (pu.j >= 0) {
                        st[2] = pu.n_mid + 1;
                        if (s.l_local > 0) st[3] = pu.head + 1 == s.l_local ? 0 : pu.head + 1;
                    } else st[1] = pu.n_local + 1;
                }
                st[4] = 0;
            }
        }
    }
}

// ---- tokens -------------------------------------------------------------------------------------------------------
// grid (Hkv * n_pass, n_cx + B n_wpart), four warps, three CTAs to an SM.  Every warp is on its own: a range of tokens, a ring of
// stages that its first lane refills, running maxima, sums and outputs; the four meet once, at the end.  Bound by the latency of
// its chain of shared-memory reads and mma per 64 tokens (a warp issues in one cycle of seven), so warps count: 8 rows of 32 KV
// heads, 4K tokens, 48 + 48 kept dims (281 MB) in 73 us with two CTAs to an SM and K and V in one stage, in 65 us with three and a
// stage for K or V, four such layers in one launch in 199 (5.7 TB/s); 562 MB of four rows of 128K tokens in 116 us, two layers in 206 (5.5 TB/s).  (Warps that shared the classes of a step met twice per step
// for its maximum and for W: 217 us there.)
// The class parts of all heads come first in the grid, the shorter window parts fill the gaps behind them.
// Class parts: a superstep is four neighbouring slots of all P classes, a stage the K rows or V rows of 16 classes as
// [slot][class][dims]; mma rows are the 16 classes, mma columns (slot, head): NT products of eight columns for HP heads (two slots
// each for four heads, all four slots in one for two).  The maximum is only worked out when some score is above the running one.
// Window parts: a stage holds 16 rows of K or V.
template <int HP>
__global__ void __launch_bounds__(32 * kMainWarps, kMainCtas) chan_main_kernel(const __grid_constant__ ChanMaps maps, Dims s, ChanPlan mp, const __grid_constant__ ChanCall call) {
    extern __shared__ __align__(128) unsigned char smem_unaligned[];
    unsigned char* smem = smem_unaligned + ((1024u - (smem_addr(smem_unaligned) & 1023u)) & 1023u);
    constexpr int NT = HP / 2, SL = 8 / HP;                // products per 16 classes, slots of a product
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int h = blockIdx.x / mp.n_pass, pass = blockIdx.x - h * mp.n_pass;
    // part `part` of layer `layer`: the class parts of all layers, then their window parts
    const int n_win_y = s.B * mp.n_wpart, n_class_y = call.n * mp.n_cx;
    const bool is_win = (int)blockIdx.y >= n_class_y;
    const int layer = is_win ? ((int)blockIdx.y - n_class_y) / n_win_y : (int)blockIdx.y / mp.n_cx;
    const int part = is_win ? mp.n_cx + (int)blockIdx.y - n_class_y - layer * n_win_y : (int)blockIdx.y - layer * mp.n_cx;
    const CacheDev& c = call.l[layer].c;
    const LayerMaps& tm_l = maps.l[layer];
    const bf16* q = call.l[layer].q;
    char* wsp = call.l[layer].ws;
    const int g_first = h * s.G + pass * mp.nh, ng = min(mp.nh, s.G - pass * mp.nh);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem) + 8 * warp;           // this warp's stages (at most 8)
    volatile int* fail = reinterpret_cast<volatile int*>(smem + 256);
    unsigned char* zero16 = smem + 272;
    float* ml_s = reinterpret_cast<float*>(smem + 288);    // [4 warps][4 heads](m, l)
    bf16* qs_s = reinterpret_cast<bf16*>(smem + 512);      // [4][d] query rows
    uint4* pt_s = reinterpret_cast<uint4*>(smem + 2048);   // [P / 16][hi, lo][lane]: the polynomials as mma A fragments, rows classes
    unsigned char* ring = smem + 2048 + (s.P >> 4) * 1024 + (size_t)warp * mp.ring;
    const int NS = is_win ? mp.ns_w : mp.ns_c, stage_bytes = is_win ? kWinStage : mp.stage_c;
    const uint32_t full_u = smem_addr(full), ring_u = smem_addr(ring), zero_u = smem_addr(zero16);
    if (tid == 0) *fail = 0;
    if (lane == 0) {
        for (int i = 0; i < NS; ++i) mbar_init(full + i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 4) reinterpret_cast<uint32_t*>(zero16)[tid] = 0;
    if (!is_win) {
        // the polynomials of every class, where the fragments want them
        for (int cls = tid; cls < s.P; cls += 32 * kMainWarps) {
            const float x = (float)(2 * cls + 1 - s.P) / (float)s.P;
            unsigned char* base = reinterpret_cast<unsigned char*>(pt_s + (cls >> 4) * 64);
            const int row = cls & 15;
            float p0 = 1.f, p1 = x;
#pragma unroll
            for (int r = 0; r < kMR; ++r) {
                const bf16 hi = __float2bfloat16_rn(p0), lo = __float2bfloat16_rn(p0 - __bfloat162float(hi));
                const int at = ((row & 7) * 4 + ((r & 7) >> 1)) * 16 + ((row >> 3) + 2 * (r >> 3)) * 4 + (r & 1) * 2;
                *reinterpret_cast<bf16*>(base + at) = hi;
                *reinterpret_cast<bf16*>(base + 512 + at) = lo;
                const float p2 = ((float)(2 * r + 3) * x * p1 - (float)(r + 1) * p0) * (1.0f / (float)(r + 2));
                p0 = p1;
                p1 = p2;
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");    // Z; rows and counters of a push
    // (only now: the kernel that this lets start takes everything before the kernel in front as finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // batch row and share: class parts by the rows' lengths, window parts alike
    int b = 0, x0 = 0, cnt = mp.n_cx;
    if (is_win) {
        b = (part - mp.n_cx) / mp.n_wpart;
    } else {
        const RowParts r = row_parts(c.state, s, mp.n_cx, part, 0);
        if (r.b == s.B) return;
        if (part == r.x0 && blockIdx.x == 0 && tid == 0) reinterpret_cast<int2*>(wsp + mp.off_p)[r.b] = make_int2(r.x0, r.cnt);      // for the last kernel
        b = r.b;
        x0 = r.x0;
        cnt = r.cnt;
    }
    const int job = (b * s.Hkv + h) * mp.n_pass + pass;
    const int n_init = c.state[kStateStride * b + 0], n_local = c.state[kStateStride * b + 1];
    const int n_mid = min(c.state[kStateStride * b + 2], s.max_mid), head = c.state[kStateStride * b + 3];
    const int nhalf = (s.d + 63) >> 6, rowb_k = 2 * s.nfk, rowb_v = 2 * s.nfv, n_ch = s.P >> 4;
    // class parts: supersteps [st0, st1), n_ch stages each; window parts: tokens [w0, w1) in runs of at most 16 rows
    const int steps = (n_mid + 4 * s.P - 1) / (4 * s.P), wq = kMainWarps * (part - x0) + warp;
    const int st0 = is_win ? 0 : (int)((long long)wq * steps / (kMainWarps * cnt)), st1 = is_win ? 0 : (int)((long long)(wq + 1) * steps / (kMainWarps * cnt));
    const int n_win = n_init + n_local, wi = kMainWarps * (part - mp.n_cx - b * mp.n_wpart) + warp;
    const int w0 = is_win ? (int)((long long)wi * n_win / (kMainWarps * mp.n_wpart)) : 0, w1 = is_win ? (int)((long long)(wi + 1) * n_win / (kMainWarps * mp.n_wpart)) : 0;
    // place of the next stage to load: superstep and chunk of 16 classes, or window token
    int ld_step = is_win ? w0 : st0, ld_ch = 0, ld_v = 0, ld_st = 0, issued = 0;
    // run of window tokens from t on: rows of one buffer
    auto win_run = [&](int t, int& buf, int& row) -> int {
        if (t < n_init) { buf = 0; row = t; return min(16, min(w1, n_init) - t); }
        const int u = t - n_init;
        buf = 1;
        row = head + u;
        if (row >= s.l_local) row -= s.l_local;
        return min(16, min(w1 - t, s.l_local - row));
    };
    auto refill = [&]() {                                  // (lane 0) loads the next stage
        const uint32_t bar = full_u + 8u * ld_st, dst = ring_u + (uint32_t)(ld_st * stage_bytes);
        if (!is_win) {
            if (ld_step >= st1) return;
            const uint32_t bytes = (uint32_t)(64 * (ld_v ? rowb_v : rowb_k));
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
            if (bytes)
                asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
                             "l"(reinterpret_cast<uint64_t>(ld_v ? &tm_l.vm : &tm_l.km)), "r"(0), "r"(ld_ch * 16), "r"(4 * ld_step), "r"(b * s.Hkv + h), "r"(bar) : "memory");
            if (ld_v && ++ld_ch == n_ch) { ld_ch = 0; ++ld_step; }
        } else {
            if (ld_step >= w1) return;
            int buf, row;
            const int n = win_run(ld_step, buf, row);
            const CUtensorMap* tm = ld_v ? (buf == 0 ? &tm_l.vi : &tm_l.vl) : (buf == 0 ? &tm_l.ki : &tm_l.kl);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(nhalf * 2048) : "memory");
            for (int hf = 0; hf < nhalf; ++hf)
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
                                 dst + (uint32_t)(hf * 2048)),
                             "l"(reinterpret_cast<uint64_t>(tm)), "r"(hf * 64), "r"(row), "r"(b * s.Hkv + h), "r"(bar) : "memory");
            if (ld_v) ld_step += n;
        }
        ld_v ^= 1;
        ++issued;
        if (++ld_st == NS) ld_st = 0;
    };
    __syncwarp();
    if (lane == 0)
        for (int i = 0; i < NS; ++i) refill();
    for (int i = tid; i < 4 * (s.d >> 3); i += 32 * kMainWarps) {
        const int g = i / (s.d >> 3), ch = i - g * (s.d >> 3);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (g < ng) v = *reinterpret_cast<const uint4*>(q + ((size_t)b * s.Hq + g_first + g) * s.d + 8 * ch);
        *reinterpret_cast<uint4*>(qs_s + g * s.d + 8 * ch) = v;
    }
    __syncthreads();

    float m_run[2], l_run[2];                              // columns 2 tq, 2 tq + 1 of this lane: heads hl, hl + 1
    m_run[0] = m_run[1] = kNegBig;
    l_run[0] = l_run[1] = 0.f;
    float acc[8][4];                                       // outputs: [16 dims][mma fragment]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const float sl2 = s.scale * kLog2e;
    const int hl = is_win || HP == 4 ? 2 * (tq & 1) : 0, tsl = HP == 4 ? tq >> 1 : tq;      // (windows: columns 0 - 3 are the heads); slot of the columns
    const bool on0 = hl < ng, on1 = hl + 1 < ng;
    int st = 0;
    uint32_t ph = 0;
    auto next_stage = [&]() { if (++st == NS) { st = 0; ph ^= 1; } };
    const int mi = lane >> 3, tok = ((mi >> 1) << 3) + (lane & 7);
    // a new maximum: per head over the lanes that hold its columns; returns the factors of what refers to the old one
    auto new_max = [&](float mx0, float mx1, auto pairs) -> float2 {
        float mn0, mn1;
        if constexpr (decltype(pairs)::value) {            // two heads: all lanes' columns
            mn0 = warp_max_redux(mx0);
            mn1 = warp_max_redux(mx1);
        } else {
            const bool odd = tq & 1;
            const float h0 = warp_max_redux(odd ? kNegBig : mx0), h1 = warp_max_redux(odd ? kNegBig : mx1);
            const float h2 = warp_max_redux(odd ? mx0 : kNegBig), h3 = warp_max_redux(odd ? mx1 : kNegBig);
            mn0 = odd ? h2 : h0;
            mn1 = odd ? h3 : h1;
        }
        mn0 = fmaxf(m_run[0], mn0);
        mn1 = fmaxf(m_run[1], mn1);
        const float2 a = make_float2(ex2(m_run[0] - mn0), ex2(m_run[1] - mn1));
        m_run[0] = mn0;
        m_run[1] = mn1;
        l_run[0] *= a.x;
        l_run[1] *= a.y;
        return a;
    };
    if (!is_win) {
        const int gcol = gq % HP, gsl = gq / HP;           // head and slot of column gq (the column of this lane's B fragments)
        const int npk = s.nfk >> 3, nchv = s.nfv >> 3, nmt = (s.nfv + 15) >> 4;
        // B fragments of q for the kept K dims (pieces of 16 bytes, two k-steps each, as in the transform kernel)
        uint32_t qk[2][2][2];
        {
            const int32_t* idf = c.idx_full_k + (size_t)h * s.nfk;
            const bf16* qrow = qs_s + gcol * s.d;
#pragma unroll
            for (int rd = 0; rd < 2; ++rd)
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const int piece = 4 * rd + tq, e0 = 8 * piece + 4 * ks;
                    const bool on = gcol < ng && piece < npk;
                    qk[rd][ks][0] = on ? pack_bf16(qrow[idf[e0]], qrow[idf[e0 + 1]]) : 0u;
                    qk[rd][ks][1] = on ? pack_bf16(qrow[idf[e0 + 2]], qrow[idf[e0 + 3]]) : 0u;
                }
        }
        // byte offsets inside a group of 16 classes: K pieces of rows gq and gq + 8, V chunks of row tok (the tensor map's swizzle:
        // chunk ^ ((row >> sh) & mask); V chunks are permuted by the slot as well)
        uint32_t k_lo[2], k_hi[2];
#pragma unroll
        for (int rd = 0; rd < 2; ++rd) {
            const int piece = 4 * rd + tq;
            k_lo[rd] = (uint32_t)(gq * rowb_k + ((piece ^ ((gq >> mp.k_sh) & mp.k_mask)) << 4));
            k_hi[rd] = (uint32_t)((gq + 8) * rowb_k + ((piece ^ (((gq + 8) >> mp.k_sh) & mp.k_mask)) << 4));
        }
        const int fsw = (tok >> mp.v_sh) & mp.v_mask;
        const bool k_on0 = tq < npk, k_on1 = 4 + tq < npk;
        const uint32_t v_row = (uint32_t)(tok * rowb_v), k_slot = (uint32_t)(16 * rowb_k), v_slot = (uint32_t)(16 * rowb_v);
        const size_t plane = (size_t)mp.slots * HP;        // a channel pair's Z or W
        const uint2* Zg = reinterpret_cast<const uint2*>(wsp + mp.off_z) + ((size_t)job * (kMR / 2) + tq) * plane + gq;
        float* Wg = reinterpret_cast<float*>(wsp + mp.off_w) + (((size_t)job * (kMR / 2) + (gq >> 1)) * plane) * 2 + (gq & 1);
        float* mWg = reinterpret_cast<float*>(wsp + mp.off_mw) + (size_t)job * (mp.slots / 4) * 4;
        uint2 za[NT], zb[NT];                              // (hi, lo) of channels 2 tq, 2 tq + 1, and 8 further on, of the superstep's columns
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            za[t] = zb[t] = make_uint2(0, 0);
            if (st0 < st1) { za[t] = Zg[(size_t)st0 * 4 * HP + 8 * t]; zb[t] = Zg[(size_t)st0 * 4 * HP + 8 * t + 4 * plane]; }
        }
#pragma unroll 1
        for (int i = st0; i < st1; ++i) {
            uint2 z0[NT], z1[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                z0[t] = za[t];
                z1[t] = zb[t];
                if (i + 1 < st1) { za[t] = Zg[(size_t)(i + 1) * 4 * HP + 8 * t]; zb[t] = Zg[(size_t)(i + 1) * 4 * HP + 8 * t + 4 * plane]; }
            }
            int vsw[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) vsw[x] = v_swz(4 * i + x, nchv) ^ fsw;
            float dw[NT][4];
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int x = 0; x < 4; ++x) dw[t][x] = 0.f;
            const int j0 = 4 * i * s.P;                    // first token of the superstep
            const bool whole = j0 + 4 * s.P <= n_mid;
#pragma unroll 1
            for (int ch = 0; ch < n_ch; ++ch) {
                const uint4 ah = pt_s[ch * 64 + lane], al = pt_s[ch * 64 + 32 + lane];
                mbar_wait_u(full_u + 8u * st, ph, fail, c.status);       // (after a time-out the walk goes on, on what is there)
                const uint32_t kt = ring_u + (uint32_t)(st * stage_bytes);
                float sc[NT][4];
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    float dm[4] = {0.f, 0.f, 0.f, 0.f}, dk[2][4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) dk[0][x] = dk[1][x] = 0.f;
                    mma_bf16(dm, ah.x, ah.y, ah.z, ah.w, z0[t].x, z1[t].x);
                    mma_bf16(dm, al.x, al.y, al.z, al.w, z0[t].x, z1[t].x);
                    mma_bf16(dm, ah.x, ah.y, ah.z, ah.w, z0[t].y, z1[t].y);
#pragma unroll
                    for (int sl = 0; sl < SL; ++sl) {
                        const bool mine = gsl == sl;
                        const uint32_t row = kt + (SL * t + sl) * k_slot;
#pragma unroll
                        for (int rd = 0; rd < 2; ++rd) {
                            if (4 * rd < npk) {
                                uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
                                if (rd == 0 ? k_on0 : k_on1) {
                                    lo = lds128(row + k_lo[rd]);
                                    hi = lds128(row + k_hi[rd]);
                                }
                                mma_bf16(dk[sl & 1], lo.x, hi.x, lo.y, hi.y, mine ? qk[rd][0][0] : 0u, mine ? qk[rd][0][1] : 0u);
                                mma_bf16(dk[sl & 1], lo.z, hi.z, lo.w, hi.w, mine ? qk[rd][1][0] : 0u, mine ? qk[rd][1][1] : 0u);
                            }
                        }
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) sc[t][x] = ((x & 1) ? on1 : on0) ? fmaf(dk[0][x] + dk[1][x], sl2, dm[x]) : 2.f * kNegBig;
                }
                __syncwarp();                              // K has been read
                if (lane == 0) refill();
                next_stage();
                if (!whole) {
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        const int js = j0 + (SL * t + tsl) * s.P + 16 * ch + gq;
                        if (js >= n_mid) sc[t][0] = sc[t][1] = 2.f * kNegBig;
                        if (js + 8 >= n_mid) sc[t][2] = sc[t][3] = 2.f * kNegBig;
                    }
                }
                float mx0 = fmaxf(sc[0][0], sc[0][2]), mx1 = fmaxf(sc[0][1], sc[0][3]);
                if (NT == 2) { mx0 = fmaxf(mx0, fmaxf(sc[NT - 1][0], sc[NT - 1][2])); mx1 = fmaxf(mx1, fmaxf(sc[NT - 1][1], sc[NT - 1][3])); }
                if (__any_sync(0xffffffffu, mx0 > m_run[0] || mx1 > m_run[1])) {
                    const float2 a = new_max(mx0, mx1, std::bool_constant<HP == 2>{});
#pragma unroll
                    for (int t = 0; t < NT; ++t) { dw[t][0] *= a.x; dw[t][1] *= a.y; dw[t][2] *= a.x; dw[t][3] *= a.y; }
#pragma unroll
                    for (int x = 0; x < 4; ++x) { acc[x][0] *= a.x; acc[x][1] *= a.y; acc[x][2] *= a.x; acc[x][3] *= a.y; }
                }
                mbar_wait_u(full_u + 8u * st, ph, fail, c.status);
                const uint32_t vt = ring_u + (uint32_t)(st * stage_bytes);
                if (!whole) {
                    // V rows past the end of the middle hold whatever was there: zero them, p = 0 does not stop a NaN
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const int sl = 2 * x + (lane >> 4), rr = lane & 15;
                        if (j0 + sl * s.P + 16 * ch + rr >= n_mid)
                            for (int y = 0; y < nchv; ++y) sts128(vt + sl * v_slot + (uint32_t)(rr * rowb_v + 16 * y), make_uint4(0, 0, 0, 0));
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                }
                // the polynomials with rows channels: the 8 x 8 blocks transposed
                const uint4 wh = make_uint4(movmatrix_trans(ah.x), movmatrix_trans(ah.z), movmatrix_trans(ah.y), movmatrix_trans(ah.w));
                const uint4 wl = make_uint4(movmatrix_trans(al.x), movmatrix_trans(al.z), movmatrix_trans(al.y), movmatrix_trans(al.w));
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    float pr[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) pr[x] = ex2(sc[t][x] - m_run[x & 1]);
                    l_run[0] += pr[0] + pr[2];
                    l_run[1] += pr[1] + pr[3];
                    uint32_t h01, l01, h23, l23;
                    split2(pr[0], pr[1], h01, l01);
                    split2(pr[2], pr[3], h23, l23);
                    const uint32_t b0 = movmatrix_trans(h01), b1 = movmatrix_trans(h23), c0 = movmatrix_trans(l01), c1 = movmatrix_trans(l23);
                    mma_bf16(dw[t], wh.x, wh.y, wh.z, wh.w, b0, b1);
                    mma_bf16(dw[t], wl.x, wl.y, wl.z, wl.w, b0, b1);
                    mma_bf16(dw[t], wh.x, wh.y, wh.z, wh.w, c0, c1);
                    // o += V^T p, slot by slot
#pragma unroll
                    for (int sl = 0; sl < SL; ++sl) {
                        const bool mine = gsl == sl;
                        const uint32_t p0 = mine ? b0 : 0u, p1 = mine ? b1 : 0u;
                        const uint32_t row = vt + (SL * t + sl) * v_slot + v_row;
#pragma unroll
                        for (int dt = 0; dt < 4; ++dt) {
                            if (dt < nmt) {
                                const int chunk = 2 * dt + (mi & 1);
                                uint32_t af[4];
                                ldmatrix_x4_trans(af, chunk < nchv ? row + (uint32_t)((chunk ^ vsw[SL * t + sl]) << 4) : zero_u);
                                mma_bf16(acc[dt], af[0], af[1], af[2], af[3], p0, p1);
                            }
                        }
                    }
                }
                __syncwarp();                              // V has been read
                if (lane == 0) refill();
                next_stage();
            }
            // W as [channel pair][slot][HP heads][channel of the pair], against the maxima so far
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                float* wo = Wg + ((size_t)i * 4 * HP + 8 * t + 2 * tq) * 2;
                if (on0) { wo[0] = dw[t][0]; wo[8 * plane] = dw[t][2]; }
                if (on1) { wo[2] = dw[t][1]; wo[8 * plane + 2] = dw[t][3]; }
            }
            if (lane < 2) *reinterpret_cast<float2*>(mWg + i * 4 + 2 * lane) = make_float2(m_run[0], m_run[1]);
        }
    } else {
        const int gcol = gq & 3;
        const bool col_on = gq < 4 && gcol < ng;
        const bf16* qrow = qs_s + gcol * s.d;
        const int npw = s.d >> 3, nmtw = (s.d + 15) >> 4;
        uint32_t qw[4][4];
#pragma unroll
        for (int rd = 0; rd < 4; ++rd) {
            const int piece = ((rd >> 1) << 3) + 2 * tq + (rd & 1);
            uint4 x = make_uint4(0, 0, 0, 0);
            if (col_on && piece < npw) x = *reinterpret_cast<const uint4*>(qrow + 8 * piece);
            qw[rd][0] = x.x; qw[rd][1] = x.y; qw[rd][2] = x.z; qw[rd][3] = x.w;
        }
        const uint32_t v_sw = (uint32_t)((tok & 7) ^ (mi & 1)) << 4;
#pragma unroll 1
        for (int t = w0; t < w1;) {
            int buf, row;
            const int rem = win_run(t, buf, row);
            mbar_wait_u(full_u + 8u * st, ph, fail, c.status);
            const uint32_t kt = ring_u + (uint32_t)(st * stage_bytes), r_lo = kt + (uint32_t)(gq * 128);
            float da[4] = {0.f, 0.f, 0.f, 0.f}, db[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int rd = 0; rd < 4; ++rd) {
                if ((rd >> 1) < nhalf) {
                    const uint32_t src = r_lo + (rd >> 1) * 2048 + (((2 * tq + (rd & 1)) ^ gq) << 4);
                    const uint4 lo = lds128(src), hi = lds128(src + 8 * 128);
                    mma_bf16(da, lo.x, hi.x, lo.y, hi.y, qw[rd][0], qw[rd][1]);
                    mma_bf16(db, lo.z, hi.z, lo.w, hi.w, qw[rd][2], qw[rd][3]);
                }
            }
            __syncwarp();
            if (lane == 0) refill();
            next_stage();
            float sc[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) sc[x] = gq + 8 * (x >> 1) < rem && tq < 2 ? (da[x] + db[x]) * sl2 : 2.f * kNegBig;
            const float mx0 = fmaxf(sc[0], sc[2]), mx1 = fmaxf(sc[1], sc[3]);
            if (__any_sync(0xffffffffu, mx0 > m_run[0] || mx1 > m_run[1])) {
                const float2 a = new_max(mx0, mx1, std::false_type{});
#pragma unroll
                for (int x = 0; x < 8; ++x) { acc[x][0] *= a.x; acc[x][1] *= a.y; acc[x][2] *= a.x; acc[x][3] *= a.y; }
            }
            float pr[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) pr[x] = ex2(sc[x] - m_run[x & 1]);
            l_run[0] += pr[0] + pr[2];
            l_run[1] += pr[1] + pr[3];
            const uint32_t b0 = movmatrix_trans(pack2(pr[0], pr[1])), b1 = movmatrix_trans(pack2(pr[2], pr[3]));
            mbar_wait_u(full_u + 8u * st, ph, fail, c.status);
            const uint32_t vt = ring_u + (uint32_t)(st * stage_bytes);
            if (rem < 16) {
                // rows past the end of the run hold whatever follows it in the cache: zero them, p = 0 does not stop a NaN
                for (int x = lane; x < (16 - rem) * 8; x += 32)
                    for (int hf = 0; hf < nhalf; ++hf) sts128(vt + hf * 2048 + (uint32_t)(rem * 8 + x) * 16, make_uint4(0, 0, 0, 0));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
            }
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
                if (mt < nmtw) {
                    uint32_t af[4];
                    ldmatrix_x4_trans(af, vt + tok * 128 + (mt >> 2) * 2048 + (v_sw ^ (uint32_t)((2 * mt & 7) << 4)));
                    mma_bf16(acc[mt], af[0], af[1], af[2], af[3], b0, b1);
                }
            }
            __syncwarp();
            if (lane == 0) refill();
            next_stage();
            t += rem;
        }
    }
    // ---------------- the warps' results side by side, then one partial result per head ----------------
    if (*fail && lane == 0)                                // a wait ran out: the copies under way land, or the bound is reached, first
        for (int i = issued - NS < 0 ? 0 : issued - NS; i < issued; ++i)
            for (uint32_t n = 0; n < (1u << 20) && !mbar_try_wait(full_u + 8u * (i % NS), (uint32_t)(i / NS) & 1u); ++n) { }
    __syncthreads();
    float* o_s = reinterpret_cast<float*>(smem + 2048);    // [warps][4][d]
    int16_t* inv = reinterpret_cast<int16_t*>(o_s + kMainWarps * 4 * s.d);       // dim -> kept position, or -1
    const int n_dims = is_win ? s.d : s.nfv;
    // sums over rows (lanes) and over the slots of a product's columns
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], o);
        l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], o);
    }
    if (!is_win) {
#pragma unroll
        for (int o = HP == 4 ? 2 : 1; o < 4; o <<= 1) {
            l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], o);
            l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], o);
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[mt][x] += __shfl_xor_sync(0xffffffffu, acc[mt][x], o);
        }
    }
    if (tq < (is_win ? 2 : NT)) {
        float* ow = o_s + warp * 4 * s.d + 2 * tq * s.d;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            const int e = 16 * mt + gq;
            if (e < n_dims) { ow[e] = acc[mt][0]; ow[s.d + e] = acc[mt][1]; }
            if (e + 8 < n_dims) { ow[e + 8] = acc[mt][2]; ow[s.d + e + 8] = acc[mt][3]; }
        }
        if (gq == 0) *reinterpret_cast<float4*>(ml_s + warp * 8 + 4 * tq) = make_float4(m_run[0], l_run[0], m_run[1], l_run[1]);
    }
    if (!is_win)
        for (int e = tid; e < s.d; e += 32 * kMainWarps) inv[e] = -1;
    __syncthreads();
    if (!is_win)
        for (int e = tid; e < s.nfv; e += 32 * kMainWarps) inv[c.idx_full_v[h * s.nfv + e]] = (int16_t)e;
    __syncthreads();
    const size_t slot = (size_t)blockIdx.x * (mp.n_cx + n_win_y) + part;
    float2* mlg = reinterpret_cast<float2*>(wsp + mp.off_ml) + slot * 4;
    float* og = reinterpret_cast<float*>(wsp + mp.off_o) + slot * 4 * s.d;
    for (int i = tid; i < 4 * s.d; i += 32 * kMainWarps) {
        const int g = i / s.d, e = i - g * s.d;
        float mx = kNegBig, v = 0.f, l = 0.f;
        if (g < ng) {
#pragma unroll
            for (int w = 0; w < kMainWarps; ++w) mx = fmaxf(mx, ml_s[w * 8 + 2 * g]);
            const int at = is_win ? e : inv[e];
#pragma unroll
            for (int w = 0; w < kMainWarps; ++w) {
                const float a = ex2(ml_s[w * 8 + 2 * g] - mx);
                l = fmaf(a, ml_s[w * 8 + 2 * g + 1], l);
                if (at >= 0) v = fmaf(a, o_s[(w * 4 + g) * s.d + at], v);
            }
        }
        og[i] = v;
        if (e == 0) mlg[g] = make_float2(mx, l);
    }
}

// Cluster per job: the parts' statistics and outputs merged, z of nq channel pairs per CTA, summed over the cluster
// through distributed shared memory, a slice of the rows of C^V per CTA, its products summed likewise, the output rows.
// After a step's push (step != 0) C^V's rows are updated on their way.
// (unbounded, the instances of 64 and 512 slots took 155 registers and one CTA to an SM: 9 to 11 % of a step)
template <int LS, bool WIDE>
__global__ void __launch_bounds__(outer_threads(WIDE), outer_ctas(LS, WIDE)) chan_out_kernel(Dims s, ChanPlan mp, const __grid_constant__ ChanCall call) {
    constexpr int S = 1 << LS, NT = outer_threads(WIDE);
    extern __shared__ __align__(16) float smz[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, CL = mp.nz, rank = CL > 1 ? (int)cluster_rank() : 0, h = blockIdx.y / mp.n_pass, pass = blockIdx.y - h * mp.n_pass;
    const int layer = blockIdx.z / s.B, b = blockIdx.z - layer * s.B, step = call.l[layer].k_new != nullptr;
    const CacheDev& c = call.l[layer].c;
    bf16* out = call.l[layer].out;
    char* wsp = call.l[layer].ws;
    const int g_first = h * s.G + pass * mp.nh, ng = min(mp.nh, s.G - pass * mp.nh), nh = mp.nh, nq = mp.nq, q0 = rank * nq;
    constexpr int fb = pf_size(S * 2);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smz);     // [8]
    volatile int* fail = reinterpret_cast<volatile int*>(smz + 16);
    float* twf = smz + 20;
    float* z_s = twf + ((2 * (tw_total(LS) + 1) + 3) & ~3);            // [nh][M] this CTA's channels' share of z
    float* g_s = z_s + nh * s.M;                           // [2 nq][k]
    float* mfin = g_s + ((2 * nq * s.k + 3) & ~3);         // [4] maxima, [4] 1 / sums
    float* oc_s = mfin + 8;                                // [4][dcv] this CTA's rows' share of o^c
    float* zw_s = oc_s + 4 * s.dcv;                        // [rows][4] z of this CTA's rows, weighted
    float* xc = zw_s + 4 * (((s.M + CL - 1) / CL + 5) & ~3);           // [dcv]
    float* f_s = xc + s.dcv;                               // [rows] basis column of the push
    int16_t* inv = reinterpret_cast<int16_t*>(f_s + (((s.M + CL - 1) / CL + 5) & ~3));      // dim -> position in D^vc, or -1
    float2* ph_s = reinterpret_cast<float2*>(inv + ((s.d + 7) & ~7));  // [k] e^{i theta n c0}
    float* cv_s = reinterpret_cast<float*>(ph_s + ((s.k + 1) & ~1));   // stages of rows of C^V
    float* fbuf = cv_s + (size_t)mp.st_out * kStageRows * s.dcv;       // [nq nh][fb]
    float* ps_s = fbuf;                                    // [row groups][4][dcv], when the transforms are over
    const int m0 = 2 * ((rank * s.k) / CL), m1 = 2 * (((rank + 1) * s.k) / CL), nv = s.dcv >> 2, nrg = NT / nv;
    float* cvg = coef_rows(c.coef_v, s, b, h, s.dcv);
    RowStream rs = {bars, cv_s, cvg + (size_t)m0 * s.dcv, m1 - m0, s.dcv, mp.st_out, (m1 - m0 + kStageRows - 1) / kStageRows};
    if (tid == 0) {
        for (int i = 0; i < mp.st_out; ++i) mbar_init(bars + i, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // rows of C^V: last written by a kernel that had ended before the main kernel let this one start
        rs.begin();
    }
    pass_twiddles<LS, NT>(twf, tid);
    for (int n = tid; n < s.k; n += NT) ph_s[n] = mid_phase(n, s);
    asm volatile("griddepcontrol.wait;" ::: "memory");    // the parts
    const int job = (b * s.Hkv + h) * mp.n_pass + pass, X = mp.n_cx + s.B * mp.n_wpart;
    const float2* ml = reinterpret_cast<const float2*>(wsp + mp.off_ml) + (size_t)blockIdx.y * X * 4;       // [part][4]
    const float* op = reinterpret_cast<const float*>(wsp + mp.off_o) + (size_t)blockIdx.y * X * 4 * s.d;     // [part][4][d]
    const float2* W = reinterpret_cast<const float2*>(wsp + mp.off_w) + ((size_t)job * (kMR / 2) + q0) * S * mp.hp;      // [q][slot][HP heads]
    const float* mW = reinterpret_cast<const float*>(wsp + mp.off_mw) + (size_t)job * (S / 4) * 4;
    const int2 rp = reinterpret_cast<const int2*>(wsp + mp.off_p)[b];      // this row's class parts: first, number
    const int n_mid = min(c.state[kStateStride * b + 2], s.max_mid), a_end = (n_mid + s.P - 1) / s.P;
    const int j_push = step ? reinterpret_cast<const int32_t*>(wsp + mp.off_j)[b] : -1;
    for (int i = tid; i < 2 * nq * s.k / 4; i += NT)
        cp_async16(g_s + 4 * i, reinterpret_cast<const float*>(wsp + mp.off_g) + (size_t)2 * q0 * s.k + 4 * i);
    const int np = rp.y + mp.n_wpart, wshift = mp.n_cx + b * mp.n_wpart - rp.y;
    auto part_at = [&](int i) { return i < rp.y ? rp.x + i : wshift + i; };
    if (tid < 32 * 4) {                                    // a warp per head
        const int g = tid >> 5, lane = tid & 31;
        float mx = kNegBig, l = 0.f;
        for (int i = lane; i < np; i += 32) mx = fmaxf(mx, ml[part_at(i) * 4 + g].x);
        mx = warp_max(mx);
        for (int i = lane; i < np; i += 32) { const float2 v = ml[part_at(i) * 4 + g]; l = fmaf(ex2(v.x - mx), v.y, l); }
        l = warp_sum(l);
        if (lane == 0) { mfin[g] = mx; mfin[4 + g] = l > 0.f ? 1.0f / l : 0.f; }
    } else {
        const int u = tid - 128;                           // a thread per dim: every dim is in D^vu or in D^vc
        if (u < s.nfv) inv[c.idx_full_v[(size_t)h * s.nfv + u]] = -1;
        else if (u < s.d) {
            const int e = c.idx_comp_v[(size_t)h * s.dcv + u - s.nfv];
            inv[e] = (int16_t)(u - s.nfv);
            if (j_push >= 0) xc[u - s.nfv] = __bfloat162float((reinterpret_cast<const bf16*>(wsp + mp.off_x) + ((size_t)b * s.Hkv + h) * s.d)[e]);
        }
    }
    if (j_push >= 0)
        for (int r = tid; r < m1 - m0; r += NT) f_s[r] = basis_value(m0 + r, j_push, s.T);
    cp_async_wait_all();
    __syncthreads();
    constexpr int RL = last_radix_log2(LS), R = 1 << RL, JL = LS - RL;
    const int lg_h = mp.hp == 4 && (nq << JL) < NT ? 1 : 0;
    for (int i = tid; i < (nq << JL) << lg_h; i += NT) {
        const int it = i >> lg_h, qi = it >> JL, j = it & ((1 << JL) - 1);
        for (int hv = i & lg_h; hv < (mp.hp >> 1); hv += 1 + lg_h) {
            float4 x[R];                                   // two heads' two channels at this thread's slots
            float2 mw[R];                                  // what they refer to
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int a = j + (r << JL);
                x[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                mw[r] = make_float2(0.f, 0.f);
                if (a < a_end) {
                    x[r] = reinterpret_cast<const float4*>(W + ((size_t)qi * S + a) * mp.hp)[hv];
                    mw[r] = reinterpret_cast<const float2*>(mW + (a >> 2) * 4)[hv];
                }
            }
#pragma unroll
            for (int g2 = 0; g2 < 2; ++g2) {
                const int g = 2 * hv + g2;
                if (g < nh) {
                    PC<1> v[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float2 y = g2 == 0 ? make_float2(x[r].x, x[r].y) : make_float2(x[r].z, x[r].w);
                        const float sc = ex2((g2 == 0 ? mw[r].x : mw[r].y) - mfin[g]);
                        const bool on = j + (r << JL) < a_end && g < ng;
                        v[r] = on ? PC<1>{PR<1>{y.x * sc}, PR<1>{y.y * sc}} : PC<1>{PR<1>{0.f}, PR<1>{0.f}};
                    }
                    dft<R, 1>(v);
                    float* base = fbuf + (qi * nh + g) * fb + pf(dif_pos<LS>(j) * 2);
#pragma unroll
                    for (int r = 0; r < R; ++r) st_pt(base + pf(r * 2), v[r]);
                }
            }
        }
    }
    // The outputs' share of this CTA, elements el0 .. el1 of [ng][d]: TP neighbouring lanes to an element take a share of the parts each
    const int n_el = ng * s.d, el0 = rank * n_el / CL, el1 = (rank + 1) * n_el / CL, lgTP = CL >= 8 ? 2 : CL >= 4 ? 1 : 0, TP = 1 << lgTP;
    float o_acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = el0 + ((tid + u * NT) >> lgTP), sub = tid & (TP - 1);
        if (i < el1) {
            const int g = i / s.d;
            const float mg = mfin[g];
            float v = 0.f;
            int x = sub;
            for (; x + 7 * TP < np; x += 8 * TP) {
                float y[8], m8[8];
#pragma unroll
                for (int w = 0; w < 8; ++w) { const int at = part_at(x + w * TP); y[w] = op[(size_t)at * 4 * s.d + i]; m8[w] = ml[at * 4 + g].x; }
#pragma unroll
                for (int w = 0; w < 8; ++w) v = fmaf(ex2(m8[w] - mg), y[w], v);
            }
#pragma unroll 4
            for (; x < np; x += TP) { const int at = part_at(x); v = fmaf(ex2(ml[at * 4 + g].x - mg), op[(size_t)at * 4 * s.d + i], v); }
            o_acc[u] = v;
        }
    }
    __syncthreads();
    fft_run<2, LS, LS, true, 1, NT>(fbuf, fb, nq * nh, twf, tid);
    // (with few bins the channel pairs of a bin go to neighbouring lanes, whose sums are added in a fixed order)
    const int lg_q = split_pairs(S / 2 * nh, nq, NT), nq_t = nq >> lg_q;
    for (int i = tid; i < ((S / 2) * nh) << lg_q; i += NT) {      // (whole warps: S is a multiple of 32 bins and pairs of them)
        const int bi = i >> lg_q, qs0 = (i & ((1 << lg_q) - 1)) * nq_t, g = bi >> (LS - 1), pr = bi & (S / 2 - 1), m = pr, mc = pr == 0 ? S / 2 : S - pr;
        float2 zm = make_float2(0.f, 0.f), zc = zm;
        if (m < s.k || mc < s.k)
#pragma unroll 2
        for (int qi = qs0; qi < qs0 + nq_t; ++qi) {
            const float* base = fbuf + (qi * nh + g) * fb;
            const float2 ya = *reinterpret_cast<const float2*>(base + pf(m * 2)), yb = *reinterpret_cast<const float2*>(base + pf(mc * 2));
            float2 am, bm, ac, bc;                         // spectra of the two channels at bins m and mc
            if (pr != 0) {
                am = make_float2(0.5f * (ya.x + yb.x), 0.5f * (ya.y - yb.y));
                bm = make_float2(0.5f * (ya.y + yb.y), 0.5f * (yb.x - ya.x));
                ac = make_float2(am.x, -am.y);
                bc = make_float2(bm.x, -bm.y);
            } else {
                am = make_float2(ya.x, 0.f); bm = make_float2(ya.y, 0.f);
                ac = make_float2(yb.x, 0.f); bc = make_float2(yb.y, 0.f);
            }
            const float sg = ((q0 + qi) & 1) ? -1.f : 1.f;
            if (m < s.k) {
                const float ga = sg * g_s[2 * qi * s.k + m], go = sg * g_s[(2 * qi + 1) * s.k + m];
                zm.x += ga * am.x - go * bm.y;
                zm.y += ga * am.y + go * bm.x;
            }
            if (mc < s.k) {
                const float ga = sg * g_s[2 * qi * s.k + mc], go = sg * g_s[(2 * qi + 1) * s.k + mc];
                zc.x += ga * ac.x - go * bc.y;
                zc.y += ga * ac.y + go * bc.x;
            }
        }
        for (int o = 1; o < (1 << lg_q); o <<= 1) {
            zm.x += __shfl_xor_sync(0xffffffffu, zm.x, o);
            zm.y += __shfl_xor_sync(0xffffffffu, zm.y, o);
            zc.x += __shfl_xor_sync(0xffffffffu, zc.x, o);
            zc.y += __shfl_xor_sync(0xffffffffu, zc.y, o);
        }
        if (qs0 == 0 && m < s.k) *reinterpret_cast<float2*>(z_s + g * s.M + 2 * m) = cmulf(zm, ph_s[m]);
        if (qs0 == 0 && mc < s.k) *reinterpret_cast<float2*>(z_s + g * s.M + 2 * mc) = cmulf(zc, ph_s[mc]);
    }
    cluster_meet(CL);                                      // all shares of z are there
    // rows of C^V against the sum of the shares
    const float inv_T = __int_as_float((127 << 23) - ((31 - __clz(s.T)) << 23));      // T is a power of two
    const float w_gen = s.norm == FA_NORM_PAPER ? 1.0f / (float)s.k : 2.f * inv_T, w_0 = s.norm == FA_NORM_PAPER ? w_gen : inv_T, w_1 = s.norm == FA_NORM_PAPER ? w_gen : 0.f;
    const int n_rows = m1 - m0;
    for (int x = tid; x < (n_rows >> 1) * nh; x += NT) {          // (rows in pairs, cos and sin of a frequency)
        const int g = x / (n_rows >> 1), r = 2 * (x - g * (n_rows >> 1)), m = m0 + r;
        const float2 v = CL == 1 ? *reinterpret_cast<const float2*>(z_s + g * s.M + m) : sum_peers2(smem_addr(z_s + g * s.M + m), CL);
        zw_s[r * 4 + g] = v.x * (m == 0 ? w_0 : w_gen);
        zw_s[(r + 1) * 4 + g] = v.y * (m == 0 ? w_1 : w_gen);
    }
    __syncthreads();
    float4 acc4[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) acc4[g] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int rg = tid / nv, vcol = tid - rg * nv;
    const float4 y = j_push >= 0 ? *reinterpret_cast<const float4*>(xc + 4 * vcol) : make_float4(0.f, 0.f, 0.f, 0.f);      // (the thread's columns are the same in every row)
    constexpr int SP = out_stages(LS, WIDE);               // stages at a time: the thread's chain through them is paid once
    for (int i = 0; i < rs.n_chunk; i += SP) {
        const float* xs[SP];
#pragma unroll
        for (int u = 0; u < SP; ++u) xs[u] = i + u < rs.n_chunk ? rs.wait(u, fail, c.status) - u * kStageRows * s.dcv : nullptr;
        const int first = i * kStageRows, rows = min(SP * kStageRows, rs.rows - first);
        if (rg < nrg) {
#pragma unroll 4
            for (int r = rg; r < rows; r += nrg) {
                const float* xr = xs[0];
#pragma unroll
                for (int u = 1; u < SP; ++u) if (r >= u * kStageRows) xr = xs[u];
                float4 x = *reinterpret_cast<const float4*>(xr + r * s.dcv + 4 * vcol);
                if (j_push >= 0) {
                    const float f = f_s[first + r];
                    x.x = fmaf(f, y.x, x.x); x.y = fmaf(f, y.y, x.y); x.z = fmaf(f, y.z, x.z); x.w = fmaf(f, y.w, x.w);
                    *reinterpret_cast<float4*>(cvg + (size_t)(m0 + first + r) * s.dcv + 4 * vcol) = x;
                }
                const float4 w4 = *reinterpret_cast<const float4*>(zw_s + (first + r) * 4);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (g < nh) {
                        const float w = g == 0 ? w4.x : g == 1 ? w4.y : g == 2 ? w4.z : w4.w;
                        acc4[g].x = fmaf(w, x.x, acc4[g].x);
                        acc4[g].y = fmaf(w, x.y, acc4[g].y);
                        acc4[g].z = fmaf(w, x.z, acc4[g].z);
                        acc4[g].w = fmaf(w, x.w, acc4[g].w);
                    }
                }
            }
        }
        rs.next(SP);
        rs.done(i, SP, tid);
    }
    if (rg < nrg) {
#pragma unroll
        for (int g = 0; g < 4; ++g) if (g < nh) *reinterpret_cast<float4*>(ps_s + (rg * nh + g) * s.dcv + 4 * vcol) = acc4[g];
    }
    __syncthreads();
    for (int i = tid; i < nh * s.dcv; i += NT) {
        float v = 0.f;
#pragma unroll 8
        for (int x = 0; x < nrg; ++x) v += ps_s[x * nh * s.dcv + i];
        oc_s[i] = v;
    }
    cluster_meet(CL);                                      // all shares of o^c are there
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = el0 + ((tid + u * NT) >> lgTP);
        float v = o_acc[u];
        for (int o = 1; o < TP; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (i < el1 && (tid & (TP - 1)) == 0) {
            const int g = i / s.d, e = i - g * s.d, at = inv[e];
            if (at >= 0) v += CL == 1 ? oc_s[g * s.dcv + at] : sum_peers(smem_addr(oc_s + g * s.dcv + at), CL);
            out[((size_t)b * s.Hq + g_first) * s.d + i] = __float2bfloat16_rn(v * mfin[4 + g]);
        }
    }
    if (CL > 1) cluster_meet(CL);                          // nobody leaves while its shares are read
}

// K^mu or V^mu as (dims, class, slot, batch * KV head): box = all dims, 16 classes, four slots.
bool mid_map(CUtensorMap* tm, const void* base, const Dims& s, int nf) {
    if (nf == 0) { memset(tm, 0, sizeof(*tm)); return true; }
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t rowb = (cuuint64_t)nf * 2;
    cuuint64_t dims[4] = {(cuuint64_t)nf, (cuuint64_t)s.P, (cuuint64_t)s.S_cap, (cuuint64_t)s.B * s.Hkv};
    cuuint64_t strides[3] = {rowb * s.S_cap, rowb, rowb * s.S_cap * s.P};
    cuuint32_t box[4] = {(cuuint32_t)nf, 16, 4, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapSwizzle sw = nf == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : nf == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : nf == 16 ? CU_TENSOR_MAP_SWIZZLE_32B
                                                                                                                    : CU_TENSOR_MAP_SWIZZLE_NONE;
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shared memory of the kernels in front of and behind the main kernel.
size_t in_smem(const Dims& s, int ls, const ChanPlan& m) {
    const size_t fft = (size_t)m.nq * m.nh * pf_size(2 << ls), stage = (size_t)m.st_in * kStageRows * s.dck;
    return sizeof(float) * (20 + ((2 * (tw_total(ls) + 1) + 3) & ~3) + (size_t)m.nh * s.M + ((2 * m.nq * s.k + 3) & ~3) + 5 * s.dck +
                            (((s.M + m.nz - 1) / m.nz + 5) & ~3) + 2 * ((s.k + 1) & ~1) + 4 * s.d + (fft > stage ? fft : stage)) + 64;
}
size_t out_smem(const Dims& s, int ls, const ChanPlan& m) {
    const size_t fft = (size_t)m.nq * m.nh * pf_size(2 << ls), ps = (size_t)outer_threads(m.wide) * 4 * m.nh;
    return sizeof(float) * (20 + ((2 * (tw_total(ls) + 1) + 3) & ~3) + (size_t)m.nh * s.M + ((2 * m.nq * s.k + 3) & ~3) + 8 + 5 * s.dcv +
                            5 * (size_t)(((s.M + m.nz - 1) / m.nz + 5) & ~3) + ((s.d + 7) & ~7) / 2 + 2 * ((s.k + 1) & ~1) + (size_t)m.st_out * kStageRows * s.dcv + (fft > ps ? fft : ps)) + 64;
}

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, int cluster, cudaStream_t st, Args... args) {
    cudaError_t err = ensure_dynamic_smem(kernel, smem);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace

// (as many as the threads of a CTA take at a time)
static int least_stages(bool wide) { return outer_threads(wide) / 128; }
// As many stages of the outer kernels' rows as a CTA's rows take and the limit of shared memory holds.
static void fit_stages(const Dims& s, int log2S, size_t limit, ChanPlan* m) {
    auto fits = [&]() { return in_smem(s, log2S, *m) <= limit && out_smem(s, log2S, *m) <= limit; };
    const int chunks = (s.M / m->nz + 2 + kStageRows - 1) / kStageRows, most = chunks < kMaxRowStages ? chunks : kMaxRowStages;
    m->st_in = m->st_out = least_stages(m->wide);
    for (; m->st_in < most; ++m->st_in) { ++m->st_in; const bool ok = fits(); --m->st_in; if (!ok) break; }
    for (; m->st_out < most; ++m->st_out) { ++m->st_out; const bool ok = fits(); --m->st_out; if (!ok) break; }
}

// When the last of n1 parts of cost a, then n2 of cost b, ends on so many slots.
static double makespan(long long n1, double a, long long n2, double b, int slots) {
    const long long full = n1 / slots, rest = n1 % slots;
    const double end1 = (rest ? full + 1 : full) * a;
    double lo = end1, hi = end1 + (n2 / slots + 2) * b;
    auto room = [&](double t) { return (long long)((t - (full + 1) * a) / b) * rest + (long long)((t - full * a) / b) * (slots - rest); };
    if (n2 == 0 || room(lo) >= n2) return lo;
    for (int i = 0; i < 24; ++i) {
        const double t = 0.5 * (lo + hi);
        (room(t) >= n2 ? hi : lo) = t;
    }
    return hi;
}

// Whether the channel form serves a layout that the transform kernel serves (period a power of two, S >= k, at most 64 kept dims
// a side, head_dim at most 128) with a multiple of four coefficients, and its plan.
bool plan_channels(const Dims& s, int log2S, int sms, ChanPlan* m) {
    memset(m, 0, sizeof(*m));
    const int S = 1 << log2S;
    m->slots = S;
    if (s.dck == 0 || s.dcv == 0 || s.nfk > 64 || s.nfv > 64 || s.nfk + s.nfv == 0 || s.d > 128) return false;
    if (s.P % 16 || s.P > 512 || s.k > S || s.P * S != s.T || s.S_cap > S || s.B > 256) return false;
    // A head's coefficients, and a pair of channels' factors, follow one another in shared memory and are read and exchanged 16 bytes at a time: whole
    // groups of four of them.  (n_coef = 2 mod 4 is left to the transform kernel, whose rows may end anywhere.)
    if (s.M % 4) return false;
    m->n_pass = (s.G + 3) / 4;
    m->nh = (s.G + m->n_pass - 1) / m->n_pass;
    m->hp = m->nh > 2 ? 4 : 2;
    // a warp's ring of K and V stages: what leaves room for three CTAs to an SM, two stages at least
    const int kt = 64 * 2 * s.nfk, vt = 64 * 2 * s.nfv;
    m->stage_c = ((kt > vt ? kt : vt) + 1023) / 1024 * 1024;
    const int head = 2048 + (s.P >> 4) * 1024, room = (75 * 1024 - 1024 - head) / kMainWarps / 1024 * 1024;
    auto stages = [&](int bytes) { return room / bytes < 2 ? 2 : room / bytes > 8 ? 8 : room / bytes; };
    m->ns_c = stages(m->stage_c);
    m->ns_w = stages(kWinStage);
    m->ring = m->ns_c * m->stage_c > m->ns_w * kWinStage ? m->ns_c * m->stage_c : m->ns_w * kWinStage;
    m->smem = head + kMainWarps * m->ring + 1024;
    if (m->smem > 227 * 1024) return false;
    auto swz = [](int nf, int* sh, int* mask) { *sh = nf == 64 ? 0 : nf == 32 ? 1 : 2; *mask = nf == 64 ? 7 : nf == 32 ? 3 : nf == 16 ? 1 : 0; };
    swz(s.nfk, &m->k_sh, &m->k_mask);
    swz(s.nfv, &m->v_sh, &m->v_mask);
    // parts of a batch row: what finishes first when the device takes the class parts and then the window parts as CTAs become free
    // (a part's bytes, and as many more as go by while it starts and ends)
    const long long heads = (long long)s.Hkv * m->n_pass, jobs = heads * s.B;
    const long long per_step = 8LL * s.P * (s.nfk + s.nfv), win_bytes = 4LL * s.d * (s.l_init + s.l_local);
    const int slots = kMainCtas * sms, steps = (s.max_mid + 4 * s.P - 1) / (4 * s.P);
    double best = 0;
    for (int cn = 1; cn == 1 || (cn <= 64 && kMainWarps * cn <= steps); ++cn)
        for (int wn = win_bytes > 0 ? 1 : 0; wn <= (win_bytes > 0 ? 8 : 0); ++wn) {
            const int q = (steps + kMainWarps * cn - 1) / (kMainWarps * cn);
            const double cost = makespan(jobs * cn, (double)kMainWarps * q * per_step + kPartCost, jobs * wn, wn ? (double)win_bytes / wn + kPartCost : 1.0, slots);
            if (best == 0 || cost < 0.98 * best) { best = cost; m->n_cx = s.B * cn; m->n_wpart = wn; }
        }
    // CTAs per cluster of the kernels in front and behind.  The device holds 15 clusters of eight CTAs of one to an SM, 33 of four,
    // 74 of two, twice that with two to an SM; a wave costs what does not depend on the split and the split's share, about four
    // times that for a job in one CTA (32 jobs of 2048 coefficients: 35 us a kernel in one wave of clusters of four, 55 in two of eight)
    // The longest transforms in CTAs of sixteen warps, one to an SM (wide), or of eight: those where two of them fit and that makes it less than three quarters of the cost (as
    // much where only the larger clusters of the wide form do not fit).  us a step of one layer / four layers, wide and not, 128 classes, cost ratio: 48 heads of three, 2048
    // coefficients 129, 124 / 363, 366 (0.75); 48 of four 137, 162 / 388, 472 (1); 48 of two 102, 108 / 281, 325 (1), 1536 88, 84 / 250, 242 (0.67); 64 of one 105, 103 / 351, 345
    // (0.67); 64 of four, 512 coefficients 112, 102 / 392, 358 (0.75, clusters of two); 32 of four, 40 coefficients 65, 71 / 190, 144 (1); 64 classes: 192 of one, 40
    // coefficients 155, 123 / 555, 405 (0.56); 96 of two, 40 76, 88 / 214, 253 (0.8), 512 118, 107 / 409, 304 (0.67).
    auto fits = [&](size_t limit) { return in_smem(s, log2S, *m) <= limit && out_smem(s, log2S, *m) <= limit; };
    constexpr size_t kHalf = 112 * 1024, kAll = 226 * 1024;
    struct Outer { int nz, occ; double cost; };
    auto outer = [&](int wide) {
        Outer best = {};
        m->wide = wide;
        m->st_in = m->st_out = least_stages(wide);
        for (m->nz = 8; m->nz >= 1; m->nz /= 2) {
            m->nq = kMR / 2 / m->nz;
            const int fit = fits(kHalf) && outer_ctas(log2S, wide) > 1 ? 2 : fits(kAll) ? 1 : 0;
            if (!fit) continue;
            const long long held = (long long)(m->nz == 8 ? 15 : m->nz == 4 ? 33 : m->nz == 2 ? 74 : 148) * sms / 148 * fit;
            const double cost = (double)((jobs + held - 1) / held) * (1.0 + 4.0 / m->nz);
            if (!best.nz || cost < best.cost) best = Outer{m->nz, fit, cost};
        }
        return best;
    };
    Outer use = outer(0);
    if (log2S == 10) {
        const Outer w = outer(1);
        if (w.nz && !(use.nz && (use.occ == 2 ? use.cost < 0.75 * w.cost : use.cost <= 0.75 * w.cost))) use = w;
        else m->wide = 0;
    }
    if (!use.nz) return false;
    m->nz = use.nz;
    m->nq = kMR / 2 / m->nz;
    fit_stages(s, log2S, use.occ == 2 && jobs * m->nz > sms ? kHalf : kAll, m);
    return true;
}

// Offsets of the channel form's areas of one layer, and their bytes.
size_t place_channels(const Dims& s, int log2S, ChanPlan* m) {
    size_t off = 0;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t jobs = (size_t)s.B * s.Hkv * m->n_pass, slots = (size_t)1 << log2S, parts = (size_t)s.Hkv * m->n_pass * (m->n_cx + s.B * m->n_wpart);
    m->off_z = off;  off = up(off + jobs * slots * (kMR / 2) * m->hp * 8);
    m->off_w = off;  off = up(off + jobs * slots * (kMR / 2) * m->hp * 8);
    m->off_mw = off; off = up(off + jobs * (slots / 4) * 16);
    m->off_ml = off; off = up(off + parts * 32);
    m->off_o = off;  off = up(off + parts * 4 * s.d * 4);
    m->off_g = off;  off = up(off + (size_t)kMR * s.k * 4);
    m->off_x = off;  off = up(off + (size_t)s.B * s.Hkv * s.d * 2);
    m->off_j = off;  off = up(off + (size_t)s.B * 4);
    m->off_p = off;  off = up(off + (size_t)s.B * 8);
    return off;
}

template <int LS, bool WIDE>
static cudaError_t launch_channels_t(const Dims& s, const ChanArgs* a, int n, const ChanPlan& one, cudaStream_t st, bool* begun) {
    *begun = false;
    if (n < 1 || n > kChanLayers) return cudaErrorInvalidValue;
    ChanPlan m = one;
    // several layers, more CTAs than two to an SM: fewer stages each, so that three fit (the sums do not depend on the number of stages)
    constexpr size_t kThird = 74 * 1024;
    if (outer_ctas(LS, WIDE) == 3 && (long long)n * s.B * s.Hkv * m.n_pass * m.nz > 2 * sm_count()) {
        m.st_in = m.st_out = least_stages(WIDE);
        if (in_smem(s, LS, m) <= kThird && out_smem(s, LS, m) <= kThird) fit_stages(s, LS, kThird, &m);
        else m = one;
    }
    const dim3 cg(m.nz, s.Hkv * m.n_pass, s.B * n), mg(s.Hkv * m.n_pass, n * (m.n_cx + s.B * m.n_wpart));
    ChanCall call = {};
    ChanMaps maps;
    call.n = n;
    const int n_bh = s.B * s.Hkv;
    for (int i = 0; i < n; ++i) {
        const CacheDev& c = a[i].c;
        call.l[i] = ChanLayer{c, static_cast<const bf16*>(a[i].q), static_cast<const bf16*>(a[i].k_new), static_cast<const bf16*>(a[i].v_new), static_cast<bf16*>(a[i].out), a[i].ws};
        LayerMaps& t = maps.l[i];
        const bool ok_i = window_map(&t.ki, c.k_init, s.l_init, s.d, n_bh, 16) & window_map(&t.vi, c.v_init, s.l_init, s.d, n_bh, 16);
        const bool ok_l = window_map(&t.kl, c.k_local, s.l_local, s.d, n_bh, 16) & window_map(&t.vl, c.v_local, s.l_local, s.d, n_bh, 16);
        if ((s.l_init > 0 && !ok_i) || (s.l_local > 0 && !ok_l)) return cudaErrorInvalidValue;
        if (!mid_map(&t.km, c.k_mid, s, s.nfk) || !mid_map(&t.vm, c.v_mid, s, s.nfv)) return cudaErrorInvalidValue;
    }
    auto launch_in = [&](auto nh) { return launch_chained(chan_in_kernel<LS, decltype(nh)::value, WIDE>, cg, dim3(outer_threads(WIDE)), in_smem(s, LS, m), m.nz, st, s, m, call); };
    cudaError_t err = m.nh == 1 ? launch_in(std::integral_constant<int, 1>{}) : m.nh == 2 ? launch_in(std::integral_constant<int, 2>{}) : launch_in(std::integral_constant<int, 4>{});
    if (err != cudaSuccess) return err;
    *begun = true;
    err = m.hp == 2 ? launch_chained(chan_main_kernel<2>, mg, dim3(32 * kMainWarps), (size_t)m.smem, 1, st, maps, s, m, call)
                    : launch_chained(chan_main_kernel<4>, mg, dim3(32 * kMainWarps), (size_t)m.smem, 1, st, maps, s, m, call);
    if (err != cudaSuccess) return err;
    return launch_chained(chan_out_kernel<LS, WIDE>, cg, dim3(outer_threads(WIDE)), out_smem(s, LS, m), m.nz, st, s, m, call);
}

// The decode calls of n layers of one layout, with k_new / v_new (not null; one pass only) each behind the push of Eq.5.  Several layers do not touch
// one another's memory.  *begun: an error came after the first launch (before it nothing has been enqueued: the device refused the
// cluster, say).
cudaError_t launch_decode_channels(const Dims& s, const ChanArgs* a, int n, const ChanPlan& m, int log2S, cudaStream_t st, bool* begun) {
    switch (log2S) {
        case 5: return launch_channels_t<5, false>(s, a, n, m, st, begun);
        case 6: return launch_channels_t<6, false>(s, a, n, m, st, begun);
        case 7: return launch_channels_t<7, false>(s, a, n, m, st, begun);
        case 8: return launch_channels_t<8, false>(s, a, n, m, st, begun);
        case 9: return launch_channels_t<9, false>(s, a, n, m, st, begun);
        case 10: return m.wide ? launch_channels_t<10, true>(s, a, n, m, st, begun) : launch_channels_t<10, false>(s, a, n, m, st, begun);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fa
