// fa_decode_attention (Eq.6), DIRECT main kernel: per token of the middle
//   s_j = q_u . K^mu_j + sum_m F[m][j] u_g[m];  online softmax;  o^u += p_j V^mu_j;
//   z[m] += p_j F[m][j];  window tokens: ordinary attention in the same softmax.
// The M basis terms of every token are summed one by one (any period, any class count):
// the reference of the GPU side and the fallback of the transform kernel.
#include <type_traits>

#include "fa_common.cuh"
#include "fa_decode_ws.cuh"

namespace fa {


// ------------------------------------------------------------- direct main --
// grid (n_split, Hkv * n_pass, B), 256 threads.  A split takes a run of middle tokens (in token order, whatever their
// classes) and a run of window tokens, in tiles of 64: four lanes share a token's sum over the frequencies and its kept
// dims, and on the way back the threads share out frequencies and groups of tokens.  The kernel is bound by its chain of
// dependent steps, so what counts is that a call has many short CTAs: 1024 fp32 tokens of one head are 16 CTAs of one
// tile instead of four CTAs that walked eight classes each with 32 of their 256 threads (compress and decode of that
// cache together: 99 -> 35 us; with the launches of the call chained and everything that does not need u in front of the wait for it: 27).
constexpr int kTile = 64, kLanes = 4;

template <int GH>
struct RunStat {
    float m[GH];   // running max, log2 units
    float l[GH];   // running sum of p over this thread's tokens
};

// Block-wide maximum of GH values per thread; result broadcast to every thread.
template <int GH>
__device__ __forceinline__ void block_max(float (&v)[GH], float* red_s /* [8][GH] */) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int g = 0; g < GH; ++g) {
        const float r = warp_max(v[g]);
        if (lane == 0) red_s[warp * GH + g] = r;
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GH; ++g) {
        float r = red_s[g];
#pragma unroll
        for (int w = 1; w < 8; ++w) r = fmaxf(r, red_s[w * GH + g]);
        v[g] = r;
    }
    __syncthreads();
}

// OCC: CTAs to an SM, by registers.  The first two (three with fewer than four heads) leave room to fetch the rows of the first tile, and form its kept-dim scores and
// basis, in front of the wait for u.  (Three with four heads come out at 80 registers by themselves; told so, the compiler's order of the loops over frequencies is up
// to 8 % slower: 320 CTAs of 1.3 K fp32 tokens 831 and 778 us.)
template <typename KV, int GH, int OCC>
__global__ void __launch_bounds__(256, OCC == 3 && GH == 4 ? 0 : OCC) decode_direct_kernel(Dims s, CacheDev c, DecodePlan p, const KV* __restrict__ q,
                                                            char* wsp) {
    constexpr bool AHEAD = OCC == 2 || (OCC == 3 && GH < 4);
    extern __shared__ float sm[];
    Ws ws = ws_view(wsp, p);
    const int split = blockIdx.x;
    const int h = blockIdx.y / p.n_pass, pass = blockIdx.y % p.n_pass;
    const int b = blockIdx.z;
    const int g_first = h * s.G + pass * GH;                 // first query head of this CTA
    const int ng = min(GH, s.G - pass * GH);
    const int tid = threadIdx.x;

    float* q_s = sm;                          // [GH][d]   scale * log2e * q, natural order
    float* qf_s = q_s + GH * s.d;             // [GH][nfk] the same gathered at D^ku
    float* u_s = qf_s + GH * s.nfk;           // [GH][M]
    float* z_s = u_s + GH * s.M;              // [GH][M]
    float* p_s = z_s + GH * s.M;              // [GH][kTile]
    float* zr_s = p_s + GH * kTile;           // [2 GH][256] partial z of the token groups
    float* red_s = zr_s + 512 * GH;           // [8][GH]
    float* o_s = red_s + 8 * GH;              // [GH][d]  final reduce
    float* acc_s = o_s + GH * s.d;            // [256][GH] cross-thread reduce of the output accumulators

    // Everything but u was there before this call: the kernel in front lets this one start when the work before it has ended.  The rows of the
    // first tile are fetched, and their kept-dim scores formed, while that kernel makes u (AHEAD).
    const int4 st4 = *reinterpret_cast<const int4*>(c.state + kStateStride * b);
    const int n_init = st4.x, n_local = st4.y, n_mid = min(st4.z, s.max_mid), head = st4.w;
    const int32_t* idf_v = c.idx_full_v + (size_t)h * s.nfv;
    const int idf_k = tid < s.nfk ? c.idx_full_k[(size_t)h * s.nfk + tid] : 0;
    // middle tokens [j0, j1) of this split; four lanes to a token; (token group, dim) map of the P.V product
    const int per = (n_mid + p.n_split - 1) / p.n_split;
    const int j0 = min(n_mid, split * per), j1 = min(n_mid, j0 + per);
    const bool p2 = (s.P & (s.P - 1)) == 0;
    const int lgP = 31 - __clz(s.P);
    auto cls_of = [&](int j) { return p2 ? j & (s.P - 1) : j % s.P; };
    auto slot_of = [&](int j) { return p2 ? j >> lgP : j / s.P; };
    const int tk = tid / kLanes, ql = tid % kLanes;
    const int ntg_mid = s.nfv > 0 ? 256 / s.nfv : 0;
    const int tg_mid = s.nfv > 0 ? tid / s.nfv : 0, e_mid = s.nfv > 0 ? tid % s.nfv : 0;
    const bool act_mid = s.nfv > 0 && tg_mid < ntg_mid;
    auto k_row = [&](int j) { return mid_row<KV>(c.k_mid, s, b, h, cls_of(j), slot_of(j), s.nfk); };
    auto v_at = [&](int j) {
        const int slot = slot_of(j);
        return ld_f(mid_row<KV>(c.v_mid, s, b, h, cls_of(j), slot, s.nfv) + v_mid_col(slot, e_mid, s.nfv, sizeof(KV) == 2 ? FA_BF16 : FA_F32));
    };
    constexpr int kPre = AHEAD ? 8 : 1;                     // values of K and of V of the first tile that a thread fetches ahead
    float k_pre[kPre], v_pre[kPre];
    if (AHEAD) {
        const KV* row = j0 + tk < j1 ? k_row(j0 + tk) : nullptr;
#pragma unroll
        for (int u = 0; u < kPre; ++u) k_pre[u] = row && ql + u * kLanes < s.nfk ? ld_f(row + ql + u * kLanes) : 0.f;
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            const int j = j0 + tg_mid + u * ntg_mid;
            v_pre[u] = act_mid && j < min(j1, j0 + kTile) ? v_at(j) : 0.f;
        }
    }

    for (int i = tid; i < GH * s.d; i += blockDim.x) {
        int g = i / s.d, e = i - g * s.d;
        q_s[i] = g < ng ? ld_f(q + ((size_t)b * s.Hq + g_first + g) * s.d + e) * s.scale * kLog2e : 0.f;
        o_s[i] = 0.f;
    }
    for (int i = tid; i < GH * s.M; i += blockDim.x) z_s[i] = 0.f;
    __syncthreads();
    if (tid < s.nfk)
#pragma unroll
        for (int g = 0; g < GH; ++g) qf_s[g * s.nfk + tid] = q_s[g * s.d + idf_k];
    __syncthreads();

    RunStat<GH> rs;
#pragma unroll
    for (int g = 0; g < GH; ++g) { rs.m[g] = kNegBig; rs.l[g] = 0.f; }
    float o_mid[GH], o_win[GH];
#pragma unroll
    for (int g = 0; g < GH; ++g) { o_mid[g] = 0.f; o_win[g] = 0.f; }

    // thread -> (token group, dim) map of the windows' P.V product
    const int ntg_win = 256 / s.d;
    const int tg_win = tid / s.d, e_win = tid % s.d;
    const bool act_win = tg_win < ntg_win;

    // after scores are known (every one of a token's four lanes has them): update the running softmax state, leave p in p_s
    bool first = true;                        // (z_s is zero)
    auto softmax_tile = [&](float (&sc)[GH], bool valid) {
        float mx[GH];
#pragma unroll
        for (int g = 0; g < GH; ++g) mx[g] = valid ? sc[g] : kNegBig;
        block_max<GH>(mx, red_s);
        float alpha[GH];
#pragma unroll
        for (int g = 0; g < GH; ++g) {
            float m_new = fmaxf(rs.m[g], mx[g]);
            alpha[g] = exp2f(rs.m[g] - m_new);
            rs.m[g] = m_new;
            const float pv = valid && ql == 0 ? exp2f(sc[g] - m_new) : 0.f;
            if (ql == 0) p_s[g * kTile + tk] = pv;
            rs.l[g] = rs.l[g] * alpha[g] + pv;      // this thread's tokens: summed over the block at the end
            o_mid[g] *= alpha[g];
            o_win[g] *= alpha[g];
        }
        if (!AHEAD || !first)
#pragma unroll
            for (int g = 0; g < GH; ++g)
                for (int m = tid; m < s.M; m += 256) z_s[g * s.M + m] *= alpha[g];
        first = false;
        __syncthreads();                        // p_s, z_s
    };
    auto lanes_sum = [&](float (&sc)[GH]) {
#pragma unroll
        for (int g = 0; g < GH; ++g) {
            sc[g] += __shfl_xor_sync(0xffffffffu, sc[g], 1);
            sc[g] += __shfl_xor_sync(0xffffffffu, sc[g], 2);
        }
    };
    // frequencies of a lane, and the way back: kz frequencies at a time, 256 / kz groups of tokens
    const int per_lane = (s.k + kLanes - 1) / kLanes;
    int kz = 32;
    while (kz < s.k && kz < 256) kz *= 2;
    const int n_grp = 256 / kz, zt = tid / kz, zn = tid % kz;
    auto kept_scores = [&](int j, float (&sc)[GH], bool ahead) {
#pragma unroll
        for (int g = 0; g < GH; ++g) sc[g] = 0.f;
        if (j >= j1) return;
        const KV* row = k_row(j);
        int e = ql;
        if (AHEAD && ahead)
#pragma unroll
            for (int u = 0; u < kPre; ++u, e += kLanes)
                if (e < s.nfk)
#pragma unroll
                    for (int g = 0; g < GH; ++g) sc[g] = fmaf(qf_s[g * s.nfk + e], k_pre[u], sc[g]);
#pragma unroll 8
        for (; e < s.nfk; e += kLanes) {
            float x = ld_f(row + e);
#pragma unroll
            for (int g = 0; g < GH; ++g) sc[g] = fmaf(qf_s[g * s.nfk + e], x, sc[g]);
        }
    };
    float sc_first[GH];
    // the basis of the first tile: a token's rotation and its lane's first frequency; a frequency's rotation and its first token
    float cd1 = 0.f, sd1 = 0.f, cr1 = 0.f, sr1 = 0.f, zc1 = 0.f, zs1 = 0.f, zr1 = 0.f, zi1 = 0.f;
    if (AHEAD) {
        kept_scores(j0 + tk, sc_first, true);
        if (s.dck > 0 && j0 + tk < j1) { basis_cs(1, j0 + tk, s.T, &cd1, &sd1); basis_cs(ql * per_lane, j0 + tk, s.T, &cr1, &sr1); }
        if (s.dcv > 0 && zn < s.k) { basis_cs(zn, 1, s.T, &zc1, &zs1); basis_cs(zn, j0 + zt * (kTile / n_grp), s.T, &zr1, &zi1); }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");     // u
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = tid; i < GH * s.M; i += blockDim.x) {
        const int g = i / s.M, m = i - g * s.M;
        u_s[i] = (g < ng && s.dck > 0) ? ws.u[((size_t)b * s.Hq + g_first + g) * s.M + m] : 0.f;
    }
    __syncthreads();
    for (int t0 = j0; t0 < j1; t0 += kTile) {
        const int j = t0 + tk;
        const bool valid = j < j1;
        const int nt = min(kTile, j1 - t0);
        float sc[GH];
        const bool first_tile = AHEAD && t0 == j0;
        if (first_tile) {
#pragma unroll
            for (int g = 0; g < GH; ++g) sc[g] = sc_first[g];
        } else {
            kept_scores(j, sc, false);
        }
        if (valid) {
            if (s.dck > 0) {
                float cd, sd;
                if (first_tile) { cd = cd1; sd = sd1; }
                else basis_cs(1, j, s.T, &cd, &sd);             // rotation per unit of n
                const int f1 = min(s.k, (ql + 1) * per_lane);
                for (int n0 = ql * per_lane; n0 < f1; n0 += 32) {
                    float cr, sr;
                    if (first_tile && n0 == ql * per_lane) { cr = cr1; sr = sr1; }
                    else basis_cs(n0, j, s.T, &cr, &sr);        // exact re-seed
                    const int n1 = min(f1, n0 + 32);
#pragma unroll 4
                    for (int n = n0; n < n1; ++n) {
#pragma unroll
                        for (int g = 0; g < GH; ++g) {
                            const float2 u = *reinterpret_cast<const float2*>(u_s + g * s.M + 2 * n);
                            sc[g] = fmaf(u.x, cr, fmaf(u.y, sr, sc[g]));
                        }
                        float t = cr * cd - sr * sd;
                        sr = fmaf(sr, cd, cr * sd);
                        cr = t;
                    }
                }
            }
        }
        lanes_sum(sc);
        softmax_tile(sc, valid);
        // o^u += p V^mu
        if (act_mid) {
            int i = tg_mid;
            if (first_tile) {
#pragma unroll
                for (int u = 0; u < kPre; ++u, i += ntg_mid) {
                    if (i < nt)
#pragma unroll
                        for (int g = 0; g < GH; ++g) o_mid[g] = fmaf(p_s[g * kTile + i], v_pre[u], o_mid[g]);
                }
            }
#pragma unroll 4
            for (; i < nt; i += ntg_mid) {
                const float x = v_at(t0 + i);
#pragma unroll
                for (int g = 0; g < GH; ++g) o_mid[g] = fmaf(p_s[g * kTile + i], x, o_mid[g]);
            }
        }
        // z[m] += p F[m][j]: thread owns a frequency and a group of the tile's tokens, walked by rotation
        if (s.dcv > 0) {
            const int gt = kTile / n_grp, i0 = zt * gt, i1 = min(nt, i0 + gt);
            for (int nb = 0; nb < s.k; nb += kz) {
                const int n = nb + zn;
                float zr[GH], zi[GH];
#pragma unroll
                for (int g = 0; g < GH; ++g) { zr[g] = 0.f; zi[g] = 0.f; }
                if (n < s.k && i0 < i1) {
                    float cd, sd, cr, sr;
                    if (AHEAD && nb == 0) { cd = zc1; sd = zs1; }
                    else basis_cs(n, 1, s.T, &cd, &sd);
                    for (int ia = i0; ia < i1; ia += 32) {
                        if (first_tile && nb == 0 && ia == i0) { cr = zr1; sr = zi1; }
                        else basis_cs(n, t0 + ia, s.T, &cr, &sr);
                        const int ib = min(i1, ia + 32);
#pragma unroll 4
                        for (int i = ia; i < ib; ++i) {
#pragma unroll
                            for (int g = 0; g < GH; ++g) {
                                float pv = p_s[g * kTile + i];
                                zr[g] = fmaf(pv, cr, zr[g]);
                                zi[g] = fmaf(pv, sr, zi[g]);
                            }
                            float t = cr * cd - sr * sd;
                            sr = fmaf(sr, cd, cr * sd);
                            cr = t;
                        }
                    }
                }
                if (n_grp == 1) {
                    if (n < s.k)
#pragma unroll
                        for (int g = 0; g < GH; ++g) { z_s[g * s.M + 2 * n] += zr[g]; z_s[g * s.M + 2 * n + 1] += zi[g]; }
                } else {
#pragma unroll
                    for (int g = 0; g < GH; ++g) { zr_s[(2 * g) * 256 + tid] = zr[g]; zr_s[(2 * g + 1) * 256 + tid] = zi[g]; }
                    __syncthreads();
                    for (int i = tid; i < 2 * GH * kz; i += 256) {
                        const int part = i / kz, f = i - part * kz;          // part = 2 g + (re, im)
                        if (nb + f < s.k) {
                            float v = 0.f;
                            for (int x = 0; x < n_grp; ++x) v += zr_s[part * 256 + x * kz + f];
                            z_s[(part >> 1) * s.M + 2 * (nb + f) + (part & 1)] += v;
                        }
                    }
                    __syncthreads();
                }
            }
        }
        __syncthreads();
    }

    // ---- window tokens [w0, w1) of this split: init rows, then the local ring --
    const int n_win = n_init + n_local;
    const int w0 = (int)((long long)split * n_win / p.n_split), w1 = (int)((long long)(split + 1) * n_win / p.n_split);
    for (int t0 = w0; t0 < w1; t0 += kTile) {
        const int t = t0 + tk;
        const bool valid = t < w1;
        auto row_of = [&](void* init, void* local, int tt) -> const KV* {
            if (tt < n_init) return win_row<KV>(init, s, b, h, s.l_init, tt);
            int r = head + (tt - n_init);
            if (r >= s.l_local) r -= s.l_local;
            return win_row<KV>(local, s, b, h, s.l_local, r);
        };
        float sc[GH];
#pragma unroll
        for (int g = 0; g < GH; ++g) sc[g] = 0.f;
        if (valid) {
            const KV* row = row_of(c.k_init, c.k_local, t);
#pragma unroll 8
            for (int e = ql; e < s.d; e += kLanes) {
                float x = ld_f(row + e);
#pragma unroll
                for (int g = 0; g < GH; ++g) sc[g] = fmaf(q_s[g * s.d + e], x, sc[g]);
            }
        }
        lanes_sum(sc);
        softmax_tile(sc, valid);
        const int nt = min(kTile, w1 - t0);
        if (act_win) {
            for (int i = tg_win; i < nt; i += ntg_win) {
                float x = ld_f(row_of(c.v_init, c.v_local, t0 + i) + e_win);
#pragma unroll
                for (int g = 0; g < GH; ++g) o_win[g] = fmaf(p_s[g * kTile + i], x, o_win[g]);
            }
        }
        __syncthreads();
    }

    // ---- reduce the output accumulators over token groups, write the partials --
#pragma unroll
    for (int g = 0; g < GH; ++g) {
        acc_s[tid * GH + g] = act_mid ? o_mid[g] : 0.f;
        const float l = warp_sum(rs.l[g]);
        if ((tid & 31) == 0) red_s[(tid >> 5) * GH + g] = l;
    }
    __syncthreads();
    for (int i = tid; i < GH * s.nfv; i += blockDim.x) {
        int g = i / s.nfv, e = i - g * s.nfv;
        float v = 0.f;
#pragma unroll 8
        for (int tg = 0; tg < ntg_mid; ++tg) v += acc_s[(tg * s.nfv + e) * GH + g];
        o_s[g * s.d + idf_v[e]] = v;
    }
    for (int i = tid; i < GH * s.M; i += blockDim.x) {
        int g = i / s.M, m = i - g * s.M;
        if (g < ng) ws.z[(((size_t)b * s.Hq + g_first + g) * p.n_part + split) * s.M + m] = z_s[i];
    }
    if (tid < ng) {
        float* ml = ws.ml + (((size_t)b * s.Hq + g_first + tid) * p.n_part + split) * 2;
        float mv = kNegBig, lv = 0.f;
#pragma unroll
        for (int g = 0; g < GH; ++g) if (g == tid) mv = rs.m[g];
#pragma unroll
        for (int w = 0; w < 8; ++w) lv += red_s[w * GH + tid];
        ml[0] = mv;
        ml[1] = lv;
    }
    __syncthreads();
    if (w1 > w0) {
#pragma unroll
        for (int g = 0; g < GH; ++g) acc_s[tid * GH + g] = act_win ? o_win[g] : 0.f;
        __syncthreads();
    }
    for (int i = tid; i < GH * s.d; i += blockDim.x) {
        int g = i / s.d, e = i - g * s.d;
        float v = o_s[i];
        if (w1 > w0)
            for (int tg = 0; tg < ntg_win; ++tg) v += acc_s[(tg * s.d + e) * GH + g];
        if (g < ng) ws.o[(((size_t)b * s.Hq + g_first + g) * p.n_part + split) * s.d + e] = v;
    }
}


static size_t direct_smem(const Dims& s, int gh) {
    return sizeof(float) * ((size_t)gh * s.d * 2 + (size_t)gh * s.nfk + 2 * (size_t)gh * s.M + (size_t)gh * kTile + 8 * gh + (size_t)(256 + 512) * gh);
}
template <typename KV, int GH, int OCC>
static cudaError_t launch_direct_t(const Dims& s, const CacheDev& c, const DecodePlan& p, const void* q, char* ws,
                                   cudaStream_t st) {
    const size_t smem = direct_smem(s, GH);
    cudaError_t err = ensure_dynamic_smem(decode_direct_kernel<KV, GH, OCC>, smem);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.n_split, s.Hkv * p.n_pass, s.B);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, decode_direct_kernel<KV, GH, OCC>, s, c, p, static_cast<const KV*>(q), ws);
}

// The fewest CTAs to an SM with which the grid takes no more waves.  Registers that a wave does not need fetch ahead; and CTAs that start while the kernel in front
// ends crowd on the SMs that it leaves first, up to this number.  The call, us, two CTAs to an SM / three (four heads): 16 CTAs (1 K tokens) 18.1/20.0,
// 72 27.4/28.6, 296 (2 K) 39.3/45.2; 304 (8 K) 146/111, 320 (a prompt of 5.8 K) 332/242, 384 (23 K) 2577/1554; of 512 53 calls 2 % faster with two, of 768 17 % slower.  One head:
// 296 CTAs (10 K tokens) 177 with as many as three to an SM, 133 with two.
static int direct_occ(const Dims& s, const DecodePlan& p) {
    const int most = p.gh == 4 ? 3 : 4, held = (int)(227 * 1024 / (direct_smem(s, p.gh) + 1024)), sms = sm_count();
    const long long ctas = (long long)p.n_split * s.Hkv * p.n_pass * s.B;
    auto waves = [&](int occ) { return (ctas + (long long)occ * sms - 1) / ((long long)occ * sms); };
    int occ = 2;
    for (int more = 3; more <= most && more <= held; ++more)
        if (waves(more) < waves(occ)) occ = more;
    return occ;
}

cudaError_t launch_decode_direct(const Dims& s, const CacheDev& c, int dtype, const DecodePlan& p, const void* q, char* ws,
                                 cudaStream_t st) {
    using std::integral_constant;
    const int occ = direct_occ(s, p);
    auto by_occ = [&](auto kv, auto heads) {
        using KV = decltype(kv);
        constexpr int GH = decltype(heads)::value;
        if (occ == 2) return launch_direct_t<KV, GH, 2>(s, c, p, q, ws, st);
        if (occ == 3) return launch_direct_t<KV, GH, 3>(s, c, p, q, ws, st);
        return launch_direct_t<KV, GH, GH == 4 ? 3 : 4>(s, c, p, q, ws, st);
    };
    auto by_heads = [&](auto kv) {
        if (p.gh == 4) return by_occ(kv, integral_constant<int, 4>{});
        if (p.gh == 2) return by_occ(kv, integral_constant<int, 2>{});
        return by_occ(kv, integral_constant<int, 1>{});
    };
    return dtype == FA_BF16 ? by_heads(__nv_bfloat16{}) : by_heads(float{});
}

}  // namespace fa
