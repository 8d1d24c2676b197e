// fa_decode_attention (Eq.6 re-associated), the two small-side products around the token loop:
//   prologue   u_g[m] = scale * log2(e) * w_m * sum_e C^K[m][e] q_g[D^kc[e]]
//   epilogue   merge the token splits, o^c[e] = sum_m w_m z[m] C^V[m][e], normalise, scatter.
// Both read their coefficient matrix exactly once; each CTA brings a tile of rows into shared
// memory with 16-byte asynchronous copies (all in flight together) and works from there.  All
// loads of partial results are issued in independent batches so that a call costs a few memory
// round trips, not one per split.  The three kernels of a decode call are chained with
// programmatic dependent launch: each waits for the work in front of it, then lets its successor start, which may
// therefore read whatever was there before the call, and waits (griddepcontrol.wait) only where it first touches what its
// predecessor wrote.  (Compress and decode of 1024 fp32 tokens of one head, five kernels that are all latency: 36.9 -> 26.6 us
// with the launches of this call chained, the direct kernel's rows and kept-dim scores in front of its wait, and an
// epilogue that fetches everything at once and, with one slice of rows, needs no ticket.)
#include "fa_common.cuh"
#include "fa_decode_ws.cuh"

namespace fa {

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------- prologue --
// grid (ceil(M / rows_pro), Hkv, B), 256 threads.  SHORT: fewest round trips and shortest chains, for a grid that is one wave; else fewest instructions and
// registers, eight CTAs to an SM.  The call, us, SHORT / else: 64 CTAs 25.6/26.4, 256 27.0/27.8, 512 29.3/29.5, 1024 38.8/38.7, 4096 84.4/78.3, 8192 107/95, 12288 200/179.
template <typename KV, bool SHORT>
__global__ void __launch_bounds__(256, SHORT ? 4 : 8) decode_prologue_kernel(Dims s, CacheDev c, DecodePlan p, const KV* __restrict__ q,
                                                              char* wsp) {
    extern __shared__ __align__(16) float sm_pro[];
    pdl_wait();                                            // coefficients, query; the workspace
    pdl_launch_dependents();
    Ws ws = ws_view(wsp, p);
    const int h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    if (blockIdx.x == 0 && tid == 0) ws.cnt[b * s.Hkv + h] = 0;
    if (s.dck == 0) return;
    const int stride = s.dck + 4;                      // row stride of the tile: 16-byte aligned, bank-skewed
    float* tile = sm_pro;                              // [rows_pro][stride]
    float* qc_s = tile + p.rows_pro * stride;          // [G][dck] gathered query
    float* q_s = qc_s + (SHORT ? s.G * s.dck : 0);     // [G][d] query rows; else [G][dck + 1] gathered query
    const int m0 = blockIdx.x * p.rows_pro;
    const int rows = min(p.rows_pro, s.M - m0);
    const float* coef = coef_rows(c.coef_k, s, b, h, s.dck) + (size_t)m0 * s.dck;
    const int vpr = s.dck >> 2;
    for (int i = tid; i < rows * vpr; i += 256) {
        int r = i / vpr, v4 = i - r * vpr;
        cp_async16(tile + r * stride + 4 * v4, coef + (size_t)r * s.dck + 4 * v4);
    }
    if constexpr (!SHORT) {                            // a thread per row and head
        const int32_t* idc = c.idx_comp_k + (size_t)h * s.dck;
        for (int i = tid; i < s.G * s.dck; i += 256) {
            const int g = i / s.dck, e = i - g * s.dck;
            q_s[g * (s.dck + 1) + e] = ld_f(q + ((size_t)b * s.Hq + h * s.G + g) * s.d + idc[e]);
        }
        cp_async_wait_all();
        __syncthreads();
        for (int t = tid; t < rows * s.G; t += 256) {
            const int g = t % s.G, r = t / s.G, m = m0 + r;
            const float *row = tile + r * stride, *qq = q_s + g * (s.dck + 1);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
            for (int e = 0; e < s.dck; e += 4) {
                a0 = fmaf(row[e], qq[e], a0);
                a1 = fmaf(row[e + 1], qq[e + 1], a1);
                a2 = fmaf(row[e + 2], qq[e + 2], a2);
                a3 = fmaf(row[e + 3], qq[e + 3], a3);
            }
            ws.u[((size_t)b * s.Hq + h * s.G + g) * s.M + m] = recon_weight(s.norm, m, s.k, s.T) * s.scale * kLog2e * ((a0 + a1) + (a2 + a3));
        }
        return;
    }
    // (whole rows of q beside the index set: gathered from memory, q would be a second round trip behind it)
    const int idx = tid < s.dck ? c.idx_comp_k[(size_t)h * s.dck + tid] : 0;
    for (int i = tid; i < s.G * s.d; i += 256) q_s[i] = ld_f(q + ((size_t)b * s.Hq + h * s.G) * s.d + i);
    __syncthreads();
    if (tid < s.dck)
        for (int g = 0; g < s.G; ++g) qc_s[g * s.dck + tid] = q_s[g * s.d + idx];
    cp_async_wait_all();
    __syncthreads();
    // eight lanes to a row, four heads at a time
    const int l8 = tid & 7;
    for (int r0 = 0; r0 < rows; r0 += 32) {
        const int r = r0 + (tid >> 3), m = m0 + r;
        for (int g0 = 0; g0 < s.G; g0 += 4) {
            float a[4] = {0.f, 0.f, 0.f, 0.f};
            if (r < rows)
#pragma unroll 3
                for (int v = l8; v < vpr; v += 8) {
                    const float4 x = *reinterpret_cast<const float4*>(tile + r * stride + 4 * v);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g0 + g < s.G) {
                            const float4 y = *reinterpret_cast<const float4*>(qc_s + (g0 + g) * s.dck + 4 * v);
                            a[g] = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, a[g]))));
                        }
                    }
                }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int g = 0; g < 4; ++g) a[g] += __shfl_xor_sync(0xffffffffu, a[g], o);
            float mine = a[0];
#pragma unroll
            for (int g = 1; g < 4; ++g) if (l8 == g) mine = a[g];
            if (r < rows && l8 < 4 && g0 + l8 < s.G)
                ws.u[((size_t)b * s.Hq + h * s.G + g0 + l8) * s.M + m] = recon_weight(s.norm, m, s.k, s.T) * s.scale * kLog2e * mine;
        }
    }
}

// ---------------------------------------------------------------- epilogue --
// grid (n_slice, Hkv, B), 256 threads.  Each CTA merges the split statistics of its KV head,
// forms the weighted z of its slice of coefficient rows and multiplies by those rows of C^V;
// the last CTA of a (b, h) to finish (atomic ticket, nobody waits) adds the slices in a fixed
// order, normalises and writes the output rows.
__host__ __device__ inline size_t epilogue_l(const Dims& s, const DecodePlan& p) {
    const size_t a = (size_t)s.G * p.n_part, b = p.n_slice == 1 ? (size_t)s.G * s.dcv : 0;
    return a > b ? a : b;
}
// SHORT: the first parts' z and o with the statistics, the product shared out over all threads, in 125 registers (two CTAs to an SM); for grids
// that fill no more.  The call, us, SHORT / else: 16 CTAs 30.9/38.0, 32 39.1/43.5, 192 83/93, 256 34.7/38.0; 384 29.5/22.0, 384 54.1/51.4, 1024 95.5/82.9, 4096 139/94.
template <typename KV, bool SHORT>
__global__ void __launch_bounds__(256, SHORT ? 2 : 5) decode_epilogue_kernel(Dims s, CacheDev c, DecodePlan p, KV* __restrict__ out,
                                                              char* wsp) {
    extern __shared__ __align__(16) float sm_epi[];
    __shared__ int last_s;
    Ws ws = ws_view(wsp, p);
    const int slice = blockIdx.x, h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    const int rows_max = (s.M + p.n_slice - 1) / p.n_slice;
    const int m0 = slice * rows_max;
    const int rows = max(0, min(rows_max, s.M - m0));
    const int stride = s.dcv + 4;
    const int ns = p.n_part;
    float* alpha_s = sm_epi;                               // [G][n_split]: first the maxima, then exp2(m - max)
    float* l_s = alpha_s + s.G * ns;                       // [G][n_split], then o^c of a CTA alone
    float* linv_s = l_s + epilogue_l(s, p);                // [G]
    float* zw_s = linv_s + s.G;                            // [G][rows_max]
    int* inv_s = reinterpret_cast<int*>(zw_s + s.G * rows_max);   // [d] dim -> slot in D^vc, or -1
    float* tile = reinterpret_cast<float*>(inv_s + s.d);   // [rows_max][stride]
    tile = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(tile) + 15) & ~uintptr_t(15));
    float* ps_s = tile + rows_max * stride;                // [row groups][4][dcv] partial o^c

    // the coefficient tile does not depend on the main kernel: start it before waiting for it
    if (s.dcv > 0) {
        const float* cv = coef_rows(c.coef_v, s, b, h, s.dcv) + (size_t)m0 * s.dcv;
        const int vpr = s.dcv >> 2;
        for (int i = tid; i < rows * vpr; i += 256) {
            int r = i / vpr, v4 = i - r * vpr;
            cp_async16(tile + r * stride + 4 * v4, cv + (size_t)r * s.dcv + 4 * v4);
        }
    }
    // (a thread per dim: every dim is in D^vu or in D^vc)
    for (int e = tid; e < s.d; e += 256) inv_s[e < s.nfv ? c.idx_full_v[(size_t)h * s.nfv + e] : c.idx_comp_v[(size_t)h * s.dcv + e - s.nfv]] = e < s.nfv ? -1 : e - s.nfv;
    pdl_wait();                                            // partial results of the main kernel are complete

    // What a thread needs of the first kPre parts comes with the statistics, in one round trip: its first entry of z, and, where this CTA
    // finishes its head alone, its first two of o (SHORT).
    const bool alone = p.n_slice == 1;
    const size_t qh0 = (size_t)b * s.Hq + h * s.G;
    auto z_of = [&](int t) { const int g = t / rows, r = t - g * rows; return ws.z + (qh0 + g) * ns * s.M + m0 + r; };
    auto o_of = [&](int t) { const int g = t / s.d, e = t - g * s.d; return ws.o + (qh0 + g) * ns * s.d + e; };
    constexpr int kPre = SHORT ? 16 : 2;
    float zp[kPre], op[2][kPre];
    if (SHORT) {
        const bool z_on = s.dcv > 0 && tid < s.G * rows;
        const float* z = z_on ? z_of(tid) : nullptr;
#pragma unroll
        for (int i = 0; i < kPre; ++i) zp[i] = z_on && i < ns ? z[(size_t)i * s.M] : 0.f;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool o_on = alone && tid + 256 * u < s.G * s.d;
            const float* o = o_on ? o_of(tid + 256 * u) : nullptr;
#pragma unroll
            for (int i = 0; i < kPre; ++i) op[u][i] = o_on && i < ns ? o[(size_t)i * s.d] : 0.f;
        }
    }
    // sum over the parts of al[sp] x[sp * stride], the first kPre of them at hand or not
    auto merge = [&](const float* x, size_t stride, const float* al, const float (&pre)[kPre], bool have) {
        float v0 = 0.f, v1 = 0.f;
        int sp = 0;
        if (SHORT && have) {
#pragma unroll
            for (int i = 0; i < kPre; i += 2) {
                if (i < ns) v0 = fmaf(al[i], pre[i], v0);
                if (i + 1 < ns) v1 = fmaf(al[i + 1], pre[i + 1], v1);
            }
            sp = min(kPre, ns);
        }
        for (; sp + 8 <= ns; sp += 8) {                    // eight independent loads in flight
            float xx[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) xx[i] = x[(size_t)(sp + i) * stride];
#pragma unroll
            for (int i = 0; i < 8; i += 2) { v0 = fmaf(al[sp + i], xx[i], v0); v1 = fmaf(al[sp + i + 1], xx[i + 1], v1); }
        }
        for (; sp < ns; ++sp) v0 = fmaf(al[sp], x[(size_t)sp * stride], v0);
        return v0 + v1;
    };
    // split statistics: one (head, split) pair per thread, then a warp per head
    for (int i = tid; i < s.G * ns; i += 256) {
        const int g = i / ns, sp = i - g * ns;
        const float2 ml = *reinterpret_cast<const float2*>(ws.ml + ((qh0 + g) * ns + sp) * 2);
        alpha_s[i] = ml.x;
        l_s[i] = ml.y;
    }
    __syncthreads();
    for (int g = tid >> 5; g < s.G; g += 8) {
        const int lane = tid & 31;
        float mx = kNegBig, L = 0.f;
        for (int sp = lane; sp < ns; sp += 32) mx = fmaxf(mx, alpha_s[g * ns + sp]);
        mx = warp_max(mx);
        for (int sp = lane; sp < ns; sp += 32) {
            const float a = exp2f(alpha_s[g * ns + sp] - mx);
            alpha_s[g * ns + sp] = a;
            L = fmaf(a, l_s[g * ns + sp], L);
        }
        L = warp_sum(L);
        if (lane == 0) linv_s[g] = L > 0.f ? 1.0f / L : 0.f;
    }
    __syncthreads();
    float* oc_s = l_s;                                     // [G][dcv] o^c of a CTA alone (room for it: epilogue_l); the sums have been read
    if (s.dcv > 0) {
        for (int t = tid; t < s.G * rows; t += 256) {
            const int g = t / rows, r = t - g * rows;
            zw_s[g * rows_max + r] = merge(z_of(t), s.M, alpha_s + g * ns, zp, t == tid) * recon_weight(s.norm, m0 + r, s.k, s.T);
        }
        cp_async_wait_all();
        __syncthreads();
        if constexpr (!SHORT) {                            // a thread per column and head
            for (int t = tid; t < s.G * s.dcv; t += 256) {
                const int g = t / s.dcv, e = t - g * s.dcv;
                const float* zw = zw_s + g * rows_max;
                float a0 = 0.f, a1 = 0.f;
                int r = 0;
                for (; r + 2 <= rows; r += 2) {
                    a0 = fmaf(zw[r], tile[r * stride + e], a0);
                    a1 = fmaf(zw[r + 1], tile[(r + 1) * stride + e], a1);
                }
                if (r < rows) a0 = fmaf(zw[r], tile[r * stride + e], a0);
                if (alone) oc_s[t] = a0 + a1;
                else ws.oc[((qh0 + g) * p.n_slice + slice) * s.dcv + e] = a0 + a1;
            }
        } else {
        // a thread takes four columns and every nrg-th row, four heads at a time; then the row groups are added in order
        const int nv = s.dcv >> 2, nrg = 256 / nv, rg = tid / nv, v = tid - rg * nv;
        for (int g0 = 0; g0 < s.G; g0 += 4) {
            const int hg = min(4, s.G - g0);
            float4 a[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) a[g] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (rg < nrg)
#pragma unroll 2
                for (int r = rg; r < rows; r += nrg) {
                    const float4 x = *reinterpret_cast<const float4*>(tile + r * stride + 4 * v);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g < hg) {
                            const float w = zw_s[(g0 + g) * rows_max + r];
                            a[g].x = fmaf(w, x.x, a[g].x);
                            a[g].y = fmaf(w, x.y, a[g].y);
                            a[g].z = fmaf(w, x.z, a[g].z);
                            a[g].w = fmaf(w, x.w, a[g].w);
                        }
                    }
                }
            if (g0 > 0) __syncthreads();
            if (rg < nrg)
#pragma unroll
                for (int g = 0; g < 4; ++g) if (g < hg) *reinterpret_cast<float4*>(ps_s + (rg * hg + g) * s.dcv + 4 * v) = a[g];
            __syncthreads();
            for (int t = tid; t < hg * s.dcv; t += 256) {
                float x = 0.f;
#pragma unroll 4
                for (int y = 0; y < nrg; ++y) x += ps_s[y * hg * s.dcv + t];
                const int g = t / s.dcv;
                if (alone) oc_s[g0 * s.dcv + t] = x;
                else ws.oc[((qh0 + g0 + g) * p.n_slice + slice) * s.dcv + t - g * s.dcv] = x;
            }
        }
        }
    }
    if (!alone) {
        // ticket
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const int done = atomicAdd(ws.cnt + b * s.Hkv + h, 1);
            last_s = (done == (int)gridDim.x - 1);
        }
        __syncthreads();
        if (!last_s) return;
        __threadfence();
    } else {
        __syncthreads();
    }
    auto finish = [&](int t, const float (&pre)[kPre], bool have) {
        const int g = t / s.d, e = t - g * s.d;
        float v = merge(o_of(t), s.d, alpha_s + g * ns, pre, have);
        const int slot = inv_s[e];
        if (slot >= 0) {
            if (alone) {
                v += oc_s[g * s.dcv + slot];
            } else {
                const float* oc = ws.oc + (qh0 + g) * p.n_slice * s.dcv + slot;
                float w0 = 0.f, w1 = 0.f;
                int sl = 0;
                for (; sl + 8 <= p.n_slice; sl += 8) {
                    float cc[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) cc[i] = __ldcg(oc + (size_t)(sl + i) * s.dcv);
#pragma unroll
                    for (int i = 0; i < 8; i += 2) { w0 += cc[i]; w1 += cc[i + 1]; }
                }
                for (; sl < p.n_slice; ++sl) w0 += __ldcg(oc + (size_t)sl * s.dcv);
                v += w0 + w1;
            }
        }
        st_f(out + (qh0 + g) * s.d + e, v * linv_s[g]);
    };
    if (SHORT) {
        if (tid < s.G * s.d) finish(tid, op[0], alone);
        if (tid + 256 < s.G * s.d) finish(tid + 256, op[1], alone);
    }
    for (int t = tid + (SHORT ? 512 : 0); t < s.G * s.d; t += 256) finish(t, op[0], false);
}

// ---------------------------------------------------------------- launchers --
// Launch with the programmatic-stream-serialization attribute: the kernel may start while its
// predecessor in the stream still runs; it synchronises with griddepcontrol.wait.
template <typename... Params, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                              Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <typename KV>
static cudaError_t launch_prologue_t(const Dims& s, const CacheDev& c, const DecodePlan& p, const void* q, char* ws,
                                     cudaStream_t st) {
    const int tiles = s.dck > 0 ? (s.M + p.rows_pro - 1) / p.rows_pro : 1;
    const bool one_wave = (long long)tiles * s.Hkv * s.B <= 4ll * sm_count();
    const size_t smem = sizeof(float) * ((size_t)p.rows_pro * (s.dck + 4) + (size_t)s.G * (one_wave ? s.dck + s.d : s.dck + 1));
    auto go = [&](auto kernel) {
        cudaError_t err = ensure_dynamic_smem(kernel, smem);
        if (err != cudaSuccess) return err;
        return launch_pdl(kernel, dim3(tiles, s.Hkv, s.B), dim3(256), smem, st, true, s, c, p, static_cast<const KV*>(q), ws);
    };
    return one_wave ? go(decode_prologue_kernel<KV, true>) : go(decode_prologue_kernel<KV, false>);
}

cudaError_t launch_decode_prologue(const Dims& s, const CacheDev& c, int dtype, const DecodePlan& p, const void* q,
                                   char* ws, cudaStream_t st) {
    if (dtype == FA_BF16) return launch_prologue_t<__nv_bfloat16>(s, c, p, q, ws, st);
    return launch_prologue_t<float>(s, c, p, q, ws, st);
}

template <typename KV>
static cudaError_t launch_epilogue_t(const Dims& s, const CacheDev& c, const DecodePlan& p, void* out, char* ws,
                                     cudaStream_t st) {
    const int rows = (s.M + p.n_slice - 1) / p.n_slice;
    const bool one_wave = (long long)p.n_slice * s.Hkv * s.B <= 2ll * sm_count();
    const size_t smem = sizeof(float) * ((size_t)s.G * p.n_part + epilogue_l(s, p) + s.G + (size_t)s.G * rows + s.d + 4 + (size_t)rows * (s.dcv + 4) +
                                         (one_wave ? 4 * 1024 : 0));      // (256 threads' four columns of four heads)
    auto go = [&](auto kernel) {
        cudaError_t err = ensure_dynamic_smem(kernel, smem);
        if (err != cudaSuccess) return err;
        return launch_pdl(kernel, dim3(p.n_slice, s.Hkv, s.B), dim3(256), smem, st, true, s, c, p, static_cast<KV*>(out), ws);
    };
    return one_wave ? go(decode_epilogue_kernel<KV, true>) : go(decode_epilogue_kernel<KV, false>);
}

cudaError_t launch_decode_epilogue(const Dims& s, const CacheDev& c, int dtype, const DecodePlan& p, void* out, char* ws,
                                   cudaStream_t st) {
    if (dtype == FA_BF16) return launch_epilogue_t<__nv_bfloat16>(s, c, p, out, ws, st);
    return launch_epilogue_t<float>(s, c, p, out, ws, st);
}

}  // namespace fa
