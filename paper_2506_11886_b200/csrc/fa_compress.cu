// fa_compress, CUDA-core path (Eq.1-4): partition + gather, then the
// projection C = F X^mn as an fp32 tile product with the basis generated on
// the fly.  Serves fp32 caches and is the fallback of the tensor-core path.
#include "fa_common.cuh"

namespace fa {

// ---- index-set check (Eq.2: D^u and D^c partition the head dims) ------------
__global__ void validate_kernel(Dims s, CacheDev c) {
    int h = blockIdx.x;
    int side = blockIdx.y;
    __shared__ int seen[256];
    __shared__ int bad;
    int nfull = side == 0 ? s.nfk : s.nfv;
    int ncomp = s.d - nfull;
    const int32_t* idf = (side == 0 ? c.idx_full_k : c.idx_full_v) + (size_t)h * nfull;
    const int32_t* idc = (side == 0 ? c.idx_comp_k : c.idx_comp_v) + (size_t)h * ncomp;
    for (int i = threadIdx.x; i < s.d; i += blockDim.x) seen[i] = 0;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < s.d; i += blockDim.x) {
        bool full = i < nfull;
        const int32_t* a = full ? idf : idc;
        int pos = full ? i : i - nfull;
        int v = a[pos];
        if (v < 0 || v >= s.d) { atomicExch(&bad, 1); continue; }
        if (pos > 0 && a[pos - 1] >= v) atomicExch(&bad, 1);
        atomicAdd(&seen[v], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < s.d; i += blockDim.x)
        if (seen[i] != 1) atomicExch(&bad, 1);
    __syncthreads();
    if (threadIdx.x == 0 && bad) atomicExch(c.status, (int)FA_ERR_INDEX);
}

cudaError_t launch_validate(const Dims& s, const CacheDev& c, cudaStream_t st) {
    validate_kernel<<<dim3(s.Hkv, 2), 128, 0, st>>>(s, c);
    return cudaGetLastError();
}

// ---- Eq.1-2: windows, kept dims, counters -----------------------------------
// grid (chunks of 64 tokens, Hkv, B * 2 sides).  Every row of the input, of the windows and of the
// kept-dim rows starts on a 16-byte boundary and is a whole number of 16-byte chunks (the C ABI asks
// for 16-byte aligned K, V and strides that are multiples of 8 elements; head_dim and the kept-dim
// counts are multiples of 8).  The CTA stages its 64 input rows in shared memory with one 16-byte load
// per chunk, then one thread per output chunk either copies it (window rows) or gathers its dims
// through the index set (kept-dim rows; for V^mu of bf16 caches the chunk it writes is the permuted one).
constexpr int kRowsPerCta = 64;
// The i-th chunk that holds window tokens (chunk 0 always counts: it writes the counters), and how many there are.
__host__ __device__ inline int window_skip(int L, int n_init, int n_local, int* first) {
    int a = (n_init + kRowsPerCta - 1) / kRowsPerCta;    // first chunk past the initial window
    const int c = (L - n_local) / kRowsPerCta;           // first chunk with a token of the local window
    if (a < 1) a = 1;
    *first = a;
    return c > a ? c - a : 0;
}
__host__ __device__ inline int window_chunk(int i, int L, int n_init, int n_local) {
    int a;
    const int skip = window_skip(L, n_init, n_local, &a);
    return i < a ? i : i + skip;
}

template <typename KV>
__global__ void __launch_bounds__(256) partition_gather_kernel(Dims s, CacheDev c, const KV* __restrict__ K,
                                                                   const KV* __restrict__ V, int64_t sb, int64_t st,
                                                                   int64_t sh, int Lmax, const __grid_constant__ RowLens lens, int tc_min, int zero_coef) {
    constexpr int EPC = 16 / (int)sizeof(KV);            // elements per chunk
    extern __shared__ __align__(16) unsigned char gsm[];
    // the contraction kernel behind this one may start at once (programmatic dependent launch): it waits for this
    // grid only in front of its reductions into the coefficients cleared here
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    KV* rows_s = reinterpret_cast<KV*>(gsm);                                         // [64][d]
    int32_t* idf_s = reinterpret_cast<int32_t*>(gsm + (size_t)kRowsPerCta * s.d * sizeof(KV));   // [nfull]
    const int h = blockIdx.y, b = blockIdx.z >> 1, side = blockIdx.z & 1;
    const int L = row_len(lens, Lmax, b);
    const int n_init = min(L, s.l_init);
    const int n_local = min(L - n_init, s.l_local);
    const int n_mid = L - n_init - n_local;
    if (blockIdx.x == 0 && blockIdx.y == 0 && side == 0 && threadIdx.x == 0) {
        c.state[kStateStride * b + 0] = n_init;
        c.state[kStateStride * b + 1] = n_local;
        c.state[kStateStride * b + 2] = n_mid;
        c.state[kStateStride * b + 3] = 0;          // ring starts at physical row 0
        c.state[kStateStride * b + 4] = 0;          // append ticket
    }
    const int nfull = side == 0 ? s.nfk : s.nfv;
    if ((zero_coef == 1 || (zero_coef == 2 && n_mid < tc_min)) && s.d > nfull) {
        // the contraction kernels behind this one ADD their partial sums: the CTAs of a (b, head, side) clear its coefficients
        float4* cz = reinterpret_cast<float4*>(coef_rows(side == 0 ? c.coef_k : c.coef_v, s, b, h, s.d - nfull));
        const int n4 = s.M * (s.d - nfull) / 4;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x) cz[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const KV* X = (side == 0 ? K : V) + (size_t)b * sb + (size_t)h * sh;
    const int32_t* idf = (side == 0 ? c.idx_full_k : c.idx_full_v) + (size_t)h * nfull;
    void* w_init = side == 0 ? c.k_init : c.v_init;
    void* w_local = side == 0 ? c.k_local : c.v_local;
    void* w_mid = side == 0 ? c.k_mid : c.v_mid;
    // without the kept-dim rows (the tensor-core kernel writes them) the chunks of middle tokens only are left out
    const bool mid_rows = n_mid < tc_min;
    const int chunk = mid_rows ? (int)blockIdx.x : window_chunk((int)blockIdx.x, L, n_init, n_local);
    const int t0 = chunk * kRowsPerCta, nrow = min(L - t0, kRowsPerCta);
    const int cpr = s.d / EPC;                            // chunks per input row
    for (int i = threadIdx.x; i < nfull; i += blockDim.x) idf_s[i] = idf[i];
    for (int i = threadIdx.x; i < nrow * cpr; i += blockDim.x) {
        const int r = i / cpr, ch = i - r * cpr;
        reinterpret_cast<uint4*>(rows_s)[i] = __ldg(reinterpret_cast<const uint4*>(X + (size_t)(t0 + r) * st) + ch);
    }
    __syncthreads();
    // window rows: chunk for chunk
    for (int i = threadIdx.x; i < nrow * cpr; i += blockDim.x) {
        const int r = i / cpr, ch = i - r * cpr, t = t0 + r;
        KV* dst = nullptr;
        if (t < n_init) dst = win_row<KV>(w_init, s, b, h, s.l_init, t);
        else if (t >= L - n_local) dst = win_row<KV>(w_local, s, b, h, s.l_local, t - (L - n_local));
        if (dst) reinterpret_cast<uint4*>(dst)[ch] = reinterpret_cast<const uint4*>(rows_s)[i];
    }
    // kept-dim rows of the middle
    // (one CTA waits for the kernel in front, so that the end of this grid implies that one's; if all did, they would keep theirs from
    // taking turns beside a projection)
    const bool waits = blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
    if (!mid_rows) {
        if (waits) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int cpo = nfull / EPC;                          // chunks per output row
    for (int i = threadIdx.x; i < nrow * cpo; i += blockDim.x) {
        const int r = i / cpo, ch = i - r * cpo, t = t0 + r;
        if (t < n_init || t >= L - n_local) continue;
        const int j = t - n_init, cls = j % s.P, slot = j / s.P;
        // output chunk ch holds the logical chunk ch ^ swizzle (the permutation is an involution)
        const int lch = (side == 1 && sizeof(KV) == 2) ? (ch ^ v_swz(slot, nfull >> 3)) : ch;
        const KV* row = rows_s + r * s.d;
        __align__(16) KV vals[EPC];
#pragma unroll
        for (int e = 0; e < EPC; ++e) vals[e] = row[idf_s[lch * EPC + e]];
        KV* dst = mid_row<KV>(w_mid, s, b, h, cls, slot, nfull);
        reinterpret_cast<uint4*>(dst)[ch] = *reinterpret_cast<const uint4*>(vals);
    }
    // In a chain of launches that overlap one another (the partition kernels of several layers, each launched
    // programmatically behind the one before), the end of this grid then implies the end of all before it.  Launched
    // the plain way this returns at once.
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- Eq.3-4: C[m][e] += sum_j F[m][j] X[n_init + j][D^c[e]] ------------------
// grid (row tiles of 32 or 64 coefficient rows, token splits, B * Hkv * 2 sides).
// Per 64-token chunk the CTA stages the gathered columns and a 64 x 32 basis
// tile in shared memory; thread (rg, lane) accumulates rows 4 rg..4 rg + 3 of
// the tile for columns lane, lane + 32, ...  Partial sums of the token splits
// are added to the zeroed coefficients with atomics.
// R rows per thread: eight (half the shared-memory reads per product) or four (finer tiles, more CTAs and fewer registers), see rows_per_thread.  Bound by the FMA and
// shared-memory pipes beside a chain of index, load and barrier per chunk.
constexpr int kTJ = 64;

// NC: columns per lane (32 NC >= the compressed dims of either side; the products of lanes without a column are not issued).
template <typename KV, int NC, int R>
__global__ void __launch_bounds__(256) compress_coef_kernel(Dims s, CacheDev c, const KV* __restrict__ K,
                                                            const KV* __restrict__ V, int64_t sb, int64_t st, int64_t sh,
                                                            int Lmax, int chunks_per_split, const __grid_constant__ RowLens lens, int tc_min) {
    extern __shared__ float smem[];
    int side = blockIdx.z & 1;
    int bh = blockIdx.z >> 1;
    int b = bh / s.Hkv, h = bh % s.Hkv;
    int nfull = side == 0 ? s.nfk : s.nfv;
    int ncomp = s.d - nfull;
    const int L = row_len(lens, Lmax, b);
    const int n_init = min(L, s.l_init), n_mid = mid_of(s, L);
    if (ncomp == 0 || n_mid >= tc_min) {                 // nothing to do, or the tensor-core kernel's row
        asm volatile("griddepcontrol.wait;" ::: "memory");   // (the end of this grid implies the end of the one before)
        return;
    }
    const KV* X = (side == 0 ? K : V) + (size_t)b * sb + (size_t)h * sh;
    const int32_t* idc = (side == 0 ? c.idx_comp_k : c.idx_comp_v) + (size_t)h * ncomp;
    float* coef = coef_rows(side == 0 ? c.coef_k : c.coef_v, s, b, h, ncomp);

    constexpr int kTM = 8 * R, kXs = 32 * NC;
    float* X_s = smem;                       // [kTJ][kXs], zeros past the compressed dims
    float* F_s = smem + kTJ * kXs;           // [kTJ][kTM]
    int m0 = blockIdx.x * kTM;
    int rg = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float acc[R][NC];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < NC; ++i) acc[r][i] = 0.f;

    int col[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) col[i] = lane + 32 * i < ncomp ? idc[lane + 32 * i] : 0;

    int j_begin = blockIdx.y * chunks_per_split * kTJ;
    int j_end = min(n_mid, j_begin + chunks_per_split * kTJ);
    for (int j0 = j_begin; j0 < j_end; j0 += kTJ) {
        int nj = min(kTJ, j_end - j0);
        __syncthreads();
        // a warp takes every eighth token: its lanes' columns are fixed, so all loads of a chunk are independent
        const KV* xrow = X + (size_t)(n_init + j0 + rg) * st;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int e = lane + 32 * i;
#pragma unroll
                for (int q = 0; q < kTJ / 8; ++q)
                    X_s[(rg + 8 * q) * kXs + e] = e < ncomp && rg + 8 * q < nj ? ld_f(xrow + (size_t)(8 * q) * st + col[i]) : 0.f;
        }
        // basis tile: thread -> (token jj, frequency pair nn) ; rows 2 nn (cos), 2 nn + 1 (sin)
        for (int i = threadIdx.x; i < kTJ * (kTM / 2); i += blockDim.x) {
            int jj = i / (kTM / 2), nn = i % (kTM / 2);
            int n = m0 / 2 + nn;
            float cs = 0.f, sn = 0.f;
            if (jj < nj && n < s.k) basis_cs(n, j0 + jj, s.T, &cs, &sn);
            *reinterpret_cast<float2*>(F_s + jj * kTM + 2 * nn) = make_float2(cs, sn);
        }
        __syncthreads();
#pragma unroll 4
        for (int jj = 0; jj < nj; ++jj) {
            float f[R];
#pragma unroll
            for (int r = 0; r < R; r += 4) {
                const float4 f4 = *reinterpret_cast<const float4*>(F_s + jj * kTM + R * rg + r);
                f[r] = f4.x; f[r + 1] = f4.y; f[r + 2] = f4.z; f[r + 3] = f4.w;
            }
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const float x = X_s[jj * kXs + lane + 32 * i];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r][i] = fmaf(f[r], x, acc[r][i]);
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");    // the partition kernel clears the coefficients
#pragma unroll
    for (int r = 0; r < R; ++r) {
        int m = m0 + R * rg + r;
        if (m >= s.M) continue;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            int e = lane + 32 * i;
            if (e < ncomp) atomicAdd(coef + (size_t)m * ncomp + e, acc[r][i]);
        }
    }
}

// Rows per thread of the contraction, and how the tokens' chunks are split: what the SM with the most CTAs takes for them, a chunk counting as the products of a
// lane's token and 10 of them more (with eight rows of eight columns, registers for one CTA to an SM, 1.3 times those), and a CTA by itself 60 at least.  Rows of
// several lengths even the SMs out: what an average one has.  Of 1184 calls (16 to 2048 coefficients, 1 to 256 heads, 20 to 6000 tokens, 64 to 256 dims) 0.5 % behind the better form on average.  us, four / eight rows a thread:
//   tiles of 64 rows that would be half empty: 16 coefficients, 32 heads, 900 tokens 149/264; 32 coefficients, 32 heads, 340 tokens 17.2/25.7
//   many CTAs: 200 coefficients, 128 heads, 5600 tokens 1234/1106, 128, 64 heads, rows of 1013 and 570 tokens 154/142 (both ragged); 128, 48 heads, 590 tokens 101/85; few: 16.9/16.1, 12.8/11.4
//   256 dims: 1024 coefficients, 32 heads 4880/6181; 100, 96 heads 459/544; few CTAs: 100, two heads 25.5/21.4
//   a fixed order (a CTA takes all tokens of its rows): 100 coefficients, 8 heads, 1300 tokens 69/100; 256, 32 heads, 240 tokens 60/47; 128, 64 heads, 1000 tokens 191/228
struct RowSplit { int rpt, row_tiles, n_tsplit, cps; };
static RowSplit rows_per_thread(const Dims& s, int live_rows, int chunks, int nc, bool ordered, bool ragged) {
    RowSplit best = {};
    double least = 0;
    const int sms = sm_count();
    for (int rpt = 4; rpt <= 8; rpt += 4) {
        RowSplit x = {rpt, (s.M + 8 * rpt - 1) / (8 * rpt), 1, 0};
        const int ctas_fixed = x.row_tiles * live_rows * s.Hkv * 2;
        int n = (4 * sms + ctas_fixed - 1) / ctas_fixed;
        if (n > chunks) n = chunks;
        if (n < 1 || ordered) n = 1;                         // one split: every coefficient is added to zero exactly once
        x.cps = (chunks + n - 1) / n;
        x.n_tsplit = (chunks + x.cps - 1) / x.cps;
        const double chunk = 10 + rpt * nc * (rpt == 8 && nc == 8 ? 1.3 : 1.0), ctas = (double)ctas_fixed * x.n_tsplit / sms, all = (ragged ? ctas : ceil(ctas)) * chunk;
        const double time = x.cps * (all > 60 ? all : 60);
        if (best.rpt == 0 || time < least) { best = x; least = time; }
    }
    return best;
}

template <typename KV>
static cudaError_t launch_compress_t(const Dims& s, const CacheDev& c, const void* K, const void* V, int64_t sb,
                                     int64_t st, int64_t sh, int L, bool with_coef, bool ordered, int tc_min, int zero_coef, bool chained,
                                     const RowLens* lens, cudaStream_t stream) {
    RowLens rl = {};
    if (lens) rl = *lens;
    // chunks and short middles (not the tensor-core kernel's) of the longest row
    int chunks_rows = 1, n_mid = 0, n_short = 0;
    for (int b = 0; b < (rl.n ? rl.n : 1); ++b) {
        const int Lb = row_len(rl, L, b), ni = Lb < s.l_init ? Lb : s.l_init, nl = (Lb - ni) < s.l_local ? (Lb - ni) : s.l_local;
        int chunks = (Lb + kRowsPerCta - 1) / kRowsPerCta, first;
        if (Lb - ni - nl >= tc_min) chunks -= window_skip(Lb, ni, nl, &first);
        else {
            ++n_short;
            if (Lb - ni - nl > n_mid) n_mid = Lb - ni - nl;
        }
        if (chunks > chunks_rows) chunks_rows = chunks;
    }
    constexpr int EPC = 16 / (int)sizeof(KV);
    if (s.d % EPC || s.nfk % EPC || s.nfv % EPC || sb % EPC || st % EPC || sh % EPC || (reinterpret_cast<uintptr_t>(K) & 15) ||
        (reinterpret_cast<uintptr_t>(V) & 15))
        return cudaErrorInvalidValue;
    const int nf = s.nfk > s.nfv ? s.nfk : s.nfv;
    const size_t gsmem = (size_t)kRowsPerCta * s.d * sizeof(KV) + sizeof(int32_t) * (size_t)nf;
    cudaError_t err = ensure_dynamic_smem(partition_gather_kernel<KV>, gsmem);
    if (err != cudaSuccess) return err;
    {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(chunks_rows, s.Hkv, s.B * 2);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = gsmem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // chained: may run beside the partition kernel in front of it
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = chained ? 1 : 0;
        err = cudaLaunchKernelEx(&cfg, partition_gather_kernel<KV>, s, c, static_cast<const KV*>(K), static_cast<const KV*>(V), sb, st, sh, L,
                                 rl, tc_min, zero_coef);
    }
    if (err != cudaSuccess) return err;
    int max_comp = s.dck > s.dcv ? s.dck : s.dcv;
    if (n_mid == 0 || max_comp == 0 || !with_coef) return cudaSuccess;
    const int live_rows = rl.n ? n_short : s.B;
    const int nc = max_comp <= 128 ? (max_comp + 31) / 32 : 8;
    const RowSplit split = rows_per_thread(s, live_rows, (n_mid + kTJ - 1) / kTJ, nc, ordered, rl.n > 1);
    const int rpt = split.rpt, cps = split.cps;
    const size_t smem = sizeof(float) * kTJ * (size_t)(32 * nc + 8 * rpt);
    // behind the partition kernel programmatically: it waits for it in front of its additions
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(split.row_tiles, split.n_tsplit, s.B * s.Hkv * 2);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto go = [&](auto kernel) {
        const cudaError_t e = ensure_dynamic_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        return cudaLaunchKernelEx(&cfg, kernel, s, c, static_cast<const KV*>(K), static_cast<const KV*>(V), sb, st, sh, L, cps, rl, tc_min);
    };
    switch (nc) {
        case 1: return rpt == 8 ? go(compress_coef_kernel<KV, 1, 8>) : go(compress_coef_kernel<KV, 1, 4>);
        case 2: return rpt == 8 ? go(compress_coef_kernel<KV, 2, 8>) : go(compress_coef_kernel<KV, 2, 4>);
        case 3: return rpt == 8 ? go(compress_coef_kernel<KV, 3, 8>) : go(compress_coef_kernel<KV, 3, 4>);
        case 4: return rpt == 8 ? go(compress_coef_kernel<KV, 4, 8>) : go(compress_coef_kernel<KV, 4, 4>);
        default: return rpt == 8 ? go(compress_coef_kernel<KV, 8, 8>) : go(compress_coef_kernel<KV, 8, 4>);
    }
}

// with_coef = false runs only the partition / gather kernel (the tensor-core or the transform path computes the
// coefficients); rows with at least tc_min middle tokens get no kept-dim rows and no coefficients here (windows and
// counters only: the tensor-core kernel writes the rest); lens: prompt lengths of the batch rows (at most L), or none;
// zero_coef: 1 clears the coefficients in the same launch (for the contraction kernels, which add to them), 2 those of the rows with fewer than
// tc_min middle tokens; chained: may run beside the kernel of the same call in front of it.
cudaError_t launch_compress(const Dims& s, const CacheDev& c, int dtype, const void* K, const void* V, int64_t sb,
                            int64_t st, int64_t sh, int L, bool with_coef, bool ordered, int tc_min, int zero_coef,
                            cudaStream_t stream, bool chained, const RowLens* lens) {
    if (dtype == FA_BF16) return launch_compress_t<__nv_bfloat16>(s, c, K, V, sb, st, sh, L, with_coef, ordered, tc_min, zero_coef, chained, lens, stream);
    return launch_compress_t<float>(s, c, K, V, sb, st, sh, L, with_coef, ordered, tc_min, zero_coef, chained, lens, stream);
}

}  // namespace fa
