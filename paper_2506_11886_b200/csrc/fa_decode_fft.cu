// Host side of the transform kernel (fa_decode_fft.cuh): which instance serves a plan, its shared memory, what fits.
#include "fa_decode_fft.cuh"

namespace fa {

int coop_pdl_state(int set) {
    constexpr int kMaxDev = 64;
    static signed char state[kMaxDev];
    static bool init = false;
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) { cudaGetLastError(); return 0; }
    std::lock_guard<std::mutex> lock(mu);
    if (!init) { for (int i = 0; i < kMaxDev; ++i) state[i] = -1; init = true; }
    if (set != -2) state[dev] = (signed char)set;
    return state[dev];
}


#define FA_FFT_LEN(GH, LS)                                                                                                        \
    extern template cudaError_t launch_fft_len<GH, LS>(const Dims&, const CacheDev&, const DecodePlan&, const void*, void*, char*, \
                                                       int, const void*, const void*, cudaStream_t);                               \
    extern template int resident_fft_len<GH, LS>(const Dims&, const DecodePlan&);
#define FA_FFT_LENS(GH) FA_FFT_LEN(GH, 5) FA_FFT_LEN(GH, 6) FA_FFT_LEN(GH, 7) FA_FFT_LEN(GH, 8) FA_FFT_LEN(GH, 9) FA_FFT_LEN(GH, 10)
FA_FFT_LENS(2)
FA_FFT_LENS(4)

template <int GH>
static cudaError_t launch_fft_ls(const Dims& s, const CacheDev& c, const DecodePlan& p, const void* q, void* out, char* ws, int step,
                                 const void* k_new, const void* v_new, cudaStream_t st) {
    switch (p.fft_log2) {
        case 5: return launch_fft_len<GH, 5>(s, c, p, q, out, ws, step, k_new, v_new, st);
        case 6: return launch_fft_len<GH, 6>(s, c, p, q, out, ws, step, k_new, v_new, st);
        case 7: return launch_fft_len<GH, 7>(s, c, p, q, out, ws, step, k_new, v_new, st);
        case 8: return launch_fft_len<GH, 8>(s, c, p, q, out, ws, step, k_new, v_new, st);
        case 9: return launch_fft_len<GH, 9>(s, c, p, q, out, ws, step, k_new, v_new, st);
        case 10: return launch_fft_len<GH, 10>(s, c, p, q, out, ws, step, k_new, v_new, st);
        default: return cudaErrorInvalidValue;
    }
}
template <int GH>
static int resident_ctas_ls(const Dims& s, const DecodePlan& p) {
    switch (p.fft_log2) {
        case 5: return resident_fft_len<GH, 5>(s, p);
        case 6: return resident_fft_len<GH, 6>(s, p);
        case 7: return resident_fft_len<GH, 7>(s, p);
        case 8: return resident_fft_len<GH, 8>(s, p);
        case 9: return resident_fft_len<GH, 9>(s, p);
        case 10: return resident_fft_len<GH, 10>(s, p);
        default: return 0;
    }
}

#ifdef FA_TIMELINE
#define FA_TL_UNIT(LS) int timeline_unit_##LS(long long* out); int spans_unit_##LS(long long* out);
FA_TL_UNIT(5) FA_TL_UNIT(6) FA_TL_UNIT(7) FA_TL_UNIT(8) FA_TL_UNIT(9) FA_TL_UNIT(10)
#endif

// True if the fused kernel of this plan can be launched as planned: a part that waits for nobody runs in
// waves; parts that wait for one another must all be resident at once (what a cooperative launch checks),
// which depends on the registers and shared memory of the compiled instance, so the runtime is asked.
bool decode_fft_launchable(const Dims& s, const DecodePlan& p) {
    if (!p.fused) return true;
    if (p.n_part <= 1) return true;
    const long long grid = (long long)p.n_part * s.Hkv * p.n_pass * s.B;
    const int resident = p.gh == 4 ? resident_ctas_ls<4>(s, p) : resident_ctas_ls<2>(s, p);
    return grid <= resident;
}

size_t decode_fft_smem_bytes(const Dims& s, int log2S, int gh, int nb, int occ, int split) {
    return (size_t)fft_smem_layout(log2S, s.k, gh, nb, s.d, occ, split, class_pairs(s.G, gh, split)).total;
}

// True if the fused kernel's staging areas hold a part's share of the coefficient rows: the rows
// of C^K in the transform buffers at the start, the merge scratch in the stage ring at the end.
bool decode_fft_fused_fits(const Dims& s, int log2S, int gh, int nb, int n_part, int occ, int split) {
    if (s.M % 4 != 0) return false;
    if (occ == 2 && log2S > 8) return false;                                           // no two-per-SM build of the long transforms
    const FftSmem L = fft_smem_layout(log2S, s.k, gh, nb, s.d, occ, split, class_pairs(s.G, gh, split));
    // at least eight rows of C^K per staged chunk (class pairs: the chunk may use the score and probability buffers too, as the kernel does)
    if (s.dck > 0 && (class_pairs(s.G, gh, split) ? (long long)((L.twf_off - L.fbuf_off) >> 2) : (long long)nb * L.fb_floats) < 8LL * s.dck) return false;
    const int ring = (L.twf_off - L.stages_off) >> 2;
    const int nrg = s.dcv ? (split ? kSplitConsumers : kConsumers) / (s.dcv >> 2) : 0;
    const int rows = (s.M / 4 + n_part - 1) / n_part * 4 + 4;
    const MergePlan m = merge_plan(ring, gh, n_part, n_part, s.d, s.dcv, nrg, rows);
    if (s.dcv > 0 && m.mch < 8) return false;                                                 // rows of C^V at a time
    return m.head + (long long)gh * n_part * s.dcv + gh * s.d <= ring;                        // the last part's merge of all parts
}

cudaError_t launch_decode_fft(const Dims& s, const CacheDev& c, int dtype, const DecodePlan& p, const void* q, void* out,
                              char* ws, const void* k_new, const void* v_new, cudaStream_t st) {
    if (dtype != FA_BF16) return cudaErrorInvalidValue;
    const int step = k_new != nullptr && v_new != nullptr ? 1 : 0;      // a fused step: the push of (k_new, v_new) rides on this launch
    if (p.gh == 4) return launch_fft_ls<4>(s, c, p, q, out, ws, step, k_new, v_new, st);
    return launch_fft_ls<2>(s, c, p, q, out, ws, step, k_new, v_new, st);
}

}  // namespace fa

#ifdef FA_TIMELINE
// The stamps of the transform length last run: of the units, the one with the latest stamp.
static int latest_unit(long long* host_out, int n, int (*const (&units)[6])(long long*)) {
    long long* buf = new long long[n];
    long long best = -1;
    int rc = 0;
    for (auto unit : units) {
        rc |= unit(buf);
        long long t = 0;
        for (int i = 0; i < n; ++i) t = buf[i] > t ? buf[i] : t;
        if (t > best) { best = t; for (int i = 0; i < n; ++i) host_out[i] = buf[i]; }
    }
    delete[] buf;
    return rc;
}
extern "C" int fa_debug_timeline(long long* host_out) {
    return latest_unit(host_out, 2 * 8 * 32, {fa::timeline_unit_5, fa::timeline_unit_6, fa::timeline_unit_7, fa::timeline_unit_8, fa::timeline_unit_9, fa::timeline_unit_10});
}
extern "C" int fa_debug_spans(long long* host_out) {
    return latest_unit(host_out, 32 * 160 * 4, {fa::spans_unit_5, fa::spans_unit_6, fa::spans_unit_7, fa::spans_unit_8, fa::spans_unit_9, fa::spans_unit_10});
}
#endif
