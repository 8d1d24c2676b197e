// The transform kernel's instances for classes of 64 slots.
#include "fa_decode_fft.cuh"

namespace fa {
#define FA_FFT_LEN(GH)                                                                                                            \
    template cudaError_t launch_fft_len<GH, 6>(const Dims&, const CacheDev&, const DecodePlan&, const void*, void*, char*, int,     \
                                                const void*, const void*, cudaStream_t);                                          \
    template int resident_fft_len<GH, 6>(const Dims&, const DecodePlan&);
FA_FFT_LEN(2)
FA_FFT_LEN(4)
#ifdef FA_TIMELINE
int timeline_unit_6(long long* out) { return (int)cudaMemcpyFromSymbol(out, g_fa_timeline, sizeof(g_fa_timeline)); }
int spans_unit_6(long long* out) { return (int)cudaMemcpyFromSymbol(out, g_fa_span, sizeof(g_fa_span)); }
#endif
}  // namespace fa
