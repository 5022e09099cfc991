// Host dispatch of the trace kernels (fft_kernels.cuh) over the complex length M: plan queries, twiddle tables,
// and the launchers, which forward to FftLaunch<M> instantiated in fft_m*.cu.
//
// Appendix A: MDC = FFT along time -> batched per-frequency products -> inverse FFT.
#include "fft_kernels.cuh"

namespace smdd {

extern template struct FftLaunch<32>;
extern template struct FftLaunch<64>;
extern template struct FftLaunch<128>;
extern template struct FftLaunch<256>;
extern template struct FftLaunch<512>;
extern template struct FftLaunch<1024>;
extern template struct FftLaunch<1536>;
extern template struct FftLaunch<2048>;
extern template struct FftLaunch<4096>;

// value of the expression for complex length M_ (MM as a constant), `other` for a length without kernels
#define SMDD_SWITCH_M(M_, other, ...)                              \
    switch (M_) {                                                 \
        case 32: { constexpr int MM = 32; return __VA_ARGS__; }     \
        case 64: { constexpr int MM = 64; return __VA_ARGS__; }     \
        case 128: { constexpr int MM = 128; return __VA_ARGS__; }   \
        case 256: { constexpr int MM = 256; return __VA_ARGS__; }   \
        case 512: { constexpr int MM = 512; return __VA_ARGS__; }   \
        case 1024: { constexpr int MM = 1024; return __VA_ARGS__; } \
        case 1536: { constexpr int MM = 1536; return __VA_ARGS__; } \
        case 2048: { constexpr int MM = 2048; return __VA_ARGS__; } \
        case 4096: { constexpr int MM = 4096; return __VA_ARGS__; } \
        default: return other;                                    \
    }

int fft_traces_per_cta(int M) { SMDD_SWITCH_M(M, 0, Team<MM>::TR) }

int fft_blocks(int M, const TraceGrid &g) { SMDD_SWITCH_M(M, 0, blocks_for<MM>(g)) }

int fft_tw_size(int M) { SMDD_SWITCH_M(M, 0, tw_size(MM)) }

void fft_tw_fill(int M, std::vector<float2> &tw) {
    const double pi = 3.14159265358979323846;
    tw.assign(fft_tw_size(M), make_float2(0.f, 0.f));
    for (int i = 0; i < (int)tw.size(); ++i) {
        int num, den;
        tw_angle(M, i, num, den);
        const double ang = 2.0 * pi * (double)num / (double)den;
        tw[i] = make_float2((float)std::cos(ang), (float)-std::sin(ang));
    }
}

cudaError_t fft_prepare(int M) { SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::prepare()) }

cudaError_t launch_rfft(int M, const FftArgs &a, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::rfft(a, st))
}

cudaError_t launch_irfft_out(int M, const FftArgs &a, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::irfft_out(a, st))
}

cudaError_t launch_residual(int M, const FftArgs &a, int nblocks_expected, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::residual(a, nblocks_expected, st))
}

cudaError_t launch_update(int M, bool keep, const FftArgs &a, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::update(keep, a, st))
}

int fft_update_ahead(int M) { SMDD_SWITCH_M(M, 0, FftLaunch<MM>::update_ahead()) }

cudaError_t launch_queue_rfft(int M, const WorkQueue &q, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::queue_rfft(q, st))
}

cudaError_t launch_queue_residual(int M, const WorkQueue &q, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::queue_residual(q, st))
}

cudaError_t launch_queue_update(int M, const WorkQueue &q, cudaStream_t st) {
    SMDD_SWITCH_M(M, cudaErrorInvalidValue, FftLaunch<MM>::queue_update(q, st))
}

}  // namespace smdd
