// k_f64_fft_lo.cu -- FP64 FFT pass kernels, radices 2^0 .. 2^7.
#include "fftq.cuh"
void mrc_fft_fill_f64_lo(FftEntry (*t)[11], FftSegEntry *ts) { fftq_fill<0>(t, ts, std::make_integer_sequence<int, 8>{}); }
