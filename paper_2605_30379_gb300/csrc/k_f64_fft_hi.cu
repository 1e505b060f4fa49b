// k_f64_fft_hi.cu -- FP64 FFT pass kernels, radices 2^8 .. 2^10.
#include "fftq.cuh"
void mrc_fft_fill_f64_hi(FftEntry (*t)[11], FftSegEntry *ts) { fftq_fill<8>(t, ts, std::make_integer_sequence<int, 3>{}); }
