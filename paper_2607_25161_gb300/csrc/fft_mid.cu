// FFT pass kernels of the grid sizes 72 to 150.
#define FSD_FFT_KERNELS
#include "fft.cuh"

namespace fsd {

template <typename T>
const FftOps<T> *fft_mid_ops(int n) {
  switch (n) {
    case 72: return FftLaunch<T, 8, 9>::ops();
    case 80: return FftLaunch<T, 8, 10>::ops();
    case 90: return FftLaunch<T, 9, 10>::ops();
    case 96: return FftLaunch<T, 8, 12>::ops();
    case 100: return FftLaunch<T, 10, 10>::ops();
    case 108: return FftLaunch<T, 9, 12>::ops();
    case 120: return FftLaunch<T, 10, 12>::ops();
    case 128: return FftLaunch<T, 8, 16>::ops();
    case 144: return FftLaunch<T, 12, 12>::ops();
    case 150: return FftLaunch<T, 10, 15>::ops();
    default: return nullptr;
  }
}
template const FftOps<float> *fft_mid_ops<float>(int);
template const FftOps<double> *fft_mid_ops<double>(int);

}  // namespace fsd
