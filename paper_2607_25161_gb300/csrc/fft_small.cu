// FFT pass kernels of the grid sizes 8 to 64.
#define FSD_FFT_KERNELS
#include "fft.cuh"

namespace fsd {

template <typename T>
const FftOps<T> *fft_small_ops(int n) {
  switch (n) {
    case 8: return FftLaunch<T, 2, 4>::ops();
    case 10: return FftLaunch<T, 2, 5>::ops();
    case 12: return FftLaunch<T, 3, 4>::ops();
    case 16: return FftLaunch<T, 4, 4>::ops();
    case 18: return FftLaunch<T, 3, 6>::ops();
    case 20: return FftLaunch<T, 4, 5>::ops();
    case 24: return FftLaunch<T, 4, 6>::ops();
    case 30: return FftLaunch<T, 5, 6>::ops();
    case 32: return FftLaunch<T, 4, 8>::ops();
    case 36: return FftLaunch<T, 6, 6>::ops();
    case 40: return FftLaunch<T, 5, 8>::ops();
    case 48: return FftLaunch<T, 6, 8>::ops();
    case 50: return FftLaunch<T, 5, 10>::ops();
    case 54: return FftLaunch<T, 6, 9>::ops();
    case 60: return FftLaunch<T, 6, 10>::ops();
    case 64: return FftLaunch<T, 8, 8>::ops();
    default: return nullptr;
  }
}
template const FftOps<float> *fft_small_ops<float>(int);
template const FftOps<double> *fft_small_ops<double>(int);

}  // namespace fsd
