// FFT pass kernels of the grid sizes 288 to 400.
#define FSD_FFT_KERNELS
#include "fft.cuh"

namespace fsd {

template <typename T>
const FftOps<T> *fft_huge_ops(int n) {
  switch (n) {
    case 288: return FftLaunch<T, 16, 18>::ops();
    case 300: return FftLaunch<T, 15, 20>::ops();
    case 320: return FftLaunch<T, 16, 20>::ops();
    case 324: return FftLaunch<T, 18, 18>::ops();
    case 360: return FftLaunch<T, 18, 20>::ops();
    case 400: return FftLaunch<T, 20, 20>::ops();
    default: return nullptr;
  }
}
template const FftOps<float> *fft_huge_ops<float>(int);
template const FftOps<double> *fft_huge_ops<double>(int);

}  // namespace fsd
