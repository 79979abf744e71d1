// FFT pass kernels of the grid sizes 160 to 270.
#define FSD_FFT_KERNELS
#include "fft.cuh"

namespace fsd {

template <typename T>
const FftOps<T> *fft_large_ops(int n) {
  switch (n) {
    case 160: return FftLaunch<T, 10, 16>::ops();
    case 162: return FftLaunch<T, 9, 18>::ops();
    case 180: return FftLaunch<T, 12, 15>::ops();
    case 192: return FftLaunch<T, 12, 16>::ops();
    case 200: return FftLaunch<T, 10, 20>::ops();
    case 216: return FftLaunch<T, 12, 18>::ops();
    case 240: return FftLaunch<T, 15, 16>::ops();
    case 256: return FftLaunch<T, 16, 16>::ops();
    case 270: return FftLaunch<T, 15, 18>::ops();
    default: return nullptr;
  }
}
template const FftOps<float> *fft_large_ops<float>(int);
template const FftOps<double> *fft_large_ops<double>(int);

}  // namespace fsd
