// Instances of the run-time any-extent FFT kernels (fft_any.cuh).  This file is
// compiled once per part (build.py), because one instance holds the line
// transforms of up to 26 lengths.
#include "fft_any.cuh"

namespace lgf {
namespace anyfft {

#if LGF_ANY_PART == 0
template struct Xy<float, 32>;
template struct Zt<float, 32>;
#elif LGF_ANY_PART == 1
template struct Xy<float, 40>;
template struct Zt<float, 64>;
#endif

}  // namespace anyfft
}  // namespace lgf
