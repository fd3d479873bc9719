// FP32 kernels of the grid sizes 8, 10, 12, 16, 18, 20, 24, 25.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<float, 8>;
template struct Sized<float, 10>;
template struct Sized<float, 12>;
template struct Sized<float, 16>;
template struct Sized<float, 18>;
template struct Sized<float, 20>;
template struct Sized<float, 24>;
template struct Sized<float, 25>;
}
