// FP32 kernels of the grid sizes 27, 30, 32, 36, 40.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<float, 27>;
template struct Sized<float, 30>;
template struct Sized<float, 32>;
template struct Sized<float, 36>;
template struct Sized<float, 40>;
}
