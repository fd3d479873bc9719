// FP64 kernels of the grid sizes 32, 36.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<double, 32>;
template struct Sized<double, 36>;
}
