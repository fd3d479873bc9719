// FP64 kernels of the grid sizes 8, 10, 12, 16, 18.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<double, 8>;
template struct Sized<double, 10>;
template struct Sized<double, 12>;
template struct Sized<double, 16>;
template struct Sized<double, 18>;
}
