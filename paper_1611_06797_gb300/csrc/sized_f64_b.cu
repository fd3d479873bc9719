// FP64 kernels of the grid sizes 20, 24, 25.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<double, 20>;
template struct Sized<double, 24>;
template struct Sized<double, 25>;
}
