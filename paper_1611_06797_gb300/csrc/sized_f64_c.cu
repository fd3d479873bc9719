// FP64 kernels of the grid sizes 27, 30.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<double, 27>;
template struct Sized<double, 30>;
}
