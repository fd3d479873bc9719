// FP64 kernels of the grid sizes 40.
#include "sized_impl.cuh"
namespace ltmp2 {
template struct Sized<double, 40>;
}
