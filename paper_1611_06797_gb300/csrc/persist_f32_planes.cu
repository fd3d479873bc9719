// FP32 persistent plane kernel of the batching form.
#define LTMP2_PERSIST_PLANES
#include "persist_impl.cuh"
namespace ltmp2 {
template struct PersistPlanes<float>;
}
