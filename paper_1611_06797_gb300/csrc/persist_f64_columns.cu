// FP64 persistent column kernel of the batching form.
#define LTMP2_PERSIST_COLUMNS
#include "persist_impl.cuh"
namespace ltmp2 {
template struct PersistColumns<double>;
}
