#include "small_form.cuh"

namespace upr {
template void small_form<true, true>(SmallRefine, cudaStream_t);
}
