#include "small_form.cuh"

namespace upr {
template void small_form<false, true>(SmallRefine, cudaStream_t);
}
