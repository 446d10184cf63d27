#include "small_form.cuh"

namespace upr {
template void small_form<false, false>(SmallRefine, cudaStream_t);
}
