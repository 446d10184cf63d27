#include "small_form.cuh"

namespace upr {
template void small_form<true, false>(SmallRefine, cudaStream_t);
}
