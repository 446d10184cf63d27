// The rule and the dispatch of the one-launch refinement of small graphs
// (small_form.cuh).  Its four forms are translation units of their own, about
// 18 s of compiling each: together in one they took 74 of a build's 78 s.
#include "kernels.h"

namespace upr {

bool small_refine_ok(const GraphDev &g, int gbits, int cbits) {
    int kbits = 1;
    while ((1ll << kbits) < g.k) kbits++;
    return g.ng == 1 && !g.sp.on() && g.n > 0 && g.n <= kSmallNodes && gbits + kbits <= 32 &&
           1 + gbits + 2 * cbits <= 63;
}

void small_refine(const SmallRefine &a, cudaStream_t s) {
    const bool unit = !a.g.vwgt, rank = a.g.k <= kRebRankK;
    if (unit && rank) small_form<true, true>(a, s);
    else if (unit) small_form<true, false>(a, s);
    else if (rank) small_form<false, true>(a, s);
    else small_form<false, false>(a, s);
}

}  // namespace upr
