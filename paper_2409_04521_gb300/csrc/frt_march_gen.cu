// frt_march_gen.cu -- the march variants of engines that may run Generalized
// Opacity members (Sec. 4.2): the moving screen and the ionised fraction's
// path, and merged rays (Sec. 3.3) when the engine also merges.  A separate
// translation unit so that the library's units compile in parallel.
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_gen(int nb, int agg, int minb) { return march_pick<3, 0>(nb, agg, minb); }

}  // namespace frt
