// frt_march_one_gen.cu -- the march variants of engines with one simulation
// that may run in Generalized Opacity mode (Sec. 4.2).
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_one_gen(int nb, int agg, int minb) { return march_pick<3, 1>(nb, agg, minb); }

}  // namespace frt
