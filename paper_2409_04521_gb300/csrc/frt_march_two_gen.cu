// frt_march_two_gen.cu -- the march variants of engines with one simulation
// that may run in Generalized Opacity mode (Sec. 4.2), with deposits of two
// words (Cells::dep).
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_two_gen(int nb, int agg, int minb) { return march_pick<3, 2>(nb, agg, minb); }

}  // namespace frt
