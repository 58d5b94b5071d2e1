// frt_march_two.cu -- the march variants of engines with one simulation whose
// deposits are two words (Cells::dep): plain, and with merged rays (Sec. 3.3).
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_two(int nb, int agg, int minb) { return march_pick<0, 2>(nb, agg, minb); }
MarchFn march_fn_two_merge(int nb, int agg, int minb) { return march_pick<1, 2>(nb, agg, minb); }

}  // namespace frt
