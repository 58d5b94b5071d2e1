// frt_march_one.cu -- the march variants of engines with one simulation:
// plain, and with merged rays (Sec. 3.3).
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_one(int nb, int agg, int minb) { return march_pick<0, 1>(nb, agg, minb); }
MarchFn march_fn_one_merge(int nb, int agg, int minb) { return march_pick<1, 1>(nb, agg, minb); }

}  // namespace frt
