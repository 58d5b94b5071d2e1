// frt_march_gen.cu -- the march variants of engines that may run Generalized
// Opacity members (Sec. 4.2): the moving screen and the ionised fraction's
// path, and merged rays (Sec. 3.3) when the engine also merges.  A separate
// translation unit so that the library's units compile in parallel.
#include "frt_march.cuh"

namespace frt {

MarchFn march_fn_gen(int nb, int agg, int minb) {
#define FRT_V(NB)                                                                   \
    if (nb == NB) {                                                                \
        if (agg == 0 && minb == 2) return k_march<NB, 0, 2, 3>;                    \
        if (agg == 0 && minb == 3) return k_march<NB, 0, 3, 3>;                    \
        if (agg == 0 && minb == 4) return k_march<NB, 0, 4, 3>;                    \
        if (agg == 1 && minb == 2) return k_march<NB, 1, 2, 3>;                    \
        if (agg == 1 && minb == 3) return k_march<NB, 1, 3, 3>;                    \
        if (agg == 1 && minb == 4) return k_march<NB, 1, 4, 3>;                    \
        if (agg == 2 && minb == 2) return k_march<NB, 2, 2, 3>;                    \
        if (agg == 2 && minb == 3) return k_march<NB, 2, 3, 3>;                    \
        if (agg == 2 && minb == 4) return k_march<NB, 2, 4, 3>;                    \
        return nullptr;                                                            \
    }
    FRT_V(1)
    FRT_V(3)
    FRT_V(4)
#undef FRT_V
#define FRT_W(NB)                                                                   \
    if (nb == NB && agg == 0) {                                                    \
        if (minb == 2) return k_march<NB, 0, 2, 3>;                                \
        if (minb == 3) return k_march<NB, 0, 3, 3>;                                \
    }
    FRT_W(2)
    FRT_W(5)
    FRT_W(6)
    FRT_W(7)
    FRT_W(8)
#undef FRT_W
    return nullptr;
}

}  // namespace frt
