// frt_launch.h -- kernel argument blocks and launchers (host side).
#pragma once
#include <string>
#include <tuple>
#include "frt_types.h"

namespace frt {

struct EmitArgs {
    Ctl *ctl;
    const SimDev *sims;
    SimAcc *acc;
    Queue q[2];
    long long cap;
    Emitters em;
    const int4 *pixtab;
    int ltab;
};

// The per-simulation constants the march needs, staged in shared
// memory; an engine with one simulation passes them with the launch.
struct MarchSim {
    int nx, ny, nz, step, l_src, l_max, active, l_merge, gen, ring0, pad1, pad2;   // ring0: this step's ring slot
    long long coff;
    float eps;
    float sig_max;          // largest sigma_b / sigma_ref of the bins
    int K[MAXL];
    float sig[MAXB], sige[MAXB], eh[MAXB];
};

struct MarchArgs {
    Ctl *ctl;
    const SimDev *sims;
    SimAcc *acc;
    int nsims;
    Queue q[2];
    long long cap;
    Emitters em;
    Cells cells;
    const int4 *pixtab;
    int ltab;
    int slab;                // output slots a warp reserves at once (run length, 32..4096)
    MarchSim one;            // the only simulation's constants (variants with ext bit 2; its step is the device's)
};

struct MergeArgs {
    Ctl *ctl;
    const SimDev *sims;
    SimAcc *acc;
    int nsims;
    Queue q[2];
    Emitters em;
    Ranges rg;
    const int4 *pixtab;
    int ltab;
    MergeWork w;
    long long cap;           // queue slots (merged rays are appended)
};

struct ChemArgs {
    Ctl *ctl;
    SimDev *sims;
    SimAcc *acc;
    int nsims;
    Cells cells;
    Ranges rg;
    int two;                 // deposits of two words (Cells::dep)
    int final_pass;          // 0: a trial pass of the Gamma - <n_HI> iteration (state unchanged)
    uint2 *status;           // host memory: the last ended step's queue slots in use, error word
};

// Where a step's kernels go: onto a stream, or into a graph as nodes that run
// one after another.  A graph is built from nodes, not by capturing a stream:
// a capture nobody asked for makes other host threads' calls fail (their use
// of the legacy stream, or a wait for the device), and theirs end it.
struct Sink {
    cudaStream_t st = nullptr;
    cudaGraph_t graph = nullptr;             // null: launched on st
    cudaGraphNode_t last[2] = {};            // the nodes the next one waits for
    int nlast = 0;
};
template <typename... P, typename... A>
cudaError_t enqueue(Sink &s, void (*k)(P...), int blocks, int threads, size_t shared, const A &...a) {
    std::tuple<P...> args(a...);
    return std::apply(
        [&](auto &...x) {
            void *ptr[] = {const_cast<void *>(static_cast<const void *>(&x))...};
            const void *f = reinterpret_cast<const void *>(k);
            if (!s.graph) return cudaLaunchKernel(f, dim3(blocks), dim3(threads), ptr, shared, s.st);
            cudaKernelNodeParams p{};
            p.func = const_cast<void *>(f);
            p.gridDim = dim3(blocks);
            p.blockDim = dim3(threads);
            p.sharedMemBytes = (unsigned)shared;
            p.kernelParams = ptr;
            cudaGraphNode_t n = nullptr;
            const cudaError_t e = cudaGraphAddKernelNode(&n, s.graph, s.last, s.nlast, &p);
            if (e == cudaSuccess) { s.last[0] = n; s.nlast = 1; }
            return e;
        },
        args);
}

// message of the last failed call that has no context (this host thread)
void set_free_error(const std::string &msg);

cudaError_t launch_pixtab(int4 *tab, int L, cudaStream_t st);
cudaError_t launch_init_cells(const SimDev *sims, int sim, Cells c, long long ncell, cudaStream_t st);
cudaError_t launch_reset(Ctl *c, SimDev *sims, SimAcc *acc, int nsims, cudaStream_t st);
cudaError_t launch_emit(const EmitArgs &a, int blocks, Sink &to);
// after a march: directions of children beyond the pixel table
cudaError_t launch_far(const EmitArgs &a, int blocks, Sink &to);
// a queue's first n records to (join: from) one array of n words per word of the record
cudaError_t launch_queue_words(const Queue &q, bool merged, long long n, uint32_t *words, bool join,
                               cudaStream_t st);
using MarchFn = void (*)(const MarchArgs);
// the march variants (nullptr if not built): with merged rays, with merged
// rays and Generalized Opacity mode, and all three for engines with one
// simulation
MarchFn march_fn_merge(int nb, int agg, int minb);
MarchFn march_fn_gen(int nb, int agg, int minb);
MarchFn march_fn_one(int nb, int agg, int minb);
MarchFn march_fn_one_merge(int nb, int agg, int minb);
MarchFn march_fn_one_gen(int nb, int agg, int minb);
MarchFn march_fn_two(int nb, int agg, int minb);
MarchFn march_fn_two_merge(int nb, int agg, int minb);
MarchFn march_fn_two_gen(int nb, int agg, int minb);
// ext: 0 plain, 1 merged rays, 3 merged rays and Generalized mode; plus 4:
// one simulation whose constants are launch arguments (its variants exist
// without aggregation; with it the general one runs); plus 8: its deposits are
// two words
bool march_variant_exists(int nb, int agg, int minb, int ext);
// opt the variant into all the dynamic shared memory a block may have
cudaError_t march_prepare(int nb, int agg, int minb, int ext);
cudaError_t launch_march(const MarchArgs &a, int nb, int agg, int minb, int blocks, int threads, Sink &to, int ext);
int march_max_blocks_per_sm(int nb, int agg, int minb, int threads, int nsims, int ext, uint32_t tile);
// blocks of the chemistry kernel that an SM holds at once
int chem_max_blocks_per_sm(int nsims);
cudaError_t launch_chem(const ChemArgs &a, int blocks, Sink &to);
// the merge step (Sec. 3.3) between the march and the chemistry
// a second stream for the merge's independent rotation pass, with the events
// that fork it from the step's stream and join it back
struct MergeSide {
    cudaStream_t st;
    cudaEvent_t fork, join;
};
cudaError_t launch_merge(const MergeArgs &a, int sm_count, Sink &to, const MergeSide *side);
cudaError_t launch_probe_merge_pixel(int level, long long n, const int32_t *d, const int32_t *Rq, bool per_ray,
                                     uint32_t *out, cudaStream_t st);
cudaError_t launch_probe_pixvec(int level, long long p0, long long n, int32_t *out, cudaStream_t st);
cudaError_t launch_probe_rates(long long n, const float *T, float *out, cudaStream_t st);
cudaError_t launch_probe_rotation(uint64_t seed, long long e, long long s, int rotate, int32_t *out, cudaStream_t st);
cudaError_t launch_probe_direction(int level, long long p0, long long n, const int32_t *Rq, const int4 *tab, int ltab,
                                   int32_t *out, cudaStream_t st);
cudaError_t launch_probe_traverse(long long n, const long long *p0, const int32_t *d, int gx, int gy, int gz,
                                  int32_t *cells, float *ds, int32_t *nseg, int32_t *esc, cudaStream_t st);

}  // namespace frt
