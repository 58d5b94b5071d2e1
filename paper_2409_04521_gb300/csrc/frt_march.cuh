// frt_march.cuh -- the fused per-ray kernel of one RT step, shared by the
// translation units that build its variants.
//
//   k_march : per ray, the one-cell march with exp(-tau) attenuation
//             (Sec. 3.1; Sec. 4.2, Eq. 13), the Eq. 17 deposit (vector
//             reductions into the per-cell buffers), escape,
//             termination, the Eq. 2-3 split and the compacted write of
//             survivors and children.
#pragma once
#include "frt_device.cuh"
#include "frt_launch.h"

namespace frt {

constexpr int NACC = 6;  // (unused), escaped, out, segments, rays in, rays out

// Warp-wide flush of lane-private tallies (lane simulation `tsim`, -1 for
// none) into the block's per-simulation fixed-point totals; clears them.
__device__ __forceinline__ void flush_tallies(float &esc, float &out, unsigned &cnt, unsigned &rout, int &tsim,
                                              unsigned long long *sh_acc) {
    const int lane = lane_id();
    const int kref = __reduce_max_sync(FULL, tsim);
    if (kref < 0) return;                                   // warp-uniform
    float v[NACC] = {0.0f, esc, out, (float)(cnt & 0xffffu), (float)(cnt >> 16), (float)rout};
    bool lead;
    int kk = tsim;
    if (__all_sync(FULL, tsim < 0 || tsim == kref)) {
        warp_sum<NACC>(v);                                  // empty lanes carry zeros
        lead = lane == 0;
        kk = kref;
    } else {
        const unsigned peers = __match_any_sync(FULL, tsim);
        peer_sum<NACC>(peers, v);
        lead = tsim >= 0 && (peers & ((1u << lane) - 1u)) == 0u;
    }
    if (lead) {
        unsigned long long *dst = sh_acc + kk * NACC;
        atomicAdd(dst + 0, fixed32(v[0]));
        atomicAdd(dst + 1, fixed32(v[1]));
        atomicAdd(dst + 2, fixed32(v[2]));
        atomicAdd(dst + 3, (unsigned long long)__float2uint_rn(v[3]));
        atomicAdd(dst + 4, (unsigned long long)__float2uint_rn(v[4]));
        atomicAdd(dst + 5, (unsigned long long)__float2uint_rn(v[5]));
    }
    esc = out = 0.0f;
    cnt = rout = 0u;
    tsim = -1;
}

// The same for the only simulation (rays out are the warp's output count).
__device__ __forceinline__ void flush_one(float &esc, float &out, unsigned &cnt, unsigned long long *sh_acc) {
    float v[2] = {esc, out};
    warp_sum<2>(v);
    const unsigned seg = __reduce_add_sync(FULL, cnt & 0xffffu), rays = __reduce_add_sync(FULL, cnt >> 16);
    if (lane_id() == 0) {
        atomicAdd(sh_acc + 1, fixed32(v[0]));
        atomicAdd(sh_acc + 2, fixed32(v[1]));
        atomicAdd(sh_acc + 3, (unsigned long long)seg);
        atomicAdd(sh_acc + 4, (unsigned long long)rays);
    }
    esc = out = 0.0f;
    cnt = 0u;
}

// shared memory of a march block: tallies and constants per simulation, then
// two tiles of ray records and the splitting lanes' rotation rows per warp
__host__ __device__ constexpr size_t march_tiles_offset(int nsims) {
    return ((size_t)nsims * (NACC * sizeof(unsigned long long) + sizeof(MarchSim)) + 127) & ~(size_t)127;
}
constexpr int ROW_BYTES = 3 * 32 * 16;
__host__ __device__ constexpr size_t march_shared_bytes(int nsims, uint32_t tile, int threads) {
    return march_tiles_offset(nsims) + (size_t)(threads / 32) * (2 * tile + ROW_BYTES);
}

// (1 - e^-t)/t for 0 <= t < 1/8, from -t: its Taylor series through t^4 (the
// next term, t^5/720, is under the single-precision epsilon there)
__device__ __forceinline__ float2 series_q2(float2 nt) {
    float2 q = __ffma2_rn(make_float2(1.0f / 120.0f, 1.0f / 120.0f), nt, make_float2(1.0f / 24.0f, 1.0f / 24.0f));
    q = __ffma2_rn(q, nt, make_float2(1.0f / 6.0f, 1.0f / 6.0f));
    q = __ffma2_rn(q, nt, make_float2(0.5f, 0.5f));
    return __ffma2_rn(q, nt, make_float2(1.0f, 1.0f));
}
__device__ __forceinline__ float series_q(float nt) {
    float q = fmaf(1.0f / 120.0f, nt, 1.0f / 24.0f);
    q = fmaf(q, nt, 1.0f / 6.0f);
    q = fmaf(q, nt, 0.5f);
    return fmaf(q, nt, 1.0f);
}

// Attenuation of the photons ph[b] entering a segment of length dse (cells)
// through a cell of optical depth per cell k = (HI at sigma_ref, sub-grid),
// with its deposits (Eq. 13, Eq. 17): v[0] = absorbed photons, v[1] =
// sum_b sigma_b N_b (1 - e^-tau_b)/kappa_b, v[2] the same weighted by the
// excess energy.  A bin with tau < 1/8 takes (1 - e^-tau)/kappa = dse q(tau)
// with the series q (no exponential, no division); with phi = N dse q it
// absorbs kappa phi and keeps N - kappa phi (one rounding).  A thicker bin
// takes the hardware exponential and the division by kappa.  SMALL: every bin
// of every lane of the warp is thin, and only the series is evaluated; the
// per-bin results are the same either way, so a ray's photons do not depend
// on the rays it shares a warp with.  HEAT: v[2] is wanted.  Bins go in pairs on the paired
// single-precision units, and the opacity enters negated, so that every
// product of the thin path is an operand of a fused multiply-add: twelve
// paired operations a pair of bins (eighteen with the opacity positive).
template <int NB, bool SMALL, bool HEAT>
__device__ __forceinline__ void seg_attenuate(float2 k, float dse, const float *sig, const float *sige, float (&ph)[NB],
                                              float (&v)[4]) {
    constexpr float NLOG2E = 1.44269504f;            // e^-tau = 2^(-tau log2 e)
    float2 w0 = make_float2(0.f, 0.f), w1 = w0, w2 = w0;
    const float2 kx2 = make_float2(-k.x, -k.x), ky2 = make_float2(-k.y, -k.y), ds2 = make_float2(dse, dse);
#pragma unroll
    for (int b = 0; b + 1 < NB; b += 2) {
        const float2 sg = make_float2(sig[b], sig[b + 1]);
        const float2 se = make_float2(sige[b], sige[b + 1]);
        const float2 nk = __ffma2_rn(kx2, sg, ky2);
        const float2 nt = __fmul2_rn(nk, ds2);
        const float2 p2 = make_float2(ph[b], ph[b + 1]);
        const float2 pd = __fmul2_rn(p2, ds2);
        float2 phin, pn;
        if (SMALL) {
            phin = __fmul2_rn(pd, series_q2(nt));
            pn = __ffma2_rn(nk, phin, p2);
            w0 = __ffma2_rn(nk, phin, w0);
        } else {
            const bool s0 = nt.x > -0.125f, s1 = nt.y > -0.125f;
            const float2 q = series_q2(make_float2(fmaxf(nt.x, -0.125f), fmaxf(nt.y, -0.125f)));
            const float2 ps = __fmul2_rn(pd, q);
            const float2 ns = __ffma2_rn(nk, ps, p2);
            const float2 l2 = __fmul2_rn(nt, make_float2(NLOG2E, NLOG2E));
            const float2 ex = make_float2(exp2_approx(l2.x), exp2_approx(l2.y));
            const float2 nx = __fmul2_rn(p2, ex);                             // what is left
            const float2 ab = __fmul2_rn(p2, __ffma2_rn(ex, make_float2(-1.0f, -1.0f), make_float2(1.0f, 1.0f)));
            const float2 na = __fmul2_rn(nk, ps);
            // (a bin in the division's lane has tau >= 1/8, so its kappa is not zero)
            phin = make_float2(s0 ? ps.x : ab.x * rcp_approx(-nk.x), s1 ? ps.y : ab.y * rcp_approx(-nk.y));
            pn = make_float2(s0 ? ns.x : nx.x, s1 ? ns.y : nx.y);
            w0 = __fadd2_rn(w0, make_float2(s0 ? na.x : -ab.x, s1 ? na.y : -ab.y));
        }
        ph[b] = pn.x;
        ph[b + 1] = pn.y;
        w1 = __ffma2_rn(sg, phin, w1);
        if (HEAT) w2 = __ffma2_rn(se, phin, w2);
    }
    v[0] = -(w0.x + w0.y);
    v[1] = w1.x + w1.y;
    v[2] = w2.x + w2.y;
    if (NB & 1) {
        const int b = NB - 1;
        const float nk = fmaf(-k.x, sig[b], -k.y);
        const float nt = nk * dse;
        float phin, a;
        if (SMALL || nt > -0.125f) {
            phin = ph[b] * dse * series_q(nt);
            a = -nk * phin;
            ph[b] = fmaf(nk, phin, ph[b]);
        } else {
            const float ex = exp2_approx(nt * NLOG2E);
            a = ph[b] * (1.0f - ex);
            phin = a * rcp_approx(-nk);
            ph[b] *= ex;
        }
        v[0] += a;
        v[1] = fmaf(sig[b], phin, v[1]);
        if (HEAT) v[2] = fmaf(sige[b], phin, v[2]);
    }
}

// What bounds it (1.45e7 rays, 4 bins, 64^3 cells, ncu): not HBM (1.2 GB in
// 398 us, 44% of the copy rate) but issue (69% busy, 706 warp instructions a
// 32 rays) and the load-store unit (60%), which the scattered reductions fill:
// 3.4e7 sectors, half its request port's cycles.  It was 647 us and 1030
// instructions with an array a word, a position update and three 64-bit
// comparisons a crossing, children made lane by lane and constants from
// shared memory.  24 warps an SM with nothing spilled beat 28 and 32.
// Phases per ray: (1) the integer walk of the whole step, (2) the opacity
// loads of every crossed cell at once, (3) attenuation and deposits.
// AGG selects how the lanes of a warp combine deposits into the same cell
// before the vector reduction: 0 none, 1 peer groups of equal keys
// (match_any + pairwise tree), 2 runs of equal consecutive keys.
// MINB is the resident-block target per SM (register budget).  EXT bit 1
// adds the rays made by the merge step (Sec. 3.3), which start from their
// merge position and carry their own distance and termination threshold;
// bit 2 adds Generalized Opacity mode (Sec. 4.2): a ray crosses the ionised
// fraction x_ion of each cell's path with the sub-grid opacity, then meets
// the moving screen, which absorbs the share rho of what reaches it
// (Eq. 18-19).  A merging engine without Generalized members runs EXT = 1
// (fewer registers: 10% less march time on the merging workloads than with
// both), an engine that may run Generalized members EXT = 3.
// ONE: an engine with one simulation (not a batch of one slot): its
// constants come with the launch (A.one: the instructions take them from
// constant memory, where a load of each from shared memory a ray and segment
// was a fifth of the load-store unit's work, the march's busiest) and its
// tallies need no simulation index.
// ONE = 2: besides, nothing reads a cell's heating and segment count
// (isothermal or Generalized, no diagnostics): its deposit is two words, half
// the buffer (128 MB at 200^3 cells, with the opacities more than the L2) and
// half the reduction's payload: 15.5 -> 14.0 ms of march in 60 steps there.
template <int NB, int AGG, int MINB, int EXT, int ONE>
__global__ void __launch_bounds__(256, MINB) k_march(const __grid_constant__ MarchArgs A) {
    constexpr bool MRG = (EXT & 1) != 0, GEN = (EXT & 2) != 0;
    // per-simulation tallies of this block (photons in 2^-32 fixed point,
    // counts as integers), then the staged constants
    extern __shared__ __align__(128) unsigned long long sh_acc[];
    __shared__ __align__(8) unsigned long long sh_bar[8][2];
    __shared__ unsigned char sh_parent[8][32];     // splitting lanes of each warp, in order
    unsigned char *const parent = sh_parent[threadIdx.x >> 5];
    MarchSim *msim = reinterpret_cast<MarchSim *>(sh_acc + A.nsims * NACC);
    const int lane = lane_id();
    for (int i = threadIdx.x; i < A.nsims * NACC; i += blockDim.x) sh_acc[i] = 0ull;
    if (ONE) {
        if (threadIdx.x < MAXL) msim[0].K[threadIdx.x] = A.one.K[threadIdx.x];
        if (threadIdx.x == 0) {
            const int s = A.sims[0].step;
            msim[0].step = s;
            msim[0].ring0 = s % A.em.ring_w;
        }
    } else {
        // a warp a simulation
        for (int i = threadIdx.x >> 5; i < A.nsims; i += blockDim.x >> 5) {
            const SimDev &S = A.sims[i];
            MarchSim &m = msim[i];
            if (lane < MAXL) m.K[lane] = S.K[lane];
            float sg = 0.0f;
            if (lane < MAXB) {
                sg = S.sig[lane];
                m.sig[lane] = sg; m.sige[lane] = S.sige[lane]; m.eh[lane] = S.eh[lane];
                if (lane >= S.nb) sg = 0.0f;
            }
            // (cross-sections are not negative: their bits order as integers)
            const unsigned mx = __reduce_max_sync(FULL, __float_as_uint(sg));
            if (lane == 0) {
                m.nx = S.nx; m.ny = S.ny; m.nz = S.nz; m.step = S.step; m.l_src = S.l_src; m.l_max = S.l_max;
                m.active = S.active; m.l_merge = S.l_merge; m.coff = S.cell_off; m.eps = S.eps_term;
                m.gen = S.gen_mode; m.ring0 = S.step % A.em.ring_w; m.pad1 = m.pad2 = 0;
                m.sig_max = __uint_as_float(mx);
            }
        }
    }
    const unsigned tile = A.q[0].tile;
    // this warp's two tiles and their barriers (one arrival each: lane 0's)
    char *const tiles = reinterpret_cast<char *>(sh_acc) + march_tiles_offset(A.nsims) +
                        (threadIdx.x >> 5) * (2 * tile + ROW_BYTES);
    int4 *const rowbuf = reinterpret_cast<int4 *>(tiles + 2 * tile);
    const unsigned tiles_s = smem_addr(tiles), bars_s = smem_addr(sh_bar[threadIdx.x >> 5]);
    if (lane == 0) {
        mbar_init(bars_s, 1);
        mbar_init(bars_s + 8, 1);
        fence_proxy_async();
    }
    __syncthreads();
    Ctl *C = A.ctl;
    if (C->err == 0) {
        const int par = C->par;
        const int step0 = ONE ? msim[0].step : 0;
        const char *const qin = A.q[par].base;
        char *const qout = A.q[par ^ 1].base;
        // queue slots stay below 2^31 (the engine's bound), so 32-bit indices
        const unsigned n = (unsigned)(C->cnt[par] + C->emit_total);
        const unsigned ntile = (n + 31u) >> 5;
        // the tile of this warp's iteration k: the warps take the tiles in turn.
        // (Runs of 8 or 32 tiles a warp keep the shells of a source and step
        // together, 2.7 of them in a tile instead of 8.2, and are 2 to 6%
        // slower: more lanes of a reduction then hit one cell.)
        const unsigned warps = gridDim.x * (blockDim.x >> 5), warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        // a cell's deposit: one vector reduction
        auto deposit = [&](int cell, float a, float g, float h, float seg) {
            if (ONE == 2) red_add_v2(reinterpret_cast<float2 *>(A.cells.dep) + cell, a, g);
            else red_add_v4(A.cells.dep + cell, a, g, h, seg);
        };
        auto tile_at = [&](unsigned k) { return k * warps + warp; };
        // warp-private run of output slots [slab, slab + slab_left), and this
        // warp's outputs and iterations so far (its output rate)
        unsigned slab = 0;
        int slab_left = 0;
        int w_out = 0, w_it = 0;
        // lane-private tallies of one simulation, flushed by the warp:
        // escaped and surviving photons, segments | rays in << 16, rays out
        float t_esc = 0.0f, t_out = 0.0f;
        unsigned t_cnt = 0u, t_rout = 0u;
        int t_sim = -1;
        auto fetch = [&](unsigned k) {                  // iteration k's tile into buffer k & 1
            const unsigned j = tile_at(k);
            if (j < ntile) bulk_load(tiles_s + (k & 1u) * tile, qin + (size_t)j * tile, tile, bars_s + 8 * (k & 1u));
        };
        if (lane == 0) {
            fetch(0);
            fetch(1);
        }
        for (unsigned tl; (tl = tile_at(w_it)) < ntile;) {
            // the tile's records, fetched two iterations ago (the copy hides
            // behind a whole iteration).  Words are read from shared memory
            // when they are needed, the unchanged ones again at the end: held
            // in registers they would spill (a dead slot's words are not used)
            const unsigned buf = w_it & 1;
            char *const rec = tiles + buf * tile;
            if (!__all_sync(FULL, mbar_wait(bars_s + 8 * buf, (w_it >> 1) & 1))) {
                // never in a working machine: report, let the other tile's copy end, stop
                if (lane == 0) {
                    atomicOr(&C->err, 16);
                    if (tile_at(w_it + 1) < ntile) mbar_wait(bars_s + 8 * (buf ^ 1), ((w_it + 1) >> 1) & 1);
                }
                break;
            }
            const uint4 *const heads = reinterpret_cast<const uint4 *>(rec);
            const uint2 *const tails = reinterpret_cast<const uint2 *>(rec + 512);
            constexpr int TW = NB >= 2 ? 2 : 1;                   // a record's dz and pixel word, in uint2 strides
            const uint4 *const merged = reinterpret_cast<const uint4 *>(rec + 128 * (6 + NB));
            const float *const mthrs = reinterpret_cast<const float *>(rec + 128 * (6 + NB) + 512);
            bool valid = false, mrg = false;
            int sim = 0;
            // (1) integer walk of this step
            int key[4];
            float ds[4];
            bool esc = false;
            {
            const uint4 ra = heads[lane];
            const uint2 rt = tails[lane * TW];
            const uint32_t e = ra.x;
            const int bi = (int)ra.y, dx = (int)ra.z, dy = (int)ra.w, dz = (int)rt.x;
            valid = 32u * tl + lane < n && rt.y != DEAD_RAY;
            mrg = MRG && valid && (e & MERGED_BIT);
            uint4 rm = make_uint4(0u, 0u, 0u, 0u);
            if (mrg) rm = merged[lane];
            int4 ec = make_int4(0, 0, 0, 0);
            if (mrg) {
                if (!ONE) sim = (int)((rm.w >> 16) & 0x7fffu);
            } else if (valid) {
                ec = __ldg(&A.em.cell[e]);
                if (!ONE) sim = ec.w;
            }
            const MarchSim &S = ONE ? A.one : msim[sim];
            const int step = ONE ? step0 : S.step;
            if (!S.active) valid = false;
            // age: cells travelled before this step.  A merged ray has moved
            // `since` steps from its merge position and had travelled its
            // constituents' mean distance when it was made.
            const int since = step - bi - 1;
            const int age = mrg ? (int)(rm.w & 0xffffu) + since : step - bi;
            if (valid && (mrg ? since < 0 : (age < 0 || age >= A.em.ring_w))) {
                atomicOr(&C->err, 2);
                valid = false;
            }
            // a queued ray is inside the box at the start of its step, so
            // its position (at most 1000 cells of 2^21) fits 32 bits
            int px, py, pz;
            if (mrg) {
                px = (int)rm.x + since * dx;
                py = (int)rm.y + since * dy;
                pz = (int)rm.z + since * dz;
            } else {
                px = ((2 * ec.x + 1) << (FRAC_BITS - 1)) + age * dx;
                py = ((2 * ec.y + 1) << (FRAC_BITS - 1)) + age * dy;
                pz = ((2 * ec.z + 1) << (FRAC_BITS - 1)) + age * dz;
            }
            // slots may be empty: every later phase visits the four slots
            // in order and skips the empty ones (negative keys)
            walk_step(valid, px, py, pz, dx, dy, dz, S.nx, S.ny, S.nz, (int)S.coff, key, ds, esc);
            }
            const MarchSim &S = ONE ? A.one : msim[sim];
            const int step = ONE ? step0 : S.step;
            int nseg = 4 + (key[0] >> 31) + (key[1] >> 31) + (key[2] >> 31) + (key[3] >> 31);
            // (2) opacities of the crossed cells (Generalized mode: also the
            // ionised fraction and the screen's share)
            float2 kc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) kc[j] = key[j] >= 0 ? __ldg(&A.cells.kap[key[j]]) : make_float2(0.f, 0.f);
            float ph[NB];
            {
                uint32_t w[2 + NB];
                load_tail<NB>(rec, lane, w);
#pragma unroll
                for (int b = 0; b < NB; ++b) ph[b] = __uint_as_float(w[2 + b]);
            }
            const bool gen = GEN && valid && S.gen;
            float xg[4], rg[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                xg[j] = 1.0f;
                rg[j] = 1.0f;
                if (GEN && gen && key[j] >= 0) { xg[j] = (float)__ldg(&A.cells.xion[key[j]]); rg[j] = __ldg(&A.cells.rho[key[j]]); }
            }
            bool screened = false;
            // (3) attenuation and deposits (Eq. 13, Eq. 17)
            int last = -1;
            float2 lastk = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float v[4] = {0.f, 0.f, 0.f, 1.0f};
                if (GEN && screened) key[j] = -1;
                const float dse = GEN ? xg[j] * ds[j] : ds[j];
                // every segment of this slot in the warp optically thin (all
                // bins' tau below 1/8): the series path, warp-uniform
                const bool thin = __all_sync(FULL, key[j] < 0 || fmaf(kc[j].x, S.sig_max, kc[j].y) * dse < 0.125f);
                if (key[j] >= 0) {
                    if (thin) seg_attenuate<NB, true, ONE != 2>(kc[j], dse, S.sig, S.sige, ph, v);
                    else seg_attenuate<NB, false, ONE != 2>(kc[j], dse, S.sig, S.sige, ph, v);
                    last = key[j];
                    lastk = kc[j];
                    if (GEN && xg[j] < 1.0f) {
                        // the screen: it absorbs the share rho of what reaches it
                        float nf = 0.0f;
#pragma unroll
                        for (int b = 0; b < NB; ++b) nf += ph[b];
                        red_add_v2(A.cells.fscr + key[j], rg[j] * nf, nf);
                        const float keep = rg[j] >= 1.0f ? 0.0f : 1.0f - rg[j];
#pragma unroll
                        for (int b = 0; b < NB; ++b) ph[b] *= keep;
                        if (rg[j] >= 1.0f) {
                            screened = true;
                            nseg = j + 1;
#pragma unroll
                            for (int i2 = 0; i2 < 4; ++i2)
                                if (i2 < j) nseg += key[i2] >> 31;
                        }
                    }
                }
                if (AGG == 0) {
                    if (key[j] >= 0) deposit(key[j], v[0], v[1], v[2], v[3]);
                } else {
                    if (__ballot_sync(FULL, key[j] >= 0) == 0u) continue;
                    if (AGG == 1) {
                        const unsigned peers = __match_any_sync(FULL, key[j]);
                        if (__any_sync(FULL, key[j] >= 0 && __popc(peers) > 1)) peer_sum<4>(peers, v);
                        if (key[j] >= 0 && (peers & ((1u << lane) - 1u)) == 0u)
                            red_add_v4(A.cells.dep + key[j], v[0], v[1], v[2], v[3]);
                    } else {
                        const bool head = run_sum<4>(key[j], v);
                        if (key[j] >= 0 && head) red_add_v4(A.cells.dep + key[j], v[0], v[1], v[2], v[3]);
                    }
                }
            }
            float s_end = 0.0f;
#pragma unroll
            for (int b = 0; b < NB; ++b) s_end += ph[b];
            int nout = 0, m = 0;
            if (GEN && screened) esc = false;
            if (valid && !esc && !(GEN && screened)) {
                const int lev = (int)(tails[lane * TW].y >> LEVEL_SHIFT);
                const float thr = mrg ? mthrs[lane] : S.eps * __ldg(&A.em.n0[heads[lane].x]) * pow2_neg(2 * (lev - S.l_src));
                if (s_end < thr) {
                    // termination: the ray's last photons stay in its last cell
                    float g = 0.f, h = 0.f;
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        const float kb = fmaf(lastk.x, S.sig[b], lastk.y);
                        if (kb > 0.0f) {
                            const float q = __fdividef(ph[b], kb);
                            g = fmaf(S.sig[b], q, g);
                            h = fmaf(S.sige[b], q, h);
                        }
                    }
                    deposit(last, s_end, g, h, 0.0f);
                } else {
                    const int age = mrg ? (int)(merged[lane].w & 0xffffu) + step - (int)heads[lane].y - 1
                                        : step - (int)heads[lane].y;
                    const int *const K = msim[sim].K;
                    while (lev + m < S.l_max && age + 1 >= K[lev + m]) ++m;
                    nout = 1 << (2 * m);
                }
            }
            // per-simulation tallies: each lane accumulates the rays of one
            // simulation for up to sixteen iterations, then the warp reduces them
            // into the block's fixed-point totals
            {
                const bool clash = !ONE && valid && t_sim >= 0 && t_sim != sim;
                if ((w_it & 15) == 15 || (!ONE && __any_sync(FULL, clash))) {
                    if (ONE) flush_one(t_esc, t_out, t_cnt, sh_acc);
                    else flush_tallies(t_esc, t_out, t_cnt, t_rout, t_sim, sh_acc);
                }
                if (valid) {
                    if (esc) t_esc += s_end;
                    if (nout) t_out += s_end;
                    t_cnt += (unsigned)nseg + (1u << 16);
                    if (!ONE) {
                        t_rout += (unsigned)nout;
                        t_sim = sim;
                    }
                }
            }
            // compacted output into the warp's run of slots: the remainder of
            // the current run first, then a new run reserved with one atomic
            // (without a split in the warp a ballot gives the positions; the
            // shuffle scan only where a lane has children)
            const unsigned outm = __ballot_sync(FULL, nout != 0);
            int k0 = __popc(outm & ((1u << lane) - 1u)), tot = __popc(outm);   // this lane's first output position
            if (__any_sync(FULL, nout > 1)) {
                const int incl = warp_incl_scan(nout);
                tot = __shfl_sync(FULL, incl, 31);
                k0 = incl - nout;
            }
            if (tot > 0) {
                const unsigned s0 = slab;
                const int left = slab_left;
                unsigned s1 = 0;
                bool fits = true;
                if (tot > left) {
                    // reserve for this warp's next iterations at its own output
                    // rate (at most 16 iterations ahead and OUT_SLAB slots), so the
                    // unused tail stays small whatever the queue's dead fraction
                    const int need = tot - left;
                    const unsigned iters_left = (ntile - tl + warps - 1u) / warps;
                    const int ahead = iters_left < 16u ? (int)iters_left : 16;
                    const int rate = (w_out + tot + w_it) / (w_it + 1);
                    const int guess = rate * ahead < A.slab ? rate * ahead : A.slab;
                    const int want = need > guess ? need : guess;
                    unsigned long long nb64 = 0;
                    if (lane == 0) nb64 = atomicAdd((unsigned long long *)&C->cnt[par ^ 1], (unsigned long long)want);
                    nb64 = __shfl_sync(FULL, nb64, 0);
                    const unsigned nbase = (unsigned)nb64;
                    if ((long long)(nb64 + want) > A.cap) {
                        if (lane == 0) atomicOr(&C->err, 1);
                        fits = false;
                        slab_left = 0;
                    } else {
                        s1 = nbase;
                        slab = nbase + need;
                        slab_left = want - need;
                    }
                } else {
                    slab = s0 + tot;
                    slab_left = left - tot;
                }
                w_out += tot;
                auto slot_of = [&](int k) -> unsigned {
                    return k < left ? s0 + (unsigned)k : s1 + (unsigned)(k - left);
                };
                if (fits && nout == 1) {
                    const unsigned o = slot_of(k0);
                    char *const t = qout + (size_t)(o >> 5) * tile;
                    __stcs(reinterpret_cast<uint4 *>(t) + (o & 31u), heads[lane]);
                    const uint2 rt = tails[lane * TW];
                    uint32_t w[2 + NB];
                    w[0] = rt.x; w[1] = rt.y;
#pragma unroll
                    for (int b = 0; b < NB; ++b) w[2 + b] = __float_as_uint(ph[b]);
                    store_tail<NB, true>(t, o & 31u, w);
                    if (mrg) {
                        char *const tm = t + 128 * (6 + NB);
                        __stcs(reinterpret_cast<uint4 *>(tm) + (o & 31u), merged[lane]);
                        __stcs(reinterpret_cast<float *>(tm + 512) + (o & 31u), mthrs[lane]);
                    }
                }
                // children: the warp makes the children of all its splitting
                // lanes together, one child a lane, whose neighbours go to
                // neighbouring slots; the splits of one depth m at a time
                // (one depth in nearly every warp).  Each splitting lane
                // writing its own four children was a fifth to a third of the
                // march: half of the warps hold a few such lanes, and every
                // lane of the warp waited through four of them.
                unsigned split = __ballot_sync(FULL, fits && nout > 1);
                while (split) {
                    const int mm = __shfl_sync(FULL, m, __ffs(split) - 1);
                    const unsigned grp = __ballot_sync(FULL, ((split >> lane) & 1u) && m == mm);
                    split &= ~grp;
                    __syncwarp();
                    // children keep their parent's sphere (Sec. 3.2): the
                    // emitter's of the birth step (whose slot of the ring the
                    // age gives: it is less than the ring's length), or the
                    // merge cell's.  Each parent's lane gets the rows and
                    // hands them over in shared memory, with its photons in
                    // its record of the tile (nobody reads it afterwards)
                    if ((grp >> lane) & 1u) {
                        parent[__popc(grp & ((1u << lane) - 1u))] = (unsigned char)lane;
                        const uint4 ra = heads[lane];
                        int4 row[3];
                        if (mrg) {
                            const SimDev &SD = A.sims[sim];
                            rotation_rows(SD.seed, (1LL << 31) + (long long)(ra.x & ~MERGED_BIT), (int)ra.y, SD.rotate, row);
                        } else {
                            int slot = msim[sim].ring0 - (step - (int)ra.y);
                            if (slot < 0) slot += A.em.ring_w;
                            const int4 *rg = A.em.ring + ((long long)ra.x * A.em.ring_w + slot) * 3;
                            row[0] = rg[0]; row[1] = rg[1]; row[2] = rg[2];
                        }
                        row[0].w = k0;
                        row[1].w = sim;
                        rowbuf[lane] = row[0];
                        rowbuf[32 + lane] = row[1];
                        rowbuf[64 + lane] = row[2];
                        const float scale = pow2_neg(2 * mm);
                        const uint2 rt = tails[lane * TW];
                        uint32_t w[2 + NB];
                        w[0] = rt.x; w[1] = rt.y;
#pragma unroll
                        for (int b = 0; b < NB; ++b) w[2 + b] = __float_as_uint(ph[b] * scale);
                        store_tail<NB, false>(rec, lane, w);
                        // these stores come before the copy that refills the
                        // tile, which goes through another proxy
                        fence_proxy_async();
                    }
                    __syncwarp();
                    const unsigned all = (unsigned)__popc(grp) << (2 * mm);
                    for (unsigned c = lane; c < all; c += 32) {
                        const int src = parent[c >> (2 * mm)];
                        const unsigned sub = c & ((1u << (2 * mm)) - 1u);
                        const uint4 pa = heads[src];
                        uint32_t cw[2 + NB];
                        load_tail<NB>(rec, src, cw);
                        const int4 rows[3] = {rowbuf[src], rowbuf[32 + src], rowbuf[64 + src]};
                        const uint32_t ppl = cw[1];
                        const int psim = rows[1].w;
                        {
                            const int plev = (int)(ppl >> LEVEL_SHIFT), L = plev + mm;
                            const bool pmrg = MRG && (pa.x & MERGED_BIT);
                            uint4 pm = make_uint4(0u, 0u, 0u, 0u);
                            if (pmrg) pm = merged[src];
                            const uint32_t pix = pmrg && (pm.w >> 31)
                                                     ? vertex_child(ONE ? A.one.l_merge : msim[psim].l_merge, ppl & PIX_MASK, plev, mm, sub)
                                                     : ((ppl & PIX_MASK) << (2 * mm)) + sub;
                            // (a level beyond the table: k_far fills the direction in)
                            int32_t cx = DIR_FAR, cy = 0, cz = 0;
                            if (L <= A.ltab) rotate_dir(rows, __ldg(&A.pixtab[level_offset(L) + pix]), cx, cy, cz);
                            else atomicOr(&C->far, 1);
                            const unsigned o = slot_of(rows[0].w + (int)sub);
                            cw[0] = (uint32_t)cz;
                            cw[1] = ((uint32_t)L << LEVEL_SHIFT) | pix;
                            char *const t = qout + (size_t)(o >> 5) * tile;
                            reinterpret_cast<uint4 *>(t)[o & 31u] = make_uint4(pa.x, pa.y, (uint32_t)cx, (uint32_t)cy);
                            store_tail<NB, false>(t, o & 31u, cw);
                            if (pmrg) {
                                char *const tm = t + 128 * (6 + NB);
                                pm.w &= 0x7fffffffu;
                                reinterpret_cast<uint4 *>(tm)[o & 31u] = pm;
                                reinterpret_cast<float *>(tm + 512)[o & 31u] = mthrs[src] * pow2_neg(2 * mm);
                            }
                        }
                    }
                }
            }
            // every lane is done with the tile: fetch the one after next into it
            __syncwarp();
            if (lane == 0) fetch(w_it + 2);
            ++w_it;
        }
        for (int k = lane; k < slab_left; k += 32) *pixel_word(A.q[par ^ 1], slab + k) = DEAD_RAY;
        if (ONE) {
            flush_one(t_esc, t_out, t_cnt, sh_acc);
            if (lane == 0 && w_out) atomicAdd(sh_acc + 5, (unsigned long long)w_out);    // rays out
        } else {
            flush_tallies(t_esc, t_out, t_cnt, t_rout, t_sim, sh_acc);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < A.nsims * NACC; i += blockDim.x) {
        const unsigned long long u = sh_acc[i];
        const double v = (i % NACC) < 3 ? (double)u * 0x1p-32 : (double)u;
        if (u != 0ull) {
            SimAcc &a = A.acc[i / NACC];
            double *dst = nullptr;
            switch (i % NACC) {
                case 0: dst = &a.p_in; break;
                case 1: dst = &a.p_esc; break;
                case 2: dst = &a.p_out; break;
                case 3: dst = &a.p_seg; break;
                case 4: dst = &a.p_rays_in; break;
                default: dst = &a.p_rays_out; break;
            }
            atomicAdd(dst, v);
        }
    }
}

// Kernel variants: every bin count with two and three blocks per SM (three:
// a quarter less time than two at six bins; four spill at every bin count and
// lose to three: 161 against 147 ms of march on the 128^3 workload); the bin
// counts of the standard spectra (1, 3, 4) also with four, and with every
// aggregation, for the autotuner.
template <int NB, int EXT, int ONE>
MarchFn march_pick_nb(int agg, int minb) {
    if (agg == 0 && minb == 2) return k_march<NB, 0, 2, EXT, ONE>;
    if (agg == 0 && minb == 3) return k_march<NB, 0, 3, EXT, ONE>;
    if constexpr (NB == 1 || NB == 3 || NB == 4) {
        if (agg == 0 && minb == 4) return k_march<NB, 0, 4, EXT, ONE>;
        if constexpr (ONE == 0) {
            if (agg == 1 && minb == 2) return k_march<NB, 1, 2, EXT, 0>;
            if (agg == 1 && minb == 3) return k_march<NB, 1, 3, EXT, 0>;
            if (agg == 1 && minb == 4) return k_march<NB, 1, 4, EXT, 0>;
            if (agg == 2 && minb == 2) return k_march<NB, 2, 2, EXT, 0>;
            if (agg == 2 && minb == 3) return k_march<NB, 2, 3, EXT, 0>;
            if (agg == 2 && minb == 4) return k_march<NB, 2, 4, EXT, 0>;
        }
    }
    return nullptr;
}
template <int EXT, int ONE>
MarchFn march_pick(int nb, int agg, int minb) {
    switch (nb) {
        case 1: return march_pick_nb<1, EXT, ONE>(agg, minb);
        case 2: return march_pick_nb<2, EXT, ONE>(agg, minb);
        case 3: return march_pick_nb<3, EXT, ONE>(agg, minb);
        case 4: return march_pick_nb<4, EXT, ONE>(agg, minb);
        case 5: return march_pick_nb<5, EXT, ONE>(agg, minb);
        case 6: return march_pick_nb<6, EXT, ONE>(agg, minb);
        case 7: return march_pick_nb<7, EXT, ONE>(agg, minb);
        case 8: return march_pick_nb<8, EXT, ONE>(agg, minb);
        default: return nullptr;
    }
}

}  // namespace frt
