// frt_kernels.cu -- the GPU kernels of one RT step and their launchers.
//
//   k_emit   : per active emitter, the step's random sphere rotation and the
//              12*4^l_src new rays at the emitter's cell centre
//              (Sec. 3.1, Eq. 1);
//   k_march  : (frt_march.cuh) per ray, the one-cell march with exp(-tau)
//              attenuation, the Eq. 17 deposit, escape, termination, the
//              Eq. 2-3 split and the compacted write of survivors and children;
//   k_chem   : per cell, Gamma from the deposits, the ionisation update of
//              Sec. 4.1 Eq. 7-10 (double precision), the temperature update
//              of Eq. 12 (single precision), kappa for the next step,
//              and the commit of the step's photon budget by its last block.
// All launches are sized on the host from capacities only; counts are read
// from device memory, so the same launches can be replayed from a CUDA graph.
#include <algorithm>
#include <cstdio>
#include "frt_march.cuh"

namespace frt {

// ---------------------------------------------------------------------------
// fixed-point pixel vector table, levels 0..L
// ---------------------------------------------------------------------------
__global__ void k_pixtab(int4 *tab, int L) {
    long long n = level_offset(L + 1);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int l = 0;
        while (level_offset(l + 1) <= i) ++l;
        tab[i] = healpix_vq(l, i - level_offset(l));
    }
}

// ---------------------------------------------------------------------------
// kappa of a cell for the next step (Sec. 4.2, Eq. 13 and the sub-grid law)
// ---------------------------------------------------------------------------
// (single precision throughout; `ionised`: the cell's neutral fraction is at
// most 1 - the ionised threshold of the sub-grid law)
__device__ __forceinline__ float2 cell_kappa(const SimDev &S, float nHf, float yf, bool ionised, float G) {
    const float kx = nHf * yf * S.ksc_f;
    float ks = 0.0f;
    if (S.mfp_mode == 1) {
        ks = S.kap_sub0;
    } else if (S.mfp_mode == 2 && ionised) {
        const float g = fmaxf(G, S.gamma_floor_f);
        const float f = powf(nHf * S.inv_nH_mean_f, S.neg_delta_exp_f) * powf(g * S.inv_gamma_ref_f, S.gamma_exp_f);
        ks = __fdividef(S.kap_sub0, f);
    }
    return make_float2(kx, ks);
}

// Generalized mode (Sec. 4.2): neutral fraction of the highly ionised part
// -- with the photo-ionisation-equilibrium law (mfp mode 3, Eq. 20-22)
// alpha (1 + chi) n_H / Gamma, else 0 -- and its opacity: n_HI sigma from
// that fraction plus the sub-grid law's 1/lambda.  A part never lit yet
// (Gamma = 0) is optically thin (the Eq. 14 guess).
__device__ __forceinline__ float gen_y_ion(const SimDev &S, float nHf, float G, float alpha) {
    if (S.mfp_mode != 3 || !(G > 0.0f)) return 0.0f;
    const float g = fmaxf(G, S.gamma_floor_f);
    return fminf(1.0f, alpha * S.chi1_f * nHf / g);
}
// case-B recombination coefficient of a Generalized-mode cell at T
__device__ __forceinline__ float gen_alpha(const SimDev &S, float T) {
    if (S.isothermal) return S.alpha_iso;
    return S.rates ? alphaB_f(T) : S.alpha_const_f;
}

// Generalized mode with evolving temperature (Sec. 4.2): dT/dt of the
// ionised part from Eq. 12 at static density -- the photo-heating of Eq. 22,
// E_pl alpha_A n_e n_HII (photo-ionisations balance case-A recombinations),
// less the cooling rates with n_HI = y_ion n_H and n_e = n_HII + chi n_H.
// Per n_H^2 inside, pref = 2 n_H / (3 k_B n_tot / n_H).
__device__ __forceinline__ float gen_dTdt_f(const SimDev &S, float T, float yion, float xe, float pref, float cc) {
    const float heat = S.pl_heat * alphaA_f(T) * xe * (1.0f - yion);
    return pref * (heat - cooling_f(T, xe, yion, 1.0f - yion, cc, S.Tcmb));
}
// Newly ionised gas enters at T_reion and mixes by mass with the gas ionised
// before; then sub-steps of the two-stage Rosenbrock scheme ROS2 (Verwer,
// Spee, Blom & Hundsdorfer 1999, gamma = 1 + 1/sqrt 2; second order for any
// Jacobian: here a one-sided difference over 10^-3 T, clipped at 0), each at
// most the step that would move T by 5% explicitly, at most 1000 (the last
// takes what is left).  L-stable: a step much longer than the relaxation
// time ends at the equilibrium temperature.
__device__ float gen_temperature_f(const SimDev &S, float T0, float x0, float dx, float x1, float yion, float nHf) {
    float T = dx > 0.0f ? (x0 * T0 + dx * S.t_reion) / x1 : T0;
    const float xe = 1.0f - yion + S.chi_f;
    const float pref = 2.0f * nHf / (3.0f * KB_F * (S.chi1_f + xe));
    const float cc = S.compton_c / nHf;
    const float gam = 1.70710678f;
    float left = S.dt_f;
    for (int k = 0; k < 1000 && left > 0.0f; ++k) {
        const float f = gen_dTdt_f(S, T, yion, xe, pref, cc);
        if (f == 0.0f) break;
        const float J = fminf((gen_dTdt_f(S, T * 1.001f, yion, xe, pref, cc) - f) / (0.001f * T), 0.0f);
        float h = left;
        if (k < 999) h = fminf(h, 0.05f * T / fabsf(f));
        const float w = 1.0f / (1.0f - gam * h * J);
        const float k1 = w * f;
        const float k2 = w * (gen_dTdt_f(S, T + h * k1, yion, xe, pref, cc) - 2.0f * k1);
        T += h * (1.5f * k1 + 0.5f * k2);
        left -= h;
    }
    return T;
}
__device__ __forceinline__ float2 gen_kappa(const SimDev &S, float nHf, float yion, float G) {
    const float kx = nHf * yion * S.ksc_f;
    float ks = 0.0f;
    if (S.mfp_mode == 1) {
        ks = S.kap_sub0;
    } else if (S.mfp_mode == 2 && G > 0.0f) {
        const float g = fmaxf(G, S.gamma_floor_f);
        const float f = powf(nHf * S.inv_nH_mean_f, S.neg_delta_exp_f) * powf(g * S.inv_gamma_ref_f, S.gamma_exp_f);
        ks = __fdividef(S.kap_sub0, f);
    }
    return make_float2(kx, ks);
}

// e = e^-r, g = (1 - e^-r)/r and h = (1 - g)/r for r >= 0 in single
// precision: Taylor series below r = 1/2, closed forms above.
__device__ __forceinline__ void relax_factors(float r, float &e, float &g, float &h) {
    const float u = fminf(fmaxf(r, 0.0f), 0.5f);
    float sg = 1.0f / 39916800.0f, sh = 1.0f / 479001600.0f;     // 1/11!, 1/12!
    const float cg[10] = {1.0f / 3628800.0f, 1.0f / 362880.0f, 1.0f / 40320.0f, 1.0f / 5040.0f, 1.0f / 720.0f,
                          1.0f / 120.0f, 1.0f / 24.0f, 1.0f / 6.0f, 0.5f, 1.0f};
    const float ch[10] = {1.0f / 39916800.0f, 1.0f / 3628800.0f, 1.0f / 362880.0f, 1.0f / 40320.0f, 1.0f / 5040.0f,
                          1.0f / 720.0f, 1.0f / 120.0f, 1.0f / 24.0f, 1.0f / 6.0f, 0.5f};
#pragma unroll
    for (int k = 0; k < 10; ++k) { sg = fmaf(sg, -u, cg[k]); sh = fmaf(sh, -u, ch[k]); }
    if (r < 0.5f) { g = sg; h = sh; e = 1.0f - r * sg; return; }
    e = __expf(-r);
    g = __fdividef(1.0f - e, r);
    h = __fdividef(1.0f - g, r);
}

__global__ void k_init_cells(const SimDev *sims, int sim, Cells c) {
    const SimDev &S = sims[sim];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < S.ncell; i += (long long)gridDim.x * blockDim.x) {
        long long g = S.cell_off + i;
        // Generalized mode starts with no ionised fraction
        double y = S.gen_mode ? 1.0 : 1.0 - S.x_init;
        c.y[g] = y;
        c.x[g] = S.gen_mode ? 0.0f : (float)S.x_init;
        c.T[g] = (float)S.T_init;
        c.gamma[g] = 0.0f;
        c.dep[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c.segcnt) c.segcnt[g] = 0;
        c.xion[g] = 0.0;
        c.rho[g] = 1.0f;
        c.fscr[g] = make_float2(0.f, 0.f);
        const float nHf = (float)c.nH[g];
        c.nHf[g] = nHf;
        c.kap[g] = S.gen_mode ? gen_kappa(S, nHf, 0.0f, 0.0f) : cell_kappa(S, nHf, (float)y, y <= S.y_thr, 0.0f);
    }
}

// the start of a run: no rays, no error, step 0, an empty photon budget (the
// marched-ray counter is kept: profiling windows difference it)
__global__ void k_reset(Ctl *C, SimDev *sims, SimAcc *acc, int nsims) {
    for (int j = threadIdx.x; j < nsims; j += blockDim.x) {
        if (!sims[j].active) continue;
        const double marched = acc[j].rays_in_total;
        acc[j] = SimAcc{};
        acc[j].rays_in_total = marched;
        sims[j].step = 0;
    }
    if (threadIdx.x == 0) {
        C->cnt[0] = C->cnt[1] = 0;
        C->par = 0;
        C->err = 0;
        C->merged = C->far = 0;                    // a step dropped between its stages may have set them
    }
}

// ---------------------------------------------------------------------------
// emission
// ---------------------------------------------------------------------------
// A warp takes 32 emitters: a lane draws one emitter's rotation, stores it in
// the ring and sums its photons; then the warp's lanes write the 32 emitters'
// rays together, one ray a lane, with the rows of its emitter from the lane
// that drew them.  Bound by the chain control words, list, cell, constants,
// draw.  (One thread an emitter wrote its 12 rays one after another, ten
// scattered words each: 25 us a step at 2e4 emitters, now 13.)
__global__ void __launch_bounds__(128) k_emit(EmitArgs A) {
    Ctl *C = A.ctl;
    if (C->err) return;
    const int par = C->par;
    const long long base = C->cnt[par];
    const long long total = C->emit_total;
    if (base + total > A.cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&C->err, 1);
        return;
    }
    const Queue q = A.q[par];
    const int n = C->n_act_emit;
    const int lane = lane_id();
    const int nr = (n + 31) & ~31;                 // whole warps
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nr; j += gridDim.x * blockDim.x) {
        double emitted = 0.0;
        int esim = -1, e = 0, s = 0, l = 0;
        unsigned off = 0;                          // queue slots stay below 2^31 (the engine's bound)
        float n0 = 0.0f;
        int4 rows[3];
        if (j < n) {
            e = A.em.act[j];
            off = (unsigned)(base + A.em.act_off[j]);
            esim = A.em.cell[e].w;
            const SimDev &S = A.sims[esim];
            s = S.step;
            l = S.l_src;
            rotation_rows(S.seed, A.em.local[e], s, S.rotate, rows);
            int4 *ring = A.em.ring + ((long long)e * A.em.ring_w + (s % A.em.ring_w)) * 3;
            ring[0] = rows[0]; ring[1] = rows[1]; ring[2] = rows[2];
            n0 = (float)(A.em.ndot[e] * S.dt * S.inv_ncast / S.nref);
            A.em.n0[e] = n0;
            double tot = 0.0;
#pragma unroll
            for (int b = 0; b < MAXB; ++b) tot += (double)(b < S.nb ? S.frac[b] * n0 : 0.0f);
            emitted = tot * (double)(12LL << (2 * l));
        } else {
            rows[0] = rows[1] = rows[2] = make_int4(0, 0, 0, 0);
        }
        // one ray: emitter of lane k (every lane of the warp takes part in
        // the shuffles), pixel p
        auto ray = [&](int k, unsigned p, bool on) {
            int4 rk[3];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                rk[r] = make_int4(__shfl_sync(FULL, rows[r].x, k), __shfl_sync(FULL, rows[r].y, k),
                                  __shfl_sync(FULL, rows[r].z, k), 0);
            const int ek = __shfl_sync(FULL, e, k), sk = __shfl_sync(FULL, s, k), lk = __shfl_sync(FULL, l, k);
            const int mk = __shfl_sync(FULL, esim, k);
            const unsigned o = __shfl_sync(FULL, off, k) + p;
            const float nk = __shfl_sync(FULL, n0, k);
            if (!on) return;
            const SimDev &S = A.sims[mk];
            int32_t dx, dy, dz;
            rotate_dir(rk, lk <= A.ltab ? __ldg(&A.pixtab[level_offset(lk) + p]) : healpix_vq(lk, p), dx, dy, dz);
            uint32_t w[2 + MAXB];
            w[0] = (uint32_t)dz;
            w[1] = ((uint32_t)lk << LEVEL_SHIFT) | p;
#pragma unroll
            for (int b = 0; b < MAXB; ++b) w[2 + b] = __float_as_uint(b < S.nb ? S.frac[b] * nk : 0.0f);
            *ray_head(q, o) = make_uint4((uint32_t)ek, (uint32_t)sk, (uint32_t)dx, (uint32_t)dy);
            store_tail_n(q, o, w);
        };
        const int here = min(32, n - (j - lane));  // emitters of this warp (its first one is j - lane < n)
        const int l0 = __shfl_sync(FULL, l, 0);
        if (__all_sync(FULL, lane >= here || l == l0)) {
            // one level: the rays of all 32 emitters as one run
            const unsigned nc = 12u << (2 * l0);
            const unsigned long long all = (unsigned long long)nc * here;
            for (unsigned long long r = lane; r < ((all + 31) & ~31ull); r += 32) {
                const bool on = r < all;
                const unsigned k = on ? (unsigned)((r >> (2 * l0)) / 12u) : 0u;
                ray((int)k, (unsigned)(r - (unsigned long long)k * nc), on);
            }
        } else {
            for (int k = 0; k < here; ++k) {
                const unsigned nc = 12u << (2 * __shfl_sync(FULL, l, k));
                for (unsigned p = lane; p < ((nc + 31u) & ~31u); p += 32) ray(k, p, p < nc);
            }
        }
        // photons emitted, summed over the warp when its emitters share a
        // simulation (one atomic per warp instead of one per emitter)
        const int kref = __reduce_max_sync(FULL, esim);
        if (kref >= 0) {
            if (__all_sync(FULL, esim < 0 || esim == kref)) {
                double v[1] = {esim == kref ? emitted : 0.0};
                warp_sum<1>(v);
                if (lane == 0) atomicAdd(&A.acc[kref].p_emit, v[0]);
            } else if (esim >= 0) {
                atomicAdd(&A.acc[esim].p_emit, emitted);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// directions of the march's children beyond the pixel table (levels that
// hardly any run reaches).  In the march itself the double-precision vector
// took 15 registers of every ray.  Launched only by engines with a member
// that can reach such a level; the march's flag says whether one did.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_far(EmitArgs A) {
    const Ctl *C = A.ctl;
    if (!C->far || C->err) return;
    const Queue q = A.q[C->par ^ 1];
    const long long n = C->cnt[C->par ^ 1];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const uint32_t pl = *pixel_word(q, i);
        if (pl == DEAD_RAY || (int)(pl >> LEVEL_SHIFT) <= A.ltab) continue;
        const uint4 a = *ray_head(q, i);
        if ((int32_t)a.z != DIR_FAR) continue;
        int4 rows[3];
        if (a.x & MERGED_BIT) {
            const SimDev &S = A.sims[(ray_merge(q, i)->w >> 16) & 0x7fffu];
            rotation_rows(S.seed, (1LL << 31) + (long long)(a.x & ~MERGED_BIT), (int)a.y, S.rotate, rows);
        } else {
            const int4 *rg = A.em.ring + ((long long)a.x * A.em.ring_w + (int)a.y % A.em.ring_w) * 3;
            rows[0] = rg[0]; rows[1] = rg[1]; rows[2] = rg[2];
        }
        int32_t dx, dy, dz;
        rotate_dir(rows, healpix_vq((int)(pl >> LEVEL_SHIFT), pl & PIX_MASK), dx, dy, dz);
        *ray_head(q, i) = make_uint4(a.x, a.y, (uint32_t)dx, (uint32_t)dy);
        *tail_word(q, 0, i) = (uint32_t)dz;
    }
}

// ---------------------------------------------------------------------------
// a queue's records to and from one array a word (checkpoints): word-major,
// in the order pixel word, emitter, birth, dx, dy, dz, photons, then the
// merged rays' position, merge word and threshold
// ---------------------------------------------------------------------------
__global__ void k_queue_words(Queue q, int merged, long long n, uint32_t *words, int join) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        uint32_t *x[6 + MAXB + 5];
        uint32_t *a = reinterpret_cast<uint32_t *>(ray_head(q, i));
        int k = 0;
        x[k++] = tail_word(q, 1, i);
        x[k++] = a; x[k++] = a + 1; x[k++] = a + 2; x[k++] = a + 3;
        x[k++] = tail_word(q, 0, i);
        for (int b = 0; b < q.nb; ++b) x[k++] = tail_word(q, 2 + b, i);
        if (merged) {
            uint32_t *m = reinterpret_cast<uint32_t *>(ray_merge(q, i));
            for (int c = 0; c < 4; ++c) x[k++] = m + c;
            x[k++] = reinterpret_cast<uint32_t *>(ray_thr(q, i));
        }
        for (int c = 0; c < k; ++c) {
            if (join) *x[c] = words[c * n + i];
            else words[c * n + i] = *x[c];
        }
    }
}

// ---------------------------------------------------------------------------
// chemistry
// ---------------------------------------------------------------------------
// double -> float rounded to nearest even, and float -> double, of
// non-negative values on the integer pipe: the conversions share the FP64
// pipe (two lanes a clock on this part), which bound the kernel -- a cell of a
// step took six double-precision operations, of which one is left.  Values
// outside the normal float range take the conversion instruction.
__device__ __forceinline__ float narrow(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    if (hi - 0x38100000u >= 0x47e00000u - 0x38100000u) return (float)v;      // not within [2^-126, 2^127)
    const unsigned f = ((hi << 3) | (lo >> 29)) - (896u << 23);
    return __uint_as_float(f + (((lo & 0x1fffffffu) + 0x0fffffffu + (f & 1u)) >> 29));
}
__device__ __forceinline__ double widen(float v) {
    const unsigned f = __float_as_uint(v);
    if (f - 0x00800000u >= 0x7f000000u) return (double)v;                    // not a positive normal number
    return __hiloint2double((int)((f >> 3) + (896u << 20)), (int)(f << 29));
}

// One sub-step of Eq. 12 at static density: heating minus cooling (per
// n_H^2), at most 5% of T (the thousandth takes what is left).
__device__ __forceinline__ void t_substep(const SimDev &S, float &T, float &left, int k, float heat, float xb, float yb,
                                          float nHf) {
    const float pref = 2.0f * nHf / (3.0f * KB_F * (1.0f + xb));
    const float cc = S.compton_c / nHf;
    const float lam = cooling_f(T, xb, yb, xb, cc, S.Tcmb);
    const float dTdt = pref * (heat - lam);
    float h = left;
    if (k < 999 && dTdt != 0.0f) h = fminf(h, 0.05f * T / fabsf(dTdt));
    T += dTdt * h;
    left -= h;
}
// Cells whose temperature needs more than T_INLINE sub-steps (those an
// ionisation front is heating take up to a hundred, most others one) wait in
// shared memory and are worked off by the whole block, each thread taking the
// next cell when its own is done: with every lane looping to its warp's
// longest, 8 to 12 of 32 lanes were active and these loops most of the kernel.
constexpr int T_INLINE = 2, T_CAP = 512;
struct TQueue {
    float T[T_CAP], left[T_CAP], heat[T_CAP], xb[T_CAP], yb[T_CAP], nH[T_CAP];
    unsigned cell[T_CAP];
    int sim[T_CAP];
    int count, next;
};
__device__ void t_drain(const ChemArgs &A, TQueue &q) {
    const int n = q.count;                         // (block-uniform: a barrier is behind the last push)
    for (;;) {
        const int w = atomicAdd(&q.next, 1);
        if (w >= n) break;
        const SimDev &S = A.sims[q.sim[w]];
        float T = q.T[w], left = q.left[w];
        const float heat = q.heat[w], xb = q.xb[w], yb = q.yb[w], nHf = q.nH[w];
        for (int k = T_INLINE; k < 1000 && left > 0.0f; ++k) t_substep(S, T, left, k, heat, xb, yb, nHf);
        A.cells.T[q.cell[w]] = T;
    }
    __syncthreads();
    if (threadIdx.x == 0) q.count = q.next = 0;
    __syncthreads();
}

// The last block of a pass ends it (kernels of their own for this were a fifth
// of a small simulation's step: one more launch a step, and one a trial pass).
// A trial pass of the Gamma - <n_HI> iteration: the next pass marches the same
// rays again, so the march's output and the step's tallies are dropped
// (emission happens once per step; the marched-ray counter keeps every pass).
// A step: its photon budget is committed, the queues change places, and the
// step's outcome goes to host memory.
__device__ void end_pass(const ChemArgs &A) {
    Ctl *C = A.ctl;
    const bool err = C->err != 0;
    if (!A.final_pass && err) return;
    for (int j = threadIdx.x; j < A.nsims; j += blockDim.x) {
        SimAcc &a = A.acc[j];
        // (written by other blocks' and kernels' atomics: read past the L1)
        const double emit = __ldcg(&a.p_emit), absd = __ldcg(&a.p_abs), esc = __ldcg(&a.p_esc), out = __ldcg(&a.p_out);
        const double seg = __ldcg(&a.p_seg), rin = __ldcg(&a.p_rays_in), rout = __ldcg(&a.p_rays_out);
        if (A.final_pass) {
            if (!err && A.sims[j].active) {
                a.emitted += emit;
                a.absorbed += absd;
                a.escaped += esc;
                a.in_flight = out;
                a.seg_last = seg;
                a.seg_total += seg;
                a.rays_live = rout;
                a.rays_in_last = rin;
                a.rays_in_total += rin;
                a.lost += __ldcg(&a.p_lost);
                A.sims[j].step += 1;
            }
            a.p_emit = 0.0;
        } else {
            a.rays_in_total += rin;
        }
        a.p_abs = a.p_esc = a.p_out = a.p_in = 0.0;
        a.p_seg = a.p_rays_in = a.p_rays_out = a.p_lost = 0.0;
    }
    if (threadIdx.x != 0) return;
    const int par = C->par;
    C->far = 0;
    if (!A.final_pass) {
        C->cnt[par ^ 1] = 0;
        return;
    }
    // the march wrote the live rays to the other queue (a merge step left
    // holes there, which the next march skips)
    long long live;
    if (err) {
        C->cnt[par ^ 1] = 0;
        live = C->cnt[par];
    } else {
        live = C->cnt[par ^ 1];
        C->cnt[par] = 0;
        C->par = par ^ 1;
    }
    C->merged = 0;
    // (each word stands for itself: the host relies on no order between them)
    *A.status = make_uint2((uint32_t)live, (uint32_t)C->err);
}

__global__ void __launch_bounds__(256) k_chem(ChemArgs A) {
    __shared__ int s_last;
    __shared__ TQueue tq;
    __shared__ int s_evolve;                       // a member's temperature evolves (Standard mode, committed pass)
    // per-simulation absorbed totals and screens' excess photons, then the
    // active cell ranges
    extern __shared__ double sh_abs[];
    double *sh_lost = sh_abs + A.nsims;
    long long *s_pref = reinterpret_cast<long long *>(sh_lost + A.nsims);
    long long *s_cell0 = s_pref + A.nsims + 1;
    int *s_sim = reinterpret_cast<int *>(s_cell0 + A.nsims);
    // Generalized mode: its flag and the atoms of a cell per unit n_H, in
    // code photons
    float *s_apn = reinterpret_cast<float *>(s_sim + A.nsims);
    int *s_gen = reinterpret_cast<int *>(s_apn + A.nsims);
    int *s_iso = s_gen + A.nsims;
    Ctl *C = A.ctl;
    const int nrng = C->n_ranges;
    if (threadIdx.x == 0) tq.count = tq.next = s_evolve = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < A.nsims; i += blockDim.x) {
        sh_abs[i] = 0.0;
        sh_lost[i] = 0.0;
        const SimDev &S = A.sims[i];
        s_apn[i] = S.apn_f;
        s_gen[i] = S.gen_mode;
        s_iso[i] = S.isothermal;
        if (A.final_pass && !S.isothermal && !S.gen_mode && S.active) s_evolve = 1;
    }
    for (int i = threadIdx.x; i <= nrng; i += blockDim.x) s_pref[i] = A.rg.pref[i];
    for (int i = threadIdx.x; i < nrng; i += blockDim.x) { s_cell0[i] = A.rg.cell0[i]; s_sim[i] = A.rg.sim[i]; }
    __syncthreads();
    const bool err = C->err != 0;
    // cell keys are 32-bit integers (the march's bound)
    const unsigned n = (unsigned)C->ncell_active;
    const int lane = lane_id();
    // absorbed photons: each thread sums its cells of one simulation in a
    // register pair (a single-precision sum and its exact rounding error,
    // Knuth's two-sum: no FP64 per cell) and adds the sum to the block's
    // total when the simulation changes and at the end (one shared-memory
    // atomic per run of cells, not one per warp and cell)
    float t_hi = 0.0f, t_lo = 0.0f;
    int t_sim = -1;
    for (unsigned base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {   // block-uniform
        const unsigned i = base + threadIdx.x;
        int sim = -1;
        float a_abs = 0.0f;
        if (i < n) {
            int lo = 0, hi = nrng;  // largest r with pref[r] <= i
            while (hi - lo > 1) {
                int mid = (lo + hi) >> 1;
                if ((unsigned)s_pref[mid] <= i) lo = mid; else hi = mid;
            }
            sim = s_sim[lo];
            const unsigned g = (unsigned)s_cell0[lo] + (i - (unsigned)s_pref[lo]);
            // every load of the cell first: the stores below would otherwise
            // hold the later loads back, one memory round trip each
            const bool gen = s_gen[sim] != 0;
            float4 d;
            if (A.two) {
                const float2 d2 = reinterpret_cast<const float2 *>(A.cells.dep)[g];
                d = make_float4(d2.x, d2.y, 0.0f, 0.0f);
            } else {
                d = A.cells.dep[g];
            }
            const float nHf = A.cells.nHf[g];
            // (an isothermal member's temperature is neither read nor written)
            const float T0 = s_iso[sim] ? 0.0f : A.cells.T[g];
            float2 fs = make_float2(0.f, 0.f);
            double xs;                     // Generalized: x_ion; Standard: neutral fraction y
            float x0f = 0.0f;
            if (gen) {
                fs = A.cells.fscr[g];
                xs = A.cells.xion[g];
            } else {
                xs = A.cells.y[g];
                x0f = A.cells.x[g];
            }
            // cleared for the next pass, where there is something to clear: most
            // cells of a large box are not lit, and their 16 (24) bytes are a
            // fifth (a third) of what the cell moves
            if (d.w != 0.0f || d.x != 0.0f || d.y != 0.0f || d.z != 0.0f) {
                if (A.two) reinterpret_cast<float2 *>(A.cells.dep)[g] = make_float2(0.f, 0.f);
                else A.cells.dep[g] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (A.cells.segcnt) A.cells.segcnt[g] = (int)d.w;
            if (gen && (fs.x != 0.0f || fs.y != 0.0f)) A.cells.fscr[g] = make_float2(0.f, 0.f);
            const SimDev &SG = A.sims[sim];
            if (gen) {
                // Generalized mode (Sec. 4.2): Gamma of the ionised part (Eq. 17
                // with ds -> x ds, V -> x V); the cell's atom balance -- photons
                // absorbed at the screen and in the ionised part less the
                // recombinations there, alpha (1 + chi) n_H^2 x V dt (Eq. 22's
                // approximation) -- moves x (Eq. 18 when the last two cancel);
                // the screen's share rho for the next pass or step
                if (!err) {
                    // single precision except the state x_ion and its
                    // complement (FP64 is a narrow pipe on this part): the
                    // atoms of the cell Ac and the photons in code units, and
                    // the recombinations per atom alpha n_H x dt
                    a_abs = d.x + fs.x;
                    // a cell no front has reached and no photon entered keeps
                    // x_ion, the neutral fraction and the ionised fraction
                    // (0, 1, 0): the rest of this branch without its
                    // double-precision arithmetic, most of the kernel's time
                    // in a large box (240 us a committed pass at 200^3 cells)
                    if ((__double2hiint(xs) | __double2loint(xs)) == 0 && a_abs == 0.0f && fs.y == 0.0f) {
                        A.cells.rho[g] = 1.0f;
                        A.cells.kap[g] = gen_kappa(SG, nHf, 0.0f, 0.0f);
                        if (A.final_pass) A.cells.gamma[g] = 0.0f;
                    } else {
                    const double x = xs;
                    const float xf = (float)x, omx = (float)(1.0 - x);
                    const float Ac = nHf * s_apn[sim];                           // atoms of a whole cell
                    const float Gf = xf > 0.0f ? d.y * SG.gscale_f / xf : 0.0f;
                    const float alpha = gen_alpha(SG, T0);
                    if (!A.final_pass) {
                        A.cells.rho[g] = fs.y > omx * Ac ? omx * Ac / fs.y : 1.0f;
                        A.cells.kap[g] = gen_kappa(SG, nHf, gen_y_ion(SG, nHf, Gf, alpha), Gf);
                    } else {
                        const float dxf = (fs.x + d.x) / Ac - alpha * nHf * xf * SG.dt_f;
                        const double x1 = fmin(fmax(x + (double)dxf, 0.0), 1.0);
                        // a screen that absorbed more photons than its cell had
                        // neutral atoms (one first reached in the last pass: its
                        // share came from a pass it was not lit in): the excess
                        // ionises nothing
                        const float sx = fs.x - omx * Ac;
                        if (sx > 0.0f) atomicAdd(&sh_lost[sim], (double)sx);
                        const float om1 = (float)(1.0 - x1), x1f = (float)x1;
                        A.cells.rho[g] = fs.y > om1 * Ac ? om1 * Ac / fs.y : 1.0f;
                        // the temperature moves with the start-of-step neutral
                        // fraction; the committed one is that of the new T
                        float yi = gen_y_ion(SG, nHf, Gf, alpha);
                        if (!SG.isothermal && x1 > 0.0) {
                            const float T1 = gen_temperature_f(SG, T0, xf, (float)(x1 - x), x1f, yi, nHf);
                            A.cells.T[g] = T1;
                            yi = gen_y_ion(SG, nHf, Gf, gen_alpha(SG, T1));
                        }
                        A.cells.xion[g] = x1;
                        A.cells.y[g] = fma(x1, (double)yi, 1.0 - x1);
                        A.cells.x[g] = x1f * (1.0f - yi);
                        A.cells.gamma[g] = Gf;
                        A.cells.kap[g] = gen_kappa(SG, nHf, yi, Gf);
                    }
                    }
                }
            } else if (!err) {
                a_abs = d.x;
                const SimDev &S = A.sims[sim];
                const float Gf = d.y * S.gscale_f;                    // Eq. 17, 1/s
                const double y0 = xs;
                const float y0f = narrow(y0);
                const float dtf = S.dt_f;
                float alpha = S.alpha_iso, Cc = S.coll_iso;
                if (!S.isothermal && S.rates) { alpha = alphaB_f(T0); Cc = collion_f(T0); }
                else if (!S.isothermal) alpha = S.alpha_const_f;
                // Eq. 7-10 with n_e re-evaluated from <x>.  With i = Gamma + C n_e,
                // b = alpha n_e, r = dt (i + b), e = e^-r, g = (1 - e)/r and
                // h = (1 - g)/r, the solution x(t) = x_eq + (x0 - x_eq) e^{-t/t_i}
                // and its time average are, for y = 1 - x,
                //   x1 = x0 e + g i dt,  y1 = y0 e + g b dt,
                //   <x> = x0 g + h i dt, <y> = y0 g + h b dt:
                // sums of positive terms, accurate however small x or y is.
                float xb = x0f, yb = y0f, ef = 1.0f, gf = 0.0f, hf = 0.0f, idt = 0.0f, bdt = 0.0f;
                for (int it = 0; it < S.chem_iters; ++it) {
                    const float ne = nHf * xb;
                    idt = (Gf + Cc * ne) * dtf;
                    bdt = alpha * ne * dtf;
                    relax_factors(idt + bdt, ef, gf, hf);
                    const float xbn = fmaf(x0f, gf, hf * idt);
                    yb = fmaf(y0f, gf, hf * bdt);
                    const bool conv = fabsf(xbn - xb) <= 1e-7f * xbn;
                    xb = xbn;
                    if (conv) break;
                }
                if (!A.final_pass) {
                    // a trial pass of the Gamma - <n_HI> iteration (Eq. 11; with
                    // the sub-grid law lambda - Gamma): the next march sees the
                    // opacity of the time-averaged state; the state is kept
                    A.cells.kap[g] = cell_kappa(S, nHf, yb, yb <= S.y_thr_dn, Gf);
                } else {
                // x1 + y1 = 1 holds to rounding: keep x1 in [0, 1]
                const float x1 = fminf(fmaf(x0f, ef, gf * idt), 1.0f);
                const double y1 = fma(y0, widen(ef), widen(gf * bdt));   // neutral fraction kept in FP64
                const float y1f = narrow(y1);
                // (the float decides unless it lies next to the threshold)
                const bool ionised = fabsf(y1f - S.y_thr_dn) > 1e-6f ? y1f < S.y_thr_dn : y1 <= S.y_thr;
                if (!S.isothermal) {
                    // Eq. 12 with static density: particle-number term, then
                    // sub-stepped heating minus cooling (per n_H^2)
                    float T = T0 * (1.0f + x0f) / (1.0f + x1);
                    const float heat = d.z * S.hscale_f * yb / nHf;
                    float left = dtf;
                    for (int k = 0; k < T_INLINE && left > 0.0f; ++k) t_substep(S, T, left, k, heat, xb, yb, nHf);
                    if (left > 0.0f) {
                        const int w = atomicAdd(&tq.count, 1);
                        tq.T[w] = T; tq.left[w] = left; tq.heat[w] = heat;
                        tq.xb[w] = xb; tq.yb[w] = yb; tq.nH[w] = nHf;
                        tq.cell[w] = g; tq.sim[w] = sim;
                    } else {
                        A.cells.T[g] = T;
                    }
                }
                A.cells.y[g] = y1;
                A.cells.x[g] = x1;
                A.cells.gamma[g] = Gf;
                A.cells.kap[g] = cell_kappa(S, nHf, y1f, ionised, Gf);
                }
            }
        }
        if (sim >= 0 && a_abs != 0.0f) {
            if (sim != t_sim) {
                if (t_sim >= 0) atomicAdd(&sh_abs[t_sim], (double)t_hi + (double)t_lo);
                t_sim = sim;
                t_hi = t_lo = 0.0f;
            }
            const float s = t_hi + a_abs, bp = s - t_hi;
            t_lo += (t_hi - (s - bp)) + (a_abs - bp);
            t_hi = s;
        }
        // an iteration pushes at most a cell a thread: drain a half-full queue
        // (and what is left after the last iteration)
        if (s_evolve) {
            __syncthreads();
            const bool drain = tq.count > T_CAP - (int)blockDim.x || n - base <= gridDim.x * blockDim.x;
            __syncthreads();
            if (drain) t_drain(A, tq);
        }
    }
    {
        // the warp's sums: one atomic when its lanes share a simulation
        const double t_abs = (double)t_hi + (double)t_lo;
        const int kref = __reduce_max_sync(FULL, t_sim);
        if (kref >= 0 && __all_sync(FULL, t_sim < 0 || t_sim == kref)) {
            double v[1] = {t_sim == kref ? t_abs : 0.0};
            warp_sum<1>(v);
            if (lane == 0 && v[0] != 0.0) atomicAdd(&sh_abs[kref], v[0]);
        } else if (t_sim >= 0 && t_abs != 0.0) {
            atomicAdd(&sh_abs[t_sim], t_abs);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < A.nsims; i += blockDim.x) {
        if (sh_abs[i] != 0.0) atomicAdd(&A.acc[i].p_abs, sh_abs[i]);
        if (sh_lost[i] != 0.0) atomicAdd(&A.acc[i].p_lost, sh_lost[i]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&C->ticket, 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (threadIdx.x == 0) C->ticket = 0u;
        end_pass(A);
    }
}

// ---------------------------------------------------------------------------
// probes: the same device functions on host-given inputs
// ---------------------------------------------------------------------------
__global__ void k_probe_pixvec(int level, long long p0, long long n, int32_t *out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int4 v = healpix_vq(level, p0 + i);
        out[3 * i] = v.x; out[3 * i + 1] = v.y; out[3 * i + 2] = v.z;
    }
}
// the single-precision rate fits of the chemistry kernel (Sec. 4.1) at n
// temperatures: alpha_B, alpha_A, C_HI and the cooling rate with unit
// electron, HI and HII fractions and no Compton term
__global__ void k_probe_rates(long long n, const float *T, float *out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float t = T[i];
        out[4 * i + 0] = alphaB_f(t);
        out[4 * i + 1] = alphaA_f(t);
        out[4 * i + 2] = collion_f(t);
        out[4 * i + 3] = cooling_f(t, 1.0f, 1.0f, 1.0f, 0.0f, 0.0f);
    }
}
__global__ void k_probe_rotation(uint64_t seed, long long e, long long s, int rotate, int32_t *out) {
    int4 r[3];
    rotation_rows(seed, e, s, rotate, r);
    for (int k = 0; k < 3; ++k) { out[3 * k] = r[k].x; out[3 * k + 1] = r[k].y; out[3 * k + 2] = r[k].z; }
}
__global__ void k_probe_direction(int level, long long p0, long long n, const int32_t *Rq, const int4 *tab, int ltab,
                                  int32_t *out) {
    int4 rows[3];
    for (int k = 0; k < 3; ++k) rows[k] = make_int4(Rq[3 * k], Rq[3 * k + 1], Rq[3 * k + 2], 0);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        long long p = p0 + i;
        int4 v = level <= ltab ? tab[level_offset(level) + p] : healpix_vq(level, p);
        int32_t dx, dy, dz;
        rotate_dir(rows, v, dx, dy, dz);
        out[3 * i] = dx; out[3 * i + 1] = dy; out[3 * i + 2] = dz;
    }
}
__global__ void k_probe_traverse(long long n, const long long *p0, const int32_t *d, int gx, int gy, int gz,
                                 int32_t *cells, float *ds, int32_t *nseg, int32_t *esc) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int key[4];
        float s[4];
        bool e = false;
        walk_step(true, (int)p0[3 * i], (int)p0[3 * i + 1], (int)p0[3 * i + 2], d[3 * i], d[3 * i + 1], d[3 * i + 2], gx,
                  gy, gz, 0, key, s, e);
        int k = 0;
        for (int j = 0; j < 4; ++j) {
            if (key[j] < 0) continue;
            const int c = key[j];
            cells[12 * i + 3 * k] = c % gx;
            cells[12 * i + 3 * k + 1] = (c / gx) % gy;
            cells[12 * i + 3 * k + 2] = c / (gx * gy);
            ds[4 * i + k] = s[j];
            ++k;
        }
        nseg[i] = k;
        esc[i] = e ? 1 : 0;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_pixtab(int4 *tab, int L, cudaStream_t st) {
    long long n = level_offset(L + 1);
    int blocks = (int)((n + 255) / 256);
    if (blocks > 65535) blocks = 65535;
    k_pixtab<<<blocks, 256, 0, st>>>(tab, L);
    return cudaGetLastError();
}
cudaError_t launch_init_cells(const SimDev *sims, int sim, Cells c, long long ncell, cudaStream_t st) {
    int blocks = (int)((ncell + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_init_cells<<<blocks, 256, 0, st>>>(sims, sim, c);
    return cudaGetLastError();
}
cudaError_t launch_reset(Ctl *c, SimDev *sims, SimAcc *acc, int nsims, cudaStream_t st) {
    k_reset<<<1, 256, 0, st>>>(c, sims, acc, nsims);
    return cudaGetLastError();
}
cudaError_t launch_emit(const EmitArgs &a, int blocks, Sink &to) { return enqueue(to, k_emit, blocks, 128, 0, a); }
cudaError_t launch_far(const EmitArgs &a, int blocks, Sink &to) { return enqueue(to, k_far, blocks, 256, 0, a); }
cudaError_t launch_queue_words(const Queue &q, bool merged, long long n, uint32_t *words, bool join,
                               cudaStream_t st) {
    if (n < 1) return cudaSuccess;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    k_queue_words<<<blocks, 256, 0, st>>>(q, merged ? 1 : 0, n, words, join ? 1 : 0);
    return cudaGetLastError();
}
// The plain variants are built here, those with merged rays in frt_merge.cu,
// the others in frt_march_gen.cu and frt_march_one*.cu.
static MarchFn march_fn(int nb, int agg, int minb, int ext) {
    if (agg == 0) {
        switch (ext) {
            case 4: return march_fn_one(nb, agg, minb);
            case 5: return march_fn_one_merge(nb, agg, minb);
            case 7: return march_fn_one_gen(nb, agg, minb);
            case 12: return march_fn_two(nb, agg, minb);
            case 13: return march_fn_two_merge(nb, agg, minb);
            case 15: return march_fn_two_gen(nb, agg, minb);
            default: break;
        }
    }
    switch (ext & 3) {
        case 0: return march_pick<0, 0>(nb, agg, minb);
        case 1: return march_fn_merge(nb, agg, minb);
        case 3: return march_fn_gen(nb, agg, minb);
        default: return nullptr;
    }
}
bool march_variant_exists(int nb, int agg, int minb, int ext) { return march_fn(nb, agg, minb, ext) != nullptr; }
// Always the device's whole opt-in limit less the kernel's static part, never
// this engine's own need: the attribute is the process's, so a smaller engine
// would take a larger one's away, and the limit without it counts the static
// part too.  A launch still asks for what its slots need.
static cudaError_t raise_shared_limit(MarchFn f) {
    int dev = 0, most = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
}
cudaError_t march_prepare(int nb, int agg, int minb, int ext) {
    MarchFn f = march_fn(nb, agg, minb, ext);
    if (!f) return cudaErrorInvalidValue;
    cudaError_t e = raise_shared_limit(f);
    MarchFn two = ext & 4 ? march_fn(nb, agg, minb, ext | 8) : f;      // a launch may take either
    if (e == cudaSuccess && two != f) e = raise_shared_limit(two);
    return e;
}
cudaError_t launch_march(const MarchArgs &a, int nb, int agg, int minb, int blocks, int threads, Sink &to, int ext) {
    MarchFn f = march_fn(nb, agg, minb, ext);
    if (!f) return cudaErrorInvalidValue;
    return enqueue(to, f, blocks, threads, march_shared_bytes(a.nsims, a.q[0].tile, threads), a);
}
int march_max_blocks_per_sm(int nb, int agg, int minb, int threads, int nsims, int ext, uint32_t tile) {
    MarchFn f = march_fn(nb, agg, minb, ext);
    if (!f) return 0;
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, threads, march_shared_bytes(nsims, tile, threads));
    return n;
}
static size_t chem_shared_bytes(int nsims) {
    return (size_t)nsims * 2 * sizeof(double) + (size_t)(2 * nsims + 1) * sizeof(long long) +
           (size_t)nsims * (3 * sizeof(int) + sizeof(float));
}
int chem_max_blocks_per_sm(int nsims) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_chem, 256, chem_shared_bytes(nsims));
    return n;
}
cudaError_t launch_chem(const ChemArgs &a, int blocks, Sink &to) {
    return enqueue(to, k_chem, blocks, 256, chem_shared_bytes(a.nsims), a);
}
cudaError_t launch_probe_pixvec(int level, long long p0, long long n, int32_t *out, cudaStream_t st) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_probe_pixvec<<<blocks, 256, 0, st>>>(level, p0, n, out);
    return cudaGetLastError();
}
cudaError_t launch_probe_rates(long long n, const float *T, float *out, cudaStream_t st) {
    const int blocks = (int)std::min<long long>((n + 255) / 256, 1024);
    k_probe_rates<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(n, T, out);
    return cudaGetLastError();
}
cudaError_t launch_probe_rotation(uint64_t seed, long long e, long long s, int rotate, int32_t *out, cudaStream_t st) {
    k_probe_rotation<<<1, 1, 0, st>>>(seed, e, s, rotate, out);
    return cudaGetLastError();
}
cudaError_t launch_probe_direction(int level, long long p0, long long n, const int32_t *Rq, const int4 *tab, int ltab,
                                   int32_t *out, cudaStream_t st) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_probe_direction<<<blocks, 256, 0, st>>>(level, p0, n, Rq, tab, ltab, out);
    return cudaGetLastError();
}
cudaError_t launch_probe_traverse(long long n, const long long *p0, const int32_t *d, int gx, int gy, int gz,
                                  int32_t *cells, float *ds, int32_t *nseg, int32_t *esc, cudaStream_t st) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_probe_traverse<<<blocks, 256, 0, st>>>(n, p0, d, gx, gy, gz, cells, ds, nseg, esc);
    return cudaGetLastError();
}

}  // namespace frt
