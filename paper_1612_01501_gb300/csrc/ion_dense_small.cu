// ion_dense_small.cu -- a small dense network stepped by one CTA: many steps per launch, one
// barrier per step (ION_FLAG_PERSISTENT, at most DENSE_SMALL cells).
//
// A step of such a network is a latency chain: V_dend -> pair sums -> gap current -> V_dend.
// Only the new V_dend needs the current; every gate, the soma, the axon and [Ca] need step-t
// values alone.  So the CTA's warps split: the pair warps (LANES lanes per cell) sum the pairs
// and finish V_dend, [Ca] and the dendritic currents, while the role warps run the rest, one
// role of 32 cells per warp and turn (about the same SFU work each).  The state lives in
// shared memory twice: everyone reads the words of step t and writes those of step t + 1, so
// one barrier separates the steps.  The functions are those of cell_step, so a cell with a
// given current gets the same bits; the currents are summed as in ion_dense.cu (centred,
// scaled, the linear part in closed form), in a fixed order: chains of four terms, folded with
// compensation every 16 columns of a lane.
//
// What bounds it: the chain (0.48 us per step with one cell) and then the instructions of one
// SM (0.54 at 32 cells, 0.86 at 64, 1.5 at 128, 2.7 at 192).  The tiled kernel with one CTA (six
// barriers, the update one thread per cell after the sums, pulses read in each step) took 2.1 at
// 64 cells.  Above 192 cells the pair warps leave too few for the roles and the network is
// better spread over the chip (the per-step launches take 2.5 us there, a grid barrier 4.4).
#include <cuda_runtime.h>

#include <algorithm>

#include "ion_dense_core.cuh"
#include "ion_kernels.cuh"

namespace ion {

constexpr int LANES = 4;        // lanes per cell in the pair warps
constexpr int BLOCK = 4;        // groups of four columns between compensated folds
constexpr int SMALL_ROLES = 8;
constexpr int SMALL_MAX_THREADS = 1024;

constexpr int LD = DENSE_SMALL; // word w of cell i at [w * LD + i]: fixed, so that addresses are immediates

// Role r of one cell: words of step t in cs, outputs into ns and, on the launch's last step,
// the output-only words into global memory.  (cs and ns point at the cell's word 0.)
__device__ __forceinline__ void small_role(int role, const PersistArgs &a, const float *cs, float *ns, int i, int64_t t,
                                           bool last) {
    const StepCommon &c = a.c;
    const ModelF &P = c.P;
    const float dt = P.dt;
    auto in = [&](int w) { return cs[w * LD]; };
    auto out = [&](int w, float v) { ns[w * LD] = v; };
    // words: 0 vd 1 vs 2 va 3 ca 4 r 5 s 6 q 7 k 8 l 9 hs 10 ns 11 xs 12 ha 13 xa 14 gcal
    switch (role) {
        case 0: out(4, relax(in(4), rate_r(in(0)), dt)); break;
        case 1:
            out(6, relax(in(6), rate_q(in(0)), dt));
            out(7, relax(in(7), rate_k(in(1)), dt));
            break;
        case 2: out(8, relax(in(8), rate_l(in(1)), dt)); break;
        case 3:
            out(9, relax(in(9), rate_hs(in(1)), dt));
            out(10, relax(in(10), rate_ns(in(1)), dt));
            break;
        case 4: out(11, relax(in(11), rate_x(in(1)), dt)); break;
        case 5: out(13, relax(in(13), rate_x(in(2)), dt)); break;
        case 6: {
            Cell cell{};
            cell.vs = in(1);
            cell.va = in(2);
            cell.ha = in(12);
            cell.xa = in(13);
            const float ma = minf_na(cell.va), va = axon_step(P, cell, ma);
            out(2, va);
            out(12, relax(cell.ha, rate_ha(cell.va), dt));
            if (last) c.S.f(F_MA)[i] = ma;
            if (!isfinite(va)) atomicOr(c.status, (uint32_t)ST_NONFINITE);
            if (c.trace != nullptr && ((t + 1) % c.trace_stride) == 0) {
                const int64_t sample = (t + 1) / c.trace_stride - 1;
                c.trace[(sample % c.trace_cap) * (int64_t)c.n + i] = va;
            }
            break;
        }
        default: {
            Cell cell{};
            cell.vd = in(0);
            cell.vs = in(1);
            cell.va = in(2);
            cell.k = in(7);
            cell.l = in(8);
            cell.hs = in(9);
            cell.ns = in(10);
            cell.xs = in(11);
            cell.gcal = in(14);
            const float ms = minf_na(cell.vs), vs = soma_step(P, cell, ms);
            out(1, vs);
            if (last) c.S.f(F_MS)[i] = ms;
            if (!isfinite(vs)) atomicOr(c.status, (uint32_t)ST_NONFINITE);
            break;
        }
    }
}

__global__ void __launch_bounds__(SMALL_MAX_THREADS) dense_small_kernel(const PersistArgs a, int pair_warps) {
    extern __shared__ __align__(16) float sd_smem[];
    const StepCommon &c = a.c;
    const int n = c.n, n4 = (n + 3) >> 2;
    const int tail = (n & 3) ? n4 - 1 : -1;     // the group of four columns that is not all real
    float *const buf = sd_smem;                 // [2][NCW][LD]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = *c.t_dev;
    for (int q = threadIdx.x; q < NCW * LD; q += blockDim.x) {
        const int w = q / LD, i = q - w * LD;
        // past the last cell: the sentinel in V_dend of both copies, never written again
        float v = PAD_VOLT;
        if (i < n) v = w == 0 ? vd_slot(c.S, t0)[i] : c.S.f(cell_word_field(w))[i];
        buf[q] = v;
        buf[NCW * LD + q] = v;                  // g_CaL (and the sentinels) stay as they are
    }
    // a pair thread's cell, its share of the columns and its pulse
    const int i = threadIdx.x / LANES, li = threadIdx.x & (LANES - 1);
    const bool pair = warp < pair_warps, mine = pair && i < n;
    const PulseAhead pa = pulse_ahead(c.pulses, i, mine);
    const int blocks = (n + 31) >> 5, role_warps = (blockDim.x >> 5) - pair_warps;
    if (a.debug_delay_ns > 0 && threadIdx.x == 0) {
        const uint64_t d0 = globaltimer_ns();
        while (globaltimer_ns() - d0 < (uint64_t)a.debug_delay_ns) __nanosleep(1000);
    }
    __syncthreads();
    const float2 negs2 = make_float2(-GJ_SCALE, -GJ_SCALE);
    for (int k = 0; k < a.n_steps; ++k) {
        const float *cs = buf + (k & 1) * (NCW * LD);
        float *ns = buf + ((k & 1) ^ 1) * (NCW * LD);
        const int64_t t = t0 + k;
        const bool last = k + 1 == a.n_steps;
        if (pair) {
            const int r = min(i, n - 1);        // lanes without a cell follow the last one
            Cell cell{};
            cell.vd = cs[r];
            cell.vs = cs[1 * LD + r];
            cell.ca = cs[3 * LD + r];
            cell.r = cs[4 * LD + r];
            cell.s = cs[5 * LD + r];
            cell.q = cs[6 * LD + r];
            const float C = cs[0] * GJ_SCALE, u = gj_u(cell.vd, C);
            const float2 c2 = make_float2(C, C), u2 = make_float2(u, u);
            float S = 0.0f, Sc = 0.0f;          // the pairs' sum
            float X = 0.0f, Xc = 0.0f;          // sum of this lane's real x_j = -u_j
            for (int m0 = li; m0 < n4; m0 += BLOCK * LANES) {
                float2 ga = make_float2(0.0f, 0.0f), gb = ga, xs = ga;
#pragma unroll
                for (int q = 0; q < BLOCK; ++q) {
                    const int m = m0 + q * LANES;
                    if (m >= n4) break;
                    const float4 v = reinterpret_cast<const float4 *>(cs)[m];
                    float2 xa = __ffma2_rn(make_float2(v.x, v.y), negs2, c2);
                    float2 xb = __ffma2_rn(make_float2(v.z, v.w), negs2, c2);
                    const float2 da = __fadd2_rn(u2, xa), db = __fadd2_rn(u2, xb);
                    const float2 qa = __fmul2_rn(da, da), qb = __fmul2_rn(db, db);
                    ga = __ffma2_rn(make_float2(ex2_approx(-qa.x), ex2_approx(-qa.y)), da, ga);
                    gb = __ffma2_rn(make_float2(ex2_approx(-qb.x), ex2_approx(-qb.y)), db, gb);
                    if (m == tail) {            // the sentinels are no part of it
                        if ((n & 3) < 2) xa.y = 0.0f;
                        if ((n & 3) < 3) xb.x = 0.0f;
                        xb.y = 0.0f;
                    }
                    xs = __fadd2_rn(xs, __fadd2_rn(xa, xb));
                }
                kahan_add(S, Sc, (ga.x + ga.y) + (gb.x + gb.y));
                kahan_add(X, Xc, xs.x + xs.y);
            }
            S -= Sc;
            X -= Xc;
#pragma unroll
            for (int off = LANES / 2; off > 0; off >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, off);
                X += __shfl_xor_sync(0xffffffffu, X, off);
            }
            const float ic = a.g * (1.0f / GJ_SCALE) * fmaf(0.8f, S, 0.2f * fmaf((float)n, u, X));
            const DendNext d = dend_step(c.P, cell, ic, pulse_current(c.pulses, pa, t));
            if (mine && li == 0) {
                ns[r] = d.vd;
                ns[3 * LD + r] = d.ca;
                ns[5 * LD + r] = relax(cell.s, rate_s(cell.ca), c.P.dt);
                if (last) {
                    c.S.f(F_ICAH)[r] = d.icah;
                    c.S.f(F_IC)[r] = ic;
                }
                if (!(isfinite(d.vd) && isfinite(d.ca))) atomicOr(c.status, (uint32_t)ST_NONFINITE);
            }
        } else {
            for (int q = warp - pair_warps; q < SMALL_ROLES * blocks; q += role_warps) {
                const int cell = (q / SMALL_ROLES) * 32 + lane;
                if (cell < n) small_role(q % SMALL_ROLES, a, cs + cell, ns + cell, cell, t, last);
            }
        }
        __syncthreads();
    }
    // the words of step t0 + n_steps back to global memory (g_CaL does not change)
    const float *fin = buf + (a.n_steps & 1) * (NCW * LD);
    float *vfin = vd_slot(c.S, t0 + a.n_steps);
    for (int q = threadIdx.x; q < (NCW - 1) * LD; q += blockDim.x) {
        const int w = q / LD, r = q - w * LD;
        if (r < n) (w == 0 ? vfin : c.S.f(cell_word_field(w)))[r] = fin[q];
    }
}

cudaError_t launch_dense_small(const PersistArgs &a, cudaStream_t st) {
    const int pair_warps = (a.c.n * LANES + 31) / 32, blocks = (a.c.n + 31) / 32;
    const int role_warps = std::min(SMALL_ROLES * blocks, SMALL_MAX_THREADS / 32 - pair_warps);
    if (role_warps < 1) return cudaErrorInvalidValue;
    const size_t smem = 2 * (size_t)NCW * LD * sizeof(float);
    return launch_k(dense_small_kernel, dim3(1), dim3(32 * (pair_warps + role_warps)), smem, st, false, a, pair_warps);
}

}  // namespace ion
