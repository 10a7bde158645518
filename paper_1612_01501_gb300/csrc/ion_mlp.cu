// ion_mlp.cu -- learned surrogate of the channel rate functions (not in the paper).
//
// A small MLP, (V, [Ca]) -> 64 tanh -> 64 tanh -> 24 outputs, stands in for the gates'
// rate functions: output 2g is logit(x_inf) of gate g (clipped to +-LOGIT_MAX), output 2g+1
// is ln(tau) (the instantaneous gates m_s, m_a have no tau; that output is masked out of
// the loss).  The logit keeps small steady states (m_inf^3 of the Na channels near rest)
// accurate in relative terms; a first fit of x_inf itself made resting cells fire.  Inputs
// and outputs are normalised (shift / scale kept with the weights).
//
// Training (ion_surrogate_train): samples V uniform in [v_lo, v_hi] and [Ca] log-uniform
// are drawn on the device (splitmix64 in counter form, Steele-Lea-Flood 2014), labelled
// by the exact FP32 rate functions of ion_model.cuh, and fitted by minibatch Adam.  Each
// minibatch is one launch of mlp_fwdbwd_kernel (forward and backward in FP32; activations
// and deltas to an L2-resident buffer) and one of mlp_wgrad_kernel (the gradient of every
// parameter over 128-sample groups, the groups added in a fixed order, then the Adam step on
// FP32 master weights), so training is deterministic.
//
// Inference runs on the tensor cores, BF16 weights and activations with FP32 accumulation:
// by default on tcgen05 with TMEM accumulators (ion_mlp_tc.cu: ion_surrogate_eval and the
// cell update); with ION_FLAG_SURROGATE_WARP_MMA the cell update below uses mma.sync
// m16n8k16 instead (kept for comparison).  Layer 1 (two
// inputs) is FP32 FMAs; the 64x64 and 64x24 layers are MMAs whose accumulator fragments
// become the next layer's A fragments in registers; tanh runs on packed bf16 pairs.
// The cell kernel evaluates one row per (cell, compartment) -- 96 rows per warp for 32
// cells -- then each lane runs the explicit-Euler update of one cell with those rates.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "ion.h"
#include "ion_kernels.cuh"
#include "ion_sim.h"

namespace ion {

constexpr int MI = ION_MLP_IN, MH = ION_MLP_HID, MO = ION_MLP_OUT;
constexpr int P_W1 = 0, P_B1 = P_W1 + MH * MI, P_W2 = P_B1 + MH, P_B2 = P_W2 + MH * MH, P_W3 = P_B2 + MH,
              P_B3 = P_W3 + MO * MH, P_TOTAL = P_B3 + MO;   // 5912 parameters, the order of ion_surrogate_weights
constexpr int MB = 128;                                      // samples per partial sum in training
constexpr float V_CENTER = -25.0f, V_HALF = 75.0f;
constexpr float LOGIT_MAX = 15.0f;

// ---- counter-based generator (splitmix64) --------------------------------------------
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ double sm64_uniform(uint64_t seed, uint64_t k) {
    return (double)(sm64_mix(seed + (k + 1) * 0x9E3779B97F4A7C15ull) >> 11) * (1.0 / 9007199254740992.0);
}

// ---- data: samples, exact targets, normalisation ---------------------------------------
__global__ void mlp_samples_kernel(int64_t n, uint64_t seed, float v_lo, float v_hi, float lc_lo, float lc_hi, float *V,
                                   float *ca) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint64_t sa = sm64_mix(seed + 0x9E3779B97F4A7C15ull), sb = sm64_mix(seed + 2 * 0x9E3779B97F4A7C15ull);
    V[k] = (float)(v_lo + (v_hi - v_lo) * sm64_uniform(sa, (uint64_t)k));
    ca[k] = (float)exp(lc_lo + (lc_hi - lc_lo) * sm64_uniform(sb, (uint64_t)k));
}

// raw targets of one (V, ca): logit(x_inf) and ln(tau) of every gate (ln tau = 0 for the
// instantaneous ones)
__device__ __forceinline__ void exact_targets(float V, float ca, float *out) {
    const Rate g[NG] = {rate_r(V), rate_s(ca), rate_q(V), rate_k(V), rate_l(V), {minf_na(V), 0.0f},
                        rate_hs(V), rate_ns(V), rate_x(V), {minf_na(V), 0.0f}, rate_ha(V), rate_x(V)};
    for (int k = 0; k < NG; ++k) {
        const float x = fminf(fmaxf(g[k].xinf, 1e-30f), 1.0f);
        const float lg = logf(x) - log1pf(-fminf(x, 1.0f - 1e-7f));
        out[2 * k] = fminf(fmaxf(lg, -LOGIT_MAX), LOGIT_MAX);
        out[2 * k + 1] = g[k].inv_tau > 0.0f ? -logf(g[k].inv_tau) : 0.0f;
    }
}

__global__ void mlp_targets_kernel(int64_t n, const float *V, const float *ca, float *T) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float o[MO];
    exact_targets(V[k], ca[k], o);
    for (int j = 0; j < MO; ++j) T[k * MO + j] = o[j];
}

// per-output sums of t and t^2 (double) over a block's share of the samples
__global__ void mlp_stats_kernel(int64_t n, const float *T, double *partial) {
    __shared__ double s1[256], s2[256];
    const int o = blockIdx.y;
    double a = 0.0, b = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const double t = T[k * MO + o];
        a += t;
        b += t * t;
    }
    s1[threadIdx.x] = a;
    s2[threadIdx.x] = b;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            s1[threadIdx.x] += s1[threadIdx.x + w];
            s2[threadIdx.x] += s2[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[((int64_t)o * gridDim.x + blockIdx.x) * 2] = s1[0];
        partial[((int64_t)o * gridDim.x + blockIdx.x) * 2 + 1] = s2[0];
    }
}

// shift = mean, scale = std (>= 1e-3) per output; masked outputs keep (0, 1)
__global__ void mlp_stats_final_kernel(int64_t n, int nblocks, const double *partial, const float *mask, float *shift,
                                       float *scale) {
    const int o = threadIdx.x;
    if (o >= MO) return;
    double a = 0.0, b = 0.0;
    for (int i = 0; i < nblocks; ++i) {
        a += partial[((int64_t)o * nblocks + i) * 2];
        b += partial[((int64_t)o * nblocks + i) * 2 + 1];
    }
    const double mean = a / (double)n;
    const double var = fmax(b / (double)n - mean * mean, 0.0);
    if (mask[o] == 0.0f) {
        shift[o] = 0.0f;
        scale[o] = 1.0f;
    } else {
        shift[o] = (float)mean;
        scale[o] = (float)fmax(sqrt(var), 1e-3);
    }
}

__global__ void mlp_normalise_kernel(int64_t n, const float *V, const float *ca, float lc_mid, float lc_half,
                                     const float *shift, const float *scale, float *X, float *T) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    X[2 * k] = (V[k] - V_CENTER) / V_HALF;
    X[2 * k + 1] = (logf(ca[k]) - lc_mid) / lc_half;
    for (int j = 0; j < MO; ++j) T[k * MO + j] = (T[k * MO + j] - shift[j]) / scale[j];
}

// ---- training: one minibatch in two launches ------------------------------------------------
// Samples of the minibatch: local index j in [0, B) maps to sample (mul * (j0 + j) + add) mod n
// (a bijection when gcd(mul, n) = 1: a cheap per-epoch reshuffle).
//
// The arithmetic of a minibatch is small (0.07 GFLOP at B = 1024) and its sums have a fixed
// order, so the time is the latency of the dependent chains and the point is to have many of
// them in flight.  The forward / backward launch takes GS = 8 samples per CTA (128 CTAs at
// B = 1024), a thread per (sample pair, hidden unit), each dot product one 64-step chain; it
// leaves the activations and the deltas in L2, one row per unit.  The gradient launch gives
// every parameter and every 128-sample group a chain of its own: a CTA stages 8 activation and
// 8 delta rows of up to 8 groups (64 KB, one round of 16-byte async copies) and holds two chains per
// thread; it adds the groups in order and takes the Adam step.  One sample per
// thread, 128 samples per CTA (8 CTAs at B = 1024) and the gradients in the same kernel
// measured 75 us per minibatch of 1024; this split 14.8 us (fwd / bwd 4.3 and gradients 5.5
// when each runs alone; the rest is the first read of what the other launch just wrote), with
// every sum in the same order, so the weights are the same bits.
constexpr int GS = 8;             // samples per CTA of the forward / backward launch
constexpr int WP = MH + 4;        // row stride of the weight copies: conflict-free 16-byte rows
constexpr int VEC_PARAMS = MH * MI + MH + MH + MO + 1;   // W1, b1, b2, b3 and the loss
constexpr int WG_GROUPS = 8;      // 128-sample groups in flight per CTA of the gradient launch
constexpr int WG_TILE = 8;        // a W2 / W3 gradient tile is 8 x 8 parameters
constexpr int WG_TILES2 = (MH / WG_TILE) * (MH / WG_TILE), WG_TILES3 = (MO / WG_TILE) * (MH / WG_TILE);
constexpr int WG_VEC = 16;        // of the other parameters per CTA
constexpr int WG_CTAS = WG_TILES2 + WG_TILES3 + (VEC_PARAMS + WG_VEC - 1) / WG_VEC;
constexpr int WG_GSTRIDE = MB + 4, WG_STRIDE = WG_GROUPS * WG_GSTRIDE + 4;   // staged group and row strides: distinct banks

struct GradArgs {
    const float *params;   // P_TOTAL
    const float *X;        // n x 2 normalised inputs
    const float *T;        // n x 24 normalised targets
    const float *mask;     // 24
    int64_t n;
    int64_t j0;
    int32_t B;
    uint64_t mul, add;
    float denom;           // B * sum(mask)
    int64_t rows;          // B rounded up to whole groups of MB samples (rows past B hold zeros)
    float *work;           // mlp_work_floats(rows): the arrays below, one after the other
};
// activations and deltas [unit][rows], inputs [2][rows], loss [rows]
__device__ __forceinline__ float *wk_h1(const GradArgs &a) { return a.work; }
__device__ __forceinline__ float *wk_h2(const GradArgs &a) { return a.work + a.rows * MH; }
__device__ __forceinline__ float *wk_d1(const GradArgs &a) { return a.work + a.rows * (2 * MH); }
__device__ __forceinline__ float *wk_d2(const GradArgs &a) { return a.work + a.rows * (3 * MH); }
__device__ __forceinline__ float *wk_d3(const GradArgs &a) { return a.work + a.rows * (4 * MH); }
__device__ __forceinline__ float *wk_x(const GradArgs &a) { return a.work + a.rows * (4 * MH + MO); }
__device__ __forceinline__ float *wk_loss(const GradArgs &a) { return a.work + a.rows * (4 * MH + MO + MI); }
static size_t mlp_work_floats(int64_t rows) { return (size_t)rows * (4 * MH + MO + MI + 1); }

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
// the 64 threads (two warps) that share a sample pair
__device__ __forceinline__ void pair_sync(int sg) { asm volatile("bar.sync %0, 64;" ::"r"(sg + 1) : "memory"); }

// Forward and backward of GS samples: 256 threads, thread (sg, u) has unit u of samples 2 sg, 2 sg + 1.
__global__ void __launch_bounds__(256) mlp_fwdbwd_kernel(const GradArgs a) {
    __shared__ __align__(16) float w2s[MH * WP], w3s[MO * WP];
    __shared__ __align__(16) float w1s[MH * MI], b1s[MH], b2s[MH], b3s[MO];
    __shared__ __align__(16) float h1[GS][MH], h2[GS][MH], d1[GS][MH], d2[GS][MH], d3[GS][MO], es[GS][MO];
    const int tid = threadIdx.x, u = tid & 63, sg = tid >> 6;
    const int64_t row0 = (int64_t)blockIdx.x * GS + 2 * sg;
    // the samples are constant data: read before the wait on the previous minibatch
    float x0[2], x1[2];
    bool valid[2];
    int64_t k[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        valid[r] = row0 + r < a.B;
        k[r] = valid[r] ? (int64_t)((a.mul * (uint64_t)(a.j0 + row0 + r) + a.add) % (uint64_t)a.n) : 0;
        x0[r] = valid[r] ? a.X[2 * k[r]] : 0.0f;
        x1[r] = valid[r] ? a.X[2 * k[r] + 1] : 0.0f;
    }
    const int so = u / MO, o = u - so * MO;   // layer 3: threads u < 48 have output o of sample 2 sg + so
    const bool out3 = u < 2 * MO;
    const bool vo = so == 0 ? valid[0] : valid[1];
    const float tgt = out3 && vo ? a.T[(so == 0 ? k[0] : k[1]) * MO + o] : 0.0f;
    const float msk = out3 ? a.mask[o] : 0.0f;
    pdl_enter();
    for (int i = tid; i < MH * MH / 4; i += 256)
        cp_async16(w2s + (i >> 4) * WP + 4 * (i & 15), a.params + P_W2 + 4 * i);
    for (int i = tid; i < MO * MH / 4; i += 256)
        cp_async16(w3s + (i >> 4) * WP + 4 * (i & 15), a.params + P_W3 + 4 * i);
    if (tid < MH * MI / 4) cp_async16(w1s + 4 * tid, a.params + P_W1 + 4 * tid);
    else if (tid < MH * MI / 4 + MH / 4) cp_async16(b1s + 4 * (tid - 32), a.params + P_B1 + 4 * (tid - 32));
    else if (tid < MH * MI / 4 + MH / 2) cp_async16(b2s + 4 * (tid - 48), a.params + P_B2 + 4 * (tid - 48));
    else if (tid < MH * MI / 4 + MH / 2 + MO / 4) cp_async16(b3s + 4 * (tid - 64), a.params + P_B3 + 4 * (tid - 64));
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();
    const int s0 = 2 * sg;
    float h1v[2], h2v[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        h1v[r] = tanhf(fmaf(w1s[2 * u], x0[r], fmaf(w1s[2 * u + 1], x1[r], b1s[u])));
        h1[s0 + r][u] = h1v[r];
    }
    pair_sync(sg);
    {
        float a0 = b2s[u], a1 = a0;
#pragma unroll
        for (int q = 0; q < MH; q += 4) {
            const float4 w = *reinterpret_cast<const float4 *>(w2s + u * WP + q);
            const float4 p = *reinterpret_cast<const float4 *>(&h1[s0][q]);
            const float4 v = *reinterpret_cast<const float4 *>(&h1[s0 + 1][q]);
            a0 = fmaf(w.w, p.w, fmaf(w.z, p.z, fmaf(w.y, p.y, fmaf(w.x, p.x, a0))));
            a1 = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, a1))));
        }
        h2v[0] = tanhf(a0);
        h2v[1] = tanhf(a1);
        h2[s0][u] = h2v[0];
        h2[s0 + 1][u] = h2v[1];
    }
    pair_sync(sg);
    if (out3) {
        float acc = b3s[o];
#pragma unroll
        for (int q = 0; q < MH; q += 4) {
            const float4 w = *reinterpret_cast<const float4 *>(w3s + o * WP + q);
            const float4 p = *reinterpret_cast<const float4 *>(&h2[s0 + so][q]);
            acc = fmaf(w.w, p.w, fmaf(w.z, p.z, fmaf(w.y, p.y, fmaf(w.x, p.x, acc))));
        }
        const float e = vo ? (acc - tgt) * msk : 0.0f;
        es[s0 + so][o] = e;
        d3[s0 + so][o] = 2.0f * e / a.denom;
    }
    pair_sync(sg);
    {
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int q = 0; q < MO; q += 4) {
            const float4 p = *reinterpret_cast<const float4 *>(&d3[s0][q]);
            const float4 v = *reinterpret_cast<const float4 *>(&d3[s0 + 1][q]);
            const float wa = w3s[q * WP + u], wb = w3s[(q + 1) * WP + u], wc = w3s[(q + 2) * WP + u],
                        wd = w3s[(q + 3) * WP + u];
            a0 = fmaf(wd, p.w, fmaf(wc, p.z, fmaf(wb, p.y, fmaf(wa, p.x, a0))));
            a1 = fmaf(wd, v.w, fmaf(wc, v.z, fmaf(wb, v.y, fmaf(wa, v.x, a1))));
        }
        d2[s0][u] = a0 * (1.0f - h2v[0] * h2v[0]);
        d2[s0 + 1][u] = a1 * (1.0f - h2v[1] * h2v[1]);
    }
    if (u < 2) {   // the sample's loss, in output order
        float loss = 0.0f;
#pragma unroll
        for (int q = 0; q < MO; ++q) loss = fmaf(es[s0 + u][q], es[s0 + u][q], loss);
        wk_loss(a)[row0 + u] = loss;
        wk_x(a)[row0 + u] = u == 0 ? x0[0] : x0[1];
        wk_x(a)[a.rows + row0 + u] = u == 0 ? x1[0] : x1[1];
    }
    pair_sync(sg);
    {
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int q = 0; q < MH; q += 4) {
            const float4 p = *reinterpret_cast<const float4 *>(&d2[s0][q]);
            const float4 v = *reinterpret_cast<const float4 *>(&d2[s0 + 1][q]);
            const float wa = w2s[q * WP + u], wb = w2s[(q + 1) * WP + u], wc = w2s[(q + 2) * WP + u],
                        wd = w2s[(q + 3) * WP + u];
            a0 = fmaf(wd, p.w, fmaf(wc, p.z, fmaf(wb, p.y, fmaf(wa, p.x, a0))));
            a1 = fmaf(wd, v.w, fmaf(wc, v.z, fmaf(wb, v.y, fmaf(wa, v.x, a1))));
        }
        d1[s0][u] = a0 * (1.0f - h1v[0] * h1v[0]);
        d1[s0 + 1][u] = a1 * (1.0f - h1v[1] * h1v[1]);
    }
    __syncthreads();
    // a unit's 8 samples are one 32-byte sector of its row: two 16-byte stores, so that every
    // sector is written once and whole (8-byte stores of each thread's own pair: 15.5 us per
    // minibatch of 1024 instead of 14.8)
    const int half = 4 * (tid & 1), unit = (tid >> 1) & 63;
    const int64_t at = (int64_t)blockIdx.x * GS + half;
    auto put = [&](float *dst, const float *src, int stride) {   // src: the unit's column, sample-major
        *reinterpret_cast<float4 *>(dst + unit * a.rows + at) =
            make_float4(src[half * stride], src[(half + 1) * stride], src[(half + 2) * stride], src[(half + 3) * stride]);
    };
    if (tid < 128) {
        put(wk_h1(a), &h1[0][unit], MH);
        put(wk_h2(a), &h2[0][unit], MH);
        if (unit < MO) put(wk_d3(a), &d3[0][unit], MO);
    } else {
        put(wk_d1(a), &d1[0][unit], MH);
        put(wk_d2(a), &d2[0][unit], MH);
    }
}

struct AdamArgs {
    GradArgs g;
    float *params, *m, *v;
    float *grad;           // non-NULL: return the gradient, no Adam step
    float lr, b1, b2, eps, c1, c2;
    float *loss;           // non-NULL: += loss sum / denom
};

// sum over a group's samples of d times h, in sample order, and the plain sum
__device__ __forceinline__ float group_dot(const float *d, const float *h) {
    float acc = 0.0f;
#pragma unroll 16
    for (int t = 0; t < MB; t += 4) {
        const float4 dd = *reinterpret_cast<const float4 *>(d + t), hh = *reinterpret_cast<const float4 *>(h + t);
        acc = fmaf(dd.w, hh.w, fmaf(dd.z, hh.z, fmaf(dd.y, hh.y, fmaf(dd.x, hh.x, acc))));
    }
    return acc;
}
__device__ __forceinline__ float group_sum(const float *d) {
    float acc = 0.0f;
#pragma unroll 16
    for (int t = 0; t < MB; t += 4) {
        const float4 dd = *reinterpret_cast<const float4 *>(d + t);
        acc += dd.x;
        acc += dd.y;
        acc += dd.z;
        acc += dd.w;
    }
    return acc;
}

// one 4-sample step of a chain
__device__ __forceinline__ float dot4(float4 d, float4 h, float acc) {
    return fmaf(d.w, h.w, fmaf(d.z, h.z, fmaf(d.y, h.y, fmaf(d.x, h.x, acc))));
}

// Gradients and the Adam step: a warp per group, lane (1 x 2 parameters of the tile, or one of
// the others).  CTAs 0..63 own an 8 x 8 tile of W2 each, 64..87 one of W3, the rest 16 of the
// other parameters (and the loss) each.
__global__ void __launch_bounds__(32 * WG_GROUPS) mlp_wgrad_kernel(const AdamArgs a) {
    extern __shared__ __align__(16) float rows_s[];   // 16 staged rows: 8 deltas, then 8 activations
    __shared__ float part[WG_GROUPS][64];
    const int lt = threadIdx.x & 31, gi = threadIdx.x >> 5, blk = blockIdx.x;
    const int64_t rows = a.g.rows;
    const int nblk = (int)(rows / MB);
    const bool tile = blk < WG_TILES2 + WG_TILES3;
    const bool w2 = blk < WG_TILES2;
    const int tb = w2 ? blk : blk - WG_TILES2;
    const int j0 = tb / (MH / WG_TILE) * WG_TILE, q0 = tb % (MH / WG_TILE) * WG_TILE;
    // this thread's parameter after the groups are added (threads < 64, < 16 of the vector CTAs)
    const int np = tile ? 64 : WG_VEC;
    int p = -1;                    // P_TOTAL: the loss
    if ((int)threadIdx.x < np) {
        if (tile) p = (w2 ? P_W2 : P_W3) + (j0 + (threadIdx.x >> 3)) * MH + q0 + (threadIdx.x & 7);
        else p = (blk - WG_TILES2 - WG_TILES3) * WG_VEC + threadIdx.x;   // list position, mapped below
    }
    const int v = tile || lt >= WG_VEC ? -1 : (blk - WG_TILES2 - WG_TILES3) * WG_VEC + lt;
    auto vec_param = [](int x) {
        if (x < MH * MI) return P_W1 + x;
        if (x < MH * MI + MH) return P_B1 + (x - MH * MI);
        if (x < MH * MI + 2 * MH) return P_B2 + (x - MH * MI - MH);
        if (x < VEC_PARAMS - 1) return P_B3 + (x - MH * MI - 2 * MH);
        return x == VEC_PARAMS - 1 ? P_TOTAL : -1;
    };
    if (!tile && p >= 0) p = vec_param(p);
    const int vp = v < 0 ? -1 : vec_param(v);
    pdl_enter();
    const bool adam = p >= 0 && p < P_TOTAL && a.grad == nullptr;
    const float m0 = adam ? a.m[p] : 0.0f, v0 = adam ? a.v[p] : 0.0f, w0 = adam ? a.params[p] : 0.0f;
    const float *dsrc = w2 ? wk_d2(a.g) : wk_d3(a.g), *hsrc = w2 ? wk_h1(a.g) : wk_h2(a.g);
    float g = 0.0f;
    for (int c0 = 0; c0 < nblk; c0 += WG_GROUPS) {
        const int here = min(WG_GROUPS, nblk - c0);
        if (tile) {
            if (gi < here) {   // this warp's group: lane = 16-byte part of the 128 samples
                const int64_t at = (int64_t)(c0 + gi) * MB + 4 * lt;
                float *dst = rows_s + gi * WG_GSTRIDE + 4 * lt;
#pragma unroll
                for (int r = 0; r < WG_TILE; ++r) {
                    cp_async16(dst + r * WG_STRIDE, dsrc + (j0 + r) * rows + at);
                    cp_async16(dst + (WG_TILE + r) * WG_STRIDE, hsrc + (q0 + r) * rows + at);
                }
            }
            cp_async_commit();
            cp_async_wait_all();
            __syncwarp();      // a warp reads what its own lanes staged
            if (gi < here) {
                const int jj = lt >> 2, qq = 2 * (lt & 3);
                const float *d = rows_s + jj * WG_STRIDE + gi * WG_GSTRIDE,
                            *h = rows_s + (WG_TILE + qq) * WG_STRIDE + gi * WG_GSTRIDE;
                float a0 = 0.0f, a1 = 0.0f;
#pragma unroll 16
                for (int t = 0; t < MB; t += 4) {
                    const float4 dd = *reinterpret_cast<const float4 *>(d + t),
                                 ha = *reinterpret_cast<const float4 *>(h + t),
                                 hb = *reinterpret_cast<const float4 *>(h + WG_STRIDE + t);
                    a0 = dot4(dd, ha, a0);
                    a1 = dot4(dd, hb, a1);
                }
                part[gi][jj * WG_TILE + qq] = a0;
                part[gi][jj * WG_TILE + qq + 1] = a1;
            }
        } else if (gi < here && vp >= 0) {
            const int64_t t0 = (int64_t)(c0 + gi) * MB;
            float acc;
            if (vp == P_TOTAL) acc = group_sum(wk_loss(a.g) + t0);
            else if (vp < P_B1) acc = group_dot(wk_d1(a.g) + (vp >> 1) * rows + t0, wk_x(a.g) + (vp & 1) * rows + t0);
            else if (vp < P_W2) acc = group_sum(wk_d1(a.g) + (vp - P_B1) * rows + t0);
            else if (vp < P_W3) acc = group_sum(wk_d2(a.g) + (vp - P_B2) * rows + t0);
            else acc = group_sum(wk_d3(a.g) + (vp - P_B3) * rows + t0);
            part[gi][lt] = acc;
        }
        __syncthreads();
        if (p >= 0)
            for (int b = 0; b < here; ++b) g += part[b][threadIdx.x];
        __syncthreads();
    }
    if (p < 0) return;
    if (p == P_TOTAL) {
        if (a.loss) *a.loss += g / a.g.denom;
        return;
    }
    if (a.grad) {
        a.grad[p] = g;
        return;
    }
    const float mm = a.b1 * m0 + (1.0f - a.b1) * g;
    const float vv = a.b2 * v0 + (1.0f - a.b2) * g * g;
    a.m[p] = mm;
    a.v[p] = vv;
    a.params[p] = w0 - a.lr * (mm / a.c1) / (sqrtf(vv / a.c2) + a.eps);
}

constexpr size_t WG_SMEM = 2 * WG_TILE * WG_STRIDE * sizeof(float);
static cudaError_t prepare_minibatch() {
    return cudaFuncSetAttribute(mlp_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WG_SMEM);
}
static cudaError_t launch_minibatch(const AdamArgs &a, bool pdl, cudaStream_t st) {
    cudaError_t e = launch_k(mlp_fwdbwd_kernel, dim3((unsigned)(a.g.rows / GS)), dim3(256), 0, st, pdl, a.g);
    if (e == cudaSuccess) e = launch_k(mlp_wgrad_kernel, dim3(WG_CTAS), dim3(32 * WG_GROUPS), WG_SMEM, st, true, a);
    return e;
}

// Glorot-uniform weights from the counter-based generator, zero biases
__global__ void mlp_init_kernel(float *params, uint64_t seed) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P_TOTAL) return;
    float a = 0.0f;
    if (p < P_B1) a = sqrtf(6.0f / (MI + MH));
    else if (p >= P_W2 && p < P_B2) a = sqrtf(6.0f / (MH + MH));
    else if (p >= P_W3 && p < P_B3) a = sqrtf(6.0f / (MH + MO));
    params[p] = a == 0.0f ? 0.0f : (float)((2.0 * sm64_uniform(sm64_mix(seed + 3), (uint64_t)p) - 1.0) * a);
}

// ---- inference on the tensor cores ---------------------------------------------------------
// Device copy of a surrogate for inference: FP32 first layer, biases and normalisation;
// BF16 64x64 and 64x24 weights with rows padded to 72 (conflict-free fragment loads).
constexpr int WS = 72;
struct MlpDev {
    float w1[MH * MI], b1[MH], b2[MH], b3[MO];
    float in_shift[MI], in_scale[MI], out_shift[MO], out_scale[MO];
    __nv_bfloat16 w2[MH * WS], w3[MO * WS];
};

__global__ void mlp_pack_kernel(const ion_surrogate_weights *w, MlpDev *d) {
    const int tid = threadIdx.x;
    for (int i = tid; i < MH * MI; i += blockDim.x) d->w1[i] = w->w1[i];
    for (int i = tid; i < MH; i += blockDim.x) {
        d->b1[i] = w->b1[i];
        d->b2[i] = w->b2[i];
    }
    for (int i = tid; i < MO; i += blockDim.x) {
        d->b3[i] = w->b3[i];
        d->out_shift[i] = w->out_shift[i];
        d->out_scale[i] = w->out_scale[i];
    }
    if (tid < MI) {
        d->in_shift[tid] = w->in_shift[tid];
        d->in_scale[tid] = w->in_scale[tid];
    }
    for (int i = tid; i < MH * WS; i += blockDim.x) {
        const int r = i / WS, c = i % WS;
        d->w2[i] = __float2bfloat16_rn(c < MH ? w->w2[r * MH + c] : 0.0f);
    }
    for (int i = tid; i < MO * WS; i += blockDim.x) {
        const int r = i / WS, c = i % WS;
        d->w3[i] = __float2bfloat16_rn(c < MH ? w->w3[r * MH + c] : 0.0f);
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}
__device__ __forceinline__ uint32_t tanh_bf16x2(uint32_t x) {
    uint32_t y;
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One warp evaluates 16 rows (one m-tile).  in0/in1: normalised inputs of rows g and g+8
// (g = lane / 4).  y[nt][0..3]: outputs (row g: cols 8nt + 2t, +1; row g+8: same), t = lane % 4.
__device__ __forceinline__ void mlp_mtile(const MlpDev &W, float a0, float a1, float c0, float c1, float (&y)[3][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // layer 1 (FP32 FMAs) -> tanh on bf16 pairs -> A fragments of layer 2
    uint32_t A[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const int cA = 16 * kk + 2 * t, cB = cA + 8;
        const float zg0 = fmaf(W.w1[2 * cA], a0, fmaf(W.w1[2 * cA + 1], a1, W.b1[cA]));
        const float zg1 = fmaf(W.w1[2 * cA + 2], a0, fmaf(W.w1[2 * cA + 3], a1, W.b1[cA + 1]));
        const float z80 = fmaf(W.w1[2 * cA], c0, fmaf(W.w1[2 * cA + 1], c1, W.b1[cA]));
        const float z81 = fmaf(W.w1[2 * cA + 2], c0, fmaf(W.w1[2 * cA + 3], c1, W.b1[cA + 1]));
        const float zg2 = fmaf(W.w1[2 * cB], a0, fmaf(W.w1[2 * cB + 1], a1, W.b1[cB]));
        const float zg3 = fmaf(W.w1[2 * cB + 2], a0, fmaf(W.w1[2 * cB + 3], a1, W.b1[cB + 1]));
        const float z82 = fmaf(W.w1[2 * cB], c0, fmaf(W.w1[2 * cB + 1], c1, W.b1[cB]));
        const float z83 = fmaf(W.w1[2 * cB + 2], c0, fmaf(W.w1[2 * cB + 3], c1, W.b1[cB + 1]));
        A[kk][0] = tanh_bf16x2(pack_bf16x2(zg0, zg1));
        A[kk][1] = tanh_bf16x2(pack_bf16x2(z80, z81));
        A[kk][2] = tanh_bf16x2(pack_bf16x2(zg2, zg3));
        A[kk][3] = tanh_bf16x2(pack_bf16x2(z82, z83));
    }
    // layer 2: 64 x 64 on the tensor cores
    float acc[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float bl = W.b2[8 * nt + 2 * t], bh = W.b2[8 * nt + 2 * t + 1];
        acc[nt][0] = bl;
        acc[nt][1] = bh;
        acc[nt][2] = bl;
        acc[nt][3] = bh;
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const __nv_bfloat16 *row = W.w2 + (8 * nt + g) * WS + 16 * kk + 2 * t;
            mma_bf16(acc[nt], A[kk], *reinterpret_cast<const uint32_t *>(row),
                     *reinterpret_cast<const uint32_t *>(row + 8));
        }
    // tanh -> A fragments of layer 3 (accumulator layout = A layout of the next MMA)
    uint32_t A3[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        A3[kk][0] = tanh_bf16x2(pack_bf16x2(acc[2 * kk][0], acc[2 * kk][1]));
        A3[kk][1] = tanh_bf16x2(pack_bf16x2(acc[2 * kk][2], acc[2 * kk][3]));
        A3[kk][2] = tanh_bf16x2(pack_bf16x2(acc[2 * kk + 1][0], acc[2 * kk + 1][1]));
        A3[kk][3] = tanh_bf16x2(pack_bf16x2(acc[2 * kk + 1][2], acc[2 * kk + 1][3]));
    }
    // layer 3: 64 x 24
#pragma unroll
    for (int nt = 0; nt < 3; ++nt) {
        const int o = 8 * nt + 2 * t;
        y[nt][0] = W.b3[o];
        y[nt][1] = W.b3[o + 1];
        y[nt][2] = W.b3[o];
        y[nt][3] = W.b3[o + 1];
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int nt = 0; nt < 3; ++nt) {
            const __nv_bfloat16 *row = W.w3 + (8 * nt + g) * WS + 16 * kk + 2 * t;
            mma_bf16(y[nt], A3[kk], *reinterpret_cast<const uint32_t *>(row),
                     *reinterpret_cast<const uint32_t *>(row + 8));
        }
    // back to physical units
#pragma unroll
    for (int nt = 0; nt < 3; ++nt) {
        const int o = 8 * nt + 2 * t;
        y[nt][0] = fmaf(y[nt][0], W.out_scale[o], W.out_shift[o]);
        y[nt][1] = fmaf(y[nt][1], W.out_scale[o + 1], W.out_shift[o + 1]);
        y[nt][2] = fmaf(y[nt][2], W.out_scale[o], W.out_shift[o]);
        y[nt][3] = fmaf(y[nt][3], W.out_scale[o + 1], W.out_shift[o + 1]);
    }
}

__device__ __forceinline__ void load_mlp(MlpDev &dst, const MlpDev *src) {
    const int4 *s = reinterpret_cast<const int4 *>(src);
    int4 *d = reinterpret_cast<int4 *>(&dst);
    for (int i = threadIdx.x; i < (int)(sizeof(MlpDev) / 16); i += blockDim.x) d[i] = s[i];
}

// ---- the cell update with learned rates ------------------------------------------------------
// 64 threads; warp w owns CPW = 16 cells [base, base + 16): rows 0..15 dendrite (V_dend,
// [Ca]), 16..31 soma (V_soma, [Ca]), 32..47 axon (V_axon, [Ca]); three m-tiles of 16 rows.
// (16 rather than 32 cells per warp doubles the warps of a launch: the kernel is bound by
// latency, not by the tensor cores.)  Lanes 0..15 then run their cells' updates.
struct SurrArgs {
    StepCommon c;
    const MlpDev *mlp;
    const float *ic;    // gap currents of this step (NULL: none)
};

// x_inf = 1 / (1 + e^{-logit}), 1 / tau = e^{-ln tau}
__device__ __forceinline__ float learned_xinf(const float *y, int gate) {
    return rcp_approx(1.0f + ex2_approx(-y[2 * gate] * 1.4426950408889634f));
}
__device__ __forceinline__ Rate learned_rate(const float *y, int gate) {
    return Rate{learned_xinf(y, gate), ex2_approx(-y[2 * gate + 1] * 1.4426950408889634f)};
}

constexpr int SURR_CPW = 16;   // cells per warp

__global__ void __launch_bounds__(64) surrogate_cell_kernel(const SurrArgs a) {
    __shared__ __align__(16) MlpDev W;
    __shared__ float ys[2][3 * SURR_CPW][MO + 1];
    pdl_enter();
    const StepCommon &c = a.c;
    load_mlp(W, a.mlp);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
    const int64_t base = ((int64_t)blockIdx.x * 2 + warp) * SURR_CPW;
    const int64_t tstep = step_index(c);
    const float *vcur = vd_cur(c);
    float *vnext = vd_next(c);
    __syncthreads();
#pragma unroll 1
    for (int mt = 0; mt < 3; ++mt) {
        const int comp = mt;                 // 0 dendrite, 1 soma, 2 axon
        const int64_t ia = base + g, ib = ia + 8;
        const float *vsrc = comp == 0 ? vcur : c.S.f(comp == 1 ? F_VSOMA : F_VAXON);
        const float va = ia < c.n ? vsrc[ia] : -60.0f, vb = ib < c.n ? vsrc[ib] : -60.0f;
        const float ca_a = ia < c.n ? c.S.f(F_CA)[ia] : 1.0f, ca_b = ib < c.n ? c.S.f(F_CA)[ib] : 1.0f;
        float y[3][4];
        mlp_mtile(W, (va - W.in_shift[0]) * W.in_scale[0], (logf(ca_a) - W.in_shift[1]) * W.in_scale[1],
                  (vb - W.in_shift[0]) * W.in_scale[0], (logf(ca_b) - W.in_shift[1]) * W.in_scale[1], y);
        const int row = comp * SURR_CPW + g;
#pragma unroll
        for (int nt = 0; nt < 3; ++nt) {
            const int o = 8 * nt + 2 * t;
            ys[warp][row][o] = y[nt][0];
            ys[warp][row][o + 1] = y[nt][1];
            ys[warp][row + 8][o] = y[nt][2];
            ys[warp][row + 8][o + 1] = y[nt][3];
        }
    }
    __syncwarp();
    const int64_t i = base + lane;
    if (lane >= SURR_CPW || i >= c.n) return;
    const Cell cell = load_cell(c.S, vcur, i);
    const float *yd = ys[warp][lane], *ysm = ys[warp][SURR_CPW + lane], *yax = ys[warp][2 * SURR_CPW + lane];
    CellRates gr;
    gr.r = learned_rate(yd, G_R);
    gr.s = learned_rate(yd, G_S);
    gr.q = learned_rate(yd, G_Q);
    gr.k = learned_rate(ysm, G_K);
    gr.l = learned_rate(ysm, G_L);
    gr.ms = Rate{learned_xinf(ysm, G_MS), 0.0f};
    gr.hs = learned_rate(ysm, G_HS);
    gr.ns = learned_rate(ysm, G_NS);
    gr.xs = learned_rate(ysm, G_XS);
    gr.ma = Rate{learned_xinf(yax, G_MA), 0.0f};
    gr.ha = learned_rate(yax, G_HA);
    gr.xa = learned_rate(yax, G_XA);
    const float ic = a.ic != nullptr ? a.ic[i] : 0.0f;
    float iapp = pulse_current(c.pulses, i, tstep);
    if (c.iapp != nullptr) iapp += c.iapp[i];
    const CellNext o = cell_step_rates(c.P, cell, ic, iapp, gr);
    finish_cell(c, tstep, vnext, i, o);
}

}  // namespace ion

using namespace ion;

// ---- host -------------------------------------------------------------------------------------
static ion_status mlp_cuda(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return ION_OK;
    return ion_fail(nullptr, ION_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

static uint64_t coprime_multiplier(uint64_t n, uint64_t seed) {
    // an odd multiplier near n * 0.618..., coprime with n (a bijection of Z_n)
    auto gcd = [](uint64_t x, uint64_t y) {
        while (y) {
            const uint64_t r = x % y;
            x = y;
            y = r;
        }
        return x;
    };
    uint64_t m = (uint64_t)(0.6180339887498949 * (double)n) + 2 * (seed % 97) + 1;
    while (gcd(m, n) != 1) ++m;
    return m;
}

extern "C" ion_status ion_surrogate_train(const ion_train_cfg *cfg, ion_surrogate_weights *w_out, float *final_loss) {
    if (!cfg || !w_out) return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_surrogate_train: NULL argument");
    const int64_t n = cfg->n_samples;
    const int B = cfg->batch;
    if (n < 256 || B < MB || B % MB != 0 || B > n || cfg->epochs < 1 || !(cfg->lr > 0) || !(cfg->v_hi > cfg->v_lo) ||
        !(cfg->ca_lo > 0) || !(cfg->ca_hi > cfg->ca_lo))
        return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_surrogate_train: bad configuration");
    cudaStream_t st = (cudaStream_t)cfg->cuda_stream;
    float *V, *ca, *X, *T, *params, *m, *v, *work, *mask, *shift, *scale, *loss;
    double *stat;
    const int sblk = 64;
    // one allocation for every buffer, cut into 256-byte aligned parts
    size_t total_bytes = 0;
    char *arena = nullptr;
    auto part = [&](size_t bytes) {
        const size_t at = total_bytes;
        total_bytes += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t oV = part(n * 4), oca = part(n * 4), oX = part(n * 8), oT = part(n * MO * 4), oparams = part(P_TOTAL * 4),
                 om = part(P_TOTAL * 4), ov = part(P_TOTAL * 4), owork = part(mlp_work_floats(B) * 4),
                 omask = part(MO * 4), oshift = part(MO * 4), oscale = part(MO * 4), oloss = part(4),
                 ostat = part((size_t)MO * sblk * 2 * 8);
    cudaError_t e = prepare_minibatch();
    if (e != cudaSuccess) return mlp_cuda(e, "ion_surrogate_train");
    e = ion_alloc(&arena, total_bytes);
    if (e != cudaSuccess) return ion_fail(nullptr, ION_ERR_OOM, "ion_surrogate_train: %s", cudaGetErrorString(e));
    V = (float *)(arena + oV);
    ca = (float *)(arena + oca);
    X = (float *)(arena + oX);
    T = (float *)(arena + oT);
    params = (float *)(arena + oparams);
    m = (float *)(arena + om);
    v = (float *)(arena + ov);
    work = (float *)(arena + owork);
    mask = (float *)(arena + omask);
    shift = (float *)(arena + oshift);
    scale = (float *)(arena + oscale);
    loss = (float *)(arena + oloss);
    stat = (double *)(arena + ostat);
    float hmask[MO];
    for (int o = 0; o < MO; ++o) hmask[o] = (o == 2 * G_MS + 1 || o == 2 * G_MA + 1) ? 0.0f : 1.0f;
    const float lc_lo = logf(cfg->ca_lo), lc_hi = logf(cfg->ca_hi);
    const float lc_mid = 0.5f * (lc_lo + lc_hi), lc_half = 0.5f * (lc_hi - lc_lo);
    const unsigned g1 = (unsigned)((n + 255) / 256);
    e = cudaMemcpyAsync(mask, hmask, sizeof hmask, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        mlp_samples_kernel<<<g1, 256, 0, st>>>(n, cfg->seed, cfg->v_lo, cfg->v_hi, lc_lo, lc_hi, V, ca);
        mlp_targets_kernel<<<g1, 256, 0, st>>>(n, V, ca, T);
        mlp_stats_kernel<<<dim3(sblk, MO), 256, 0, st>>>(n, T, stat);
        mlp_stats_final_kernel<<<1, 32, 0, st>>>(n, sblk, stat, mask, shift, scale);
        mlp_normalise_kernel<<<g1, 256, 0, st>>>(n, V, ca, lc_mid, lc_half, shift, scale, X, T);
        mlp_init_kernel<<<(P_TOTAL + 255) / 256, 256, 0, st>>>(params, cfg->seed);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(m, 0, P_TOTAL * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(v, 0, P_TOTAL * 4, st);
    const int64_t steps_per_epoch = n / B;
    const int64_t total = steps_per_epoch * cfg->epochs;
    const float denom = (float)B * 22.0f;
    int64_t step = 0;
    for (int ep = 0; ep < cfg->epochs && e == cudaSuccess; ++ep) {
        const uint64_t mul = coprime_multiplier((uint64_t)n, cfg->seed + ep);
        const uint64_t add = (uint64_t)(ep * 7919) % (uint64_t)n;
        if (ep == cfg->epochs - 1) e = cudaMemsetAsync(loss, 0, 4, st);
        for (int64_t b = 0; b < steps_per_epoch && e == cudaSuccess; ++b, ++step) {
            // cosine decay of the step size to 1 % over the run
            const double frac = total > 1 ? (double)step / (double)(total - 1) : 1.0;
            const float lr = (float)(cfg->lr * (0.01 + 0.99 * 0.5 * (1.0 + cos(M_PI * frac))));
            const double k = (double)(step + 1);
            const float c1 = (float)(1.0 - pow(0.9, k)), c2 = (float)(1.0 - pow(0.999, k));
            AdamArgs aa{{params, X, T, mask, n, b * B, B, mul, add, denom, B, work},
                        params, m, v, nullptr, lr, 0.9f, 0.999f, 1e-8f, c1, c2, ep == cfg->epochs - 1 ? loss : nullptr};
            // the first launch reads the samples that the kernels before it wrote: an ordinary one
            e = launch_minibatch(aa, step > 0, st);
        }
    }
    float hl = 0.0f;
    if (e == cudaSuccess) e = cudaMemcpyAsync(w_out, params, P_TOTAL * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w_out->out_shift, shift, MO * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w_out->out_scale, scale, MO * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hl, loss, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(arena);
    if (e != cudaSuccess) return ion_fail(nullptr, ION_ERR_CUDA, "ion_surrogate_train: %s", cudaGetErrorString(e));
    // input normalisation: x' = (x - shift) * scale with x = (V, ln [Ca])
    w_out->in_shift[0] = V_CENTER;
    w_out->in_scale[0] = 1.0f / V_HALF;
    w_out->in_shift[1] = lc_mid;
    w_out->in_scale[1] = 1.0f / lc_half;
    if (final_loss) *final_loss = hl / (float)steps_per_epoch;
    return ION_OK;
}

extern "C" ion_status ion_surrogate_grad(const ion_surrogate_weights *w, const float *x, const float *t,
                                         const float *mask, int32_t B, ion_surrogate_weights *grad, float *loss) {
    if (!w || !x || !t || !mask || !grad || B < 1)
        return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_surrogate_grad: bad arguments");
    const int64_t rows = ((int64_t)B + MB - 1) / MB * MB;
    float msum = 0.0f;
    for (int o = 0; o < MO; ++o) msum += mask[o];
    if (!(msum > 0)) return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_surrogate_grad: empty mask");
    float *params = nullptr, *X = nullptr, *T = nullptr, *M = nullptr, *work = nullptr, *g = nullptr, *L = nullptr;
    cudaError_t e = ion_alloc(&params, P_TOTAL * 4);
    if (e == cudaSuccess) e = ion_alloc(&X, (size_t)B * 8);
    if (e == cudaSuccess) e = ion_alloc(&T, (size_t)B * MO * 4);
    if (e == cudaSuccess) e = ion_alloc(&M, MO * 4);
    if (e == cudaSuccess) e = ion_alloc(&work, mlp_work_floats(rows) * 4);
    if (e == cudaSuccess) e = ion_alloc(&g, P_TOTAL * 4);
    if (e == cudaSuccess) e = ion_alloc(&L, 4);
    if (e == cudaSuccess) e = cudaMemcpy(params, w, P_TOTAL * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(X, x, (size_t)B * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(T, t, (size_t)B * MO * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(M, mask, MO * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(L, 0, 4);
    const float denom = (float)B * msum;
    if (e == cudaSuccess) e = prepare_minibatch();
    if (e == cudaSuccess) {
        AdamArgs aa{{params, X, T, M, B, 0, B, 1, 0, denom, rows, work}, params, nullptr, nullptr, g, 0, 0, 0, 0, 1, 1, L};
        e = launch_minibatch(aa, false, nullptr);
    }
    float hl = 0.0f;
    if (e == cudaSuccess) e = cudaMemcpy(grad, g, P_TOTAL * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&hl, L, 4, cudaMemcpyDeviceToHost);
    cudaFree(params);
    cudaFree(X);
    cudaFree(T);
    cudaFree(M);
    cudaFree(work);
    cudaFree(g);
    cudaFree(L);
    if (e != cudaSuccess)
        return ion_fail(nullptr, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "ion_surrogate_grad: %s",
                        cudaGetErrorString(e));
    if (loss) *loss = hl;
    return ION_OK;
}

// Upload a surrogate (host struct) as the packed inference copies: the warp-MMA layout
// (*d_out, may be NULL) and the tcgen05 layout (*d_tc).
ion_status ion_mlp_upload(const ion_surrogate_weights *w, void **d_out, void **d_tc, cudaStream_t st) {
    ion_surrogate_weights *dw = nullptr;
    MlpDev *d = nullptr;
    void *t = nullptr;
    cudaError_t e = ion_alloc(&dw, sizeof *dw);
    if (e == cudaSuccess && d_out) e = ion_alloc(&d, sizeof *d);
    if (e == cudaSuccess) e = ion_alloc(&t, surrogate_tc_weights_bytes());
    if (e == cudaSuccess) e = cudaMemcpyAsync(dw, w, sizeof *dw, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && d_out) {
        mlp_pack_kernel<<<1, 256, 0, st>>>(dw, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = surrogate_tc_pack(dw, t, st);
    if (e == cudaSuccess) e = surrogate_tc_prepare();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(dw);
    if (e != cudaSuccess) {
        cudaFree(d);
        cudaFree(t);
        return ion_fail(nullptr, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "surrogate upload: %s",
                        cudaGetErrorString(e));
    }
    if (d_out) *d_out = d;
    *d_tc = t;
    return ION_OK;
}

extern "C" ion_status ion_surrogate_eval(const ion_surrogate_weights *w, const float *V, const float *ca, int64_t n,
                                         float *out) {
    if (!w || !V || !ca || !out || n < 1) return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_surrogate_eval: bad arguments");
    void *t = nullptr;
    ion_status st = ion_mlp_upload(w, nullptr, &t, nullptr);
    if (st != ION_OK) return st;
    float *dV = nullptr, *dc = nullptr, *dout = nullptr;
    uint32_t *dstat = nullptr;
    cudaError_t e = ion_alloc(&dV, n * 4);
    if (e == cudaSuccess) e = ion_alloc(&dc, n * 4);
    if (e == cudaSuccess) e = ion_alloc(&dout, n * MO * 4);
    if (e == cudaSuccess) e = ion_alloc(&dstat, 4);
    if (e == cudaSuccess) e = cudaMemset(dstat, 0, 4);
    if (e == cudaSuccess) e = cudaMemcpy(dV, V, n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dc, ca, n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = launch_mlp_eval_tc(t, n, dV, dc, dout, dstat, nullptr);
    uint32_t hstat = 0;
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, n * MO * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&hstat, dstat, 4, cudaMemcpyDeviceToHost);
    cudaFree(dV);
    cudaFree(dc);
    cudaFree(dout);
    cudaFree(dstat);
    cudaFree(t);
    if (e != cudaSuccess)
        return ion_fail(nullptr, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "ion_surrogate_eval: %s",
                        cudaGetErrorString(e));
    if (hstat & ST_TIMEOUT) return ion_fail(nullptr, ION_ERR_TIMEOUT, "ion_surrogate_eval: a tensor-core wait timed out");
    return ION_OK;
}

// ---- a simulation handle with learned rates -----------------------------------------------------
// Per step: the gap-junction kernel writes the currents (split mode), then the surrogate
// cell kernel runs the MLP and the update.
static cudaError_t surrogate_step(ion_sim *s, int k_off, const float *iapp) {
    const StepCommon c = ion_step_common(s, k_off, iapp);
    cudaError_t e = cudaSuccess;
    if (s->kind == ION_DENSE_UNIFORM) {
        DenseArgs a{};
        a.c = c;
        a.g = s->g;
        a.kahan = 1;
        a.fuse = 0;
        a.ic_out = s->d_ic;
        e = launch_dense_step(a, s->dense_R, s->dense_W, s->dense_GJ, s->st);
        s->launches++;
    } else if (s->kind == ION_CSR) {
        CsrArgs a{};
        a.c = c;
        ion_csr_fill(s, a, s->csr_staged == 1);
        a.fuse = 0;
        a.ic_out = s->d_ic;
        e = ion_launch_csr(s, a);
        s->launches++;
    }
    if (e != cudaSuccess) return e;
    s->launches++;
    const float *ic = s->kind == ION_NO_GJ ? nullptr : s->d_ic;
    const StepCommon cu = ion_update_common(s, c);
    if (!(s->flags & ION_FLAG_SURROGATE_WARP_MMA)) 
        return launch_surrogate_tc(cu, s->d_mlp_tc, ic, (int)std::min<int64_t>(s->debug_delay_ns, 7), s->st);
    SurrArgs sa{cu, (const MlpDev *)s->d_mlp, ic};
    return launch_k(surrogate_cell_kernel, dim3((unsigned)((s->n + 2 * SURR_CPW - 1) / (2 * SURR_CPW))), dim3(64), 0,
                    s->st, c.pdl != 0, sa);
}

ion_status ion_setup_surrogate(ion_sim *s, const ion_params *p) {
    if (!p->surrogate) return ion_fail(nullptr, ION_ERR_INVALID_ARG, "surrogate: no weights");
    ion_status st = ion_mlp_upload((const ion_surrogate_weights *)p->surrogate, &s->d_mlp, &s->d_mlp_tc, s->st);
    if (st != ION_OK) return st;
    if (s->kind != ION_NO_GJ && !s->d_ic) {
        cudaError_t e = ion_alloc(&s->d_ic, (size_t)s->n_pad * sizeof(float));
        if (e != cudaSuccess) return ion_fail(nullptr, ION_ERR_OOM, "surrogate: %s", cudaGetErrorString(e));
    }
    s->step_override = surrogate_step;
    s->lps = s->kind == ION_NO_GJ ? 1 : 2;
    return ION_OK;
}
