// ion_matrix.cu -- dense N x N weight-matrix connectivity (the programmed connectivity of
// Sec. 2.3 with every pair stored):
//   Ic_i = sum_j W[i][j] (0.8 e^{-dV^2/100} + 0.2) dV,  dV = V_dend,i - V_dend,j.
// The weights are stored padded to n_pad columns (zeros beyond n), so a padded column
// contributes exactly zero.  Every step streams the whole matrix (4 B per pair: 268 MB at
// 8192 cells), so the kernel is bound by memory.
//
// One CTA of 16 warps per SM owns n / SMs rows (the same number within one, so every SM
// streams the same bytes).  A warp owns 512 columns of every GR-th of these rows: its 16
// transformed V_dend values per lane stay in registers, each row costs it four coalesced
// 16-byte weight loads per lane and nothing else, and the weights of the next R rows are in
// flight (up to 128 KB per SM).  The first R rows are requested before the wait on the
// previous step.  A row's lane sums are combined by a fixed butterfly, its column splits in
// order with compensation; then one thread per row runs the update from state words that
// cp.async brought in meanwhile.
//
// The rows are walked in opposite directions on even and odd steps: what the last step left in
// L2 (part of its last rows) is read first, before it is evicted.
//
// At 8192 cells: 41.7 us per step (0.95 of the measured copy rate); eight rows per CTA of 8
// warps (1024 CTAs, each staging and transforming all of V_dend first, evict-first loads, one
// direction) 65.8.  Keeping a fixed share of the rows in L2 by cache hints (20 to 40 % loaded
// evict-last, the rest evict-first) measured 42.8 to 45.7: the plain loads stay.
#include <cuda_runtime.h>

#include <algorithm>

#include "ion.h"
#include "ion_async.cuh"
#include "ion_dense_core.cuh"
#include "ion_kernels.cuh"

namespace ion {

constexpr int MX_WARPS = 16, MX_THREADS = 32 * MX_WARPS, MX_COLS = 512;   // columns of a warp

struct MatrixShape {
    int32_t rows;     // rows per CTA (<= MX_THREADS: one thread updates each)
    int32_t GJ, GR;   // column splits, row groups (GJ x GR <= MX_WARPS)
};
static MatrixShape matrix_shape(int n, int n_pad, int sms) {
    MatrixShape s;
    s.rows = std::min(MX_THREADS, std::max(1, (n + sms - 1) / sms));
    s.GJ = std::min(MX_WARPS, (n_pad + MX_COLS - 1) / MX_COLS);
    s.GR = MX_WARPS / s.GJ;
    return s;
}
// u of the rows, [rows][GJ] partial sums and their compensations, the rows' state words
static size_t matrix_smem_bytes(const MatrixShape &s) { return (size_t)s.rows * (1 + 2 * s.GJ + NCW) * sizeof(float); }

template <int R>
__global__ void __launch_bounds__(MX_THREADS, 1) matrix_step_kernel(const MatrixArgs a, const MatrixShape S) {
    extern __shared__ __align__(16) float mx_smem[];
    float *u_s = mx_smem, *part = u_s + S.rows, *comp = part + S.rows * S.GJ, *cs = comp + S.rows * S.GJ;
    const StepCommon &c = a.c;
    const int n = c.n, n_pad = c.n_pad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = blockIdx.x * S.rows, here = min(S.rows, n - row0);
    const int rg = warp / S.GJ, sp = warp - rg * S.GJ;
    const int nr = rg < S.GR && rg < here ? (here - rg + S.GR - 1) / S.GR : 0;   // rows of this warp
    auto row = [&](int k) { return rg + (c.par ? nr - 1 - k : k) * S.GR; };       // k-th row in step order
    const int span = S.GJ * MX_COLS, n_tiles = (n_pad + span - 1) / span;
    float4 w[R][4];
    int col = sp * MX_COLS + 4 * lane;   // this lane's first column; + 128 q, q = 0..3
    auto load = [&](int slot, int k) {
        const float *p = a.W + (int64_t)(row0 + row(k)) * n_pad + col;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            w[slot][q] = col + 128 * q < n_pad ? __ldg(reinterpret_cast<const float4 *>(p + 128 * q))
                                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (k < nr) load(k, k);
    const int mine = threadIdx.x;
    const bool has_row = mine < here;
    const PulseAhead pa = pulse_ahead(c.pulses, row0 + mine, has_row);
    pdl_enter();
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    const float m = vcur[0];
    stage_cells(cs, c.S, vcur, row0, S.rows, n);
    if (has_row) u_s[mine] = (vcur[row0 + mine] - m) * GJ_SCALE;
    float iapp = pulse_current(c.pulses, pa, t);
    if (c.iapp != nullptr && has_row) iapp += c.iapp[row0 + mine];
    __syncthreads();
    const float2 c08 = make_float2(0.8f, 0.8f), c02 = make_float2(0.2f, 0.2f);
    const float2 negm2 = make_float2(-m, -m), negs2 = make_float2(-GJ_SCALE, -GJ_SCALE);
    for (int tile = 0; tile < n_tiles; ++tile, col += span) {
        float2 x[8];   // -u of this lane's columns (padding: the sentinel, far from any cell)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float4 v = make_float4(PAD_VOLT, PAD_VOLT, PAD_VOLT, PAD_VOLT);
            if (col + 128 * q < n_pad) v = *reinterpret_cast<const float4 *>(vcur + col + 128 * q);
            x[2 * q] = __fmul2_rn(__fadd2_rn(make_float2(v.x, v.y), negm2), negs2);
            x[2 * q + 1] = __fmul2_rn(__fadd2_rn(make_float2(v.z, v.w), negm2), negs2);
        }
        if (tile > 0)
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (k < nr) load(k, k);
        for (int k0 = 0; k0 < nr; k0 += R) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const int k = k0 + j;
                if (k < nr) {
                    const int r = row(k);
                    const float ui = u_s[r];
                    const float2 u2 = make_float2(ui, ui);
                    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 da = __fadd2_rn(u2, x[2 * q]), db = __fadd2_rn(u2, x[2 * q + 1]);
                        const float2 qa = __fmul2_rn(da, da), qb = __fmul2_rn(db, db);
                        const float2 ea = make_float2(ex2_approx(-qa.x), ex2_approx(-qa.y));
                        const float2 eb = make_float2(ex2_approx(-qb.x), ex2_approx(-qb.y));
                        const float2 ta = __fmul2_rn(__ffma2_rn(ea, c08, c02), da);
                        const float2 tb = __fmul2_rn(__ffma2_rn(eb, c08, c02), db);
                        acc = __ffma2_rn(ta, make_float2(w[j][q].x, w[j][q].y), acc);
                        acc = __ffma2_rn(tb, make_float2(w[j][q].z, w[j][q].w), acc);
                    }
                    if (k + R < nr) load(j, k + R);
                    float v = acc.x + acc.y;
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                    if (lane == 0) {   // further column tiles (n > 8192) are added with compensation
                        float ks = tile > 0 ? part[r * S.GJ + sp] : 0.0f, kc = tile > 0 ? comp[r * S.GJ + sp] : 0.0f;
                        kahan_add(ks, kc, v);
                        part[r * S.GJ + sp] = ks;
                        comp[r * S.GJ + sp] = kc;
                    }
                }
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
    if (!has_row) return;
    float ks = 0.0f, kc = 0.0f;
    for (int q = 0; q < S.GJ; ++q) kahan_add(ks, kc, part[mine * S.GJ + q] - comp[mine * S.GJ + q]);
    const float ic = (ks - kc) * (1.0f / GJ_SCALE);
    const CellNext o = cell_step(c.P, staged_cell(cs, S.rows, mine), ic, iapp);
    finish_cell(c, t, vd_next(c), row0 + mine, o);
}

cudaError_t prepare_matrix_step() {
    const int smem = MX_THREADS * (1 + 2 * MX_WARPS + NCW) * (int)sizeof(float);   // the largest shape's
    cudaError_t e = cudaFuncSetAttribute(matrix_step_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(matrix_step_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(matrix_step_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

template <int R>
static cudaError_t matrix_launch_R(const MatrixArgs &a, int sms, cudaStream_t st) {
    const MatrixShape s = matrix_shape(a.c.n, a.c.n_pad, sms);
    const int grid = (a.c.n + s.rows - 1) / s.rows;
    return launch_k(matrix_step_kernel<R>, dim3(grid), dim3(MX_THREADS), matrix_smem_bytes(s), st, a.c.pdl != 0, a, s);
}
// R: rows whose weights a warp has in flight
cudaError_t launch_matrix_step(const MatrixArgs &a, int R, int sms, cudaStream_t st) {
    switch (R) {
        case 1: return matrix_launch_R<1>(a, sms, st);
        case 2: return matrix_launch_R<2>(a, sms, st);
        case 4: return matrix_launch_R<4>(a, sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ion
