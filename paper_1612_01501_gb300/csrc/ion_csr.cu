// ion_csr.cu -- sparse (CSR) gap-junction step and the stand-alone cell update.
//
// Algorithm 1 over a programmed weight matrix (Sec. 2.3): for every stored connection
// e = (i, j) of row i,
//   Ic_i += w_e (0.8 e^{-dV^2/100} + 0.2) dV,  dV = V_dend,i - V_dend,j.
// A CTA of 256 threads owns `rows` consecutive rows (1..256, chosen from the mean degree
// so that the grid keeps every SM busy).  Phase 1: groups of SW lanes (SW = 1..32) walk
// one row's edges; with 16-byte aligned arrays each lane reads four consecutive indices
// and weights per 16-byte load, and four V_dend gathers are in flight per lane; the SW
// lane sums are combined with shuffles in a fixed order.  Phase 2: one thread per row
// runs the explicit-Euler cell update with that row's current (fused variant), so the
// cell work runs on full warps whatever SW is.
#include <cuda_runtime.h>

#include <algorithm>

#include "ion_async.cuh"
#include "ion_csr_core.cuh"
#include "ion_kernels.cuh"

namespace ion {

// One CTA of 256 threads owns `rows` consecutive rows (rows <= 256).  Phase 1: groups of
// SW lanes take the rows round-robin; phase 2: thread t updates row t.  For long rows (16-byte
// loads of four 32-bit or eight 16-bit columns; csr_direct has the rule and its figures) and the
// stand-alone primitive; the rest runs csr_direct_step_kernel.  LIN: linear junctions, on 16-bit
// columns only.
template <int SW, bool VEC, bool HAS_W, bool C16, bool LIN>
__global__ void __launch_bounds__(256) csr_step_kernel(const CsrArgs a, int rows) {
    static_assert(!LIN || C16, "linear junctions run on the 16-bit column layout");
    __shared__ float ic_s[256];
    pdl_enter();
    const StepCommon &c = a.c;
    const int n = c.n;
    const int row0 = blockIdx.x * rows;
    const int64_t t = step_index(c);
    const float *vcur = a.vd_in != nullptr ? a.vd_in : vd_cur(c);
    float *vnext = a.fuse ? vd_next(c) : nullptr;
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int iters = (rows + nsub - 1) / nsub;          // the same for every lane (shuffles below)
    // a row's bounds and V_dend are loaded one row ahead (see the chunked variant)
    auto bounds = [&](int it, int &e0, int &e1, float &vi) {
        const int rr = sub + it * nsub, i = row0 + rr;
        e0 = e1 = 0;
        vi = 0.0f;
        if (it < iters && rr < rows && i < n) {
            e0 = a.row_ptr[i];
            e1 = a.row_ptr[i + 1];
            vi = vcur[i];
        }
    };
    int e0n, e1n;
    float vin;
    bounds(0, e0n, e1n, vin);
    for (int it = 0; it < iters; ++it) {
        const int rr = sub + it * nsub;
        const int e0 = e0n, e1 = e1n;
        const float vi = vin;
        bounds(it + 1, e0n, e1n, vin);
        float acc = 0.0f;
        if (e1 > e0) {   // rows past the end (and empty rows) have e0 == e1
            if (C16)
                acc = csr_row_sum16<SW, HAS_W, false, LIN>(a.col16, a.w, e0, e1, vi, li, VjGlobal{vcur});
            else
                acc = csr_row_sum<SW, VEC, HAS_W>(vcur, a.col, a.w, e0, e1, vi, li);
        }
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < rows) ic_s[rr] = (HAS_W ? acc : acc * a.g) * (1.0f / GJ_SCALE);
    }
    __syncthreads();
    if ((int)threadIdx.x >= rows) return;
    const int i = row0 + threadIdx.x;
    if (i >= n) return;
    const float ic = ic_s[threadIdx.x];
    if (!a.fuse) {
        a.ic_out[i] = ic;
        return;
    }
    const Cell cell = load_cell(c.S, vcur, i);
    float iapp = pulse_current(c.pulses, i, t);
    if (c.iapp != nullptr) iapp += c.iapp[i];
    const CellNext o = cell_step(c.P, cell, ic, iapp);
    finish_cell(c, t, vnext, i, o);
}

template <int SW, bool VEC, bool HAS_W, bool C16 = false, bool LIN = false>
static cudaError_t launch_csr_T(const CsrArgs &a, int rows, cudaStream_t st) {
    const int grid = (a.c.n + rows - 1) / rows;
    return launch_k(csr_step_kernel<SW, VEC, HAS_W, C16, LIN>, dim3(grid), dim3(256), 0, st, a.c.pdl != 0, a, rows);
}
template <int SW>
static cudaError_t launch_csr_SW(const CsrArgs &a, int rows, cudaStream_t st) {
    if (a.lin) {
        if (a.col16 == nullptr) return cudaErrorInvalidValue;
        return a.w != nullptr ? launch_csr_T<SW, true, true, true, true>(a, rows, st)
                              : launch_csr_T<SW, true, false, true, true>(a, rows, st);
    }
    if (a.col16 != nullptr)   // 16-byte aligned indices (and weights, both the handle's own)
        return a.w != nullptr ? launch_csr_T<SW, true, true, true>(a, rows, st) : launch_csr_T<SW, true, false, true>(a, rows, st);
    const bool vec = ((uintptr_t)a.col % 16 == 0) && (a.w == nullptr || (uintptr_t)a.w % 16 == 0);
    if (a.w != nullptr) return vec ? launch_csr_T<SW, true, true>(a, rows, st) : launch_csr_T<SW, false, true>(a, rows, st);
    return vec ? launch_csr_T<SW, true, false>(a, rows, st) : launch_csr_T<SW, false, false>(a, rows, st);
}

// rows: rows per CTA (1..256); SW: lanes per row.
cudaError_t launch_csr_step(const CsrArgs &a, int SW, int rows, cudaStream_t st) {
    if (rows < 1 || rows > 256) return cudaErrorInvalidValue;
    switch (SW) {
        case 1: return launch_csr_SW<1>(a, rows, st);
        case 2: return launch_csr_SW<2>(a, rows, st);
        case 4: return launch_csr_SW<4>(a, rows, st);
        case 8: return launch_csr_SW<8>(a, rows, st);
        case 16: return launch_csr_SW<16>(a, rows, st);
        case 32: return launch_csr_SW<32>(a, rows, st);
        default: return cudaErrorInvalidValue;
    }
}

// Prefer L1 over shared memory for the V_dend gathers (the kernel uses 1 KB of shared).
template <int SW>
static void carveout_SW() {
    auto prefer_l1 = [](auto *k) { cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 0); };
    prefer_l1(csr_step_kernel<SW, true, true, false, false>);
    prefer_l1(csr_step_kernel<SW, false, true, false, false>);
    prefer_l1(csr_step_kernel<SW, true, false, false, false>);
    prefer_l1(csr_step_kernel<SW, false, false, false, false>);
    prefer_l1(csr_step_kernel<SW, true, true, true, false>);
    prefer_l1(csr_step_kernel<SW, true, false, true, false>);
    prefer_l1(csr_step_kernel<SW, true, true, true, true>);
    prefer_l1(csr_step_kernel<SW, true, false, true, true>);
}
cudaError_t prepare_csr_step() {
    carveout_SW<1>();
    carveout_SW<2>();
    carveout_SW<4>();
    carveout_SW<8>();
    carveout_SW<16>();
    carveout_SW<32>();
    return cudaGetLastError();
}

// ---- the direct step: V_dend gathered through L1 / L2 ---------------------------------------
// Where it runs (short rows, small networks) a step is a few dependent memory latencies long,
// so everything that does not change between steps (the row's bounds, its first SHORT_E columns
// and weights per lane, its pulse) is read before the wait on the previous step; after it the
// V_dend gathers and the rows' state words (cp.async) go out together.  Arrays borrowed from the
// caller (a.borrowed) are read after the wait: the caller may rewrite them on the handle's
// stream between two calls, and only the wait orders this kernel after such a write.  A row of
// more than a.long_rounds rounds (a multiple of the mean row) is finished by its whole warp:
// 65 536 cells, k = 10, 8 rows of 3000 edges: 75.7 us per step with SW lanes for every row, 26.6
// now.  256 threads, SW lanes per row, four gathers in flight per lane; then one thread per row
// runs the update.  C16: 16-bit columns.  LIN: linear junctions, w (V_i - V_j).
// 65 536 cells, k = 10: 5.5 us per step (4 lanes, 128 rows per CTA); the kernel that read
// bounds, columns, gathers, state and pulses one after the other took 9.5 (7.1 tuned).
constexpr int SHORT_E = 4;

template <int SW, bool HAS_W, bool LIN, bool C16>
__global__ void __launch_bounds__(256) csr_direct_step_kernel(const CsrArgs a, int rows) {
    extern __shared__ __align__(16) float sh_smem[];
    float *ic_s = sh_smem, *cs = sh_smem + 256;
    const StepCommon &c = a.c;
    const int n = c.n, row0 = blockIdx.x * rows;
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW;
    constexpr int NSUB = 256 / SW;
    uint32_t e = 0, e1 = 0;   // unsigned: the look-ahead below may pass 2^31
    int j[SHORT_E];
    float w[HAS_W ? SHORT_E : 1];
    auto column = [&](uint32_t q) { return C16 ? (int)__ldg(a.col16 + q) : __ldg(a.col + q); };
    auto columns = [&]() {      // SHORT_E columns and weights from e on
#pragma unroll
        for (int k = 0; k < SHORT_E; ++k)
            if (e + k * SW < e1) {
                j[k] = column(e + k * SW);
                if (HAS_W) w[k] = __ldg(a.w + e + k * SW);
            }
    };
    auto head = [&](int rr) {   // bounds, first columns and weights of row rr of the CTA
        const int i = row0 + rr;
        e = e1 = 0;
        if (rr < rows && i < n) {
            e = (uint32_t)__ldg(a.row_ptr + i) + li;
            e1 = (uint32_t)__ldg(a.row_ptr + i + 1);
        }
        columns();
    };
    // an edge's term added to a sum, the last product fused into it (one rounding, as gj_edge2)
    auto add = [&](float s, float vi, float vj, float wt) {
        const float d = vi - vj;
        if (LIN) return HAS_W ? fmaf(wt, d, s) : s + d;
        const float du = d * GJ_SCALE, f = fmaf(0.8f, ex2_approx(-du * du), 0.2f);
        return fmaf(HAS_W ? wt * f : f, du, s);
    };
    if (!a.borrowed) head(sub);
    const int mine = threadIdx.x;
    const bool has_row = mine < rows && row0 + mine < n;
    const PulseAhead pa = pulse_ahead(c.pulses, row0 + mine, has_row && a.fuse);
    pdl_enter();
    if (a.borrowed) head(sub);
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    if (a.fuse && has_row) {
#pragma unroll
        for (int q = 0; q < NCW; ++q)
            cp_async4(cs + q * rows + mine, (q == 0 ? vcur : c.S.f(cell_word_field(q))) + row0 + mine);
    }
    cp_async_commit();
    for (int rr = sub; rr - sub < rows; rr += NSUB) {   // the same trip count in every lane
        if (rr != sub) head(rr);
        const int i = row0 + rr;
        const float vi = rr < rows && i < n ? vcur[i] : 0.0f;
        float acc = 0.0f;
        for (int round = 0; e < e1 && (SW == 32 || round < a.long_rounds); ++round) {
            float v[SHORT_E];
#pragma unroll
            for (int k = 0; k < SHORT_E; ++k)
                if (e + k * SW < e1) v[k] = __ldg(vcur + j[k]);
            float part[2] = {0.0f, 0.0f};   // two short chains
#pragma unroll
            for (int k = 0; k < SHORT_E; ++k)
                if (e + k * SW < e1) part[k >> 1] = add(part[k >> 1], vi, v[k], HAS_W ? w[k] : 1.0f);
            acc += part[0] + part[1];
            e += SHORT_E * SW;
            columns();
        }
        if (SW < 32) {   // rows with edges left (lane 0 of the row has e = its first one)
            const int lane = threadIdx.x & 31;
            for (uint32_t left = __ballot_sync(0xffffffffu, li == 0 && e < e1); left != 0; left &= left - 1) {
                const int src = __ffs(left) - 1;
                const uint32_t first = __shfl_sync(0xffffffffu, e, src), end = __shfl_sync(0xffffffffu, e1, src);
                const float vl = __shfl_sync(0xffffffffu, vi, src);
                float sum = 0.0f;
                for (uint32_t q = first + lane; q < end; q += SHORT_E * 32) {
                    int jl[SHORT_E];
                    float v[SHORT_E], wl[SHORT_E];
#pragma unroll
                    for (int k = 0; k < SHORT_E; ++k) {
                        const bool in = q + k * 32 < end;
                        jl[k] = in ? column(q + k * 32) : 0;
                        wl[k] = in && HAS_W ? __ldg(a.w + q + k * 32) : 1.0f;
                    }
#pragma unroll
                    for (int k = 0; k < SHORT_E; ++k)
                        if (q + k * 32 < end) v[k] = __ldg(vcur + jl[k]);
                    float part[2] = {0.0f, 0.0f};
#pragma unroll
                    for (int k = 0; k < SHORT_E; ++k)
                        if (q + k * 32 < end) part[k >> 1] = add(part[k >> 1], vl, v[k], wl[k]);
                    sum += part[0] + part[1];
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
                if (lane == src) acc += sum;
            }
        }
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < rows) ic_s[rr] = (HAS_W ? acc : acc * a.g) * (LIN ? 1.0f : 1.0f / GJ_SCALE);
    }
    cp_async_wait_all();
    __syncthreads();
    if (!has_row) return;
    const int i = row0 + mine;
    if (!a.fuse) {
        a.ic_out[i] = ic_s[mine];
        return;
    }
    float iapp = pulse_current(c.pulses, pa, t);
    if (c.iapp != nullptr) iapp += c.iapp[i];
    const CellNext o = cell_step(c.P, staged_cell(cs, rows, mine), ic_s[mine], iapp);
    finish_cell(c, t, vd_next(c), i, o);
}

template <int SW, bool C16>
static cudaError_t launch_direct_T(const CsrArgs &a, int rows, cudaStream_t st) {
    const dim3 grid((a.c.n + rows - 1) / rows), block(256);
    const size_t smem = (256 + (size_t)NCW * rows) * sizeof(float);
    const bool pdl = a.c.pdl != 0;
    if (a.lin)
        return a.w != nullptr ? launch_k(csr_direct_step_kernel<SW, true, true, C16>, grid, block, smem, st, pdl, a, rows)
                              : launch_k(csr_direct_step_kernel<SW, false, true, C16>, grid, block, smem, st, pdl, a, rows);
    return a.w != nullptr ? launch_k(csr_direct_step_kernel<SW, true, false, C16>, grid, block, smem, st, pdl, a, rows)
                          : launch_k(csr_direct_step_kernel<SW, false, false, C16>, grid, block, smem, st, pdl, a, rows);
}
template <int SW>
static cudaError_t launch_direct_SW(const CsrArgs &a, int rows, cudaStream_t st) {
    return a.col16 != nullptr ? launch_direct_T<SW, true>(a, rows, st) : launch_direct_T<SW, false>(a, rows, st);
}
// rows: rows per CTA (1..256); SW: lanes per row.
cudaError_t launch_csr_direct_step(const CsrArgs &a, int SW, int rows, cudaStream_t st) {
    if (rows < 1 || rows > 256) return cudaErrorInvalidValue;
    switch (SW) {
        case 1: return launch_direct_SW<1>(a, rows, st);
        case 2: return launch_direct_SW<2>(a, rows, st);
        case 4: return launch_direct_SW<4>(a, rows, st);
        case 8: return launch_direct_SW<8>(a, rows, st);
        case 16: return launch_direct_SW<16>(a, rows, st);
        case 32: return launch_direct_SW<32>(a, rows, st);
        default: return cudaErrorInvalidValue;
    }
}

// ---- column-chunked variant: V_dend staged in shared memory -------------------------------
// For large networks the V_dend gathers of a random graph touch a different L1 line per
// lane.  Here the column space is cut into chunks of CSR_CHUNK floats (128 KB); each
// CTA (one per SM, 1024 threads) owns `rows` consecutive rows and, chunk by chunk,
// stages V_dend[chunk] into shared memory with one bulk copy and sums the edges of its
// rows whose columns fall in that chunk (the per-row chunk boundaries are precomputed:
// mid[(c-1) * n + i] is the first edge of row i in chunk c).  The gathers then hit shared
// memory while the indices and weights stream from HBM.
// Networks with the compact layout run the sliced kernel (ion_csr_sliced.cu) instead; this one
// serves the columns as given (32-bit), the opt-in bank order and layouts beyond 32-bit offsets.
template <int SW, bool VEC, bool HAS_W, bool C16, bool LIN = false>
__global__ void __launch_bounds__(1024) csr_chunk_step_kernel(const CsrArgs a, int rows, const int32_t *mid,
                                                              int n_chunks) {
    static_assert(!LIN || C16, "linear junctions run on the 16-bit column layout");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *vs = reinterpret_cast<float *>(smem_raw);
    const int nb = min(CSR_CHUNK, a.c.n_pad);
    float *ic_s = vs + nb;
    __shared__ __align__(8) uint64_t bar;
    pdl_enter();
    const StepCommon &c = a.c;
    const int n = c.n;
    const int row0 = blockIdx.x * rows;
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    float *vnext = vd_next(c);
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int iters = (rows + nsub - 1) / nsub;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    for (int r = threadIdx.x; r < rows; r += blockDim.x) ic_s[r] = 0.0f;
    __syncthreads();
    for (int ch = 0; ch < n_chunks; ++ch) {
        const int c0 = ch * CSR_CHUNK;
        const int len = min(CSR_CHUNK, c.n_pad - c0);
        if (threadIdx.x == 0) {
            mbar_expect_tx(&bar, (uint32_t)len * 4u);
            bulk_g2s(vs, vcur + c0, (uint32_t)len * 4u, &bar);
        }
        const bool landed = mbar_wait_bounded(&bar, (uint32_t)(ch & 1));
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) {
                atomicOr(c.status, (uint32_t)ST_TIMEOUT);
                (void)mbar_wait_bounded(&bar, (uint32_t)(ch & 1));
            }
            return;
        }
        // The bounds of a row's segment in this chunk and its V_dend.  With 16 or more lanes
        // per row (long rows, few rows per group) they are loaded two rows ahead and the
        // next row's index (and weight) stream is requested into L2 one row ahead, so that
        // each row waits on an L2 latency rather than on two HBM latencies.
        auto bounds = [&](int it, int &e0, int &e1, float &vi) {
            const int rr = sub + it * nsub, i = row0 + rr;
            e0 = e1 = 0;
            vi = 0.0f;
            if (it < iters && rr < rows && i < n) {
                e0 = ch == 0 ? a.row_ptr[i] : mid[(int64_t)(ch - 1) * n + i];
                e1 = ch == n_chunks - 1 ? a.row_ptr[i + 1] : mid[(int64_t)ch * n + i];
                vi = vcur[i];
            }
        };
        constexpr bool AHEAD = SW >= 16;
        int e0n = 0, e1n = 0, e0m = 0, e1m = 0;
        float vin = 0.0f, vim = 0.0f;
        if (AHEAD) {
            bounds(0, e0n, e1n, vin);
            bounds(1, e0m, e1m, vim);
        }
        for (int it = 0; it < iters; ++it) {
            const int rr = sub + it * nsub;
            int e0, e1;
            float vi;
            if (AHEAD) {
                e0 = e0n;
                e1 = e1n;
                vi = vin;
                e0n = e0m;
                e1n = e1m;
                vin = vim;
                bounds(it + 2, e0m, e1m, vim);
                if (li == 0 && e1n > e0n) {   // the next row's stream, in whole 16-byte groups
                    if (C16) {   // col16 is padded to whole 16-byte groups
                        const int64_t b0 = ((int64_t)e0n * 2) & ~(int64_t)15, b1 = ((int64_t)e1n * 2 + 15) & ~(int64_t)15;
                        bulk_prefetch_l2(reinterpret_cast<const char *>(a.col16) + b0, (uint32_t)(b1 - b0));
                    } else {     // 32-bit columns: the last partial group is left out
                        const int64_t b0 = ((int64_t)e0n * 4) & ~(int64_t)15, b1 = ((int64_t)e1n * 4) & ~(int64_t)15;
                        if (b1 > b0) bulk_prefetch_l2(reinterpret_cast<const char *>(a.col) + b0, (uint32_t)(b1 - b0));
                    }
                    if (HAS_W) {
                        const int64_t b0 = ((int64_t)e0n * 4) & ~(int64_t)15, b1 = ((int64_t)e1n * 4) & ~(int64_t)15;
                        if (b1 > b0) bulk_prefetch_l2(reinterpret_cast<const char *>(a.w) + b0, (uint32_t)(b1 - b0));
                    }
                }
            } else {
                bounds(it, e0, e1, vi);
            }
            float acc = 0.0f;
            if (e1 > e0) {   // rows past the end (and empty segments) have e0 == e1
                if (C16)
                    acc = csr_row_sum16<SW, HAS_W, true, LIN>(a.col16, a.w, e0, e1, vi, li, VjChunk{vs});
                else
                    acc = csr_row_sum_smem<SW, VEC, HAS_W>(vs, c0, a.col, a.w, e0, e1, vi, li);
            }
#pragma unroll
            for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (li == 0 && rr < rows) ic_s[rr] += acc;
        }
        // all reads of this chunk are done before the next bulk copy overwrites it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
    }
    for (int rr = threadIdx.x; rr < rows; rr += blockDim.x) {
        const int i = row0 + rr;
        if (i >= n) break;
        const float ic = (HAS_W ? ic_s[rr] : ic_s[rr] * a.g) * (1.0f / GJ_SCALE);
        const Cell cell = load_cell(c.S, vcur, i);
        float iapp = pulse_current(c.pulses, i, t);
        if (c.iapp != nullptr) iapp += c.iapp[i];
        const CellNext o = cell_step(c.P, cell, ic, iapp);
        finish_cell(c, t, vnext, i, o);
    }
}

// the chunk and the rows' currents
size_t csr_chunk_smem_bytes(int n_pad, int rows) {
    return (size_t)(n_pad < CSR_CHUNK ? n_pad : CSR_CHUNK) * sizeof(float) + (size_t)rows * sizeof(float);
}

template <int SW, bool VEC, bool HAS_W, bool C16 = false, bool LIN = false>
static cudaError_t chunk_T(const CsrArgs &a, int rows, const int32_t *mid, int n_chunks, bool prepare,
                           cudaStream_t st) {
    const size_t smem = csr_chunk_smem_bytes(a.c.n_pad, rows);
    if (prepare)
        return allow_smem(csr_chunk_step_kernel<SW, VEC, HAS_W, C16, LIN>, smem);
    const int grid = (a.c.n + rows - 1) / rows;
    return launch_k(csr_chunk_step_kernel<SW, VEC, HAS_W, C16, LIN>, dim3(grid), dim3(1024), smem, st,
                    a.c.pdl != 0, a, rows, mid, n_chunks);
}
template <int SW>
static cudaError_t chunk_SW(const CsrArgs &a, int rows, const int32_t *mid, int n_chunks, bool prepare,
                            cudaStream_t st) {
    const bool vec = ((uintptr_t)a.col % 16 == 0) && (a.w == nullptr || (uintptr_t)a.w % 16 == 0);
    if (prepare) {   // set the limit on every instantiation the launch may pick
        cudaError_t e = chunk_T<SW, true, true>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, false, true>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, true, false>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, false, false>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, true, true, true>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, true, false, true>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, true, true, true, true>(a, rows, mid, n_chunks, true, st);
        if (e == cudaSuccess) e = chunk_T<SW, true, false, true, true>(a, rows, mid, n_chunks, true, st);
        return e;
    }
    if (a.lin) {
        if (a.col16 == nullptr) return cudaErrorInvalidValue;
        return a.w != nullptr ? chunk_T<SW, true, true, true, true>(a, rows, mid, n_chunks, false, st)
                              : chunk_T<SW, true, false, true, true>(a, rows, mid, n_chunks, false, st);
    }
    if (a.col16 != nullptr)
        return a.w != nullptr ? chunk_T<SW, true, true, true>(a, rows, mid, n_chunks, false, st)
                              : chunk_T<SW, true, false, true>(a, rows, mid, n_chunks, false, st);
    if (a.w != nullptr)
        return vec ? chunk_T<SW, true, true>(a, rows, mid, n_chunks, false, st)
                   : chunk_T<SW, false, true>(a, rows, mid, n_chunks, false, st);
    return vec ? chunk_T<SW, true, false>(a, rows, mid, n_chunks, false, st)
               : chunk_T<SW, false, false>(a, rows, mid, n_chunks, false, st);
}

// rows: rows per CTA (1..1024); mid: (n_chunks - 1) x n interior chunk boundaries.
cudaError_t launch_csr_chunk_step(const CsrArgs &a, int SW, int rows, const int32_t *mid, int n_chunks, bool prepare,
                                  cudaStream_t st) {
    if (rows < 1 || rows > 1024 || n_chunks < 1) return cudaErrorInvalidValue;
    switch (SW) {
        case 1: return chunk_SW<1>(a, rows, mid, n_chunks, prepare, st);
        case 2: return chunk_SW<2>(a, rows, mid, n_chunks, prepare, st);
        case 4: return chunk_SW<4>(a, rows, mid, n_chunks, prepare, st);
        case 8: return chunk_SW<8>(a, rows, mid, n_chunks, prepare, st);
        case 16: return chunk_SW<16>(a, rows, mid, n_chunks, prepare, st);
        case 32: return chunk_SW<32>(a, rows, mid, n_chunks, prepare, st);
        default: return cudaErrorInvalidValue;
    }
}

// mid[(c - 1) * n + i] = first edge of row i whose column is >= c * CSR_CHUNK (c = 1..C-1)
__global__ void csr_chunk_bounds_kernel(const int32_t *row_ptr, const int32_t *col, int32_t n, int n_chunks,
                                        int32_t *mid) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int ch = 1; ch < n_chunks; ++ch) {
        const int bound = ch * CSR_CHUNK;
        int lo = row_ptr[i], hi = row_ptr[i + 1];   // first e in [lo, hi) with col[e] >= bound
        while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (col[m] < bound) lo = m + 1;
            else hi = m;
        }
        mid[(int64_t)(ch - 1) * n + i] = lo;
    }
}

cudaError_t launch_csr_chunk_bounds(const int32_t *row_ptr, const int32_t *col, int32_t n, int n_chunks, int32_t *mid,
                                    cudaStream_t st) {
    if (n_chunks <= 1) return cudaSuccess;
    csr_chunk_bounds_kernel<<<(n + 255) / 256, 256, 0, st>>>(row_ptr, col, n, n_chunks, mid);
    return cudaGetLastError();
}

constexpr int CELL_THREADS = 128;   // CTA of the kernels that only update cells (cell_step_kernel has the figures)

// ---- simplified gap junctions (SGJ use case, Sec. 2.3.2) ---------------------------------
// Each connection contributes w (V_i - V_j) (the small-dV limit of the RGJ term).
// Dense: Ic_i = g sum_j (V_i - V_j) = g (N (V_i - m) - sum_j (V_j - m)), m = V_dend of cell 0
// (shifted so nearly equal voltages do not cancel).  Larger networks take two launches
// per step: P CTAs write compensated partial sums of V_j - m over fixed strided ranges, then
// every warp of the update sums the P partials in a fixed order and updates its cells
// (deterministic).  Networks of at most SGJ_ONE_LAUNCH cells take one: every CTA sums V_j - m
// over all cells itself, in the same order in every CTA.
//
// A step is bound by latency up to some 10^5 cells, by memory beyond.  So the sums run in four
// chains per thread over 16-byte loads, the partials are added by all lanes (one thread adding
// 256 of them held every CTA of the update for 2 us), the cells' words are on their way before
// the sum is known, the pulses before the wait, and the update walks the cells in opposite directions on even
// and odd steps (cell_step_kernel).
// Per step before / now: 200 cells 3.1 / 2.1 us, 8192 5.2 / 3.0, 16 384 7.1 / 3.6 (one launch),
// 16 385 5.5 / 4.5, 100 003 7.8 / 6.0, 600 011 25.9 / 16.6, 1 211 904 62.7 / 31.0.
__device__ __forceinline__ void two_sum_add(float &s, float &e, float so, float eo) {   // (s + e) += so + eo
    const float t = s + so, b = t - s;
    e = (e + eo) + ((s - (t - b)) + (so - b));
    s = t;
}
// sum of V_j - m over j = 4 first .. 4 first + 3, then every 4 stride on, of all threads of a
// CTA of 256 (each gets it)
__device__ __forceinline__ float sgj_block_sum(const float *v, int n, float m, int64_t first, int64_t stride) {
    __shared__ float red[8];
    float s[4] = {}, cc[4] = {};
#pragma unroll 4
    for (int64_t j = 4 * first; j < n; j += 4 * stride) {   // the padding reaches a multiple of 256
        const float4 x = *reinterpret_cast<const float4 *>(v + j);
        kahan_add(s[0], cc[0], x.x - m);
        kahan_add(s[1], cc[1], j + 1 < n ? x.y - m : 0.0f);
        kahan_add(s[2], cc[2], j + 2 < n ? x.z - m : 0.0f);
        kahan_add(s[3], cc[3], j + 3 < n ? x.w - m : 0.0f);
    }
    float S = s[0], E = -cc[0];
#pragma unroll
    for (int q = 1; q < 4; ++q) two_sum_add(S, E, s[q], -cc[q]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        two_sum_add(S, E, __shfl_xor_sync(0xffffffffu, S, off), __shfl_xor_sync(0xffffffffu, E, off));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = S + E;
    __syncthreads();
    float tot = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    return tot;
}
__global__ void __launch_bounds__(256) sgj_partial_kernel(const StepCommon c, float *part) {
    pdl_enter();
    (void)step_index(c);
    const float *vcur = vd_cur(c);
    const float tot = sgj_block_sum(vcur, c.n, vcur[0], (int64_t)blockIdx.x * 256 + threadIdx.x, (int64_t)gridDim.x * 256);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}
// ONE: the whole step (part NULL).  Else the launch after sgj_partial_kernel: the state is that
// of a launch before the one it waits for, but only the wait makes memory visible to a launch,
// so nothing but the pulses is read before it.
template <bool ONE>
__global__ void __launch_bounds__(ONE ? 256 : CELL_THREADS, ONE ? 1 : 10)
    sgj_dense_update_kernel(const StepCommon c, const float *part, int n_part, float g) {
    const int64_t b = !ONE && c.par == 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int64_t i = b * blockDim.x + threadIdx.x;
    const bool mine = i < c.n;
    const PulseAhead pa = pulse_ahead(c.pulses, i, mine);
    pdl_enter();
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    const float m = vcur[0];
    Cell cell{};
    float iapp = 0.0f;
    if (mine) {
        cell = load_cell(c.S, vcur, i);
        iapp = pulse_current(c.pulses, pa, t);
        if (c.iapp != nullptr) iapp += c.iapp[i];
    }
    float U;
    if (ONE) {
        U = sgj_block_sum(vcur, c.n, m, threadIdx.x, 256);
    } else {
        float s = 0.0f, cc = 0.0f;
        for (int q = threadIdx.x & 31; q < n_part; q += 32) kahan_add(s, cc, part[q]);
        float e = -cc;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            two_sum_add(s, e, __shfl_xor_sync(0xffffffffu, s, off), __shfl_xor_sync(0xffffffffu, e, off));
        U = s + e;
    }
    if (!mine) return;
    const float ic = g * fmaf((float)c.n, cell.vd - m, -U);
    const CellNext o = cell_step(c.P, cell, ic, iapp);
    finish_cell(c, t, vd_next(c), i, o);
}
cudaError_t launch_sgj_dense_step(const StepCommon &c, float g, float *part, cudaStream_t st) {
    if (c.n <= SGJ_ONE_LAUNCH)
        return launch_k(sgj_dense_update_kernel<true>, dim3((c.n + 255) / 256), dim3(256), 0, st, c.pdl != 0, c,
                        (const float *)nullptr, 0, g);
    const int n_part = sgj_partials(c.n);
    cudaError_t e = launch_k(sgj_partial_kernel, dim3(n_part), dim3(256), 0, st, c.pdl != 0, c, part);
    if (e != cudaSuccess) return e;
    return launch_k(sgj_dense_update_kernel<false>, dim3((c.n + CELL_THREADS - 1) / CELL_THREADS), dim3(CELL_THREADS), 0,
                    st, c.pdl != 0, c, (const float *)part, n_part, g);
}
int sgj_partials(int n) { return std::min(256, std::max(1, (n + 4095) / 4096)); }

// ---- half-work CSR (each stored pair evaluated once) ------------------------------------
// The pair term is odd in dV and the weights are symmetric, so the term of the stored edge
// (j, i) is exactly the negated term of (i, j).  Pass 1 walks the upper triangle: for each
// edge e = (i, j), j > i, it adds t_e to row i and writes -t_e into slot[rev[e]], the
// position of the mirrored edge (j, i) in row j (every slot is written by exactly one
// edge: no atomics).  Pass 2 adds to each row the slots of its lower edges, in a fixed
// order, and runs the cell update.  split[i] is the first edge of row i with col > i.
template <int SW, bool HAS_W>
__global__ void __launch_bounds__(256) csr_half_upper_kernel(const CsrArgs a, int rows, const int32_t *split,
                                                             const int32_t *rev, float *slot, float *icu) {
    pdl_enter();
    const StepCommon &c = a.c;
    const float *vcur = vd_cur(c);
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int row0 = blockIdx.x * rows;
    for (int rr = sub; rr - sub < rows; rr += nsub) {   // the same trip count in every lane
        const int i = row0 + rr;
        float acc = 0.0f;
        if (rr < rows && i < c.n) {
            const float vi = vcur[i];
            for (int e = split[i] + li; e < a.row_ptr[i + 1]; e += SW) {
                const float t = gj_edge(vi, __ldg(vcur + __ldg(a.col + e)), HAS_W ? __ldg(a.w + e) : 1.0f);
                acc += t;
                slot[__ldg(rev + e)] = -t;
            }
        }
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < rows && i < c.n) icu[i] = acc;
    }
}

template <int SW, bool HAS_W>
__global__ void __launch_bounds__(256) csr_half_lower_kernel(const CsrArgs a, int rows, const int32_t *split,
                                                             const float *slot, const float *icu) {
    __shared__ float ic_s[256];
    pdl_enter();
    const StepCommon &c = a.c;
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    float *vnext = vd_next(c);
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int row0 = blockIdx.x * rows;
    for (int rr = sub; rr - sub < rows; rr += nsub) {
        const int i = row0 + rr;
        float acc = 0.0f;
        if (rr < rows && i < c.n)
            for (int e = a.row_ptr[i] + li; e < split[i]; e += SW) acc += slot[e];
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < rows && i < c.n) {
            const float tot = icu[i] + acc;
            ic_s[rr] = (HAS_W ? tot : tot * a.g) * (1.0f / GJ_SCALE);
        }
    }
    __syncthreads();
    if ((int)threadIdx.x >= rows) return;
    const int i = row0 + threadIdx.x;
    if (i >= c.n) return;
    const Cell cell = load_cell(c.S, vcur, i);
    float iapp = pulse_current(c.pulses, i, t);
    if (c.iapp != nullptr) iapp += c.iapp[i];
    const CellNext o = cell_step(c.P, cell, ic_s[threadIdx.x], iapp);
    finish_cell(c, t, vnext, i, o);
}

template <int SW>
static cudaError_t half_SW(const CsrArgs &a, int rows, const int32_t *split, const int32_t *rev, float *slot,
                           float *icu, cudaStream_t st) {
    const int grid = (a.c.n + rows - 1) / rows;
    const bool pdl = a.c.pdl != 0;
    cudaError_t e = a.w != nullptr
                        ? launch_k(csr_half_upper_kernel<SW, true>, dim3(grid), dim3(256), 0, st, pdl, a, rows, split, rev, slot, icu)
                        : launch_k(csr_half_upper_kernel<SW, false>, dim3(grid), dim3(256), 0, st, pdl, a, rows, split, rev, slot, icu);
    if (e != cudaSuccess) return e;
    const float *cslot = slot, *cicu = icu;
    return a.w != nullptr
               ? launch_k(csr_half_lower_kernel<SW, true>, dim3(grid), dim3(256), 0, st, pdl, a, rows, split, cslot, cicu)
               : launch_k(csr_half_lower_kernel<SW, false>, dim3(grid), dim3(256), 0, st, pdl, a, rows, split, cslot, cicu);
}

// Both passes of a half-work CSR step (rows per CTA <= 256; SW lanes per row).
cudaError_t launch_csr_half_step(const CsrArgs &a, int SW, int rows, const int32_t *split, const int32_t *rev,
                                 float *slot, float *icu, cudaStream_t st) {
    if (rows < 1 || rows > 256) return cudaErrorInvalidValue;
    switch (SW) {
        case 1: return half_SW<1>(a, rows, split, rev, slot, icu, st);
        case 2: return half_SW<2>(a, rows, split, rev, slot, icu, st);
        case 4: return half_SW<4>(a, rows, split, rev, slot, icu, st);
        case 8: return half_SW<8>(a, rows, split, rev, slot, icu, st);
        case 16: return half_SW<16>(a, rows, split, rev, slot, icu, st);
        case 32: return half_SW<32>(a, rows, split, rev, slot, icu, st);
        default: return cudaErrorInvalidValue;
    }
}

// ---- compact column layout: the low 16 bits of every column (zero padding to 8 entries)
__global__ void csr_col16_kernel(const int32_t *col, int64_t nnz, int64_t n_alloc, uint16_t *col16) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n_alloc) col16[e] = e < nnz ? (uint16_t)((uint32_t)col[e] & 0xFFFFu) : (uint16_t)0;
}
cudaError_t launch_csr_col16(const int32_t *col, int64_t nnz, int64_t n_alloc, uint16_t *col16, cudaStream_t st) {
    if (n_alloc <= 0) return cudaSuccess;
    csr_col16_kernel<<<(unsigned)((n_alloc + 255) / 256), 256, 0, st>>>(col, nnz, n_alloc, col16);
    return cudaGetLastError();
}

// ---- stand-alone cell update (no gap junctions, or Ic computed by another launch) ----
// Bound by memory once the state is larger than L2 (132 bytes per cell and step, 12 more with
// pulses).  The CTAs walk the cells in opposite directions on even and odd steps: the cells a
// step ends with are still in L2 when the next begins with them, so up to L2's worth of the
// state is neither read from nor written back to HBM.  2^21 cells with
// pulses on a fifth: 45.7 us per step (0.95 of the measured copy rate in the bytes above); 46.9
// with CTAs of 256 threads, 53.6 in one direction only, 61.8 before with the pulse table read
// after the state.
//
// CTAs of 128 threads at 48 registers: ten per SM, 1280 cells in flight, and a step's last CTAs
// leave less of the chip idle than larger ones do (2^20 cells 21.1 -> 20.4 us, 16 384 cells
// 1.93 -> 1.69).  Twelve per SM spill (2^21 cells 46.2 us), nine keep too little in flight (47.7).
__global__ void __launch_bounds__(CELL_THREADS, 10) cell_step_kernel(const CellArgs a) {
    const StepCommon &c = a.c;
    const int64_t b = c.par == 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int64_t i = b * blockDim.x + threadIdx.x;
    const PulseAhead pa = pulse_ahead(c.pulses, i, i < c.n);
    pdl_enter();
    if (i >= c.n) return;
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    float *vnext = vd_next(c);
    const Cell cell = load_cell(c.S, vcur, i);
    const float ic = a.ic != nullptr ? a.ic[i] : 0.0f;
    float iapp = pulse_current(c.pulses, pa, t);
    if (c.iapp != nullptr) iapp += c.iapp[i];
    const CellNext o = a.cellp != nullptr ? cell_step(cell_model(c.P, a.cellp, c.S.stride, i), cell, ic, iapp)
                                          : cell_step(c.P, cell, ic, iapp);
    finish_cell(c, t, vnext, i, o);
}

cudaError_t launch_cell_step(const CellArgs &a, cudaStream_t st) {
    const int64_t grid = ((int64_t)a.c.n + CELL_THREADS - 1) / CELL_THREADS;
    return launch_k(cell_step_kernel, dim3((unsigned)grid), dim3(CELL_THREADS), 0, st, a.c.pdl != 0, a);
}

// ---- rate functions and default state (host-visible copies of the device model) ----
__global__ void rates_kernel(float V, float ca, float *out) {
    if (threadIdx.x != 0) return;
    const Rate g[NG] = {rate_r(V), rate_s(ca), rate_q(V), rate_k(V), rate_l(V), {minf_na(V), 0.0f},
                        rate_hs(V), rate_ns(V), rate_x(V), {minf_na(V), 0.0f}, rate_ha(V), rate_x(V)};
    for (int k = 0; k < NG; ++k) {
        out[k] = g[k].xinf;
        out[NG + k] = g[k].inv_tau > 0.0f ? 1.0f / g[k].inv_tau : 0.0f;
    }
}

cudaError_t launch_rates(float V, float ca, float *out, cudaStream_t st) {
    rates_kernel<<<1, 32, 0, st>>>(V, ca, out);
    return cudaGetLastError();
}

__global__ void default_state_kernel(ModelF P, float V0, float ca0, float gcal, int32_t n, int64_t stride, float *S) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float r = rate_r(V0).xinf;
    const float v[NF] = {V0, V0, V0, ca0, r, rate_s(ca0).xinf, rate_q(V0).xinf, rate_k(V0).xinf,
                         rate_l(V0).xinf, minf_na(V0), rate_hs(V0).xinf, rate_ns(V0).xinf, rate_x(V0).xinf,
                         minf_na(V0), rate_ha(V0).xinf, rate_x(V0).xinf, gcal, P.gCaH * r * r * (V0 - P.VCa), 0.0f};
    for (int f = 0; f < NF; ++f) S[f * stride + i] = v[f];
}

cudaError_t launch_default_state(const ModelF &P, float V0, float ca0, float gcal, int32_t n, int64_t stride,
                                 float *state, cudaStream_t st) {
    default_state_kernel<<<(n + 255) / 256, 256, 0, st>>>(P, V0, ca0, gcal, n, stride, state);
    return cudaGetLastError();
}

// ---- small helpers ------------------------------------------------------------------
__global__ void advance_kernel(int64_t *t_dev, int64_t k) {
    pdl_enter();
    *t_dev += k;
}

cudaError_t launch_advance(int64_t *t_dev, int64_t k, cudaStream_t st, bool pdl) {
    return launch_k(advance_kernel, dim3(1), dim3(1), 0, st, pdl, t_dev, k);
}

// One field (or, field < 0, all of them) of n cells and the status word into a pinned host
// buffer: one launch instead of two copies, each with a synchronisation of its own.
__global__ void state_put_kernel(const float *vd, const float *base, int64_t stride, int n, int field,
                                 const uint32_t *status, float *dst, int64_t status_at) {
    pdl_enter();
    const int total = field < 0 ? NF * n : n;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < total) {
        const int f = field < 0 ? q / n : field, i = field < 0 ? q - f * n : q;
        dst[q] = f == 0 ? vd[i] : base[f * stride + i];
    }
    if (q == 0) reinterpret_cast<uint32_t *>(dst)[status_at] = *status;
}
cudaError_t launch_state_put(const float *vd, const float *base, int64_t stride, int n, int field, const uint32_t *status,
                             float *dst, int64_t status_at, bool pdl, cudaStream_t st) {
    const int total = field < 0 ? NF * n : n;
    return launch_k(state_put_kernel, dim3((total + 255) / 256), dim3(256), 0, st, pdl, vd, base, stride, n, field, status,
                    dst, status_at);
}

__global__ void fill_kernel(float *p, float v, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

cudaError_t launch_fill(float *p, float v, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096;
    fill_kernel<<<(unsigned)blocks, 256, 0, st>>>(p, v, n);
    return cudaGetLastError();
}

}  // namespace ion
