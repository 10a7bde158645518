// ion_batch.cu -- many independent networks advanced together, a few launches per time step.
//
// Parameter sweeps run many small networks of uneven sizes and densities.  Each network
// b gets a segment of the state arrays starting at seg_b (a multiple of 256 cells, the
// tail padded like a single network's V_dend), so networks can stage their V_dend with one
// 16-byte aligned bulk copy.  The work of a step is a list of tiles (network, first row,
// rows): a dense tile is blocks of 8 warps x R rows of one network against all of that
// network's columns (the single-network pair loop, ion_dense_core.cuh), a CSR tile is up to
// 256 rows, from the network's sliced rows where its V_dend is staged; every tile then runs
// the explicit-Euler update of its rows.  The networks are dealt to up to three chains of
// launches that run side by side (dense and CSR networks have kernels of their own), and
// within a chain tiles are ordered by decreasing cost so the hardware scheduler packs the
// long ones first; the launches of K steps are captured into one CUDA graph and replayed.
// ion_autotune times the tile shapes and keeps the fastest.
//
// What bounds it: the dense chains' pair loops and the updates between them (256 networks: the
// dense launches keep the XU pipe 53 % and issue 63 % busy, the CSR launch is bound by latency
// beside them).  A sweep of 96 networks of 32-4096 cells, us per step: 20.3 (the 48 dense networks
// alone 17.5, the 48 CSR ones 8.8); one launch per step with fixed tiles, 16-bit rows with heads
// and tails, state and pulses read after the sums took 30.4.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <vector>

#include "ion.h"
#include "ion_csr_core.cuh"
#include "ion_dense_core.cuh"
#include "ion_kernels.cuh"
#include "ion_sim.h"

namespace ion {

enum TileKind : int32_t { TILE_DENSE = 0, TILE_CSR = 1 };
// CSR tile modes: every weight of the network equals T.g; 16-bit network-local columns
// (col16); the network's V_dend staged in shared memory (with TILE_C16); its rows stored in
// slices (with TILE_STAGE_V)
enum TileMode : int32_t { TILE_UNIFORM_W = 1, TILE_C16 = 2, TILE_STAGE_V = 4, TILE_SLICED = 8 };

struct BatchTile {
    int32_t kind;
    int32_t seg;     // first cell of the network's segment
    int32_t n;       // cells of the network
    int32_t n_pad;   // padded length of the segment (multiple of 256)
    int32_t row0;    // first row (global cell index) of the tile
    int32_t rows;    // rows of the tile
    int32_t sw;      // CSR: lanes per row
    float g;         // dense: pair weight; CSR with TILE_UNIFORM_W: every edge weight
    int32_t mode;    // CSR: TileMode bits
    int32_t slice0;  // TILE_SLICED: the network's first slice
};

struct BatchArgs {
    StepCommon c;    // c.n = padded total, c.S = state over the padded index space
    const BatchTile *tiles;
    const int32_t *row_ptr;   // padded-index CSR of every CSR network (other rows empty)
    const int32_t *col;
    const uint16_t *col16;    // network-local columns (TILE_C16 networks)
    const float *w;
    const uint4 *scols;       // sliced columns (and weights) of the staged CSR networks
    const float4 *sw;
    const int32_t *soff;      // first round of each slice, and the end
    int32_t kahan;
    int32_t rows_max;         // rows of the largest tile (<= 256: one thread updates each)
    int32_t vbuf;             // floats of the V_dend buffer
};

// ---- sliced rows of a staged CSR network -----------------------------------------------------
// As in ion_csr_sliced.cu, without the sort and the bank order: a slice is 32 / SW consecutive
// rows of one network, SW lanes per row, its columns stored round by round (8 edges of every
// lane, 512 contiguous bytes), padded with the row's own column (dV = 0: adds exactly 0).  A
// row's sum depends on its edges and SW alone, not on the tile or piece it is computed in, so
// the per-step and the persistent kernel give the same bits.
template <bool HAS_W>
struct SliceAhead {
    static constexpr int D = HAS_W ? 2 : 4;   // rounds in flight per lane
    uint4 q[D];
    float4 wa[HAS_W ? D : 1], wb[HAS_W ? D : 1];
    int e0, n;                                // first round, rounds
    __device__ __forceinline__ void load(int j, int round, const uint4 *cols, const float4 *w) {
        const int lane = threadIdx.x & 31;
        q[j] = __ldg(cols + (int64_t)round * 32 + lane);
        if (HAS_W) {
            wa[j] = __ldg(w + (int64_t)round * 64 + lane);
            wb[j] = __ldg(w + (int64_t)round * 64 + 32 + lane);
        }
    }
    // the header and first rounds of a slice
    __device__ __forceinline__ void begin(int slice, const int32_t *off, const uint4 *cols, const float4 *w) {
        e0 = __ldg(off + slice);
        n = __ldg(off + slice + 1) - e0;
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (j < n) load(j, e0 + j, cols, w);
    }
};
// Currents of rows [r0, r0 + rows) of a network (local rows) into ic_s; `ah` holds this warp's
// first slice already (slice_begin below).
template <bool HAS_W>
__device__ __forceinline__ void slice_rows(SliceAhead<HAS_W> &ah, int slice0, int lsw, int n, int r0, int rows,
                                           const int32_t *off, const uint4 *cols, const float4 *w, const float *vs,
                                           float g, float *ic_s) {
    constexpr int D = SliceAhead<HAS_W>::D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = 32 >> lsw, s0 = r0 / per, ns = (r0 + rows - 1) / per - s0 + 1;
    const VjSliced vj{vs};
    for (int s = warp; s < ns; s += 8) {
        if (s != warp) ah.begin(slice0 + s0 + s, off, cols, w);
        const int i = (s0 + s) * per + (lane >> lsw);
        const float vi = vs[min(i, n - 1)];
        float ks = 0.0f, kc = 0.0f;           // compensated over groups of D rounds
        for (int k = 0; k < ah.n; k += D) {
            float blk = 0.0f;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                if (k + j < ah.n) blk += csr_group16<HAS_W>(ah.q[j], ah.wa[HAS_W ? j : 0], ah.wb[HAS_W ? j : 0], vi, vj);
                if (k + D + j < ah.n) ah.load(j, ah.e0 + k + D + j, cols, w);
            }
            kahan_add(ks, kc, blk);
        }
        float acc = ks - kc;
        for (int o = (1 << lsw) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((lane & ((1 << lsw) - 1)) == 0 && i >= r0 && i < r0 + rows)
            ic_s[i - r0] = (HAS_W ? acc : acc * g) * (1.0f / GJ_SCALE);
    }
}
// This warp's first slice of rows [r0, ...) of a network
template <bool HAS_W>
__device__ __forceinline__ void slice_begin(SliceAhead<HAS_W> &ah, int slice0, int lsw, int r0, int rows,
                                            const int32_t *off, const uint4 *cols, const float4 *w) {
    const int per = 32 >> lsw, warp = threadIdx.x >> 5, s0 = r0 / per, ns = (r0 + rows - 1) / per - s0 + 1;
    if (warp < ns) ah.begin(slice0 + s0 + warp, off, cols, w);
}

// The same sums, one round loaded ahead, for the persistent kernel: groups of rounds in flight
// there (two kinds of rows and the pair loop in one kernel) spilled 440 to 560 bytes a thread, in
// the dense pieces' loops too, and a step of two 64-cell dense networks took 4.9 us; now 3.6.
template <bool HAS_W>
__device__ __forceinline__ void slice_rows_short(int slice0, int lsw, int n, int r0, int rows, const int32_t *off,
                                                 const uint4 *cols, const float4 *w, const float *vs, float g,
                                                 float *ic_s) {
    constexpr int D = SliceAhead<HAS_W>::D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = 32 >> lsw, s0 = r0 / per, ns = (r0 + rows - 1) / per - s0 + 1;
    const VjSliced vj{vs};
    for (int s = warp; s < ns; s += 8) {
        const int e0 = __ldg(off + slice0 + s0 + s), ne = __ldg(off + slice0 + s0 + s + 1) - e0;
        const int i = (s0 + s) * per + (lane >> lsw);
        const float vi = vs[min(i, n - 1)];
        const uint4 *pc = cols + (int64_t)e0 * 32 + lane;
        const float4 *pw = HAS_W ? w + (int64_t)e0 * 64 + lane : w;
        float ks = 0.0f, kc = 0.0f, blk = 0.0f;
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (ne > 0) q = __ldg(pc);
#pragma unroll 1
        for (int k = 0; k < ne; ++k) {
            const uint4 now = q;
            float4 wa, wb;
            if (HAS_W) {
                wa = __ldg(pw);
                wb = __ldg(pw + 32);
                pw += 64;
            }
            pc += 32;
            if (k + 1 < ne) q = __ldg(pc);
            blk += csr_group16<HAS_W>(now, wa, wb, vi, vj);
            if ((k & (D - 1)) == D - 1 || k + 1 == ne) {
                kahan_add(ks, kc, blk);
                blk = 0.0f;
            }
        }
        float acc = ks - kc;
        for (int o = (1 << lsw) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((lane & ((1 << lsw) - 1)) == 0 && i >= r0 && i < r0 + rows)
            ic_s[i - r0] = (HAS_W ? acc : acc * g) * (1.0f / GJ_SCALE);
    }
}

// The sliced columns (and weights) from the networks' 16-bit rows: a warp per slice.
struct SliceDesc {
    int32_t row, rows;   // first row (padded index), rows (<= 32 / SW)
    int32_t seg, lsw;
};
__global__ void __launch_bounds__(128) batch_slice_fill_kernel(const SliceDesc *desc, int n_slices, const int32_t *off,
                                                               const int32_t *row_ptr, const uint16_t *col16,
                                                               const float *w, uint16_t *cols, float *wout) {
    const int s = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (s >= n_slices) return;
    const SliceDesc d = desc[s];
    const int rr = lane >> d.lsw, sw = 1 << d.lsw, li = lane & (sw - 1);
    const bool has = rr < d.rows;
    const int i = d.row + (has ? rr : 0);
    const int b = row_ptr[i], e = has ? row_ptr[i + 1] : b;
    const int64_t r0 = off[s];
    const int rounds = off[s + 1] - (int)r0;
    const uint16_t self = (uint16_t)(i - d.seg);
    for (int k = 0; k < rounds; ++k)
        for (int t = 0; t < 8; ++t) {
            const int x = b + (k * sw + li) * 8 + t;
            const bool real = x < e;
            cols[((r0 + k) * 32 + lane) * 8 + t] = real ? col16[x] : self;
            if (wout) wout[((r0 + k) * 64 + (t >> 2) * 32 + lane) * 4 + (t & 3)] = real ? w[x] : 0.0f;
        }
}

// A row's sum by SW lanes, each lane's part of it; a row of more than eight rounds (64 SW edges) by
// its whole warp, one such row after the other (its sum in the row's lane 0).  All lanes of the
// warp call it; e0 == e1: no row.
template <int SW, bool HAS_W, class VJ>
__device__ __forceinline__ float batch_row16(const uint16_t *col16, const float *w, int e0, int e1, float vi, int li,
                                             VJ vj) {
    const bool far = SW < 32 && e1 - e0 > 64 * SW;
    float acc = far || e0 == e1 ? 0.0f : csr_row_sum16<SW, HAS_W, false>(col16, w, e0, e1, vi, li, vj);
    if (SW < 32) {
        const int lane = threadIdx.x & 31;
        for (uint32_t left = __ballot_sync(0xffffffffu, far && li == 0); left != 0; left &= left - 1) {
            const int src = __ffs(left) - 1;
            float sum = csr_row_sum16<32, HAS_W, false>(col16, w, __shfl_sync(0xffffffffu, e0, src),
                                                        __shfl_sync(0xffffffffu, e1, src),
                                                        __shfl_sync(0xffffffffu, vi, src), lane, vj);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            if (lane == src) acc = sum;
        }
    }
    return acc;
}

// CSR rows of a TILE_C16 tile: 16-bit local columns, V_dend from `vj`
template <int SW, bool HAS_W, class VJ>
__device__ __forceinline__ void batch_csr_rows16(const BatchArgs &a, const BatchTile &T, const float *vcur, VJ vj,
                                                 float *ic_s) {
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int iters = (T.rows + nsub - 1) / nsub;
    int e0n = 0, e1n = 0;   // the next row's bounds and V_dend, loaded one row ahead
    float vin = 0.0f;
    if (sub < T.rows) {
        e0n = a.row_ptr[T.row0 + sub];
        e1n = a.row_ptr[T.row0 + sub + 1];
        vin = vcur[T.row0 + sub];
    }
    for (int it = 0; it < iters; ++it) {
        const int rr = sub + it * nsub;
        const int e0 = e0n, e1 = e1n;
        const float vi = vin;
        if (rr + nsub < T.rows) {
            e0n = a.row_ptr[T.row0 + rr + nsub];
            e1n = a.row_ptr[T.row0 + rr + nsub + 1];
            vin = vcur[T.row0 + rr + nsub];
        }
        const bool has = rr < T.rows;
        float acc = batch_row16<SW, HAS_W>(a.col16, a.w, has ? e0 : 0, has ? e1 : 0, vi, li, vj);
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < T.rows) ic_s[rr] = (HAS_W ? acc : acc * T.g) * (1.0f / GJ_SCALE);
    }
}
template <int SW, class VJ>
__device__ __forceinline__ void batch_csr_rows16_w(const BatchArgs &a, const BatchTile &T, const float *vcur, VJ vj,
                                                   float *ic_s) {
    if (T.mode & TILE_UNIFORM_W) batch_csr_rows16<SW, false>(a, T, vcur, vj, ic_s);
    else batch_csr_rows16<SW, true>(a, T, vcur, vj, ic_s);
}
template <class VJ>
__device__ __forceinline__ void batch_csr_tile16(const BatchArgs &a, const BatchTile &T, const float *vcur, VJ vj,
                                                 float *ic_s) {
    switch (T.sw) {
        case 1: batch_csr_rows16_w<1>(a, T, vcur, vj, ic_s); break;
        case 2: batch_csr_rows16_w<2>(a, T, vcur, vj, ic_s); break;
        case 4: batch_csr_rows16_w<4>(a, T, vcur, vj, ic_s); break;
        case 8: batch_csr_rows16_w<8>(a, T, vcur, vj, ic_s); break;
        case 16: batch_csr_rows16_w<16>(a, T, vcur, vj, ic_s); break;
        default: batch_csr_rows16_w<32>(a, T, vcur, vj, ic_s); break;
    }
}

template <int SW>
__device__ __forceinline__ void batch_csr_rows(const BatchArgs &a, const BatchTile &T, const float *vcur, float *ic_s) {
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    const int iters = (T.rows + nsub - 1) / nsub;
    const bool vec = ((uintptr_t)a.col % 16 == 0) && ((uintptr_t)a.w % 16 == 0);
    int e0n = 0, e1n = 0;   // the next row's bounds and V_dend, loaded one row ahead
    float vin = 0.0f;
    if (sub < T.rows) {
        e0n = a.row_ptr[T.row0 + sub];
        e1n = a.row_ptr[T.row0 + sub + 1];
        vin = vcur[T.row0 + sub];
    }
    for (int it = 0; it < iters; ++it) {
        const int rr = sub + it * nsub;
        const int e0 = e0n, e1 = e1n;
        const float vi = vin;
        if (rr + nsub < T.rows) {
            e0n = a.row_ptr[T.row0 + rr + nsub];
            e1n = a.row_ptr[T.row0 + rr + nsub + 1];
            vin = vcur[T.row0 + rr + nsub];
        }
        float acc = 0.0f;
        if (rr < T.rows)
            acc = vec ? csr_row_sum<SW, true, true>(vcur, a.col, a.w, e0, e1, vi, li)
                      : csr_row_sum<SW, false, true>(vcur, a.col, a.w, e0, e1, vi, li);
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < T.rows) ic_s[rr] = acc * (1.0f / GJ_SCALE);
    }
}

// ---- the per-step kernels ------------------------------------------------------------------
// What both do around the row currents: the tile's pulses are read before the wait on the
// previous step (neither they nor the tile list change between steps), its rows' state words
// travel to shared memory while the sums run, and one thread per row updates its cell.
struct TileRow {
    int64_t i;            // this thread's cell
    bool has;
    PulseAhead pa;
};
__device__ __forceinline__ TileRow tile_row(const BatchArgs &a, const BatchTile &T) {
    const bool has = (int)threadIdx.x < T.rows;
    const int64_t i = T.row0 + (int64_t)threadIdx.x;
    return {i, has, pulse_ahead(a.c.pulses, i, has)};
}
__device__ __forceinline__ void tile_stage(const BatchArgs &a, const TileRow &r, const float *vcur, float *cs) {
    if (r.has)
#pragma unroll
        for (int w = 0; w < NCW; ++w)
            cp_async4(cs + w * a.rows_max + threadIdx.x, (w == 0 ? vcur : a.c.S.f(cell_word_field(w))) + r.i);
    cp_async_commit();
}
__device__ __forceinline__ void tile_update(const BatchArgs &a, const TileRow &r, int64_t t, const float *cs, float ic) {
    float iapp = pulse_current(a.c.pulses, r.pa, t);
    if (a.c.iapp != nullptr) iapp += a.c.iapp[r.i];
    const CellNext o = cell_step(a.c.P, staged_cell(cs, a.rows_max, threadIdx.x), ic, iapp);
    finish_cell(a.c, t, vd_next(a.c), r.i, o);
}

// Dense tiles, 8 warps: blocks of 8 row groups of R rows against the network's staged columns.
template <int R>
__global__ void __launch_bounds__(256) batch_dense_kernel(const BatchArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ float red_s[32], red_c[32];
    const BatchTile T = a.tiles[blockIdx.x];
    const StepCommon &c = a.c;
    const TileRow row = tile_row(a, T);
    float *cs = reinterpret_cast<float *>(smem_raw) + a.vbuf + 8 * R;
    const DenseSmem sm = dense_smem(smem_raw, T.n_pad);   // one tile: n_pad <= 8192
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_enter();
    const float *vcur = vd_cur(c), *net_v = vcur + T.seg;
    if (threadIdx.x == 0) issue_tile(sm, net_v, T.n_pad, 0, bar);
    tile_stage(a, row, vcur, cs);
    const int64_t t = step_index(c);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mine = threadIdx.x;
    const float C = net_v[0] * GJ_SCALE;
    const int local0 = T.row0 - T.seg;
    uint32_t uses[2] = {0u, 0u};
    float U = 0.0f, ic = 0.0f;
    for (int sub = 0; sub < T.rows; sub += 8 * R) {
        float ui[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int rr = sub + warp * R + r;
            ui[r] = rr < T.rows ? gj_u(net_v[local0 + rr], C) : 0.0f;
        }
        float tot[R], Us, Uc;
        if (!gj_pass<R, 1, true>(sm, sub == 0 ? net_v : nullptr, T.n, T.n_pad, bar, uses, C, ui, 0, lane, a.kahan, tot, Us, Uc,
                           sub == 0)) {
            if (threadIdx.x == 0) {
                atomicOr(c.status, (uint32_t)ST_TIMEOUT);
                (void)mbar_wait_bounded(&bar[0], uses[0] & 1u);
            }
            cp_async_wait_all();
            return;
        }
        if (sub > 0) __syncthreads();   // the last block's partial sums have been read
        gj_reduce<R, 1>(sm, tot, Us, Uc, warp, 0, lane, red_s, red_c);
        if (sub == 0) U = gj_sum_u(red_s, red_c);
        const int rr = mine - sub;      // the thread that owns a row of this block takes its current
        if (row.has && rr >= 0 && rr < 8 * R) ic = row_current<1>(sm, rr, gj_u(cs[mine], C), T.n, U, T.g);
    }
    if (row.has) tile_update(a, row, t, cs, ic);
}

// CSR tiles (and networks without junctions)
__global__ void __launch_bounds__(256) batch_csr_kernel(const BatchArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ float ic_s[256];
    const BatchTile T = a.tiles[blockIdx.x];
    const StepCommon &c = a.c;
    const TileRow row = tile_row(a, T);
    float *vs = reinterpret_cast<float *>(smem_raw), *cs = vs + a.vbuf;
    const bool staged = (T.mode & TILE_STAGE_V) != 0, uniform = (T.mode & TILE_UNIFORM_W) != 0;
    const bool sliced = (T.mode & TILE_SLICED) != 0;
    const int lsw = 31 - __clz(T.sw), local0 = T.row0 - T.seg;
    // the first slice of this warp, before the wait too
    SliceAhead<false> au;
    SliceAhead<true> aw;
    if (sliced && uniform) slice_begin(au, T.slice0, lsw, local0, T.rows, a.soff, a.scols, a.sw);
    else if (sliced) slice_begin(aw, T.slice0, lsw, local0, T.rows, a.soff, a.scols, a.sw);
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_enter();
    const float *vcur = vd_cur(c);
    if (staged && threadIdx.x == 0) {   // the network's V_dend (n_pad <= TJ floats)
        mbar_expect_tx(&bar, (uint32_t)T.n_pad * 4u);
        bulk_g2s(vs, vcur + T.seg, (uint32_t)T.n_pad * 4u, &bar);
    }
    tile_stage(a, row, vcur, cs);
    const int64_t t = step_index(c);
    if (staged) {
        const bool landed = threadIdx.x >= 32 || mbar_wait_bounded(&bar, 0u);
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) {
                atomicOr(c.status, (uint32_t)ST_TIMEOUT);
                (void)mbar_wait_bounded(&bar, 0u);
            }
            cp_async_wait_all();
            return;
        }
        if (!sliced) batch_csr_tile16(a, T, vcur, VjSliced{vs}, ic_s);
        else if (uniform) slice_rows(au, T.slice0, lsw, T.n, local0, T.rows, a.soff, a.scols, a.sw, vs, T.g, ic_s);
        else slice_rows(aw, T.slice0, lsw, T.n, local0, T.rows, a.soff, a.scols, a.sw, vs, T.g, ic_s);
    } else if (T.mode & TILE_C16) {
        batch_csr_tile16(a, T, vcur, VjGlobal{vcur + T.seg}, ic_s);
    } else {
        switch (T.sw) {
            case 1: batch_csr_rows<1>(a, T, vcur, ic_s); break;
            case 2: batch_csr_rows<2>(a, T, vcur, ic_s); break;
            case 4: batch_csr_rows<4>(a, T, vcur, ic_s); break;
            case 8: batch_csr_rows<8>(a, T, vcur, ic_s); break;
            case 16: batch_csr_rows<16>(a, T, vcur, ic_s); break;
            default: batch_csr_rows<32>(a, T, vcur, ic_s); break;
        }
    }
    cp_async_wait_all();
    __syncthreads();
    if (row.has) tile_update(a, row, t, cs, ic_s[threadIdx.x]);
}

// ---- persistent form: many steps of every network in one cooperative launch -------------
// The host cuts every network into pieces of at most 256 rows (one piece for a network
// whose work fits a CTA's share of a step, several for the large ones) and deals the
// pieces out to CTAs that are all resident at once.  Each CTA walks its pieces once per
// step.  Before reading network b's V_dend(t) it waits (bounded) until every piece of b
// has finished step t - 1: each piece adds 1 to b's arrival counter when its rows' states
// and V_dend(t + 1) are written, so b is ready for step k of the launch once its counter
// holds k x (pieces of b).  No CTA ever waits on a later step than its own, so the CTA
// with the oldest step always progresses: the launch cannot deadlock, and no grid-wide
// barrier is needed.  The pair loop, the CSR row sums and the cell update are those of
// the per-step kernels (the same lanes per row give the same sums, whatever the rows per
// warp), so the states equal those of the per-step launches bit for bit.
struct PersistItem {
    int32_t kind;     // TILE_DENSE or TILE_CSR
    int32_t net;      // network (index of its arrival counter)
    int32_t seg, n, n_pad;
    int32_t row0;     // first row (padded cell index)
    int32_t rows;     // 1..256
    int32_t pieces;   // pieces of this network (arrivals per step)
    int32_t sw;       // CSR: lanes per row
    int32_t mode;     // CSR: TileMode bits
    int32_t slice0;   // TILE_SLICED: the network's first slice
    float g;
};

struct BatchPersistArgs {
    StepCommon c;              // par = -1; the launch runs steps *t_dev .. *t_dev + n_steps - 1
    const PersistItem *items;  // every CTA's pieces, CTA after CTA
    const int32_t *cta_off;    // [gridDim.x + 1] first piece of each CTA
    const int32_t *row_ptr;
    const uint16_t *col16;
    const float *w;
    const uint4 *scols;        // as in BatchArgs
    const float4 *sw;
    const int32_t *soff;
    uint32_t *cnt;             // arrival counter per network (zeroed before the launch)
    uint32_t *abort_flag;      // set by a CTA whose wait gave up (zeroed before the launch)
    uint64_t timeout_ns;
    int32_t n_steps;
    int32_t vbuf;              // floats of the staged V_dend buffer (>= n_pad of staged networks)
    int32_t kahan;
    int64_t debug_delay_ns;    // test hook: CTA 0 sleeps this long before its first piece
};

// Bounded wait until *cnt has reached target (mod 2^32), by one thread.  On timeout sets
// the timeout status bit and the abort word; returns false on timeout or abort.
__device__ __forceinline__ bool wait_arrivals(const uint32_t *cnt, uint32_t target, uint32_t *abort_flag,
                                              uint64_t timeout_ns, uint32_t *status) {
    if (arrivals_reached(ld_acquire_gpu(cnt), target)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        if (arrivals_reached(ld_acquire_gpu(cnt), target)) return true;
        if ((it & 63u) == 0u) {
            if (ld_acquire_gpu(abort_flag) != 0u) return false;
            if (globaltimer_ns() - t0 > timeout_ns || it > (1u << 30)) {
                atomicOr(status, (uint32_t)ST_TIMEOUT);
                atomicExch(abort_flag, 1u);
                return false;
            }
        }
    }
}

// Rows [row0, row0 + rows) of a CSR piece with 16-bit local columns: SW lanes per row,
// row voltages from vrow(local row), neighbour voltages from vj.
template <int SW, bool HAS_W, class VR, class VJ>
__device__ __forceinline__ void persist_csr_rows(const BatchPersistArgs &a, const PersistItem &P, VR vrow, VJ vj,
                                                 float *ic_s) {
    const int sub = threadIdx.x / SW, li = threadIdx.x % SW, nsub = blockDim.x / SW;
    for (int rr = sub; rr - sub < P.rows; rr += nsub) {   // the same trip count in every lane
        int e0 = 0, e1 = 0;
        float vi = 0.0f;
        if (rr < P.rows) {
            const int i = P.row0 + rr;
            e0 = a.row_ptr[i];
            e1 = a.row_ptr[i + 1];
            vi = vrow(i - P.seg);
        }
        float acc = batch_row16<SW, HAS_W>(a.col16, a.w, e0, e1, vi, li, vj);
#pragma unroll
        for (int off = SW / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (li == 0 && rr < P.rows) ic_s[rr] = (HAS_W ? acc : acc * P.g) * (1.0f / GJ_SCALE);
    }
}
template <class VR, class VJ>
__device__ __forceinline__ void persist_csr_piece(const BatchPersistArgs &a, const PersistItem &P, VR vrow, VJ vj,
                                                  float *ic_s) {
#define ION_CSR_SW(SWV)                                                                    \
    if (P.mode & TILE_UNIFORM_W) persist_csr_rows<SWV, false>(a, P, vrow, vj, ic_s);       \
    else persist_csr_rows<SWV, true>(a, P, vrow, vj, ic_s);
    switch (P.sw) {
        case 1: ION_CSR_SW(1) break;
        case 2: ION_CSR_SW(2) break;
        case 4: ION_CSR_SW(4) break;
        case 8: ION_CSR_SW(8) break;
        case 16: ION_CSR_SW(16) break;
        default: ION_CSR_SW(32) break;
    }
#undef ION_CSR_SW
}

struct VRowSmem {
    const float *v;
    __device__ __forceinline__ float operator()(int j) const { return v[j]; }
};
struct VRowCG {
    const float *v;
    __device__ __forceinline__ float operator()(int j) const { return __ldcg(v + j); }
};

// 256 threads: 8 warps; dense pieces run 8 x R rows at a time.  Three CTAs per SM: a piece is a
// chain of latencies, and fewer, larger shares of the networks wait for fewer others.  us per step
// with four / three: 12 dense networks of 1792 cells 19.2 / 11.6, two networks of 500 5.2 / 4.4, 96
// networks of 32-4096 cells 43 / 45.
template <int R>
__global__ void __launch_bounds__(256, 3) batch_persist_kernel(const BatchPersistArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ float red_s[32], red_c[32];
    __shared__ float ic_s[256];
    __shared__ int ok_sh;
    float *vb = reinterpret_cast<float *>(smem_raw);   // the piece's network's V_dend(t)
    float *part = vb + a.vbuf;                          // 8 R row partials
    const StepCommon &c = a.c;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int it0 = a.cta_off[blockIdx.x], it1 = a.cta_off[blockIdx.x + 1];
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int64_t t0 = *c.t_dev;
    uint32_t phase = 0;
    if (a.debug_delay_ns > 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        const uint64_t d0 = globaltimer_ns();
        while (globaltimer_ns() - d0 < (uint64_t)a.debug_delay_ns) __nanosleep(1000);
    }
    for (int k = 0; k < a.n_steps; ++k) {
        const int64_t t = t0 + k;
        const float *vcur = vd_slot(c.S, t);
        float *vnext = vd_slot(c.S, t + 1);
        for (int it = it0; it < it1; ++it) {
            const PersistItem P = a.items[it];
            const bool staged = P.kind == TILE_DENSE || (P.mode & TILE_STAGE_V);
            if (threadIdx.x == 0) {
                // network P.net finished step t - 1 (the launch's own earlier steps only)
                int ok = k == 0 || wait_arrivals(a.cnt + P.net, (uint32_t)k * (uint32_t)P.pieces, a.abort_flag,
                                                 a.timeout_ns, c.status);
                if (ok && staged) {
                    // the acquire above (or stream order) made the writes visible to this
                    // thread; order them before the bulk copy's async-proxy reads
                    asm volatile("fence.proxy.async;" ::: "memory");
                    mbar_expect_tx(&bar, (uint32_t)P.n_pad * 4u);
                    bulk_g2s(vb, vcur + P.seg, (uint32_t)P.n_pad * 4u, &bar);
                }
                ok_sh = ok;
            }
            __syncthreads();
            if (!ok_sh) return;
            if (staged) {
                const bool landed = mbar_wait_bounded(&bar, phase & 1u);
                phase++;
                if (__syncthreads_or(!landed)) {
                    if (threadIdx.x == 0) {
                        atomicOr(c.status, (uint32_t)ST_TIMEOUT);
                        atomicExch(a.abort_flag, 1u);
                        (void)mbar_wait_bounded(&bar, (phase - 1u) & 1u);
                    }
                    return;
                }
            }
            if (P.kind == TILE_DENSE) {
                const DenseSmem sm{vb, P.n_pad, 1, part};
                const float C = vb[0] * GJ_SCALE;
                for (int sub = 0; sub < P.rows; sub += 8 * R) {
                    const int local0 = P.row0 - P.seg + sub;
                    const int srows = min(8 * R, P.rows - sub);
                    float ui[R];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        ui[r] = (warp * R + r < srows) ? gj_u(vb[local0 + warp * R + r], C) : 0.0f;
                    uint32_t uses[2] = {0u, 0u};
                    float tot[R], Us, Uc;
                    (void)gj_pass<R, 1>(sm, nullptr, P.n, P.n_pad, nullptr, uses, C, ui, 0, lane, a.kahan, tot,
                                        Us, Uc);
                    gj_reduce<R, 1>(sm, tot, Us, Uc, warp, 0, lane, red_s, red_c);
                    const float U = gj_sum_u(red_s, red_c);
                    if ((int)threadIdx.x < srows)
                        ic_s[sub + threadIdx.x] = row_current<1>(sm, threadIdx.x,
                                                                 gj_u(vb[local0 + threadIdx.x], C),
                                                                 P.n, U, P.g);
                    __syncthreads();   // part[] is rewritten by the next row block
                }
            } else if (P.mode & TILE_SLICED) {
                const int lsw = 31 - __clz(P.sw), r0 = P.row0 - P.seg;
                if (P.mode & TILE_UNIFORM_W)
                    slice_rows_short<false>(P.slice0, lsw, P.n, r0, P.rows, a.soff, a.scols, a.sw, vb, P.g, ic_s);
                else
                    slice_rows_short<true>(P.slice0, lsw, P.n, r0, P.rows, a.soff, a.scols, a.sw, vb, P.g, ic_s);
            } else if (P.mode & TILE_STAGE_V) {
                persist_csr_piece(a, P, VRowSmem{vb}, VjSliced{vb}, ic_s);
            } else {
                persist_csr_piece(a, P, VRowCG{vcur + P.seg}, VjGlobalCG{vcur + P.seg}, ic_s);
            }
            __syncthreads();
            // the explicit-Euler update of the piece's rows, one thread per cell (a thread
            // reads its cell's step-t words before writing any of them)
            for (int rr = threadIdx.x; rr < P.rows; rr += blockDim.x) {
                const int64_t i = P.row0 + rr;
                const float vd = staged ? vb[i - P.seg] : __ldcg(vcur + i);
                float iapp = pulse_current(c.pulses, i, t);
                if (c.iapp != nullptr) iapp += c.iapp[i];
                const CellNext o = cell_step(c.P, load_cell(c.S, vcur, i, vd), ic_s[rr], iapp);
                finish_cell(c, t, vnext, i, o);
            }
            // every thread's reads of vb come before the next piece's bulk refill of it
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            // the CTA's writes (ordered before the barrier above) precede the arrival
            if (threadIdx.x == 0) red_release_gpu_add(a.cnt + P.net, 1u);
        }
    }
}

// gather / scatter between the user's numbering (consecutive cells) and the segments
__global__ void batch_gather_kernel(const float *state, int64_t stride, const int32_t *map, int64_t n_user,
                                    int32_t vd_slot_field, float *out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_user) return;
    const int64_t src = map[j];
    for (int f = 0; f < NF; ++f) {
        const int slot = (f == 0) ? vd_slot_field : f;
        out[(int64_t)f * n_user + j] = state[(int64_t)slot * stride + src];
    }
}
__global__ void batch_scatter_kernel(float *state, int64_t stride, const int32_t *map, int64_t n_user,
                                     int32_t vd_slot_field, const float *in) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_user) return;
    const int64_t dst = map[j];
    for (int f = 0; f < NF; ++f) {
        const int slot = (f == 0) ? vd_slot_field : f;
        state[(int64_t)slot * stride + dst] = in[(int64_t)f * n_user + j];
    }
}

}  // namespace ion

using namespace ion;

// ---- host side -------------------------------------------------------------------------
struct BatchNet {
    int32_t kind, n, n_pad, seg;
    float g;          // dense: pair weight; CSR with uniform weights: every edge weight
    int64_t e0, nnz;  // CSR edges in the global arrays
    int sw;
    int slice0 = 0;         // sliced CSR: first slice
    bool sliced = false;    // CSR: rows in slices
    bool uniform = false;   // CSR: every weight bitwise equal (g)
    bool c16 = false;       // CSR: 16-bit network-local columns in col16
};

constexpr int BATCH_CHAINS = 4;

struct BatchExt {
    std::vector<BatchNet> nets;
    // persistent form (ION_FLAG_PERSISTENT): pieces dealt out to the CTAs of one
    // cooperative launch, per-network arrival counters + the abort word, and the graph of
    // one launch (counter reset, kernel, step-counter advance) for the last step count
    bool persistent = false;
    PersistItem *d_items = nullptr;
    int32_t *d_cta_off = nullptr;
    uint32_t *d_pcnt = nullptr;     // n_nets counters, then the abort word
    int p_grid = 0, p_vbuf = 256, p_pieces = 0;
    int p_R = 0;                    // dense rows per warp of the persistent kernel (0: choose)
    cudaGraphExec_t p_graph = nullptr;
    int64_t p_graph_steps = 0;
    bool p_graph_refused = false;
    std::vector<int32_t> h_map;     // user cell -> padded cell
    BatchTile *d_tiles = nullptr;
    int n_tiles = 0;
    // The networks are independent, so their tiles are dealt to a few chains of launches that
    // run side by side: the latency of one chain's step (launch, V_dend copies, the last
    // tiles' updates) overlaps another chain's work.  Chain 0 runs on the handle's stream, the
    // others on side streams forked from it before, and joined after, the steps of a call.
    struct Chain {
        bool dense = false;
        int off = 0, n = 0;             // tiles
        int vbuf = 256, rows_max = 32;  // shared memory of its launches
    };
    std::vector<Chain> chains;
    std::vector<Chain> whole;           // the same tiles, one list per kind: runs on one stream
    int one_steps = 0;                  // direct runs of up to so many steps are
    bool on_one = false;                // the present run is one
    cudaStream_t side[BATCH_CHAINS - 1] = {};
    cudaEvent_t ev_fork = nullptr, ev_join[BATCH_CHAINS - 1] = {};
    bool forked_now = false;            // the next step is the first after a fork
    int R = 4;                      // dense rows per warp (rows per dense tile = 8 R)
    int csr_rows = 256;             // rows per CSR tile (fewer where rows are long)
    int sw_scale = 0;               // 0: lanes per row from the degree; +-1: twice / half that
    int max_dense_pad = 256;
    // sliced rows of the staged CSR networks, for the lanes per row of sw_scale `slice_scale`
    std::vector<int32_t> h_rp;      // row_ptr over the padded cells
    uint16_t *d_scols = nullptr;
    float *d_sw = nullptr;
    int32_t *d_soff = nullptr;
    int slice_scale = -2;           // none built yet
    float *d_tmp = nullptr;         // 19 x n_user staging for state I/O
};

static BatchExt *ext_of(ion_sim *s) { return static_cast<BatchExt *>(s->ext); }

static int csr_sw_for(double deg, int scale) {
    int sw, rows;
    ion_choose_csr_shape(deg, &sw, &rows);
    if (scale > 0 && sw < 32) sw *= 2;
    if (scale < 0 && sw > 1) sw /= 2;
    return sw;
}

// Lanes per row of a sliced network: rows of about four rounds or more, so that the last round's
// padding stays small.
static int slice_sw_for(double deg, int scale) {
    int sw = 1;
    while (sw < 32 && 64 * sw <= deg) sw *= 2;
    if (scale > 0 && sw < 32) sw *= 2;
    if (scale < 0 && sw > 1) sw /= 2;
    return sw;
}

static bool net_staged(const BatchExt *X, const BatchNet &b) {
    return b.kind == ION_CSR && b.c16 && b.n_pad <= X->max_dense_pad;   // fits the launches' shared memory
}

// A slice lasts as long as its longest row, with the few lanes of a mean row.  Networks with a
// row of more than four times the mean's rounds (at least four) keep their 16-bit rows: more lanes
// per row, a whole warp for the long ones (batch_row16), no slices.  us per step of six networks
// of 4000 cells, k = 10, two cells with 2000 partners each: sliced 61, so 6.8.
static bool net_sliced(const BatchExt *X, const BatchNet &b, int sw) {
    if (!net_staged(X, b)) return false;
    const int most = 4 * std::max(1, (int)std::ceil((double)b.nnz / b.n / (8 * sw)));
    for (int r = b.seg; r < b.seg + b.n; ++r)
        if (X->h_rp[(size_t)r + 1] - X->h_rp[(size_t)r] > 8 * sw * most) return false;
    return true;
}

// The sliced layout for the current lanes-per-row scale (kept while that does not change).
static ion_status batch_build_slices(ion_sim *s) {
    BatchExt *X = ext_of(s);
    if (X->slice_scale == X->sw_scale) return ION_OK;
    std::vector<SliceDesc> desc;
    std::vector<int32_t> off;
    int64_t tot = 0;
    bool weights = false;
    for (BatchNet &b : X->nets) {
        const double deg = b.n > 0 ? (double)b.nnz / b.n : 0.0;
        b.sliced = net_sliced(X, b, slice_sw_for(deg, X->sw_scale));
        if (b.kind == ION_CSR) b.sw = b.sliced ? slice_sw_for(deg, X->sw_scale) : csr_sw_for(deg, X->sw_scale);
        if (!b.sliced) continue;
        weights = weights || !b.uniform;
        b.slice0 = (int)desc.size();
        int lsw = 0;
        while ((1 << lsw) < b.sw) ++lsw;
        const int per = 32 >> lsw;
        for (int r = 0; r < b.n; r += per) {
            const int here = std::min(per, b.n - r);
            int most = 0;
            for (int q = 0; q < here; ++q) most = std::max(most, X->h_rp[(size_t)b.seg + r + q + 1] - X->h_rp[(size_t)b.seg + r + q]);
            desc.push_back({b.seg + r, here, b.seg, lsw});
            off.push_back((int32_t)tot);
            tot += (most + 8 * b.sw - 1) / (8 * b.sw);
            if (tot >= INT32_MAX / 64) return ion_fail(s, ION_ERR_INVALID_ARG, "batch: too many edges");
        }
    }
    off.push_back((int32_t)tot);
    cudaError_t e = cudaStreamSynchronize(s->st);
    ion_drop_graphs(s);   // captured steps hold the old arrays
    cudaFree(X->d_scols);
    cudaFree(X->d_sw);
    cudaFree(X->d_soff);
    X->d_scols = nullptr;
    X->d_sw = nullptr;
    X->d_soff = nullptr;
    X->slice_scale = -2;
    if (!desc.empty()) {
        SliceDesc *d_desc = nullptr;
        const size_t rounds = (size_t)std::max<int64_t>(tot, 1);
        if (e == cudaSuccess) e = ion_alloc(&X->d_scols, rounds * 512);
        if (e == cudaSuccess && weights) e = ion_alloc(&X->d_sw, rounds * 1024);
        if (e == cudaSuccess) e = ion_alloc(&X->d_soff, off.size() * sizeof(int32_t));
        if (e == cudaSuccess) e = ion_alloc(&d_desc, desc.size() * sizeof(SliceDesc));
        if (e == cudaSuccess) e = cudaMemcpy(X->d_soff, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(d_desc, desc.data(), desc.size() * sizeof(SliceDesc), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            batch_slice_fill_kernel<<<(unsigned)((desc.size() + 3) / 4), 128, 0, s->st>>>(
                d_desc, (int)desc.size(), X->d_soff, s->d_rowptr, s->d_col16, s->d_w, X->d_scols, X->d_sw);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
        cudaFree(d_desc);
    }
    if (e != cudaSuccess)
        return ion_fail(s, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "batch slices: %s", cudaGetErrorString(e));
    X->slice_scale = X->sw_scale;
    return ION_OK;
}

// Work per tile: a tile pays about 3 us of latency (its V_dend copy, its rows' update) whatever
// it computes, so small networks get several row blocks per tile and short rows more rows;
// while there are too few tiles to fill the chip, fewer.  Measured (96 networks of 32-4096
// cells, us per step): 80 000 pairs per dense tile 20.1, one row block 20.9, 160 000: 21.4;
// 12 networks: 20 000 pairs 5.5, 80 000: 8.6.
constexpr double DENSE_TILE_PAIRS = 80000.0, DENSE_TILE_LEAST = 16000.0;
constexpr double CSR_TILE_EDGES = 32768.0, CSR_TILE_LEAST = 2048.0;
// Chains: two for the dense networks (one: 24.0 us per step, three: as two), one for the rest.
constexpr int DENSE_CHAINS = 2, CSR_CHAINS = 1;
static_assert(DENSE_CHAINS + CSR_CHAINS <= BATCH_CHAINS, "one stream per chain");

// Build (or rebuild) the tile list for the current shape parameters.
static ion_status batch_plan(ion_sim *s) {
    BatchExt *X = ext_of(s);
    const ion_status ss = batch_build_slices(s);
    if (ss != ION_OK) {
        X->n_tiles = 0;   // the slices a tile list would refer to are gone: stepping is refused
        cudaFree(X->d_tiles);
        X->d_tiles = nullptr;
        return ss;
    }
    std::vector<BatchTile> tiles;
    std::vector<double> cost;
    std::vector<int> tile_net;
    double pairs = 0.0, edges = 0.0;
    for (const BatchNet &b : X->nets) (b.kind == ION_DENSE_UNIFORM ? pairs : edges) += b.kind == ION_DENSE_UNIFORM ? (double)b.n * b.n_pad : (double)b.nnz;
    const double dense_work = std::min(DENSE_TILE_PAIRS, std::max(DENSE_TILE_LEAST, pairs / (4 * s->sms)));
    const double csr_work = std::min(CSR_TILE_EDGES, std::max(CSR_TILE_LEAST, edges / s->sms));
    for (size_t net = 0; net < X->nets.size(); ++net) {
        const BatchNet &b = X->nets[net];
        if (b.kind == ION_DENSE_UNIFORM) {
            const int blocks = std::min(256 / (8 * X->R), std::max(1, (int)(dense_work / ((double)8 * X->R * b.n_pad) + 0.5)));
            const int drows = 8 * X->R * blocks;
            for (int r = 0; r < b.n; r += drows) {
                BatchTile T{TILE_DENSE, b.seg, b.n, b.n_pad, b.seg + r, std::min(drows, b.n - r), 0, b.g, 0, 0};
                tiles.push_back(T);
                tile_net.push_back((int)net);
                cost.push_back((double)T.rows * b.n_pad);
            }
        } else {
            const double deg = b.n > 0 ? (double)b.nnz / b.n : 0.0;
            int mode = (b.uniform ? TILE_UNIFORM_W : 0) | (b.c16 ? TILE_C16 : 0);
            if (net_staged(X, b)) mode |= TILE_STAGE_V | (b.sliced ? TILE_SLICED : 0);
            int crows = X->csr_rows;
            while (crows > 32 && crows * deg > csr_work) crows = (crows + 1) / 2;
            for (int r = 0; r < b.n; r += crows) {
                BatchTile T{TILE_CSR, b.seg, b.n, b.n_pad, b.seg + r, std::min(crows, b.n - r),
                            b.kind == ION_CSR ? b.sw : 1, b.uniform ? b.g : 0.0f, mode, b.slice0};
                tiles.push_back(T);
                tile_net.push_back((int)net);
                cost.push_back(3.0 * T.rows * deg + 60.0 * T.rows);
            }
        }
    }
    // deal the networks to chains: dense and CSR ones apart (different kernels), each kind's
    // networks largest first to the lighter of its chains
    std::vector<double> net_cost(X->nets.size(), 0.0);
    for (size_t k = 0; k < tiles.size(); ++k) net_cost[(size_t)tile_net[k]] += cost[k];
    std::vector<int> chain_of(X->nets.size(), 0);
    X->chains.clear();
    for (int dense = 1; dense >= 0; --dense) {
        std::vector<int> own;
        for (size_t b = 0; b < X->nets.size(); ++b)
            if ((X->nets[b].kind == ION_DENSE_UNIFORM) == (dense == 1)) own.push_back((int)b);
        if (own.empty()) continue;
        std::stable_sort(own.begin(), own.end(), [&](int a, int b) { return net_cost[(size_t)a] > net_cost[(size_t)b]; });
        const int nc = std::min<int>((int)own.size(), dense ? DENSE_CHAINS : CSR_CHAINS), c0 = (int)X->chains.size();
        std::vector<double> load((size_t)nc, 0.0);
        for (int q = 0; q < nc; ++q) {
            X->chains.emplace_back();
            X->chains.back().dense = dense == 1;
        }
        for (int b : own) {
            const int q = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            load[(size_t)q] += net_cost[(size_t)b];
            chain_of[(size_t)b] = c0 + q;
        }
    }
    std::vector<int> order(tiles.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const int ca = chain_of[(size_t)tile_net[(size_t)a]], cb = chain_of[(size_t)tile_net[(size_t)b]];
        return ca != cb ? ca < cb : cost[a] > cost[b];
    });
    std::vector<BatchTile> sorted(tiles.size());
    for (size_t k = 0; k < order.size(); ++k) {
        const BatchTile &T = sorted[k] = tiles[order[k]];
        BatchExt::Chain &C = X->chains[(size_t)chain_of[(size_t)tile_net[(size_t)order[k]]]];
        if (C.n++ == 0) C.off = (int)k;
        if (T.kind == TILE_DENSE || (T.mode & TILE_STAGE_V)) C.vbuf = std::max(C.vbuf, T.n_pad);
        C.rows_max = std::max(C.rows_max, T.rows);
    }
    X->whole.clear();
    for (const BatchExt::Chain &C : X->chains) {   // the chains of a kind lie one after the other
        if (X->whole.empty() || X->whole.back().dense != C.dense) {
            X->whole.push_back(C);
            continue;
        }
        BatchExt::Chain &W = X->whole.back();
        W.n += C.n;
        W.vbuf = std::max(W.vbuf, C.vbuf);
        W.rows_max = std::max(W.rows_max, C.rows_max);
    }
    // Forking and joining costs the host 4 to 5 us per call, more than the chains save in a few
    // steps.  us per step of a call of k steps, chains / one stream: two dense networks of 64 cells
    // 9.1 / 5.3 (k = 1), 4.1 / 3.7 (40); twelve of 1792 14.7 / 12.4 (1), 11.4 / 10.9 (4), 10.0 / 10.6
    // (10); a dense and a CSR network of 500 9.6 / 7.8 (1), 6.5 / 7.0 (2); 96 networks of 32-4096 33.2
    // / 35.5 (1).
    const double total = std::accumulate(net_cost.begin(), net_cost.end(), 0.0);
    X->one_steps = total > 6.0e7 ? 0 : X->whole.size() > 1 ? 1 : (int)sorted.size() <= s->sms ? INT32_MAX : 4;
    s->lps = (int64_t)X->chains.size();
    cudaError_t e = cudaStreamSynchronize(s->st);
    ion_drop_graphs(s);   // the captured steps hold the old tile list
    if (e == cudaSuccess && X->d_tiles) e = cudaFree(X->d_tiles);
    X->d_tiles = nullptr;   // until a new list is in place, stepping is refused
    X->n_tiles = 0;
    if (e == cudaSuccess) e = ion_alloc(&X->d_tiles, std::max<size_t>(1, sorted.size()) * sizeof(BatchTile));
    if (e == cudaSuccess)
        e = cudaMemcpy(X->d_tiles, sorted.data(), sorted.size() * sizeof(BatchTile), cudaMemcpyHostToDevice);
    if (e != cudaSuccess)
        return ion_fail(s, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "batch plan: %s", cudaGetErrorString(e));
    X->n_tiles = (int)sorted.size();
    return ION_OK;
}

// dynamic shared memory of a chain's launches: a network's V_dend, the dense row partials and
// the tile's cell words
static size_t batch_smem(const BatchExt *X, const BatchExt::Chain &C) {
    return ((size_t)C.vbuf + (C.dense ? 8 * X->R : 0) + (size_t)NCW * C.rows_max) * sizeof(float);
}

static cudaError_t batch_allow_smem(bool dense, int R, size_t need) {
    if (!dense) return allow_smem(batch_csr_kernel, need);
    switch (R) {
        case 1: return allow_smem(batch_dense_kernel<1>, need);
        case 2: return allow_smem(batch_dense_kernel<2>, need);
        case 4: return allow_smem(batch_dense_kernel<4>, need);
        default: return allow_smem(batch_dense_kernel<8>, need);
    }
}
static cudaError_t batch_launch(const BatchArgs &a, bool dense, int R, int tiles, size_t smem, bool pdl, cudaStream_t st) {
    const dim3 grid(tiles), block(256);
    if (!dense) return launch_k(batch_csr_kernel, grid, block, smem, st, pdl, a);
    switch (R) {
        case 1: return launch_k(batch_dense_kernel<1>, grid, block, smem, st, pdl, a);
        case 2: return launch_k(batch_dense_kernel<2>, grid, block, smem, st, pdl, a);
        case 4: return launch_k(batch_dense_kernel<4>, grid, block, smem, st, pdl, a);
        case 8: return launch_k(batch_dense_kernel<8>, grid, block, smem, st, pdl, a);
        default: return cudaErrorInvalidValue;
    }
}

static cudaError_t batch_step(ion_sim *s, int k_off, const float *iapp) {
    BatchExt *X = ext_of(s);
    if (X->d_tiles == nullptr) return cudaErrorInvalidResourceHandle;   // no tile list: a failed re-plan
    BatchArgs a{};
    a.c = ion_step_common(s, k_off, iapp);
    a.row_ptr = s->d_rowptr;
    a.col = s->d_col;
    a.col16 = s->d_col16;
    a.w = s->d_w;
    a.scols = reinterpret_cast<const uint4 *>(X->d_scols);
    a.sw = reinterpret_cast<const float4 *>(X->d_sw);
    a.soff = X->d_soff;
    a.kahan = 1;
    cudaError_t e = cudaSuccess;
    const std::vector<BatchExt::Chain> &run = X->on_one ? X->whole : X->chains;
    for (size_t q = 0; q < run.size() && e == cudaSuccess; ++q) {
        const BatchExt::Chain &C = run[q];
        a.tiles = X->d_tiles + C.off;
        a.rows_max = C.rows_max;
        a.vbuf = C.vbuf;
        // a side stream's first launch follows the fork event, not a kernel: an ordinary launch
        const bool pdl = a.c.pdl && !(q > 0 && X->forked_now);
        e = batch_launch(a, C.dense, X->R, C.n, batch_smem(X, C), pdl, q == 0 || X->on_one ? s->st : X->side[q - 1]);
        s->launches++;
    }
    X->forked_now = false;
    return e;
}

// Before the steps of a captured graph or of a direct run: the side streams start after the
// handle's stream; after them the handle's stream continues when every chain is done.  A direct run
// of few steps stays on the handle's stream (one_steps).
static cudaError_t batch_fork(ion_sim *s, int steps, bool captured) {
    BatchExt *X = ext_of(s);
    X->on_one = !captured && steps <= X->one_steps;
    s->forked = !X->on_one && X->chains.size() > 1;
    X->forked_now = s->forked;
    if (!s->forked) return cudaSuccess;
    cudaError_t e = cudaEventRecord(X->ev_fork, s->st);
    for (size_t q = 1; q < X->chains.size() && e == cudaSuccess; ++q) e = cudaStreamWaitEvent(X->side[q - 1], X->ev_fork, 0);
    return e;
}
static cudaError_t batch_join(ion_sim *s) {
    BatchExt *X = ext_of(s);
    cudaError_t e = cudaSuccess;
    for (size_t q = 1; s->forked && q < X->chains.size(); ++q) {   // every side stream joins, also after an error
        cudaError_t e1 = cudaEventRecord(X->ev_join[q - 1], X->side[q - 1]);
        if (e1 == cudaSuccess) e1 = cudaStreamWaitEvent(s->st, X->ev_join[q - 1], 0);
        if (e == cudaSuccess) e = e1;
    }
    return e;
}

// ---- persistent form: planning and launch ----------------------------------------------
template <int R>
static cudaError_t persist_kernel_attr(size_t smem, int *per_sm) {
    cudaError_t e = allow_smem(batch_persist_kernel<R>, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, batch_persist_kernel<R>, 256, smem);
    return e;
}
static cudaError_t persist_attr(int R, size_t smem, int *per_sm) {
    switch (R) {
        case 1: return persist_kernel_attr<1>(smem, per_sm);
        case 2: return persist_kernel_attr<2>(smem, per_sm);
        case 4: return persist_kernel_attr<4>(smem, per_sm);
        default: return cudaErrorInvalidValue;
    }
}
static const void *persist_fn(int R) {
    switch (R) {
        case 1: return (const void *)batch_persist_kernel<1>;
        case 2: return (const void *)batch_persist_kernel<2>;
        default: return (const void *)batch_persist_kernel<4>;
    }
}
static size_t persist_smem(const BatchExt *X) { return (size_t)X->p_vbuf * 4 + 8 * X->p_R * 4; }

// Rows per warp of the persistent kernel's dense pieces where none are asked for: a row's sum is the
// same whatever R.  Two keep a small network's chain short, four share the column loads once
// the pairs fill the chip.  us per step with 2 / 4: one network of 2000 cells 6.2 / 8.0, of 300 4.2 /
// 4.7, twelve of 1792 (4e7 pairs) 11.6 / 11.8, 48 of 32-4096 beside 48 CSR ones (1e8) 45 / 35.
static int persist_rows(const BatchExt *X) {
    double pairs = 0.0;
    for (const BatchNet &b : X->nets)
        if (b.kind == ION_DENSE_UNIFORM) pairs += (double)b.n * b.n_pad;
    return pairs > 6.0e7 ? 4 : 2;
}

// Cut the networks into pieces and deal them out to the CTAs of one resident grid.
// Work per row: a dense row costs its network's padded width in pair evaluations (plus a
// constant for its update), a CSR row 3 units per edge and 60 for its update; a piece
// also pays its staging.  A network becomes several pieces when its work exceeds a CTA's
// share of the total (and pieces hold at most 256 rows); pieces go largest first to the
// least loaded CTA.  Each CTA handles the pieces of networks split over several CTAs
// first, so that their arrivals come early in every step.
static ion_status batch_persist_plan(ion_sim *s) {
    BatchExt *X = ext_of(s);
    X->p_vbuf = X->max_dense_pad;
    int per_sm = 0;
    cudaError_t e = persist_attr(X->p_R, persist_smem(X), &per_sm);
    if (e != cudaSuccess || per_sm < 1)
        return ion_fail(s, ION_ERR_UNSUPPORTED, "persistent batch: no resident CTA (%s)", cudaGetErrorString(e));
    const int grid = per_sm * s->sms;
    struct Net { double per_row, fixed; int rows_align; };
    std::vector<Net> nc(X->nets.size());
    double total = 0.0;
    for (size_t b = 0; b < X->nets.size(); ++b) {
        const BatchNet &x = X->nets[b];
        // sliced rows: two slices or more per piece (twelve networks of 2000 cells, k = 24: 5.1 us
        // per step, one slice 8.5, eight 6.6)
        if (x.kind == ION_DENSE_UNIFORM) nc[b] = {(double)x.n_pad + 64.0, 2048.0 + x.n_pad, 8 * X->p_R};
        else nc[b] = {3.0 * (x.n > 0 ? (double)x.nnz / x.n : 0.0) + 60.0, 2048.0 + 0.5 * x.n_pad,
                      x.sliced ? 2 * (32 / x.sw) : 32};
        total += nc[b].per_row * x.n + nc[b].fixed;
    }
    const double share = total / grid;
    struct Piece { PersistItem it; double cost; };
    std::vector<Piece> pieces;
    for (size_t b = 0; b < X->nets.size(); ++b) {
        const BatchNet &x = X->nets[b];
        const double cost = nc[b].per_row * x.n;
        int k = std::max((x.n + 255) / 256, (int)std::ceil(cost / (0.8 * share)));
        k = std::max(1, std::min(k, x.n));
        int rows = (x.n + k - 1) / k;
        const int al = nc[b].rows_align;
        rows = std::min(256, (rows + al - 1) / al * al);
        k = (x.n + rows - 1) / rows;
        for (int r = 0; r < x.n; r += rows) {
            PersistItem it{};
            it.kind = x.kind == ION_DENSE_UNIFORM ? TILE_DENSE : TILE_CSR;
            it.net = (int32_t)b;
            it.seg = x.seg;
            it.n = x.n;
            it.n_pad = x.n_pad;
            it.row0 = x.seg + r;
            it.rows = std::min(rows, x.n - r);
            it.pieces = k;
            it.g = x.g;
            if (x.kind != ION_DENSE_UNIFORM) {
                it.sw = x.sw;
                it.mode = (x.uniform ? TILE_UNIFORM_W : 0) | (x.c16 ? TILE_C16 : 0);
                it.slice0 = x.slice0;
                if (net_staged(X, x)) it.mode |= TILE_STAGE_V | (x.sliced ? TILE_SLICED : 0);
            }
            pieces.push_back({it, nc[b].per_row * it.rows + nc[b].fixed});
        }
    }
    std::vector<int> order(pieces.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return pieces[a].cost > pieces[b].cost; });
    std::vector<double> load((size_t)grid, 0.0);
    std::vector<std::vector<int>> own((size_t)grid);
    for (int q : order) {
        const size_t c = (size_t)(std::min_element(load.begin(), load.end()) - load.begin());
        load[c] += pieces[q].cost;
        own[c].push_back(q);
    }
    std::vector<PersistItem> items;
    std::vector<int32_t> off((size_t)grid + 1, 0);
    for (int c = 0; c < grid; ++c) {
        std::vector<int> &L = own[(size_t)c];
        std::stable_sort(L.begin(), L.end(), [&](int a, int b) {
            const PersistItem &A = pieces[a].it, &B = pieces[b].it;
            if ((A.pieces > 1) != (B.pieces > 1)) return A.pieces > 1;
            return A.row0 < B.row0;
        });
        for (int q : L) items.push_back(pieces[q].it);
        off[(size_t)c + 1] = (int32_t)items.size();
    }
    e = cudaStreamSynchronize(s->st);
    if (X->p_graph) {
        cudaGraphExecDestroy(X->p_graph);
        X->p_graph = nullptr;
        X->p_graph_steps = 0;
    }
    cudaFree(X->d_items);
    cudaFree(X->d_cta_off);
    X->d_items = nullptr;
    X->d_cta_off = nullptr;
    X->p_grid = 0;
    if (e == cudaSuccess) e = ion_alloc(&X->d_items, std::max<size_t>(1, items.size()) * sizeof(PersistItem));
    if (e == cudaSuccess) e = ion_alloc(&X->d_cta_off, off.size() * sizeof(int32_t));
    if (e == cudaSuccess && !X->d_pcnt) e = ion_alloc(&X->d_pcnt, (X->nets.size() + 1) * sizeof(uint32_t));
    if (e == cudaSuccess && !items.empty())
        e = cudaMemcpy(X->d_items, items.data(), items.size() * sizeof(PersistItem), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(X->d_cta_off, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess)
        return ion_fail(s, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "persistent batch plan: %s",
                        cudaGetErrorString(e));
    X->p_grid = grid;
    X->p_pieces = (int)items.size();
    return ION_OK;
}

// One launch of n_steps steps: counters and abort word cleared, the cooperative kernel,
// then the device step counter advanced.
static cudaError_t persist_enqueue(ion_sim *s, int n_steps, bool capture) {
    BatchExt *X = ext_of(s);
    BatchPersistArgs a{};
    a.c = ion_step_common(s, 0, nullptr);
    a.c.par = -1;   // many steps per launch: the slots follow the device counter
    a.items = X->d_items;
    a.cta_off = X->d_cta_off;
    a.row_ptr = s->d_rowptr;
    a.col16 = s->d_col16;
    a.w = s->d_w;
    a.scols = reinterpret_cast<const uint4 *>(X->d_scols);
    a.sw = reinterpret_cast<const float4 *>(X->d_sw);
    a.soff = X->d_soff;
    a.cnt = X->d_pcnt;
    a.abort_flag = X->d_pcnt + X->nets.size();
    a.timeout_ns = s->barrier_timeout_ns;
    a.n_steps = n_steps;
    a.vbuf = X->p_vbuf;
    a.kahan = 1;
    a.debug_delay_ns = s->debug_delay_ns;
    cudaError_t e = cudaMemsetAsync(X->d_pcnt, 0, (X->nets.size() + 1) * sizeof(uint32_t), s->st);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    if (capture) {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(X->p_grid);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = persist_smem(X);
        cfg.stream = s->st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelExC(&cfg, persist_fn(X->p_R), args);
    } else {
        e = cudaLaunchCooperativeKernel(persist_fn(X->p_R), dim3(X->p_grid), dim3(256), args, persist_smem(X), s->st);
    }
    if (e != cudaSuccess) return e;
    return launch_advance(s->d_t, n_steps, s->st);
}

// The captured launch holds the pulse table and trace ring of its capture: dropped with
// the per-step graphs whenever those change.
static void batch_persist_drop(ion_sim *s) {
    BatchExt *X = ext_of(s);
    if (X && X->p_graph) {
        cudaGraphExecDestroy(X->p_graph);
        X->p_graph = nullptr;
        X->p_graph_steps = 0;
    }
}

// ion_step of a persistent batch: one graph replay (or, where a capture is refused, one
// direct cooperative launch) per 2^22 steps.
static ion_status batch_persist_run(ion_sim *s, int64_t n_steps, const float *iapp) {
    (void)iapp;
    BatchExt *X = ext_of(s);
    if (X->d_items == nullptr || X->p_grid == 0) return ion_fail(s, ION_ERR_CUDA, "persistent batch: no plan");
    int64_t done = 0;
    while (done < n_steps) {
        const int chunk = (int)std::min<int64_t>(n_steps - done, 1 << 22);
        cudaError_t e = cudaSuccess;
        if (!X->p_graph_refused && X->p_graph_steps != chunk) {
            if (X->p_graph) cudaGraphExecDestroy(X->p_graph);
            X->p_graph = nullptr;
            X->p_graph_steps = 0;
            cudaGraph_t g = nullptr;
            e = cudaStreamBeginCapture(s->st, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                const cudaError_t e1 = persist_enqueue(s, chunk, true);
                const cudaError_t e2 = cudaStreamEndCapture(s->st, &g);
                e = e1 != cudaSuccess ? e1 : e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&X->p_graph, g, 0);
            if (g) cudaGraphDestroy(g);
            if (e == cudaSuccess) {
                X->p_graph_steps = chunk;
            } else {   // no cooperative launches in graphs here: launch directly from now on
                (void)cudaGetLastError();
                X->p_graph = nullptr;
                X->p_graph_refused = true;
            }
        }
        if (X->p_graph != nullptr && X->p_graph_steps == chunk) e = cudaGraphLaunch(X->p_graph, s->st);
        else e = persist_enqueue(s, chunk, false);
        s->launches += 2;
        if (e != cudaSuccess) return ion_fail(s, ION_ERR_CUDA, "persistent batch launch: %s", cudaGetErrorString(e));
        done += chunk;
    }
    return ION_OK;
}

// What the launches of the current tile list (batch_plan) need before they can be captured.
static ion_status batch_prepare(ion_sim *s) {
    BatchExt *X = ext_of(s);
    cudaError_t e = cudaSuccess;
    for (size_t q = 0; q < X->whole.size() && e == cudaSuccess; ++q)   // as large as any chain's need
        e = batch_allow_smem(X->whole[q].dense, X->R, batch_smem(X, X->whole[q]));
    if (e == cudaSuccess && !X->ev_fork) e = cudaEventCreateWithFlags(&X->ev_fork, cudaEventDisableTiming);
    for (size_t q = 1; q < X->chains.size() && e == cudaSuccess; ++q) {
        if (!X->side[q - 1]) e = cudaStreamCreateWithFlags(&X->side[q - 1], cudaStreamNonBlocking);
        if (e == cudaSuccess && !X->ev_join[q - 1]) e = cudaEventCreateWithFlags(&X->ev_join[q - 1], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) return ion_fail(s, ION_ERR_CUDA, "batch setup: %s", cudaGetErrorString(e));
    return ION_OK;
}

// state I/O in the user's numbering
ion_status ion_batch_read(ion_sim *s, int32_t field, float *out) {
    BatchExt *X = ext_of(s);
    const int64_t nu = (int64_t)X->h_map.size();
    const int vd = (s->t & 1) ? 19 : 0;
    batch_gather_kernel<<<(unsigned)((nu + 255) / 256), 256, 0, s->st>>>(s->d_state, s->stride, s->d_map, nu, vd,
                                                                        X->d_tmp);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e == cudaSuccess) {
        if (field == ION_FIELD_ALL)
            e = cudaMemcpy(out, X->d_tmp, (size_t)NF * nu * sizeof(float), cudaMemcpyDeviceToHost);
        else
            e = cudaMemcpy(out, X->d_tmp + (int64_t)field * nu, (size_t)nu * sizeof(float), cudaMemcpyDeviceToHost);
    }
    if (e != cudaSuccess) return ion_fail(s, ION_ERR_CUDA, "batch read: %s", cudaGetErrorString(e));
    return ION_OK;
}

ion_status ion_batch_write(ion_sim *s, int32_t field, const float *in) {
    BatchExt *X = ext_of(s);
    const int64_t nu = (int64_t)X->h_map.size();
    const int vd = (s->t & 1) ? 19 : 0;
    cudaError_t e = cudaSuccess;
    if (field != ION_FIELD_ALL) {   // read-modify-write of the one field through the staging buffer
        batch_gather_kernel<<<(unsigned)((nu + 255) / 256), 256, 0, s->st>>>(s->d_state, s->stride, s->d_map, nu, vd,
                                                                            X->d_tmp);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
        if (e == cudaSuccess)
            e = cudaMemcpy(X->d_tmp + (int64_t)field * nu, in, (size_t)nu * sizeof(float), cudaMemcpyHostToDevice);
    } else {
        e = cudaMemcpy(X->d_tmp, in, (size_t)NF * nu * sizeof(float), cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) {
        batch_scatter_kernel<<<(unsigned)((nu + 255) / 256), 256, 0, s->st>>>(s->d_state, s->stride, s->d_map, nu, vd,
                                                                             X->d_tmp);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) return ion_fail(s, ION_ERR_CUDA, "batch write: %s", cudaGetErrorString(e));
    return ION_OK;
}

int32_t ion_batch_map_cell(ion_sim *s, int64_t user_cell) {
    BatchExt *X = ext_of(s);
    if (user_cell < 0 || user_cell >= (int64_t)X->h_map.size()) return -1;
    return X->h_map[(size_t)user_cell];
}

static void batch_free(ion_sim *s) {
    BatchExt *X = ext_of(s);
    if (!X) return;
    s->drop_hook = nullptr;
    if (X->p_graph) cudaGraphExecDestroy(X->p_graph);
    for (int q = 0; q < BATCH_CHAINS - 1; ++q) {   // their work is joined to the handle's stream, which is idle
        if (X->side[q]) cudaStreamDestroy(X->side[q]);
        if (X->ev_join[q]) cudaEventDestroy(X->ev_join[q]);
    }
    if (X->ev_fork) cudaEventDestroy(X->ev_fork);
    cudaFree(X->d_items);
    cudaFree(X->d_cta_off);
    cudaFree(X->d_pcnt);
    cudaFree(X->d_tiles);
    cudaFree(X->d_scols);
    cudaFree(X->d_sw);
    cudaFree(X->d_soff);
    cudaFree(X->d_tmp);
    cudaFree(s->d_map);
    s->d_map = nullptr;
    delete X;
    s->ext = nullptr;
}

extern "C" ion_status ion_create_batch(int32_t n_nets, const ion_net *nets, const ion_conn *conns,
                                       const ion_params *params, const float *init_state, ion_sim **out) {
    if (!out) return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: NULL out");
    *out = nullptr;
    if (n_nets < 1 || !nets || !conns || !params)
        return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: bad arguments");
    if (params->flags & (ION_FLAG_SURROGATE | ION_FLAG_SPLIT | ION_FLAG_SGJ))
        return ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: flags not supported for batches");
    if ((params->flags & ION_FLAG_PERSISTENT) && (params->flags & ION_FLAG_CSR_AS_GIVEN))
        return ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: a persistent batch needs the compact CSR layout");
    if (params->cell_params)
        return ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: per-cell constants not supported for batches");
    // validate and lay out
    std::vector<BatchNet> bn((size_t)n_nets);
    int64_t seg = 0, n_user = 0, nnz_total = 0;
    int max_pad = 256;
    for (int b = 0; b < n_nets; ++b) {
        const ion_net &N = nets[b];
        if (N.n_cells < 1 || (N.kind != ION_DENSE_UNIFORM && N.kind != ION_CSR && N.kind != ION_NO_GJ))
            return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: network %d: bad size or kind", b);
        if (N.kind == ION_DENSE_UNIFORM && N.n_cells > TJ)
            return ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: dense network %d has %d > %d cells", b,
                            N.n_cells, TJ);
        if (N.kind == ION_DENSE_UNIFORM && !std::isfinite(conns[b].g_c))
            return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: network %d: g_c not finite", b);
        if (N.kind == ION_CSR) {
            if (conns[b].mem != ION_HOST)
                return ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: network %d: CSR must be host memory", b);
            ion_status st = ion_validate_csr(N.n_cells, &conns[b]);
            if (st != ION_OK) return st;
        }
        BatchNet &x = bn[(size_t)b];
        x.kind = N.kind;
        x.n = N.n_cells;
        x.n_pad = (N.n_cells + PAD_J - 1) / PAD_J * PAD_J;
        x.seg = (int32_t)seg;
        x.g = N.kind == ION_DENSE_UNIFORM ? conns[b].g_c : 0.0f;
        x.e0 = nnz_total;
        x.nnz = N.kind == ION_CSR ? conns[b].nnz : 0;
        if (N.kind == ION_CSR && !(params->flags & ION_FLAG_CSR_AS_GIVEN)) {
            // compact layout: 16-bit local columns; one scalar when every weight is bitwise equal
            x.c16 = N.n_cells <= 65536;
            const ion_conn &C = conns[b];
            x.uniform = true;
            x.g = C.g_c;
            if (C.weight && x.nnz > 0) {
                uint32_t b0, be;
                std::memcpy(&b0, C.weight, sizeof b0);
                for (int64_t q = 1; q < x.nnz && x.uniform; ++q) {
                    std::memcpy(&be, C.weight + q, sizeof be);
                    x.uniform = be == b0;
                }
                x.g = C.weight[0];
            }
        }
        if (N.kind == ION_DENSE_UNIFORM || (x.c16 && x.n_pad <= TJ)) max_pad = std::max(max_pad, x.n_pad);
        seg += x.n_pad;
        n_user += x.n;
        nnz_total += x.nnz;
        if (seg >= (1 << 30) || nnz_total >= INT32_MAX)
            return ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: batch too large");
    }
    // create an empty single-network handle of the padded size, then turn it into a batch
    ion_net whole{(int32_t)seg, ION_NO_GJ};
    ion_params p = *params;
    p.flags &= ~(uint32_t)ION_FLAG_PERSISTENT;
    ion_sim *s = nullptr;
    ion_status st = ion_create(&whole, nullptr, &p, nullptr, &s);
    if (st != ION_OK) return st;
    auto fail = [&](ion_status code) {
        ion_destroy(s);
        return code;
    };
    BatchExt *X = new BatchExt();
    s->ext = X;
    s->extra_free = batch_free;
    X->nets = bn;
    X->max_dense_pad = max_pad;
    X->h_map.resize((size_t)n_user);
    {
        int64_t u = 0;
        for (const BatchNet &x : bn)
            for (int i = 0; i < x.n; ++i) X->h_map[(size_t)u++] = x.seg + i;
    }
    const ion_tune *tu = (const ion_tune *)params->tune;
    if (tu && tu->dense_rows_per_warp > 0) X->R = X->p_R = tu->dense_rows_per_warp;
    if (tu && tu->csr_rows_per_cta > 0) X->csr_rows = tu->csr_rows_per_cta;
    if (tu && tu->csr_lanes_scale != 0) X->sw_scale = tu->csr_lanes_scale > 0 ? 1 : -1;
    if ((X->R != 1 && X->R != 2 && X->R != 4 && X->R != 8) || X->csr_rows < 1 || X->csr_rows > 256)
        return fail(ion_fail(nullptr, ION_ERR_INVALID_ARG, "ion_create_batch: bad tile shape override"));
    // global CSR over the padded index space
    std::vector<int32_t> rp((size_t)seg + 1, 0), col((size_t)std::max<int64_t>(nnz_total, 1));
    std::vector<float> w((size_t)std::max<int64_t>(nnz_total, 1));
    std::vector<uint16_t> col16((size_t)(nnz_total + 8), 0);   // padded to whole 16-byte groups
    bool any16 = false;
    for (int b = 0; b < n_nets; ++b) {
        const BatchNet &x = bn[(size_t)b];
        if (x.kind != ION_CSR) continue;
        const ion_conn &C = conns[b];
        any16 = any16 || x.c16;
        for (int i = 0; i < x.n; ++i) rp[(size_t)x.seg + i + 1] = C.row_ptr[i + 1] - C.row_ptr[i];
        for (int64_t e = 0; e < x.nnz; ++e) {
            col[(size_t)(x.e0 + e)] = x.seg + C.col_idx[e];
            w[(size_t)(x.e0 + e)] = C.weight ? C.weight[e] : C.g_c;
            if (x.c16) col16[(size_t)(x.e0 + e)] = (uint16_t)C.col_idx[e];
        }
    }
    for (size_t i = 0; i < (size_t)seg; ++i) rp[i + 1] += rp[i];
    X->h_rp = rp;
    // the per-row counts above were placed in network order, so the prefix sum lines the
    // edges up with x.e0 (segments are laid out in network order)
    s->own_csr = true;   // before the allocations, so that a partial failure frees them
    cudaError_t e = ion_alloc(&s->d_rowptr, rp.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = ion_alloc(&s->d_col, col.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = ion_alloc(&s->d_w, w.size() * sizeof(float));
    if (e == cudaSuccess && any16) e = ion_alloc(&s->d_col16, col16.size() * sizeof(uint16_t));
    if (e == cudaSuccess) e = ion_alloc(&s->d_map, X->h_map.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = ion_alloc(&X->d_tmp, (size_t)NF * n_user * sizeof(float));
    if (e != cudaSuccess) return fail(ion_fail(nullptr, ION_ERR_OOM, "ion_create_batch: %s", cudaGetErrorString(e)));
    s->nnz = nnz_total;
    e = cudaMemcpy(s->d_rowptr, rp.data(), rp.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(s->d_col, col.data(), col.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(s->d_w, w.data(), w.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && any16)
        e = cudaMemcpy(s->d_col16, col16.data(), col16.size() * sizeof(uint16_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(s->d_map, X->h_map.data(), X->h_map.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return fail(ion_fail(nullptr, ION_ERR_CUDA, "ion_create_batch: %s", cudaGetErrorString(e)));
    s->kind = ION_CSR;   // the generic paths see a CSR handle; stepping is overridden
    s->n_user = n_user;
    s->step_override = batch_step;
    s->fork_hook = batch_fork;
    s->join_hook = batch_join;
    s->prepare_hook = nullptr;
    // every V_dend padding cell holds the sentinel (the default state wrote V_0 there)
    for (const BatchNet &x : X->nets) {
        if (x.n_pad > x.n) {
            e = launch_fill(s->d_state + x.seg + x.n, PAD_VOLT, x.n_pad - x.n, s->st);
            if (e == cudaSuccess) e = launch_fill(s->d_state + 19 * s->stride + x.seg + x.n, PAD_VOLT, x.n_pad - x.n, s->st);
            if (e != cudaSuccess) return fail(ion_fail(nullptr, ION_ERR_CUDA, "ion_create_batch: %s", cudaGetErrorString(e)));
        }
    }
    if (init_state) {
        st = ion_batch_write(s, ION_FIELD_ALL, init_state);
        if (st != ION_OK) return fail(st);
    }
    st = batch_plan(s);
    if (st == ION_OK) st = batch_prepare(s);
    if (st != ION_OK) return fail(st);
    if (params->flags & ION_FLAG_PERSISTENT) {
        int coop = 0;
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, s->device);
        if (!coop) return fail(ion_fail(nullptr, ION_ERR_UNSUPPORTED, "ion_create_batch: no cooperative launches"));
        X->persistent = true;
        s->flags |= ION_FLAG_PERSISTENT;
        if (X->p_R == 0) X->p_R = persist_rows(X);
        else if (X->p_R == 8) X->p_R = 2;   // a shape of the per-step launches only
        st = batch_persist_plan(s);
        if (st != ION_OK) return fail(st);
        s->run_override = batch_persist_run;
        s->drop_hook = batch_persist_drop;
    }
    *out = s;
    return ION_OK;
}

// ---- autotuner ------------------------------------------------------------------------------
// Times candidate launch shapes on the handle's own network(s), `steps` time steps each
// (direct launches, CUDA events), and keeps the fastest.  The state and step count are
// saved before and restored after, so tuning does not advance the simulation.
static ion_status time_steps(ion_sim *s, int steps, float *ms) {
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    const int64_t t_save = s->t;
    cudaEventRecord(a, s->st);
    const uint32_t flags = s->flags;
    s->flags |= ION_FLAG_NO_GRAPH;
    ion_status st = ion_step(s, steps, nullptr);
    s->flags = flags;
    cudaEventRecord(b, s->st);
    cudaError_t e = cudaEventSynchronize(b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    (void)t_save;
    if (st != ION_OK) return st;
    if (e != cudaSuccess) return ion_fail(s, ION_ERR_CUDA, "autotune timing: %s", cudaGetErrorString(e));
    return ION_OK;
}

static ion_status autotune_persist_batch(ion_sim *s, int32_t steps, ion_tune *chosen);

extern "C" ion_status ion_autotune(ion_sim *s, int32_t steps, ion_tune *chosen) {
    if (!s || steps < 1) return ion_fail(s, ION_ERR_INVALID_ARG, "ion_autotune: bad arguments");
    if (s->ext && s->run_override == batch_persist_run) return autotune_persist_batch(s, steps, chosen);
    if (s->run_override) return ion_fail(s, ION_ERR_UNSUPPORTED, "ion_autotune: persistent handles are not tuned");
    // save the state and the step counter
    float *save = nullptr;
    const size_t bytes = (size_t)20 * s->stride * sizeof(float);
    cudaError_t e = cudaStreamSynchronize(s->st);
    if (e == cudaSuccess) e = ion_alloc(&save, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(save, s->d_state, bytes, cudaMemcpyDeviceToDevice);
    if (e != cudaSuccess) {
        cudaFree(save);
        return ion_fail(s, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "ion_autotune: %s",
                        cudaGetErrorString(e));
    }
    const int64_t t0 = s->t;
    auto restore = [&]() {
        cudaStreamSynchronize(s->st);
        cudaMemcpy(s->d_state, save, bytes, cudaMemcpyDeviceToDevice);
        cudaMemcpy(s->d_t, &t0, sizeof t0, cudaMemcpyHostToDevice);
        s->t = t0;
    };
    float best = 1e30f;
    ion_tune bt{};
    ion_status st = ION_OK;
    if (s->ext && s->step_override == batch_step) {
        BatchExt *X = ext_of(s);
        const int Rs[] = {1, 2, 4, 8};
        const int rows[] = {64, 128, 256};
        const int scales[] = {0, 1, -1};
        int bR = X->R, brows = X->csr_rows, bsc = X->sw_scale;
        for (int R : Rs)
            for (int r : rows)
                for (int sc : scales) {
                    X->R = R;
                    X->csr_rows = r;
                    X->sw_scale = sc;
                    st = batch_plan(s);
                    if (st == ION_OK) st = batch_prepare(s);
                    float ms = 0;
                    if (st == ION_OK) st = time_steps(s, steps, &ms);
                    restore();
                    if (st != ION_OK) break;
                    if (ms < best) {
                        best = ms;
                        bR = R;
                        brows = r;
                        bsc = sc;
                    }
                }
        X->R = bR;
        X->csr_rows = brows;
        X->sw_scale = bsc;
        if (st == ION_OK) st = batch_plan(s);
        if (st == ION_OK) st = batch_prepare(s);
        bt.dense_rows_per_warp = bR;
        bt.dense_warps = 8;
        bt.dense_col_splits = 1;
        bt.csr_rows_per_cta = brows;
        bt.csr_lanes_scale = bsc;     // scale of the degree-based choice: 0, +1 (x2), -1 (/2)
    } else if (s->kind == ION_DENSE_UNIFORM) {
        int R0, W0, G0;
        ion_choose_dense_shape(s->n, s->sms, &R0, &W0, &G0);
        struct Shape { int R, W, GJ; };
        std::vector<Shape> cand = {{R0, W0, G0}};
        const int Rs[] = {1, 2, 4, 6, 8};
        const int GJs[] = {1, 2, 4};
        for (int R : Rs)
            for (int GJ : GJs)
                for (int GR = 1; GR <= 32; ++GR) {
                    const int W = GR * GJ;
                    if (W * 32 > dense_max_threads(R) || W < 8) continue;
                    const long rows_cta = (long)GR * R;
                    const long grid = (s->n + rows_cta - 1) / rows_cta;
                    const long cost = ((grid + s->sms - 1) / s->sms) * (rows_cta + 4);
                    const long grid0 = (s->n + (long)(W0 / G0) * R0 - 1) / ((long)(W0 / G0) * R0);
                    const long cost0 = ((grid0 + s->sms - 1) / s->sms) * ((long)(W0 / G0) * R0 + 4);
                    if (cost <= cost0 * 11 / 10 && cand.size() < 12 && !(R == R0 && W == W0 && GJ == G0))
                        cand.push_back({R, W, GJ});
                }
        Shape bs = cand[0];
        for (const Shape &c : cand) {
            if (prepare_dense_step(c.R, c.W, c.GJ, s->n_pad) != cudaSuccess) continue;
            s->dense_R = c.R;
            s->dense_W = c.W;
            s->dense_GJ = c.GJ;
            float ms = 0;
            st = time_steps(s, steps, &ms);
            restore();
            if (st != ION_OK) break;
            if (ms < best) {
                best = ms;
                bs = c;
            }
        }
        s->dense_R = bs.R;
        s->dense_W = bs.W;
        s->dense_GJ = bs.GJ;
        prepare_dense_step(bs.R, bs.W, bs.GJ, s->n_pad);
        bt.dense_rows_per_warp = bs.R;
        bt.dense_warps = bs.W;
        bt.dense_col_splits = bs.GJ;
    } else if (s->kind == ION_DENSE_MATRIX) {
        int bR = s->dense_R;
        for (int R : {1, 2, 4}) {
            s->dense_R = R;
            float ms = 0;
            st = time_steps(s, steps, &ms);
            restore();
            if (st != ION_OK) break;
            if (ms < best) {
                best = ms;
                bR = R;
            }
        }
        s->dense_R = bR;
        bt.dense_rows_per_warp = bR;
        bt.dense_warps = 8;
        bt.dense_col_splits = 1;
    } else if (s->kind == ION_CSR) {
        const int SWs[] = {1, 2, 4, 8, 16, 32};
        const int rows[] = {32, 64, 128, 256};
        int bsw = s->csr_SW, brows = s->csr_rows, bstaged = s->csr_staged;
        int b_csw = s->csr_chunk_SW;
        const int sw0 = s->csr_SW;
        int sl0 = 0;   // the sliced layout's own choice of lanes per row
        for (int staged = 0; staged <= 1 && st == ION_OK; ++staged) {
            if (staged) {
                if (ion_setup_csr_staging(s, 2) != ION_OK || s->csr_staged == 0) break;
                if (s->sl.cols) sl0 = 1 << s->sl.lsw;
            } else {
                s->csr_staged = 0;
            }
            const int mode = s->csr_staged;
            for (int sw : SWs) {
                if (sl0 ? (sw * 2 < sl0 || sw > sl0 * 2) : (sw * 4 < sw0 || sw > sw0 * 4)) continue;   // near the default
                for (int r : rows) {
                    if (staged && r != rows[0]) continue;     // staged: rows per CTA fixed by the SM count
                    if (sl0) {   // the layout holds the lanes per row: built again
                        s->csr_chunk_SW = sw;
                        st = sw == 1 << s->sl.lsw ? ION_OK : ion_build_sliced(s, sw);
                        if (st != ION_OK) break;
                    } else if (staged) {
                        s->csr_chunk_SW = sw;
                        st = ion_prepare_csr_chunk(s);
                        if (st != ION_OK) break;
                    } else {
                        s->csr_SW = sw;
                        s->csr_rows = r;
                    }
                    float ms = 0;
                    st = time_steps(s, steps, &ms);
                    restore();
                    if (st != ION_OK) break;
                    if (ms < best) {
                        best = ms;
                        bstaged = mode;
                        if (staged) b_csw = sw;
                        else {
                            bsw = sw;
                            brows = r;
                        }
                    }
                }
            }
        }
        s->csr_SW = bsw;
        s->csr_rows = brows;
        s->csr_staged = bstaged;
        s->csr_chunk_SW = b_csw;
        if (sl0 && st == ION_OK && (!bstaged || b_csw != 1 << s->sl.lsw))
            st = ion_build_sliced(s, bstaged ? b_csw : sl0);   // the best lanes (or the default) again
        if (sl0 && !s->sl.cols) s->csr_staged = 0;   // a failed rebuild: the direct kernel
        bt.csr_lanes_per_row = bstaged ? b_csw : bsw;
        bt.csr_rows_per_cta = bstaged ? (sl0 ? s->sl.rows : s->csr_chunk_rows) : brows;
        bt.csr_staging = bstaged ? 2 : 1;
    }
    ion_drop_graphs(s);
    cudaFree(save);
    if (st != ION_OK) return st;
    if (chosen) *chosen = bt;
    return ION_OK;
}

// Persistent batches: rows per warp of the dense pieces (1, 2 or 4), each timed over
// `steps` steps of one launch, the state and step count restored after each.
static ion_status autotune_persist_batch(ion_sim *s, int32_t steps, ion_tune *chosen) {
    BatchExt *X = ext_of(s);
    float *save = nullptr;
    const size_t bytes = (size_t)20 * s->stride * sizeof(float);
    cudaError_t e = cudaStreamSynchronize(s->st);
    if (e == cudaSuccess) e = ion_alloc(&save, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(save, s->d_state, bytes, cudaMemcpyDeviceToDevice);
    if (e != cudaSuccess) {
        cudaFree(save);
        return ion_fail(s, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "ion_autotune: %s",
                        cudaGetErrorString(e));
    }
    const int64_t t0 = s->t;
    float best = 1e30f;
    int bR = X->p_R;
    ion_status st = ION_OK;
    for (int R : {1, 2, 4}) {
        X->p_R = R;
        st = batch_persist_plan(s);
        if (st != ION_OK) break;
        cudaEvent_t a, b;
        cudaEventCreate(&a);
        cudaEventCreate(&b);
        cudaEventRecord(a, s->st);
        st = batch_persist_run(s, steps, nullptr);
        cudaEventRecord(b, s->st);
        float ms = 0.0f;
        e = cudaEventSynchronize(b);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
        cudaEventDestroy(a);
        cudaEventDestroy(b);
        cudaMemcpy(s->d_state, save, bytes, cudaMemcpyDeviceToDevice);
        cudaMemcpy(s->d_t, &t0, sizeof t0, cudaMemcpyHostToDevice);
        s->t = t0;
        if (st != ION_OK) break;
        if (e != cudaSuccess) {
            st = ion_fail(s, ION_ERR_CUDA, "ion_autotune: %s", cudaGetErrorString(e));
            break;
        }
        if (ms < best) {
            best = ms;
            bR = R;
        }
    }
    X->p_R = bR;
    if (st == ION_OK) st = batch_persist_plan(s);
    cudaFree(save);
    if (st != ION_OK) return st;
    if (chosen) {
        *chosen = ion_tune{};
        chosen->dense_rows_per_warp = bR;
        chosen->dense_warps = 8;
        chosen->dense_col_splits = 1;
        chosen->csr_rows_per_cta = X->csr_rows;
    }
    return ION_OK;
}
