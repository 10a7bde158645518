// ion_csr_sliced.cu -- the staged CSR step on a sliced layout: V_dend in shared memory, every
// warp's edges one contiguous stream.
//
// A CTA of 1024 threads (one per SM) owns `rows` consecutive rows.  V_dend is staged in shared
// memory: whole when it fits beside the rows' own data, else in even chunks through two
// buffers, the next chunk landing while one is summed.  Within a (chunk, CTA) the rows are
// sorted by their edge count there and cut into slices of 32 / SW rows, one warp per slice,
// SW lanes per row.  A slice's columns are stored round by round: a round is 8 edges of every
// lane, 32 x 16 bytes read by one coalesced load, so a warp walks one stream without row
// bounds, heads, tails or a remainder loop; the sort keeps the padding of a slice's shorter
// rows small (sorted sliced ELLPACK, Kreutzer et al. 2014).  A row far longer than the mean
// gets more lanes, up to the whole warp: a warp walking it with SW lanes would hold every
// other warp at the chunk's barrier (65 536 cells, k = 100, 8 rows of 3000 edges: 37.5 us per
// step with the mean row's lanes, 10.3 now, 10.0 without such rows).  Columns are 16-bit
// offsets into the staged buffer; padding entries point at the row's own V_dend behind the
// buffers (dV = 0: they add exactly 0).
//
// Bank order: one gather reads entry t of all 32 lanes, from 32 random banks about 3.5
// wavefronts, and these bound the sums.  The order of a lane's edges is free, so the fill
// orders them for distinct banks in each gather (sliced_fill_kernel).
//
// The connectivity and the pulse table do not change between steps, so a warp's first rounds and
// its row's pulse are loaded before the wait on the previous step; the rows' state words are
// fetched while the chunks land.
//
// What bounds it: at 65 536 cells, k = 100, a step is 10.2 us: 1.8 us from the previous step's
// end to the first chunk in shared memory, 3 x 1.7 us of sums (issue: 8 warps per scheduler,
// about half of it slice bookkeeping), 1.2 us of update, 1.5 us to the next step.  The chunked
// kernel it replaced (16 lanes per row-and-chunk segment of 50 edges, chunks in turn through
// one buffer, pulses and state read at the end) took 19.6 us; 9 001 cells with k = 1000 and a
// weight per edge went from 12.2 to 9.9 us.  Tried and left out: rounds of 4 edges per lane
// (less padding, 7 % slower), slice headers in shared memory (10 % slower), two threads per
// cell in the update (1.4 against 1.2 us).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ion.h"
#include "ion_csr_core.cuh"
#include "ion_kernels.cuh"
#include "ion_sim.h"

namespace ion {

constexpr int SL_THREADS = 1024, SL_WARPS = SL_THREADS / 32;
constexpr size_t SL_SMEM = 227 * 1024 - 1024;   // dynamic shared memory of a CTA

// An entry of L.rowid: a row of the CTA (L.rows: none) and its slice's lanes per row (log2).
constexpr int ROW_BITS = 10;
static_assert(SL_THREADS <= 1 << ROW_BITS, "rows and the none mark fit the row bits");
__host__ __device__ constexpr uint16_t row_entry(int row, int lsw) { return (uint16_t)(row | lsw << ROW_BITS); }
__host__ __device__ constexpr int entry_row(uint16_t v) { return v & ((1 << ROW_BITS) - 1); }
__host__ __device__ constexpr int entry_lsw(uint16_t v) { return v >> ROW_BITS; }

struct SliceItem {
    int32_t e0, e1;  // first round and end (as loaded: nothing waits on them before they are used)
    uint16_t row;    // this lane's entry of L.rowid
    __device__ __forceinline__ int n() const { return e1 - e0; }
};

__device__ __forceinline__ void cp_async16_sl(void *smem_dst, const void *gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}

template <bool HAS_W, bool LIN>
__global__ void __launch_bounds__(SL_THREADS, 1) csr_sliced_step_kernel(const CsrArgs a, const SliceLayout L) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    // rounds in flight per lane: 64 bytes of columns, or 32 and 64 of weights, of the 64
    // registers a thread may have
    constexpr int D = HAS_W ? 2 : 4;
    float *vs = reinterpret_cast<float *>(smem_raw);
    float *own = vs + L.nbuf * L.chunk, *ic_s = own + L.rows + 4, *cs = ic_s + L.rows + 4;
    const StepCommon &c = a.c;
    const int n = c.n, row0 = blockIdx.x * L.rows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int passes = L.nsl / SL_WARPS;   // slices per (chunk, CTA): whole passes, the last ones empty
    // this warp's slices: base of (chunk 0, pass 0), then pass by pass and chunk by chunk (the
    // arrays end with two chunks' worth of empty slices, so the look-ahead needs no bounds)
    int next_base = blockIdx.x * L.nsl + warp, next_p = 0;
    auto next_item = [&]() {
        SliceItem it;
        it.e0 = __ldg(L.off + next_base);
        it.e1 = __ldg(L.off + next_base + 1);
        it.row = __ldg(L.rowid + ((next_base << (5 - L.lsw)) + (lane >> L.lsw)));
        next_base += ++next_p == passes ? (int)gridDim.x * L.nsl - (passes - 1) * SL_WARPS : SL_WARPS;
        if (next_p == passes) next_p = 0;
        return it;
    };
    uint4 q[D];
    float4 wa[HAS_W ? D : 1], wb[HAS_W ? D : 1];
    // (rounds x 64 below 2^31: checked when the layout is built)
    auto stream = [&](const SliceItem &it) { return L.cols + (it.e0 * 32 + lane); };
    auto wstream = [&](const SliceItem &it) { return HAS_W ? L.w + (it.e0 * 64 + lane) : L.w; };
    auto load = [&](int j, const uint4 *p, const float4 *w) {   // round j of the stream at p, w
        q[j] = __ldcs(p + j * 32);
        if (HAS_W) {
            wa[j] = __ldcs(w + j * 64);
            wb[j] = __ldcs(w + j * 64 + 32);
        }
    };
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    // connectivity and pulses do not change between steps: read before the wait
    SliceItem cur = next_item(), nxt = next_item();
    {
        const uint4 *p = stream(cur);
        const float4 *w = wstream(cur);
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (j < cur.n()) load(j, p, w);
    }
    const int mine = threadIdx.x;   // this thread's row (rows <= SL_THREADS)
    const bool has_row = mine < L.rows && row0 + mine < n;
    const PulseAhead pa = pulse_ahead(c.pulses, row0 + mine, has_row && a.fuse);
    __syncthreads();
    pdl_enter();
    const float *vcur = vd_cur(c);
    auto issue = [&](int ch) {
        const int c0 = ch * L.chunk, b = ch % L.nbuf;
        const uint32_t bytes = (uint32_t)min(L.chunk, c.n_pad - c0) * 4u;
        mbar_expect_tx(&bar[b], bytes);
        bulk_g2s(vs + b * L.chunk, vcur + c0, bytes, &bar[b]);
    };
    if (threadIdx.x == 0)
        for (int ch = 0; ch < min(L.nbuf, L.n_chunks); ++ch) issue(ch);
    const int64_t t = step_index(c);
    if (mine <= L.rows) {   // [rows]: the row of slice positions that have none
        ic_s[mine] = 0.0f;
        own[mine] = has_row ? vcur[row0 + mine] : 0.0f;
    }
    if (L.stage && a.fuse) {   // the rows' state words, 16 bytes (4 rows) at a time
        const int q4 = L.rows >> 2;
        for (int i = threadIdx.x; i < NCW * q4; i += SL_THREADS) {
            const int w = i / q4, r = 4 * (i - w * q4);
            if (row0 + r < c.n_pad)
                cp_async16_sl(cs + w * L.rows + r, (w == 0 ? vcur : c.S.f(cell_word_field(w))) + row0 + r);
        }
        cp_async_commit();
    }
    float iapp = 0.0f;
    if (has_row && a.fuse) {
        iapp = pulse_current(c.pulses, pa, t);
        if (c.iapp != nullptr) iapp += c.iapp[row0 + mine];
    }
    __syncthreads();
    for (int ch = 0; ch < L.n_chunks; ++ch) {
        const int b = ch % L.nbuf;
        const uint32_t phase = (uint32_t)(ch / L.nbuf) & 1u;
        // one warp polls, the others wait at the barrier (all 32 polling took two thirds of the
        // kernel's issue slots)
        const bool landed = warp != 0 || mbar_wait_bounded(&bar[b], phase);
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) {   // wait (bounded) for the copies still in flight, then leave
                if (c.status != nullptr) atomicOr(c.status, (uint32_t)ST_TIMEOUT);
                (void)mbar_wait_bounded(&bar[b], phase);
                if (L.nbuf > 1 && ch + 1 < L.n_chunks)
                    (void)mbar_wait_bounded(&bar[b ^ 1], (uint32_t)((ch + 1) / L.nbuf) & 1u);
            }
            cp_async_wait_all();
            return;
        }
        const VjSliced vj{vs + b * L.chunk};
        for (int p = 0; p < passes; ++p) {
            const SliceItem nn = next_item();   // the slice after next: its header arrives meanwhile
            const int rr = entry_row(cur.row), sw = 1 << entry_lsw(cur.row);
            const float vi = own[rr];
            float ks = 0.0f, kc = 0.0f;   // compensated over groups of D rounds
            const uint4 *pc = stream(cur);
            const float4 *wc = wstream(cur);
            for (int left = cur.n();; left -= D) {
                const bool last = left <= D;   // then the next slice's first rounds are requested
                pc = last ? stream(nxt) : pc + D * 32;
                if (HAS_W) wc = last ? wstream(nxt) : wc + D * 64;
                const int more = last ? nxt.n() : left - D;
                float blk = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    if (j < left) blk += csr_group16<HAS_W, LIN>(q[j], wa[HAS_W ? j : 0], wb[HAS_W ? j : 0], vi, vj);
                    if (j < more) load(j, pc, wc);
                }
                kahan_add(ks, kc, blk);
                if (last) break;
            }
            float acc = ks - kc;
            for (int off = sw >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if ((lane & (sw - 1)) == 0) ic_s[rr] += acc;
            cur = nxt;
            nxt = nn;
        }
        if (ch + 1 == L.n_chunks) cp_async_wait_all();   // the staged state words, before the barrier below
        __syncthreads();
        if (threadIdx.x == 0 && ch + L.nbuf < L.n_chunks) {   // every read of this buffer is done
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(ch + L.nbuf);
        }
    }
    auto current = [&](int r) { return (HAS_W ? ic_s[r] : ic_s[r] * a.g) * (1.0f / GJ_SCALE); };
    if (!has_row) return;
    const int i = row0 + mine;
    if (!a.fuse) {
        a.ic_out[i] = current(mine);
        return;
    }
    const Cell cell = L.stage ? staged_cell(cs, L.rows, mine) : load_cell(c.S, vcur, i, own[mine]);
    const CellNext o = cell_step(c.P, cell, current(mine), iapp);
    finish_cell(c, t, vd_next(c), i, o);
}

static size_t sliced_smem_bytes(const SliceLayout &L) {
    return ((size_t)L.nbuf * L.chunk + (size_t)(2 + (L.stage ? NCW : 0)) * L.rows + 8) * sizeof(float);
}

template <bool HAS_W, bool LIN>
static cudaError_t sliced_T(const CsrArgs &a, const SliceLayout &L, bool prepare, cudaStream_t st) {
    if (prepare)
        return cudaFuncSetAttribute(csr_sliced_step_kernel<HAS_W, LIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)SL_SMEM);
    const int grid = (a.c.n + L.rows - 1) / L.rows;
    return launch_k(csr_sliced_step_kernel<HAS_W, LIN>, dim3(grid), dim3(SL_THREADS), sliced_smem_bytes(L), st,
                    a.c.pdl != 0, a, L);
}
static cudaError_t sliced(const CsrArgs &a, const SliceLayout &L, bool prepare, cudaStream_t st) {
    if (L.w != nullptr) return a.lin ? sliced_T<true, true>(a, L, prepare, st) : sliced_T<true, false>(a, L, prepare, st);
    return a.lin ? sliced_T<false, true>(a, L, prepare, st) : sliced_T<false, false>(a, L, prepare, st);
}
cudaError_t launch_csr_sliced_step(const CsrArgs &a, const SliceLayout &L, cudaStream_t st) {
    return sliced(a, L, false, st);
}

// First edge of row i with a column of chunk ch or later: the lower bound of ch * chunk in the
// sorted row (ch = 0 .. n_chunks: bound[ch * n + i]).
__global__ void sliced_bounds_kernel(const int32_t *row_ptr, const int32_t *col, int32_t n, int chunk, int n_chunks,
                                     int32_t *bound) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int b = row_ptr[i], e = row_ptr[i + 1];
    bound[i] = b;
    bound[(int64_t)n_chunks * n + i] = e;
    for (int ch = 1; ch < n_chunks; ++ch) {
        int lo = b, hi = e;
        while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (col[m] < ch * chunk) lo = m + 1;
            else hi = m;
        }
        bound[(int64_t)ch * n + i] = lo;
    }
}

// Columns (and weights) of every slice from the sorted CSR, in an order that spreads the banks
// of each gather: one warp per slice, a thread per slice lane.  Every lane sorts its edges by
// bank (`order`, as many entries as `cols`, receives them); then, gather by gather, the lanes
// take turns (from a lane that moves on by one each time) to pick an edge whose bank no lane
// before has taken; a lane without one puts in a padding entry if it has any left, else any
// edge.
__global__ void __launch_bounds__(128) sliced_fill_kernel(const int32_t *bound, const int32_t *col, const float *w,
                                                          int32_t n, int grid, SliceLayout L, int64_t slices,
                                                          uint16_t *cols, float *wout, uint16_t *order) {
    __shared__ uint16_t cnt_s[4][32][32], pos_s[4][32][32];   // [warp][bank][lane]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = (int64_t)blockIdx.x * 4 + warp;
    if (base >= slices) return;
    const int ch = (int)(base / ((int64_t)grid * L.nsl)), cta = (int)(base / L.nsl % grid);
    const uint16_t row = L.rowid[(base << (5 - L.lsw)) + (lane >> L.lsw)];
    const int rr = entry_row(row), sw = 1 << entry_lsw(row), li = lane & (sw - 1);
    const int64_t r0 = L.off[base];
    const int T = 8 * (int)(L.off[base + 1] - r0);   // entries of every lane
    auto at = [&](int t) { return ((r0 + (t >> 3)) * 32 + lane) * 8 + (t & 7); };
    auto wat = [&](int t) { return ((r0 + (t >> 3)) * 64 + ((t >> 2) & 1) * 32 + lane) * 4 + (t & 3); };
    uint16_t (*cnt)[32] = cnt_s[warp], (*pos)[32] = pos_s[warp];
    for (int b = 0; b < 32; ++b) cnt[b][lane] = 0;
    int e0 = 0, e1 = 0;
    uint16_t self = 0;
    if (rr != L.rows) {
        const int i = cta * L.rows + rr;
        e0 = bound[(int64_t)ch * n + i];
        e1 = bound[(int64_t)(ch + 1) * n + i];
        self = (uint16_t)((L.nbuf - ch % L.nbuf) * L.chunk + rr);
    }
    int left = 0;                  // this lane's edges not yet placed
    for (int k = e0 + li; k < e1; k += sw, ++left) cnt[(col[k] - ch * L.chunk) & 31][lane]++;
    uint32_t avail = 0, many = 0;  // banks it still has edges of, and at least two
    int run = 0;
    for (int b = 0; b < 32; ++b) {
        pos[b][lane] = (uint16_t)run;
        run += cnt[b][lane];
        if (cnt[b][lane]) avail |= 1u << b;
        if (cnt[b][lane] > 1) many |= 1u << b;
    }
    for (int k = e0 + li; k < e1; k += sw) {
        const int b = (col[k] - ch * L.chunk) & 31;
        order[at(pos[b][lane]++)] = (uint16_t)(k - e0);
    }
    for (int t = 0; t < T; ++t) {   // pos[b] now ends bank b's edges: they are taken from the end
        uint32_t taken = 0;
        int pick = -1;              // bank of this lane's entry (-1: padding)
        for (int s = 0; s < 32; ++s) {
            const int l = (s + t) & 31;
            const uint32_t av = __shfl_sync(0xffffffffu, avail, l), mn = __shfl_sync(0xffffffffu, many, l) & ~taken;
            const int slack = __shfl_sync(0xffffffffu, T - t - left, l);   // > 0: padding entries left
            const uint32_t free = av & ~taken;
            // scan the banks from one that moves on too, so that no bank is always used up first
            // (banks with several edges first: a choice is left for later gathers)
            const uint32_t from = mn ? mn : (free ? free : (slack > 0 ? 0u : av));
            const uint32_t rot = __funnelshift_r(from, from, l + t);
            const int b = rot ? (__ffs(rot) - 1 + l + t) & 31 : -1;
            if (b >= 0) taken |= 1u << b;
            if (l == lane) pick = b;
        }
        if (pick >= 0) {
            const int x = --pos[pick][lane];
            const int more = --cnt[pick][lane];
            if (more <= 1) many &= ~(1u << pick);
            if (more == 0) avail &= ~(1u << pick);
            --left;
            const int k = e0 + order[at(x)];
            cols[at(t)] = (uint16_t)(col[k] - ch * L.chunk);
            if (wout) wout[wat(t)] = w[k];
        } else {
            cols[at(t)] = self;
            if (wout) wout[wat(t)] = 0.0f;
        }
    }
}

}  // namespace ion

using namespace ion;

// Rows per CTA, chunks, buffers and lanes per row of a network of n cells (lanes 0: choose).
// One CTA per SM; up to 512 rows the rows' state words are staged too.  A V_dend that fits is
// one chunk, a longer one even chunks in two buffers.  Lanes per row: enough slices for the 32
// warps of the CTA, as long as a row keeps about 8 edges per lane and chunk.
SliceLayout ion_plan_sliced(int32_t n, int32_t n_pad, int64_t nnz, int sms, int lanes) {
    SliceLayout L{};
    L.rows = (std::min(SL_THREADS - 4, std::max(1, (n + sms - 1) / sms)) + 3) / 4 * 4;   // a thread per row, and one more
    L.stage = L.rows <= SL_THREADS / 2;
    const int cap = (int)(SL_SMEM / sizeof(float)) - (2 + (L.stage ? NCW : 0)) * L.rows - 8;
    L.nbuf = n_pad <= cap ? 1 : 2;
    L.chunk = n_pad;
    L.n_chunks = 1;
    if (L.nbuf == 2) {
        const int most = cap / 2 / PAD_J * PAD_J;
        L.n_chunks = (n_pad + most - 1) / most;
        L.chunk = ((n_pad + L.n_chunks - 1) / L.n_chunks + PAD_J - 1) / PAD_J * PAD_J;
        L.n_chunks = (n_pad + L.chunk - 1) / L.chunk;   // the rounding may leave fewer
    }
    const double seg = (double)nnz / n / L.n_chunks;
    L.lsw = 0;
    if (lanes > 0)
        while (L.lsw < 5 && (1 << L.lsw) < lanes) L.lsw++;
    else
        while (L.lsw < 5 && (L.rows << (L.lsw + 1)) <= SL_THREADS && (8 << (L.lsw + 1)) <= seg) L.lsw++;
    const int per = 32 >> L.lsw;
    L.nsl = (L.rows + per * SL_WARPS - 1) / (per * SL_WARPS) * SL_WARPS;   // whole passes of the 32 warps
    // twice the mean rounds, at least four: no row of a random graph is near it
    L.most_rounds = std::max(4, 2 * (int)std::ceil(seg / (8 << L.lsw)));
    return L;
}

// Lanes (log2) of a row with `edges` edges in a chunk
static int row_lsw(const SliceLayout &L, int32_t edges) {
    int lsw = L.lsw;
    while (lsw < 5 && edges > (8 << lsw) * L.most_rounds) ++lsw;
    return lsw;
}

void ion_free_sliced(ion_sim *s) {
    cudaFree((void *)s->sl.cols);
    cudaFree((void *)s->sl.w);
    cudaFree((void *)s->sl.off);
    cudaFree((void *)s->sl.rowid);
    s->sl = SliceLayout{};
}

// Build the layout on the handle (host CSR copied to the device: columns sorted and in range).
// Leaves s->sl empty, with ION_OK, where the round offsets would not fit 32 bits.
ion_status ion_build_sliced(ion_sim *s, int lanes) {
    ion_free_sliced(s);
    SliceLayout L = ion_plan_sliced(s->n, s->n_pad, s->nnz, s->sms, lanes);
    const int n = s->n, C = L.n_chunks, grid = (n + L.rows - 1) / L.rows, per0 = 32 >> L.lsw;
    int32_t *d_bound = nullptr;
    uint16_t *d_order = nullptr;
    auto done = [&](cudaError_t e) {
        cudaFree(d_bound);
        cudaFree(d_order);
        if (e == cudaSuccess) return ION_OK;
        ion_free_sliced(s);
        return ion_fail(nullptr, e == cudaErrorMemoryAllocation ? ION_ERR_OOM : ION_ERR_CUDA, "CSR sliced layout: %s",
                        cudaGetErrorString(e));
    };
    cudaError_t e = ion_alloc(&d_bound, (size_t)(C + 1) * n * sizeof(int32_t));
    if (e != cudaSuccess) return done(e);
    sliced_bounds_kernel<<<(n + 255) / 256, 256, 0, s->st>>>(s->d_rowptr, s->d_col, n, L.chunk, C, d_bound);
    std::vector<int32_t> bound((size_t)(C + 1) * n);
    e = cudaMemcpyAsync(bound.data(), d_bound, bound.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, s->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) return done(e);
    auto edges_at = [&](int ch, int i) { return bound[(size_t)(ch + 1) * n + i] - bound[(size_t)ch * n + i]; };
    // slices per (chunk, CTA): rows of different lanes are in slices of their own
    for (int ch = 0; ch < C; ++ch)
        for (int b = 0; b < grid; ++b) {
            int rows_of[6] = {}, need = 0;
            for (int i = b * L.rows; i < std::min(n, (b + 1) * L.rows); ++i) rows_of[row_lsw(L, edges_at(ch, i))]++;
            for (int l = 0; l <= 5; ++l) need += (rows_of[l] + (32 >> l) - 1) / (32 >> l);
            L.nsl = std::max(L.nsl, (need + SL_WARPS - 1) / SL_WARPS * SL_WARPS);
        }
    const int64_t slices = (int64_t)C * grid * L.nsl;
    const int64_t pad = 2 * (int64_t)grid * L.nsl;   // empty slices behind the last, for the look-ahead
    if ((slices + pad) * 32 >= INT32_MAX) return done(cudaSuccess);   // keep the unsliced layout
    std::vector<int32_t> off((size_t)(slices + pad) + 1);
    std::vector<uint16_t> rowid((size_t)(slices + pad) * per0, row_entry(L.rows, L.lsw));
    std::vector<int32_t> order((size_t)L.rows), first;   // rows by falling edge count (a counting sort)
    int64_t tot = 0;
    for (int ch = 0; ch < C; ++ch)
        for (int b = 0; b < grid; ++b) {
            const int r0 = b * L.rows, here = std::min(L.rows, n - r0);
            auto edges = [&](int r) { return edges_at(ch, r0 + r); };
            int32_t most = 0;
            for (int r = 0; r < here; ++r) most = std::max(most, edges(r));
            first.assign((size_t)most + 2, 0);
            for (int r = 0; r < here; ++r) first[(size_t)(most - edges(r)) + 1]++;
            for (int32_t k = 0; k <= most; ++k) first[(size_t)k + 1] += first[(size_t)k];
            for (int r = 0; r < here; ++r) order[(size_t)first[(size_t)(most - edges(r))]++] = r;
            for (int q = 0, at = 0; q < L.nsl; ++q) {   // at: the next row of the sorted order
                const int64_t base = ((int64_t)ch * grid + b) * L.nsl + q;
                off[(size_t)base] = (int32_t)tot;
                if (at >= here) continue;
                const int32_t longest = edges(order[(size_t)at]);
                const int lsw = row_lsw(L, longest), rep = 1 << (lsw - L.lsw);   // entries of a row
                tot += (longest + (8 << lsw) - 1) / (8 << lsw);
                if (tot >= INT32_MAX / 64) return done(cudaSuccess);   // keep the unsliced layout
                for (int x = 0; x < per0; ++x) {
                    const int r = at + x / rep;
                    const bool mine = r < here && row_lsw(L, edges(order[(size_t)r])) == lsw;
                    rowid[(size_t)base * per0 + x] = row_entry(mine ? order[(size_t)r] : L.rows, lsw);
                }
                for (int x = 0; x < 32 >> lsw && at < here && row_lsw(L, edges(order[(size_t)at])) == lsw; ++x) ++at;
            }
        }
    std::fill(off.begin() + slices, off.end(), (int32_t)tot);
    const size_t rounds = (size_t)std::max<int64_t>(tot, 1);
    uint16_t *cols = nullptr, *rid = nullptr;
    float *w = nullptr;
    int32_t *doff = nullptr;
    e = ion_alloc(&cols, rounds * 512);
    s->sl.cols = reinterpret_cast<const uint4 *>(cols);
    if (e == cudaSuccess && s->d_w) e = ion_alloc(&w, rounds * 1024);
    s->sl.w = reinterpret_cast<const float4 *>(w);
    if (e == cudaSuccess) e = ion_alloc(&doff, off.size() * sizeof(int32_t));
    s->sl.off = doff;
    if (e == cudaSuccess) e = ion_alloc(&rid, rowid.size() * sizeof(uint16_t));
    s->sl.rowid = rid;
    if (e == cudaSuccess) e = ion_alloc(&d_order, rounds * 512);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(doff, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s->st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(rid, rowid.data(), rowid.size() * sizeof(uint16_t), cudaMemcpyHostToDevice, s->st);
    L.cols = s->sl.cols;
    L.w = s->sl.w;
    L.off = s->sl.off;
    L.rowid = s->sl.rowid;
    for (int lin = 0; lin < 2 && e == cudaSuccess; ++lin) {   // both junctions' kernels
        CsrArgs probe{};
        probe.lin = lin;
        e = sliced(probe, L, true, s->st);
    }
    if (e == cudaSuccess) {
        s->sl = L;
        sliced_fill_kernel<<<(unsigned)((slices + 3) / 4), 128, 0, s->st>>>(d_bound, s->d_col, s->d_w, n, grid, L, slices,
                                                                           cols, w, d_order);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);   // the host arrays are released on return
    return done(e);
}
