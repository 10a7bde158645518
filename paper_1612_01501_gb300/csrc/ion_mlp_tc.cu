// ion_mlp_tc.cu -- inference of the learned rate-function surrogate (not in the paper) on
// the fifth-generation tensor cores: tcgen05.mma with TMEM accumulators.
//
// The surrogate is the MLP of ion_mlp.cu: (V, ln[Ca]) -> 64 tanh -> 64 tanh -> 24 outputs
// (logit x_inf and ln tau of every gate).  A CTA of 128 threads owns 128 cells and
// evaluates the MLP for their three compartments (V_dend, V_soma, V_axon, each with the
// cell's [Ca]) as three 128-row tiles: row t of every tile is cell t of the CTA, so thread
// t ends up holding all three compartments' rates and runs that cell's explicit-Euler
// update itself.  The tiles are pipelined through two operand buffers: while the tensor core
// works on one compartment the threads run another's layer 1, epilogue or update, so that
// of the six completions only the first is waited for with nothing to do.  (The floor is the
// 192 tanh.bf16x2 of a cell: 5.0 us per step at 65 536 cells.  One tile after the other, the
// update at the end, this launch took 14.4 us of a step there; pipelined 13.4; with the TMEM
// allocation and its permit's release before the weights' copy 11.2: the next CTA of an SM
// does not start while one holds the permit.  All three tiles through a layer together needs
// a third operand buffer, and then only three CTAs share an SM.)
//   layer 1 (2 -> 64) in FP32 on the CUDA cores, tanh on packed bf16 pairs, written to
//     shared memory as the three BF16 A operands of layer 2;
//   layer 2 (64 x 64): four tcgen05.mma.kind::f16 (M = 128, N = 64, K = 16 each, BF16 in,
//     FP32 accumulation) into TMEM columns 0..63, issued by one thread and completed
//     through one tcgen05.commit on an mbarrier;
//   every thread reads its row of each tile back (tcgen05.ld, lane = row), adds the bias,
//     applies tanh and writes the tile's BF16 A operand of layer 3 over its layer-2 one;
//   layer 3 (64 x 24, padded to N = 32): four MMAs into TMEM columns 0..31 (over the
//     layer-2 results, already read), one commit, read back and mapped to physical units.
// Operands use the canonical K-major layout without swizzling: 8-row x 16-byte core
// matrices of 128 contiguous bytes, core matrix (row group g, K chunk c) at byte
// (8 g + c) 128, so the K-direction core-matrix stride (leading byte offset) is 128 B and
// the row-group stride (stride byte offset) 1024 B.
// Every wait is bounded: a tensor-core completion that does not arrive within ~0.5 s sets
// the timeout status bit.  A warp whose wait ran out neither reads the accumulators nor writes
// the operands from there on, and thread 0 issues nothing once its own has; at the end the CTA
// waits (again bounded) once more for what is in flight, frees its TMEM and returns without
// having stored a word: its cells keep step t.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "ion.h"
#include "ion_kernels.cuh"
#include "ion_sim.h"

namespace ion {
namespace tc {

constexpr int ROWS = 128;        // M of every MMA: rows (cells) per CTA
constexpr int KH = 64;           // hidden width (K of layers 2 and 3)
constexpr int N2 = 64, N3 = 32;  // layer 2 outputs; layer 3 outputs (24) padded to a multiple of 16
constexpr int NOUT = ION_MLP_OUT;
constexpr uint32_t TMEM_COLS = 128;   // buffer b: layer 2 in columns [64 b, 64 b + 64), layer 3 in the first 32 of them
constexpr float LOG2E = 1.4426950408889634f;

__host__ __device__ constexpr int core_off(int row, int kchunk) {
    return ((row >> 3) * (KH / 8) + kchunk) * 128 + (row & 7) * 16;
}

// Weights as the kernels use them (packed once per handle by mlp_tc_pack_kernel).
struct Weights {
    __nv_bfloat16 w2[N2 * KH];   // B of layer 2 (row = output unit), core-matrix layout
    __nv_bfloat16 w3[N3 * KH];   // B of layer 3, rows 24..31 zero
    float w1[2 * KH], b1[KH], b2[N2], b3[N3];
    float in_shift[2], in_scale[2], out_shift[N3], out_scale[N3];
};
struct Smem {
    __nv_bfloat16 a[2][ROWS * KH];    // A of layer 2, then of layer 3, per buffer
    Weights W;
    uint64_t bar[2];                  // completions of a buffer's MMAs
    uint64_t wbar;                    // the weights' copy
    uint32_t tmem;
};
static_assert(sizeof(Weights) % 16 == 0, "weights are copied 16 bytes at a time");
static_assert(offsetof(Smem, W) % 16 == 0, "16-byte aligned operands");

// ---- tcgen05 / TMEM primitives (inline PTX) ------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem] x B[smem]^T, both K-major; accumulate = 0 overwrites D
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrive once on `bar` when every MMA this thread issued before has completed
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 consecutive 32-bit columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: start address, leading (K-direction) and stride
// (row-group) byte offsets, descriptor version 1, no swizzling.
__device__ __forceinline__ uint64_t smem_desc(const void *p, uint32_t lbo, uint32_t sbo) {
    const uint32_t a = smem_u32(p);
    return (uint64_t)((a >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
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

// Hand buffer b to the tensor core (all threads): its generic writes are ordered before the
// asynchronous reads, then thread 0 issues the layer's four K = 16 steps and the commit, unless one
// of its own waits has run out (`ok`: those before it have then not been seen to complete).
// issued[b] counts thread 0's layers.  withhold: test hook, the commit is left out, so that the
// wait for this layer runs out.
__device__ __forceinline__ void tc_issue(Smem &sm, int b, const __nv_bfloat16 *B, uint32_t idesc, bool ok,
                                         uint32_t (&issued)[2], bool withhold) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && ok) {
        issued[b]++;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < KH / 16; ++kk)
            tc_mma(sm.tmem + b * N2, smem_desc(sm.a[b] + kk * 16 * 8, 128, 1024), smem_desc(B + kk * 16 * 8, 128, 1024),
                   idesc, kk > 0 ? 1u : 0u);
        if (!withhold) tc_commit(&sm.bar[b]);
    }
}
// Wait (bounded) for the layer last issued on buffer b; false, in every lane of the warp, if a lane
// of it did not see the completion in time, or (ok) an earlier wait of the warp ran out.
__device__ __forceinline__ bool tc_wait(Smem &sm, int b, uint32_t phase, bool ok) {
    if (!ok) return false;
    const bool done = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.bar[b], phase));
    tc_fence_after();
    return done;
}

// Layer 1 of one row of tile c: z = W1 x + b1 (FP32), tanh on bf16 pairs, into A (core-matrix layout).
__device__ __forceinline__ void layer1_row(Smem &sm, int c, int row, float x0, float x1) {
    char *abase = reinterpret_cast<char *>(sm.a[c]);
#pragma unroll
    for (int kc = 0; kc < KH / 8; ++kc) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int j = 8 * kc + 2 * h;
            const float z0 = fmaf(sm.W.w1[2 * j], x0, fmaf(sm.W.w1[2 * j + 1], x1, sm.W.b1[j]));
            const float z1 = fmaf(sm.W.w1[2 * j + 2], x0, fmaf(sm.W.w1[2 * j + 3], x1, sm.W.b1[j + 1]));
            w[h] = tanh_bf16x2(pack_bf16x2(z0, z1));
        }
        *reinterpret_cast<uint4 *>(abase + core_off(row, kc)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Layer-2 epilogue of this thread's row of tile c: + b2, tanh, into the tile's A operand
// of layer 3 (over its layer-2 operand, which the completed MMAs no longer read).
__device__ __forceinline__ void layer2_epilogue(Smem &sm, int c, uint32_t lane_addr, int row) {
    char *abase = reinterpret_cast<char *>(sm.a[c]);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        float v[32];
        tc_ld32(lane_addr + 32 * half, v);
        tc_wait_ld();
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) {
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int j = 8 * kc + 2 * h;
                w[h] = tanh_bf16x2(pack_bf16x2(v[j] + sm.W.b2[32 * half + j], v[j + 1] + sm.W.b2[32 * half + j + 1]));
            }
            *reinterpret_cast<uint4 *>(abase + core_off(row, 4 * half + kc)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// CTA prologue: TMEM columns (warp 0), weights into shared memory by one bulk copy, mbarriers.
// The weights are waited for where they are first read (wbar).
__device__ __forceinline__ void tc_setup(Smem &sm, const Weights *Wg) {
    if (threadIdx.x < 32) {
        tmem_alloc(&sm.tmem, TMEM_COLS);
        tmem_relinquish();
    } else if (threadIdx.x == 32) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        mbar_init(&sm.wbar, 1);
        fence_mbar_init();
        mbar_expect_tx(&sm.wbar, (uint32_t)sizeof(Weights));
        bulk_g2s(&sm.W, Wg, (uint32_t)sizeof(Weights), &sm.wbar);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}
__device__ __forceinline__ void tc_teardown(Smem &sm) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(sm.tmem, TMEM_COLS);
}

// The lane of TMEM this thread reads back, in buffer b
__device__ __forceinline__ uint32_t tc_lane(const Smem &sm, int b) {
    return sm.tmem + b * N2 + ((uint32_t)(32 * (threadIdx.x >> 5)) << 16);
}
// The 24 outputs of this thread's row of buffer b in physical units (layer 3 done)
__device__ __forceinline__ void tc_outputs(Smem &sm, int b, float (&y)[NOUT]) {
    float v[32];
    tc_ld32(tc_lane(sm, b), v);
    tc_wait_ld();
#pragma unroll
    for (int o = 0; o < NOUT; ++o) y[o] = fmaf(v[o] + sm.W.b3[o], sm.W.out_scale[o], sm.W.out_shift[o]);
}
// After the last wait (all threads): true if every wait of the CTA succeeded.  Else reports the
// timeout and waits once more (bounded) for the layers and the copy in flight, so that the TMEM they
// write can be freed.
__device__ __forceinline__ bool tc_finish(Smem &sm, bool ok, uint32_t *status, const uint32_t (&issued)[2]) {
    if (!__syncthreads_or(!ok)) return true;
    if (threadIdx.x == 0) {
        if (status != nullptr) atomicOr(status, (uint32_t)ST_TIMEOUT);
        for (int b = 0; b < 2; ++b)
            if (issued[b] > 0) (void)mbar_wait_bounded(&sm.bar[b], (issued[b] - 1u) & 1u);
        (void)mbar_wait_bounded(&sm.wbar, 0u);
    }
    return false;
}

__device__ __forceinline__ float learned_xinf(const float (&y)[NOUT], int gate) {
    return rcp_approx(1.0f + ex2_approx(-y[2 * gate] * LOG2E));
}
__device__ __forceinline__ Rate learned_rate(const float (&y)[NOUT], int gate) {
    return Rate{learned_xinf(y, gate), ex2_approx(-y[2 * gate + 1] * LOG2E)};
}

}  // namespace tc

struct SurrTcArgs {
    StepCommon c;
    const tc::Weights *W;
    const float *ic;    // gap currents of this step (NULL: none)
    int32_t withhold;   // test hook: CTA 0 leaves out its withhold-th commit (0: none)
};

// The cell update with learned rates: 128 cells per CTA, three tensor-core tiles (dendrite and
// axon through buffer 0, soma through buffer 1).
__global__ void __launch_bounds__(128) surrogate_tc_kernel(const SurrTcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    tc::Smem &sm = *reinterpret_cast<tc::Smem *>(smem_raw);
    const StepCommon &c = a.c;
    const int64_t i = (int64_t)blockIdx.x * tc::ROWS + threadIdx.x;
    const bool valid = i < c.n;
    tc::tc_setup(sm, a.W);   // weights, TMEM and pulses are not step data: before the dependency wait
    const PulseAhead pa = pulse_ahead(c.pulses, i, valid);
    pdl_enter();
    const int64_t t = step_index(c);
    const float *vcur = vd_cur(c);
    float *vnext = vd_next(c);
    Cell cell{};
    cell.vd = cell.vs = cell.va = -60.0f;
    cell.ca = 1.0f;
    if (valid) cell = load_cell(c.S, vcur, i);
    const float ic = valid && a.ic != nullptr ? a.ic[i] : 0.0f;
    float iapp = pulse_current(c.pulses, pa, t);
    if (c.iapp != nullptr && valid) iapp += c.iapp[i];
    const int row = threadIdx.x, hook = blockIdx.x == 0 ? a.withhold : 0;
    const float dt = c.P.dt;
    auto x0 = [&](float V) { return (V - sm.W.in_shift[0]) * sm.W.in_scale[0]; };
    constexpr uint32_t L2 = tc::idesc_bf16(tc::ROWS, tc::N2), L3 = tc::idesc_bf16(tc::ROWS, tc::N3);
    float y[tc::NOUT];
    // The new words stay in registers until every completion has been seen: nothing of a cell is
    // stored if one does not arrive (0.2 us of a step's 21.4 at 65 536 cells, k = 100).
    DendNext d{};
    float r1 = 0.0f, s1 = 0.0f, q1 = 0.0f, ms = 0.0f, vs = 0.0f, k1 = 0.0f, l1 = 0.0f, hs1 = 0.0f, ns1 = 0.0f, xs1 = 0.0f;
    uint32_t issued[2] = {0u, 0u};
    bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.wbar, 0u));   // the weights
    const float x1 = (logf(cell.ca) - sm.W.in_shift[1]) * sm.W.in_scale[1];
    tc::layer1_row(sm, 0, row, x0(cell.vd), x1);
    tc::tc_issue(sm, 0, sm.W.w2, L2, ok, issued, hook == 1);
    tc::layer1_row(sm, 1, row, x0(cell.vs), x1);
    tc::tc_issue(sm, 1, sm.W.w2, L2, ok, issued, hook == 2);
    ok = tc::tc_wait(sm, 0, 0u, ok);
    if (ok) tc::layer2_epilogue(sm, 0, tc::tc_lane(sm, 0), row);
    tc::tc_issue(sm, 0, sm.W.w3, L3, ok, issued, hook == 3);
    ok = tc::tc_wait(sm, 1, 0u, ok);
    if (ok) tc::layer2_epilogue(sm, 1, tc::tc_lane(sm, 1), row);
    tc::tc_issue(sm, 1, sm.W.w3, L3, ok, issued, hook == 4);
    // dendrite: its outputs, then the axon's layer 1 into the buffer they leave
    ok = tc::tc_wait(sm, 0, 1u, ok);
    if (ok) {
        tc::tc_outputs(sm, 0, y);
        tc::layer1_row(sm, 0, row, x0(cell.va), x1);
    }
    tc::tc_issue(sm, 0, sm.W.w2, L2, ok, issued, hook == 5);
    if (ok) {
        d = dend_step(c.P, cell, ic, iapp);
        r1 = relax(cell.r, tc::learned_rate(y, G_R), dt);
        s1 = relax(cell.s, tc::learned_rate(y, G_S), dt);
        q1 = relax(cell.q, tc::learned_rate(y, G_Q), dt);
    }
    // soma
    ok = tc::tc_wait(sm, 1, 1u, ok);
    if (ok) {
        tc::tc_outputs(sm, 1, y);
        ms = tc::learned_xinf(y, G_MS);
        vs = soma_step(c.P, cell, ms);
        k1 = relax(cell.k, tc::learned_rate(y, G_K), dt);
        l1 = relax(cell.l, tc::learned_rate(y, G_L), dt);
        hs1 = relax(cell.hs, tc::learned_rate(y, G_HS), dt);
        ns1 = relax(cell.ns, tc::learned_rate(y, G_NS), dt);
        xs1 = relax(cell.xs, tc::learned_rate(y, G_XS), dt);
    }
    // axon
    ok = tc::tc_wait(sm, 0, 0u, ok);
    if (ok) tc::layer2_epilogue(sm, 0, tc::tc_lane(sm, 0), row);
    tc::tc_issue(sm, 0, sm.W.w3, L3, ok, issued, hook == 6);
    ok = tc::tc_wait(sm, 0, 1u, ok);
    if (ok) tc::tc_outputs(sm, 0, y);
    const bool all = tc::tc_finish(sm, ok, c.status, issued);
    tc::tc_teardown(sm);
    if (!all || !valid) return;
    const float ma = tc::learned_xinf(y, G_MA), va = axon_step(c.P, cell, ma);
    vnext[i] = d.vd;
    c.S.f(F_CA)[i] = d.ca;
    c.S.f(F_ICAH)[i] = d.icah;
    c.S.f(F_IC)[i] = ic;
    c.S.f(F_R)[i] = r1;
    c.S.f(F_S)[i] = s1;
    c.S.f(F_Q)[i] = q1;
    c.S.f(F_VSOMA)[i] = vs;
    c.S.f(F_MS)[i] = ms;
    c.S.f(F_K)[i] = k1;
    c.S.f(F_L)[i] = l1;
    c.S.f(F_HS)[i] = hs1;
    c.S.f(F_NS)[i] = ns1;
    c.S.f(F_XS)[i] = xs1;
    c.S.f(F_VAXON)[i] = va;
    c.S.f(F_MA)[i] = ma;
    c.S.f(F_HA)[i] = relax(cell.ha, tc::learned_rate(y, G_HA), dt);
    c.S.f(F_XA)[i] = relax(cell.xa, tc::learned_rate(y, G_XA), dt);
    if (!(isfinite(d.vd) && isfinite(d.ca) && isfinite(vs) && isfinite(va))) atomicOr(c.status, (uint32_t)ST_NONFINITE);
    if (c.par >= 0 && (int)(t & 1) != c.par) atomicOr(c.status, (uint32_t)ST_SLOT);
    if (c.trace != nullptr && ((t + 1) % c.trace_stride) == 0) {
        const int64_t sample = (t + 1) / c.trace_stride - 1;
        c.trace[(sample % c.trace_cap) * (int64_t)c.n + i] = va;
    }
}

// Batched evaluation: out[k * 24 + o] for n (V, [Ca]) pairs, 128 per CTA.
__global__ void __launch_bounds__(128) mlp_eval_tc_kernel(const tc::Weights *Wg, int64_t n, const float *V,
                                                          const float *ca, float *out, uint32_t *status) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    tc::Smem &sm = *reinterpret_cast<tc::Smem *>(smem_raw);
    tc::tc_setup(sm, Wg);
    const int64_t k = (int64_t)blockIdx.x * tc::ROWS + threadIdx.x;
    const bool valid = k < n;
    const uint32_t lane = tc::tc_lane(sm, 0);
    uint32_t issued[2] = {0u, 0u};
    float y[tc::NOUT];
    bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.wbar, 0u));   // the weights
    const float x0 = valid ? (V[k] - sm.W.in_shift[0]) * sm.W.in_scale[0] : 0.0f;
    const float x1 = valid ? (logf(ca[k]) - sm.W.in_shift[1]) * sm.W.in_scale[1] : 0.0f;
    tc::layer1_row(sm, 0, threadIdx.x, x0, x1);
    tc::tc_issue(sm, 0, sm.W.w2, tc::idesc_bf16(tc::ROWS, tc::N2), ok, issued, false);
    ok = tc::tc_wait(sm, 0, 0u, ok);
    if (ok) tc::layer2_epilogue(sm, 0, lane, threadIdx.x);
    tc::tc_issue(sm, 0, sm.W.w3, tc::idesc_bf16(tc::ROWS, tc::N3), ok, issued, false);
    ok = tc::tc_wait(sm, 0, 1u, ok);
    if (ok) tc::tc_outputs(sm, 0, y);
    if (tc::tc_finish(sm, ok, status, issued) && valid)
#pragma unroll
        for (int o = 0; o < tc::NOUT; ++o) out[k * tc::NOUT + o] = y[o];
    tc::tc_teardown(sm);
}

// Pack a host-layout surrogate (ion_surrogate_weights, FP32, row-major [out][in]) into the
// kernels' layout: BF16 layer-2/3 weights in core-matrix order, the rest FP32.
__global__ void mlp_tc_pack_kernel(const ion_surrogate_weights *w, tc::Weights *d) {
    for (int i = threadIdx.x; i < tc::N2 * tc::KH; i += blockDim.x) {
        const int r = i / tc::KH, k = i % tc::KH;
        d->w2[tc::core_off(r, k / 8) / 2 + (k % 8)] = __float2bfloat16_rn(w->w2[r * tc::KH + k]);
    }
    for (int i = threadIdx.x; i < tc::N3 * tc::KH; i += blockDim.x) {
        const int r = i / tc::KH, k = i % tc::KH;
        d->w3[tc::core_off(r, k / 8) / 2 + (k % 8)] = __float2bfloat16_rn(r < tc::NOUT ? w->w3[r * tc::KH + k] : 0.0f);
    }
    for (int i = threadIdx.x; i < 2 * tc::KH; i += blockDim.x) d->w1[i] = w->w1[i];
    for (int i = threadIdx.x; i < tc::KH; i += blockDim.x) {
        d->b1[i] = w->b1[i];
        d->b2[i] = w->b2[i];
    }
    for (int i = threadIdx.x; i < tc::N3; i += blockDim.x) {
        const bool real = i < tc::NOUT;
        d->b3[i] = real ? w->b3[i] : 0.0f;
        d->out_shift[i] = real ? w->out_shift[i] : 0.0f;
        d->out_scale[i] = real ? w->out_scale[i] : 0.0f;
    }
    if (threadIdx.x < 2) {
        d->in_shift[threadIdx.x] = w->in_shift[threadIdx.x];
        d->in_scale[threadIdx.x] = w->in_scale[threadIdx.x];
    }
}

// Shared memory requested per CTA: at least 56 KB, so that at most four CTAs share an SM
// and their TMEM allocations (128 of the SM's 512 columns each) never have to wait.
static constexpr size_t kTcSmem = sizeof(tc::Smem) > 56 * 1024 ? sizeof(tc::Smem) : 56 * 1024;
size_t surrogate_tc_smem() { return kTcSmem; }
size_t surrogate_tc_weights_bytes() { return sizeof(tc::Weights); }

cudaError_t surrogate_tc_prepare() {
    cudaError_t e = cudaFuncSetAttribute(surrogate_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_eval_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
    return e;
}

cudaError_t surrogate_tc_pack(const ion_surrogate_weights *d_w, void *d_out, cudaStream_t st) {
    mlp_tc_pack_kernel<<<1, 256, 0, st>>>(d_w, static_cast<tc::Weights *>(d_out));
    return cudaGetLastError();
}

cudaError_t launch_surrogate_tc(const StepCommon &c, const void *W, const float *ic, int withhold, cudaStream_t st) {
    SurrTcArgs a{c, static_cast<const tc::Weights *>(W), ic, withhold};
    return launch_k(surrogate_tc_kernel, dim3((unsigned)((c.n + tc::ROWS - 1) / tc::ROWS)), dim3(tc::ROWS), kTcSmem,
                    st, c.pdl != 0, a);
}

cudaError_t launch_mlp_eval_tc(const void *W, int64_t n, const float *V, const float *ca, float *out,
                               uint32_t *status, cudaStream_t st) {
    mlp_eval_tc_kernel<<<(unsigned)((n + tc::ROWS - 1) / tc::ROWS), tc::ROWS, kTcSmem, st>>>(
        static_cast<const tc::Weights *>(W), n, V, ca, out, status);
    return cudaGetLastError();
}

}  // namespace ion
