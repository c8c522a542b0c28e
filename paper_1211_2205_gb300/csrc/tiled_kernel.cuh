// Tiled half-step pass for the 2D real P_N system in FP32 (sm_103a).
//
// One CTA owns a TX x TY tile of point indices, shared by the four staggered
// grids (section 4.1); each consumer thread owns RB rows of a pair of points
// (x, x + 1).  A pass updates the components of one parity (odd l: grids G21
// (R) and G12 (I); even l: G11 (R) and G22 (I)) from the half-grid
// differences (eq. central_differences) of the other parity, weighted by
// -Mx/dx and -My/dy, followed by the exact sub-step u <- a u + b (W + q)
// (eq. sub_step_solution).
//
// Streaming by moment order.  Input components of order l' are visited in
// the paper's real order (m' = l', l'-2, ...; R then I).  Writing m = l - 2q,
// Lemma 2 says input (l', q') reaches only the outputs
//     (l'-1, q'-1), (l'-1, q'), (l'+1, q'), (l'+1, q'+1)
// of the same kind through Mx and of the other kind through My.  So while
// the inputs of order l' stream by in increasing q', register windows per
// kind hold the accumulators W of the two previous-order and the two
// next-order targets in reach:
//   * a previous-order target is complete once input q'+1 has been seen and
//     is finalised right there (its old value arrives through the ring);
//   * a next-order target has received all contributions of this order once
//     input q'+1 has been seen; its partial sum goes to a per-thread slice of
//     shared memory and comes back when order l'+2 streams by.
// Every input value is read from HBM once, every output read and written
// once; the differences of an input are formed once per point.
//
// Data movement: two producer warps walk a host-built stage list and issue
// the TMA boxes (cp.async.bulk.tensor.3d) of each stage into a ring of
// shared-memory stages guarded by mbarriers (full: transaction bytes, empty:
// one arrival per consumer warp).  A stage is one step of the consumer loop:
// slots for the R and I input of (l', q') and the R and I output finalised
// there.  Input boxes are BX x (TY+1) (one-point halo, x start aligned to 16
// bytes); output boxes TX x TY.  The I input that m' = 0 does not have is a
// box wholly outside the tensor, which TMA fills with zeros (no memory
// traffic), so the consumers need no case for it.  Boundary conditions live
// in ghost cells (section 4.2), which the lanes at the grid's edge write with
// the boundary values they copy.  Every wait is bounded: on expiry the kernel raises an
// error flag, waits (bounded) for its copies in flight, and returns.
//
// What bounds it.  At N = 39 on 1024^2 the memory: 865 us per pass, 5.97 TB/s
// of algorithmic traffic, 90 % of a plain copy's rate.  At low orders and on
// grids that L2 holds, the chain of a consumer warp's steps: its instructions,
// their latency and their fetch (two dozen steps in flight on an SM are not
// enough to hide it).  So a step is as short as it goes:
//   * it carries the differences of the previous input, not four accumulators
//     (a target's sum is completed where it is finalised, in the same order
//     of additions), so one copy of the loop body serves every step;
//   * its branches are uniform by construction (votes, redux): no
//     reconvergence code; boundary work is predicated stores behind one
//     branch;
//   * a stage's weights (each twice, as an f32x2 pair), offset and source
//     address are one record, read before the stage's barrier;
//   * a thread takes several adjacent rows of a pair where the warps are
//     enough (tiled.cu): the fixed part is shared and d_y needs one load per
//     row;
//   * both kinds run the same code (three 4-byte loads per d_x instead of a
//     template on the x shift): two copies missed the instruction cache.
// Against the kernel before (four accumulators, a branch per case, a separate
// kernel for the boundary copies, one warp issuing every box): P_13 512^2 59 ->
// 39 us per pass, P_9 1501 x 1099 150 -> 103, N = 3 at 1024^2 35 -> 19, P_39
// 1024^2 925 -> 862, the 16-instance batch 358 -> 224.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "pdl.h"

namespace starmap {
namespace tiled {

constexpr int TX = 64;                  // tile width: 32 lanes x 2 points
constexpr int VEC = 4;                  // 16 bytes of FP32: TMA x alignment
constexpr int BX = TX + VEC;            // input box width (halo + alignment)
constexpr int MAX_STAGES = 15;          // ring depth limit (the host fills the shared memory up to it)
constexpr int PRODUCER_WARPS = 2;       // one issues the input boxes, one the output boxes

// A tile of NB_ bands of RB_ rows, a consumer warp per band and output kind;
// MINB_: resident CTAs per SM the registers are limited for; DUP_: each
// weight twice in shared memory (an f32x2 pair ready to use), else once.
template <int RB_, int NB_, int MINB_, bool DUP_>
struct Shape {
    static constexpr int RB = RB_, NB = NB_, MINB = MINB_;
    static constexpr bool DUP = DUP_;
    static constexpr int TY = RB * NB;              // tile height
    static constexpr int BYI = TY + 1;              // input box height (halo)
    static constexpr int IN_BYTES = BX * BYI * 4;
    static constexpr int OUT_BYTES = TX * TY * 4;
    static constexpr int IN_SLOT = ((IN_BYTES + 127) / 128) * 128;    // slot strides in bytes
    static constexpr int OUT_SLOT = ((OUT_BYTES + 127) / 128) * 128;
    // a stage (one consumer step) holds the input R, input I, output R, output I boxes
    static constexpr int STAGE_BYTES = 2 * IN_SLOT + 2 * OUT_SLOT;
    static constexpr int CONSUMER_WARPS = 2 * NB;   // per output kind (R, I), one warp per band
    static constexpr int CONSUMERS = CONSUMER_WARPS * 32;
    static constexpr int THREADS = CONSUMERS + 32 * PRODUCER_WARPS;
    static constexpr int PART_BYTES = RB * CONSUMERS * 8;             // partial sums of one q
    static constexpr int REC_BYTES = DUP ? 80 : 48;                   // record of a stage and kind in shared memory
};
constexpr int MAXN = 63;
// Shared memory: full[MAX_STAGES], empty[MAX_STAGES], abort flag, the stages
// each producer had issued when it gave up (drain), a scratch word (warm_line); partial sums;
// tables; ring.  (A step may read one q past the partial sums: table values
// that nothing uses.)
constexpr int PART_OFF = 256;
constexpr int SCRATCH_OFF = PART_OFF - 4;
static_assert(2 * MAX_STAGES * 8 + 4 * (1 + PRODUCER_WARPS) <= SCRATCH_OFF, "the barrier area");
constexpr unsigned long long WAIT_NS = 2000000000ull;   // bounded waits: 2 s

struct OutGrid {
    float* base;        // point (0,0) of component 0
    long cstride;       // elements between components
    const float* coef;  // decay coefficients [cls][4][ny][cp]
    int nx, ny;
    int cp;             // row pitch of coefficients and sources (even, >= nx)
};

struct Params {
    CUtensorMap maps[4];        // input R, input I, output R, output I
    OutGrid out[2];             // output grids: R, I
    long pitch;
    int p[2];
    int tiles_x;
    int skew;                   // tile order (tile_column)
    int N, P;                   // moment order, pass parity (1 odd, 0 even)
    int which;                  // 0 half-step coefficients, 1 full-step
    int nclasses;               // 2 = isotropic (class 0: l = 0, 1: l >= 1), else class = l
    int nstages;
    int nring;                  // stages in the ring (2 .. MAX_STAGES)
    int top;                    // highest output order finalised: N, or N - 1 when every order-N
                                // component is frozen (a closure sets them)
    const int4* stages;         // per stage: component (in its grid) of slot 0..3, -1 if absent (an absent
                                // I input: a component outside the tensor, a box of zeros)
    const float4* rec[2];       // per output kind K, per stage: (P0 x, P0 y, Np x, Np y) of the previous
                                // input of the order, (Pm x, Pm y, N0 x, N0 y) of the stage's input (x:
                                // -Mx/dx, y: -My/dy; zero if absent), and as integers (element offset
                                // of the target completed / 32, or -1; 0; address of its source or 0)
    int* err;                   // bounded-wait failure flag
    int smem_rec_off[2], smem_stage_off, smem_ring_off;     // byte offsets in dynamic smem
    int any_src[2];             // per output kind: whether any finalised component has a source
    int many_src;               // whether half of the targets or more have one
    const float* pf_src[2];     // per output kind: the source array its finalisations read, if it
                                // has exactly one (prefetched into L2 with the decay pairs), else null
};

__host__ __device__ constexpr int nq_of(int l) { return l < 0 ? 0 : l / 2 + 1; }
__host__ __device__ constexpr bool has_imag(int l, int q) { return l - 2 * q >= 1; }

// ---------------------------------------------------------------------------
// PTX helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// The same by 32-bit shared addresses.
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}\n" : "=r"(p));
    return p != 0;
}

// Wait for a barrier phase with a time limit; on expiry raise the CTA's
// abort flag and the global error flag.
__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (global_ns() - t0 > WAIT_NS) {
            *abort_flag = 1;
            atomicExch(err, 1);
            return false;
        }
    }
    return true;
}

// Offsets of the right / upper neighbour of the staggered outputs read from
// the input grid of kind k (0 = R, 1 = I) in pass P.
__device__ __forceinline__ void input_shift(int P, int k, int px, int py, int& sx, int& sy) {
    // input grids: odd pass (P=1) R -> G11, I -> G22; even pass R -> G21, I -> G12
    const int g = P == 1 ? (k == 0 ? 0 : 3) : (k == 0 ? 1 : 2);
    const bool xnode = g & 1, ynode = g & 2;
    sx = xnode ? 1 - px : px;
    sy = ynode ? 1 - py : py;
}

// Packed pair of FP32 values (point A in the low half, point B in the high
// half) and the f32x2 arithmetic of sm_100-family parts.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_make(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_split(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 lds2(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ f2 ldg2(const float* p) { return __ldg(reinterpret_cast<const f2*>(p)); }
__device__ __forceinline__ f2 zero2() { return 0ull; }


// The source address of a finalise entry.
__device__ __forceinline__ const float* source_of(const int4& f) {
    return reinterpret_cast<const float*>(((unsigned long long)(unsigned)f.w << 32) | (unsigned)f.z);
}

// Slots of a stage: byte offsets of the R / I input boxes and the R / I output boxes.
template <class S>
__host__ __device__ constexpr int slot_off(int slot) {
    return slot < 2 ? slot * S::IN_SLOT : 2 * S::IN_SLOT + (slot - 2) * S::OUT_SLOT;
}

// The weighted differences of one q step for a pair of points: x and y hold
// the weights of the targets Pm, P0, N0, Np for d_x and d_y.  Nn starts here
// (Np is the first contribution to its target from this order).
__device__ __forceinline__ void add_targets(f2 dx, f2 dy, const f2 (&x)[4], const f2 (&y)[4], f2& Pc, f2& Pn, f2& Nc,
                                            f2& Nn) {
    Pc = f2_fma(x[0], dx, Pc);
    Pn = f2_fma(x[1], dx, Pn);
    Nc = f2_fma(x[2], dx, Nc);
    Nn = f2_fma(x[3], dx, zero2());
    Pc = f2_fma(y[0], dy, Pc);
    Pn = f2_fma(y[1], dy, Pn);
    Nc = f2_fma(y[2], dy, Nc);
    Nn = f2_fma(y[3], dy, Nn);
}

// The weights of a step (cp[0]: x, cp[1]: y), each as an f32x2 pair.
__device__ __forceinline__ void load_weights(const float4* cp, f2 (&x)[4], f2 (&y)[4]) {
    const float4 a = cp[0], b = cp[1];
    x[0] = f2_make(a.x, a.x); x[1] = f2_make(a.y, a.y); x[2] = f2_make(a.z, a.z); x[3] = f2_make(a.w, a.w);
    y[0] = f2_make(b.x, b.x); y[1] = f2_make(b.y, b.y); y[2] = f2_make(b.z, b.z); y[3] = f2_make(b.w, b.w);
}

// Shared memory by 32-bit address (the consumers' inner loop).
template <int OFF>
__device__ __forceinline__ f2 ld8(uint32_t a) {
    f2 v;
    asm volatile("ld.shared.b64 %0, [%1+%2];" : "=l"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float ld4(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ void ld16(uint32_t a, f2& x, f2& y) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(x), "=l"(y) : "r"(a), "n"(OFF));
}
__device__ __forceinline__ int4 ld16i(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
template <int OFF>
__device__ __forceinline__ void st8(uint32_t a, f2 v) {
    asm volatile("st.shared.b64 [%0+%1], %2;" ::"r"(a), "n"(OFF), "l"(v));
}
// The four weights of one half of a stage record, as f32x2 pairs.
template <bool DUP, int HALF>
__device__ __forceinline__ void ld_weights(uint32_t a, f2 (&w)[4]) {
    if constexpr (DUP) {
        ld16<32 * HALF>(a, w[0], w[1]);
        ld16<32 * HALF + 16>(a, w[2], w[3]);
    } else {
        f2 p[2];
        ld16<16 * HALF>(a, p[0], p[1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float u, v;
            f2_split(p[i], u, v);
            w[2 * i] = f2_make(u, u);
            w[2 * i + 1] = f2_make(v, v);
        }
    }
}

// A value every lane holds, as the compiler can see (the batch reads its
// parameters from shared memory): branches on it need no reconvergence.
__device__ __forceinline__ int uni(int v) { return __reduce_max_sync(0xffffffffu, v); }

// wait_bounded for a whole warp: all lanes take part and leave together.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err) {
    auto test = [&]() -> bool {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        return __all_sync(0xffffffffu, ok != 0);
    };
    if (test()) return true;
    const unsigned long long t0 = global_ns();
    while (!test()) {
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        if (__any_sync(0xffffffffu, global_ns() - t0 > WAIT_NS)) {
            *abort_flag = 1;
            atomicExch(err, 1);
            return false;
        }
    }
    return true;
}
// One arrival of the warp (all lanes' reads before it).
__device__ __forceinline__ void arrive_warp(uint32_t bar, int lane) {
    __syncwarp();
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}\n" ::"r"(bar),
                 "r"(lane)
                 : "memory");
}

// Global stores of the lanes with i < n (predicated: as branches they cost
// more than the stores).
template <int I>
__device__ __forceinline__ void st8_if(float* p, f2 v, int n) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\t@p st.global.b64 [%0], %1;\n\t}\n" ::"l"(p), "l"(v), "r"(n), "n"(I));
}
template <int I>
__device__ __forceinline__ void st4_if(float* p, float v, int n) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\t@p st.global.f32 [%0], %1;\n\t}\n" ::"l"(p), "f"(v), "r"(n), "n"(I));
}

// v, with its origin hidden: what is computed from it is not hoisted out of
// the loops, where it would hold registers.
__device__ __forceinline__ int here(int v) { asm volatile("" : "+r"(v)); return v; }
__device__ __forceinline__ long here(long v) { asm volatile("" : "+l"(v)); return v; }

// f(row) for the rows of a thread, the row a compile-time constant (an immediate offset).
template <class F, int... I>
__device__ __forceinline__ void each_row(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}

// Column of tile `tile` in row `row`: in raster order, or (skew) each row
// starting one column further than the row before, so that a CTA's strided
// run of tiles does not stay in one column (the edge columns cost more).
__device__ __forceinline__ int tile_column(const Params& prm, int tile, int row) {
    int c = tile - row * prm.tiles_x;
    if (prm.skew) c = (c + row) % prm.tiles_x;
    return c;
}

// Consumer warps of one CTA: the tiles t0, t0 + tstride, ... (ntl of them).
// Warp w handles rows RB band .. RB band + RB - 1 (band = w % NB) of the tile
// for the targets of kind K = w / NB (0: R outputs, 1: I outputs), lane l the
// points A = x0 + 2 l and B = A + 1.  Targets of kind K take d_x of the
// inputs of kind K (slot K, through Mx) and d_y of the other kind's (slot
// 1 - K, through My).  sxK, syK: shifts of the right / upper operand of kind
// K's input (input_shift).
//
// Step q of order lp has the differences of input (lp, q) at hand and, in
// registers, those of input (lp, q - 1); it completes the previous-order
// target (lp - 1, q - 1) (partial sum, then input q - 1, then input q) and
// what order lp adds to the next-order target (lp + 1, q).
template <class S>
__device__ __forceinline__ void consume(const Params& prm, int K, int sxK, int syK, int t0, int tstride, int ntl) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int RB = S::RB;
    constexpr auto ROWS = std::make_integer_sequence<int, RB>{};
    constexpr int PI = S::CONSUMERS * 8;                // bytes between a thread's partial sums of two rows
    constexpr int PQ = RB * PI;                         // and of two q
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 2 * MAX_STAGES * 8);
    const uint32_t base = smem_u32(smem);
    const uint32_t ring = base + prm.smem_ring_off;
    const int NR = uni(prm.nring);
    const int tid = threadIdx.x;
    const int lane = tid & 31, band = (tid >> 5) % S::NB;
    const uint32_t part = base + PART_OFF + 8 * tid;    // entry (q, i) at part + q PQ + i PI
    // byte offsets inside a stage, row i of the thread at + 4 i BX (+ 4 i TX):
    // the aligned pair and the single value of d_x, the lower operands of
    // d_y (both boxes start one row below the first row that is read from
    // below, so d_y always takes box rows r and r + 1), the old value
    const int ox = slot_off<S>(K) + 4 * ((RB * band + (syK == 0 ? 1 : 0)) * BX + 2 * lane + (sxK == 0 ? VEC - 1 : 0));
    const int oy = slot_off<S>(1 - K) + 4 * (RB * band * BX + 2 * lane + (sxK == 0 ? 0 : VEC));
    const int ou = slot_off<S>(2 + K) + 4 * (RB * band * TX + 2 * lane);
    const OutGrid& G = prm.out[K];
    const int N = uni(prm.N), first = 1 - uni(prm.P);   // first input order: even l' for the odd pass
    const int top = uni(prm.top), ncls = uni(prm.nclasses);
    const bool any_src = uni(prm.any_src[K]) != 0;
    // whether an axis of the output grid keeps copies (section 4.2: every axis but an extrapolation axis
    // of nodes); periodic -1 <- n - 1, n <- 0; extrapolation -1 <- 0, n <- n - 1; corners by both rules
    const int px = prm.p[0], py = prm.p[1];
    const bool hx = px || (prm.P == 1) == (K == 1), hy = py || K == 0;
    int r = 0;                                          // ring slot and phase of the next stage
    uint32_t ph = 0;
    int done = 0;                                       // stages consumed
    for (int tl = 0; tl < ntl; ++tl) {
        const int tile = t0 + tl * tstride;
        const int trow = tile / prm.tiles_x;
        const int gx = tile_column(prm, tile, trow) * TX + 2 * lane;
        const int gy = trow * S::TY + RB * band;
        // rows in which the lane stores both points, or A alone (the last column of an odd width)
        const int nrow = max(0, min(RB, G.ny - gy));
        const int both = gx + 1 < G.nx ? nrow : 0, lone = gx + 1 == G.nx ? nrow : 0;
        // ghost-cell copies of the warp's points: along x the lane's copy of A (or B: cb) lands xo
        // elements from A in xrow rows (xo2: a second one, in a grid narrower than three); along y row il
        // of the warp is copied to row -1 and row ir to row ny (-1: neither)
        int xo = 0, xo2 = 0;
        bool cb = false;
        if (hx) {
            const int xl = px ? G.nx - 1 : 0, xr = px ? 0 : G.nx - 1;
            const bool l = xl == gx || xl == gx + 1, r = xr == gx || xr == gx + 1;
            xo = l ? -1 - gx : r ? G.nx - gx : 0;
            cb = (l ? xl : xr) != gx;
            if (l && r) xo2 = G.nx - gx;
        }
        const int xrow = xo != 0 ? nrow : 0;
        int il = -1, ir = -1;
        if (hy) {
            il = (py ? G.ny - 1 : 0) - gy;
            ir = (py ? 0 : G.ny - 1) - gy;
            if (il < 0 || il >= RB) il = -1;
            if (ir < 0 || ir >= RB) ir = -1;
        }
        il = uni(il);
        ir = uni(ir);
        const bool tiny = __any_sync(0xffffffffu, xo2 != 0);
        const bool edge = __any_sync(0xffffffffu, lone != 0 || xrow != 0 || tiny || il >= 0 || ir >= 0);
        float* const dst0 = G.base + (long)(gy + 1) * prm.pitch + gx;   // point A of row 0 in component 0
        // coefficient / source index of point A of row 0, and the last row's offset in rows; points
        // outside the grid read a valid place and are never stored
        const long c0 = (long)min(gy, G.ny - 1) * G.cp + min(gx, G.cp - 2);
        const int cmax = max(G.ny - 1 - gy, 0);
        uint32_t rec = base + prm.smem_rec_off[K];      // the stage's record
        int cls = -1;
        f2 aL[RB], bL[RB];                              // decay pairs (a, b) of the outputs being finalised
        f2 W[RB];                                       // sum of the target being completed
        // The stage's barrier and its release, which follows the stores of what the stage's values went into:
        // a load from the ring that is merely issued can be passed by the arrival, and the next box (async
        // proxy) then lands before it reads.  (Released at once, one half-warp of one row in 10^6 stages read
        // the next round's values on 1501 x 1099 cells; a proxy fence instead costs 3 % of a P_13 pass.)
        auto wait = [&]() -> bool { return wait_warp(base + 8 * r, ph, abort_flag, prm.err); };
        auto release = [&]() {
            arrive_warp(base + 8 * (MAX_STAGES + r), lane);
            ++done;
            if (++r == NR) { r = 0; ph ^= 1u; }
        };
        // differences of the stage's input
        auto differences = [&](uint32_t t, f2 (&dx)[RB], f2 (&dy)[RB]) {
            const uint32_t tx = t + ox, ty = t + oy;
            f2 lo = ld8<0>(ty);
            each_row([&](auto i) {
                const f2 hi = ld8<4 * (i + 1) * BX>(ty);
                dy[i] = f2_sub(hi, lo);
                lo = hi;
                const float a = ld4<4 * i * BX>(tx), b = ld4<4 * i * BX + 4>(tx), c = ld4<4 * i * BX + 8>(tx);
                dx[i] = f2_make(b - a, c - b);
            }, ROWS);
        };
        // row `row` of v to the ghost row whose point A is at g, with its own copies along x
        auto copy_row = [&](f2 c, const f2 (&v)[RB], int row, float* g) {
            each_row([&](auto i) { if (row == i) c = v[i]; }, ROWS);
            float c0, c1;
            f2_split(c, c0, c1);
            st8_if<0>(g, c, both);
            st4_if<0>(g, c0, lone);
            st4_if<0>(g + xo, cb ? c1 : c0, xrow);
            if (tiny && xo2 != 0) g[xo2] = (px ? 0 : G.nx - 1) == gx ? c0 : c1;
        };
        // u <- a u + b (W + q) of the target whose sum is W; f: its offset and source
        auto finalise = [&](const int4& f, const f2 (&u)[RB]) {
            if (any_src) {
                if (__any_sync(0xffffffffu, (f.z | f.w) != 0)) {
                    const float* sp = source_of(f) + c0;
                    const int cm = here(cmax);
#pragma unroll
                    for (int i = 0; i < RB; ++i) W[i] = f2_add(W[i], ldg2(sp + min(i, cm) * G.cp));
                }
            }
            float* dst = dst0 + 32 * (long)f.x;         // 64-bit: states beyond 2^31 values
            const long pitch = here(prm.pitch);
            f2 v[RB];
#pragma unroll
            for (int i = 0; i < RB; ++i) v[i] = f2_fma(aL[i], u[i], f2_mul(bL[i], W[i]));
            float* d = dst;
            each_row([&](auto i) { st8_if<i>(d, v[i], both); d += pitch; }, ROWS);
            if (edge) {
                d = dst;
                each_row([&](auto i) {
                    float v0, v1;
                    f2_split(v[i], v0, v1);
                    st4_if<i>(d, v0, lone);
                    st4_if<i>(d + xo, cb ? v1 : v0, xrow);
                    d += pitch;
                }, ROWS);
                if (tiny && xo2 != 0) {
                    d = dst;
                    for (int i = 0; i < RB; ++i, d += pitch) {
                        float v0, v1;
                        f2_split(v[i], v0, v1);
                        if (i < nrow) d[xo2] = (px ? 0 : G.nx - 1) == gx ? v0 : v1;
                    }
                }
                if (il >= 0) copy_row(v[0], v, il, dst - (long)(gy + 1) * pitch);
                if (ir >= 0) copy_row(v[0], v, ir, dst + (long)(G.ny - gy) * pitch);
            }
        };
        // a step with an input and a target to complete: differences of the
        // previous input in, of this one out in (dx, dy)
        auto full_step = [&](uint32_t pq, f2 (&dx)[RB], f2 (&dy)[RB]) -> bool {
            f2 w[4], Nn[RB], u[RB];
            ld_weights<S::DUP, 0>(rec, w);              // P0 and Np of the previous input
#pragma unroll
            for (int i = 0; i < RB; ++i) {
                W[i] = f2_fma(w[0], dx[i], W[i]);
                Nn[i] = f2_fma(w[2], dx[i], zero2());
                W[i] = f2_fma(w[1], dy[i], W[i]);
                Nn[i] = f2_fma(w[3], dy[i], Nn[i]);
            }
            ld_weights<S::DUP, 1>(rec, w);              // Pm and N0 of this input
            const int4 f = ld16i(rec + S::REC_BYTES - 16);
            rec += S::REC_BYTES;
            if (!wait()) return false;
            const uint32_t t = ring + r * S::STAGE_BYTES;
            differences(t, dx, dy);
            each_row([&](auto i) { u[i] = ld8<4 * i * TX>(t + ou); }, ROWS);
#pragma unroll
            for (int i = 0; i < RB; ++i) {
                W[i] = f2_fma(w[0], dx[i], W[i]);
                Nn[i] = f2_fma(w[2], dx[i], Nn[i]);
                W[i] = f2_fma(w[1], dy[i], W[i]);
                Nn[i] = f2_fma(w[3], dy[i], Nn[i]);
            }
            finalise(f, u);
            each_row([&](auto i) {
                W[i] = ld8<i * PI>(pq);
                st8<i * PI>(pq, Nn[i]);
            }, ROWS);
            release();
            return true;
        };
        if (first == 1)                         // the even pass completes order 0 after order 1 alone: no partial sums yet
            each_row([&](auto i) { st8<i * PI>(part, zero2()); }, ROWS);
        // input orders, then (lp > N) the outputs of the order above the last input order
        for (int lp = first;; lp += 2) {
            const bool body = lp <= N;
            if (!body && lp - 1 > top) break;
            const int want = ncls == 2 ? min(lp - 1, 1) : lp - 1;
            if (want >= 0 && want != cls) {
                // used one step later at the earliest (or at once in the last order)
                cls = want;
                const long plane = here((long)G.cp * G.ny);
                const int cm = here(cmax);
                const float* ca = G.coef + ((long)cls * 4 + 2 * prm.which) * plane + c0;
                const float* cb = ca + plane;
#pragma unroll
                for (int i = 0; i < RB; ++i) aL[i] = ldg2(ca + min(i, cm) * G.cp);
#pragma unroll
                for (int i = 0; i < RB; ++i) bL[i] = ldg2(cb + min(i, cm) * G.cp);
            }
            uint32_t pq = part;                 // partial sums of the step
            int left;                           // steps that only complete a target
            f2 dx[RB], dy[RB];
            if (body) {
                // q = 0: no target of order lp - 1 to complete yet
                f2 w[4], Nn[RB];
                ld_weights<S::DUP, 1>(rec, w);
                rec += S::REC_BYTES;
                if (!wait()) return;
                differences(ring + r * S::STAGE_BYTES, dx, dy);
                each_row([&](auto i) {
                    Nn[i] = f2_fma(w[3], dy[i], f2_fma(w[2], dx[i], zero2()));
                    W[i] = ld8<i * PI>(pq);
                    st8<i * PI>(pq, Nn[i]);
                }, ROWS);
                release();
                for (int q = nq_of(lp) - 1; q > 0; --q) {
                    pq += PQ;
                    if (!full_step(pq, dx, dy)) return;
                }
                left = lp & 1;                  // an odd order's last target has no further input
            } else {
                left = nq_of(lp - 1);
#pragma unroll
                for (int i = 0; i < RB; ++i) dx[i] = dy[i] = zero2();
                each_row([&](auto i) { W[i] = ld8<i * PI>(pq); }, ROWS);
            }
            for (; left > 0; --left) {
                f2 w[4], Nn[RB], u[RB];
                ld_weights<S::DUP, 0>(rec, w);
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    W[i] = f2_fma(w[0], dx[i], W[i]);
                    Nn[i] = f2_fma(w[2], dx[i], zero2());
                    W[i] = f2_fma(w[1], dy[i], W[i]);
                    Nn[i] = f2_fma(w[3], dy[i], Nn[i]);
                }
                const int4 f = ld16i(rec + S::REC_BYTES - 16);
                rec += S::REC_BYTES;
                if (!wait()) return;
                const uint32_t t = ring + r * S::STAGE_BYTES;
                each_row([&](auto i) { u[i] = ld8<4 * i * TX>(t + ou); }, ROWS);
                if (__any_sync(0xffffffffu, f.x >= 0)) finalise(f, u);
                release();
                pq += PQ;
                if (body) {
                    if (lp < N) each_row([&](auto i) { st8<i * PI>(pq, Nn[i]); }, ROWS);
                } else {
                    each_row([&](auto i) { W[i] = ld8<i * PI>(pq); }, ROWS);
                }
            }
            if (!body) break;
        }
        // every tile consumes exactly the stages the producers issue for it
        if (done != (tl + 1) * prm.nstages) {
            atomicExch(prm.err, 1);
            return;
        }
    }
}

// The end of a producer warp (h: which) that gave up after arming `issued`
// stages.  The CTA must not leave, nor re-use its barriers, with copies in
// flight, and a stage's full barrier needs both producers, of which one may
// be ahead of the other by up to a ring.  So each waits for the other's count
// (-1 until it gives up too), arrives, without a box, at what the other armed
// alone, and waits for the last ring of stages, which now completes when its
// copies land.  (The stages armed by one producer are of the current round:
// it armed them after their slots had drained.)  One limit for all of it,
// which a producer that had issued everything lets run out: its copies are
// older than that then.  (A count from that one as well, stored at the end of
// every pass, changed the code of the issuing loop: the beam's pass, 102 us,
// took 1 to 2 % longer.)  The consumers' own waits end by the abort flag, or
// with what has landed, in an error either way.
__device__ __forceinline__ void drain(uint64_t* full, int NR, volatile int* issued_by, int h, int issued) {
    static_assert(PRODUCER_WARPS == 2, "one other producer");
    const unsigned long long t0 = global_ns();
    issued_by[h] = issued;
    while (issued_by[1 - h] < 0)
        if (global_ns() - t0 > WAIT_NS) return;
    const int all = max(issued, issued_by[1 - h]);
    for (int G = issued; G < all; ++G) mbar_arrive(&full[G % NR]);
    for (int G = max(0, all - NR); G < all; ++G)
        while (!mbar_try_wait(&full[G % NR], (G / NR) & 1))
            if (global_ns() - t0 > WAIT_NS) return;
}

// The 32 bytes at a into L1: a 4-byte copy to a word that nothing reads
// (prefetch.global.L1 brought half the gain).
__device__ __forceinline__ void warm_line(const float* a, uint32_t scratch) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(scratch), "l"(a) : "memory");
}

// Tiles t0, t0 + tstride, ... < tend of one pass, through one continuous
// pipeline: the producer walks a global stage index over all of them (the
// first stages of the next tile are in flight while the consumers finish
// the current one), the consumers step through the tiles in the same order.
// maps: the pass's four tensor maps (in parameter or global memory: TMA
// reads them from there); prm: everything else.  first_call: the CTA's
// first call (a later call invalidates and re-initialises the barriers; the
// caller synchronises the CTA in between).
template <class S, bool WARM>
__device__ __forceinline__ void tiled_tiles(const Params& prm, const CUtensorMap* maps, int t0, int tstride, int tend,
                                            bool first_call) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + MAX_STAGES;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + MAX_STAGES);
    const int NR = prm.nring;
    const uint32_t base = smem_u32(smem), ring = base + prm.smem_ring_off;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int ntl = t0 < tend ? (tend - t0 + tstride - 1) / tstride : 0;

    // warm the TMA descriptor cache while the barriers and tables are set up
    if (warp == S::CONSUMER_WARPS && lane < 4)
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(maps + lane)) : "memory");
    if (tid == 0) {
        for (int r = 0; r < MAX_STAGES; ++r) {      // every barrier: a batch's items differ in depth
            if (!first_call) {
                mbar_inval(&full[r]);
                mbar_inval(&empty[r]);
            }
            mbar_init(&full[r], PRODUCER_WARPS);
            mbar_init(&empty[r], S::CONSUMER_WARPS);
        }
        for (int k = 0; k <= PRODUCER_WARPS; ++k) abort_flag[k] = k == 0 ? 0 : -1;      // and the stages issued
        fence_mbar_init();
    }
    // stage the records and the stage list in shared memory
    for (int k = 0; k < 2; ++k) {
        unsigned char* rec = smem + prm.smem_rec_off[k];
        for (int i = tid; i < 3 * prm.nstages; i += S::THREADS) {
            const float4 w = __ldg(prm.rec[k] + i);
            const int stage = i / 3, part = i % 3;
            float4* d = reinterpret_cast<float4*>(rec + stage * S::REC_BYTES);
            if (!S::DUP || part == 2) {
                d[S::DUP ? 4 : part] = w;
            } else {
                d[2 * part] = make_float4(w.x, w.x, w.y, w.y);
                d[2 * part + 1] = make_float4(w.z, w.z, w.w, w.w);
            }
        }
    }
    {
        int4* st = reinterpret_cast<int4*>(smem + prm.smem_stage_off);
        for (int i = tid; i < prm.nstages; i += S::THREADS) st[i] = __ldg(prm.stages + i);
    }
    __syncthreads();
    if (first_call) {
        // everything above reads host-written data only; the state is read
        // and written below, after the previous kernel of the stream is done
        pdl_trigger();
        pdl_wait();
    }

    int sxR, syR, sxI, syI;
    input_shift(prm.P, 0, prm.p[0], prm.p[1], sxR, syR);
    input_shift(prm.P, 1, prm.p[0], prm.p[1], sxI, syI);

    if (warp < S::CONSUMER_WARPS) {
        const int K = warp / S::NB;
        const int syK = K == 0 ? syR : syI;
        // (the two kinds' inputs lie on opposite x grids: sxI = 1 - sxR)
        consume<S>(prm, K, K == 0 ? sxR : sxI, syK, t0, tstride, ntl);
        return;
    }

    // --------------------------------------------------------- producers
    // Producer warp h issues the two input boxes (h = 0) or the two output
    // boxes (h = 1) of every stage of the CTA's tiles (stage k of local tile
    // tl in ring slot r, ring round u): it waits for the slot to drain, arms
    // its share of the slot's byte count and issues the boxes.  (With one
    // warp for all four boxes a stage took about 800 cycles to issue, which
    // set the pace of every pass.)
    const int h = warp - S::CONSUMER_WARPS;
    const int2* s_comp = reinterpret_cast<const int2*>(smem + prm.smem_stage_off) + h;
    const CUtensorMap* mR = maps + 2 * h;
    const CUtensorMap* mI = maps + 2 * h + 1;
    const uint32_t box_bytes = h == 0 ? S::IN_BYTES : S::OUT_BYTES;
    const int oR = slot_off<S>(2 * h), oI = slot_off<S>(2 * h + 1);
    const int nst = prm.nstages;
    int r = 0, u = 0, issued = 0;
    bool ok = true;
    // WARM: the output warp also has the values that the consumers load one by
    // one (a source of every target, the decay pairs of every order) brought
    // into L1, a ring of stages before they are used: such a load stood in the
    // chain of steps with its whole latency.
    const uint32_t scratch = base + SCRATCH_OFF;
    // A row of 64 values at any alignment: 9 x 32 bytes, or, for the tiles of ten rows, which leave L1 little
    // room, 3 x 128 (whose other sectors then come from L2).  us per pass, none / 9 / 3: 150^2 P_39 164 / 98 to 103
    // / 114, 300^2 331 / 237 / 220, 512^2 P_9 42 / 40 / 38.  (Loads into registers a step or two ahead, by the
    // consumers: 174 to 179; prefetch.global.L1: 128.)
    constexpr int STEP = S::RB == 1 ? 8 : 32, PER = TX / STEP + 1;
    constexpr int LINES = (PER * S::TY + 31) / 32;
    for (int tl = 0; tl < ntl && ok; ++tl) {
        // box origins (tensor coordinates x' = x + VEC, row = y + 1)
        const int tile = t0 + tl * tstride;
        const int trow = tile / prm.tiles_x;
        const int x0 = tile_column(prm, tile, trow) * TX, y0 = trow * S::TY;
        const int bxR = h == 0 ? x0 + (sxR == 0 ? 0 : VEC) : x0 + VEC, byR = h == 0 ? y0 + (syR == 0 ? 0 : 1) : y0 + 1;
        const int bxI = h == 0 ? x0 + (sxI == 0 ? 0 : VEC) : x0 + VEC, byI = h == 0 ? y0 + (syI == 0 ? 0 : 1) : y0 + 1;
        int k = 0;
        int order_at = 0, next = 1 - prm.P;             // the stage at which input order `next` starts
        int line[2][LINES];                             // the lane's 32 bytes of the tile's rows from row y0 on, per kind
        if constexpr (WARM)
#pragma unroll
            for (int kind = 0; kind < 2; ++kind)
#pragma unroll
                for (int j = 0; j < LINES; ++j) {
                    const OutGrid& Gk = prm.out[kind];
                    const int e = lane + 32 * j, row = min(min(e / PER, S::TY - 1), Gk.ny - 1 - y0);
                    line[kind][j] = row * Gk.cp + min(x0 + min(STEP * (e % PER), TX - 1), Gk.cp - 1);
                }
        auto issue = [&](int kend) {
            for (; k < kend && ok; ++k) {
                const int2 c = s_comp[2 * k];
                if (u > 0 && !wait_warp(base + 8 * (MAX_STAGES + r), (u - 1) & 1, abort_flag, prm.err)) {
                    ok = false;
                    break;
                }
                const uint32_t dst = ring + r * S::STAGE_BYTES, bar = base + 8 * r;
                if (elect_one()) {
                    expect_tx(bar, ((c.x >= 0 ? 1u : 0u) + (c.y >= 0 ? 1u : 0u)) * box_bytes);
                    if (c.x >= 0) tma_box(dst + oR, mR, bxR, byR, c.x, bar);
                    if (c.y >= 0) tma_box(dst + oI, mI, bxI, byI, c.y, bar);
                }
                if constexpr (WARM) if (h == 1) {
                    auto warm = [&](const float* a, int kind) {
#pragma unroll
                        for (int j = 0; j < LINES; ++j)
                            warm_line(a + (long)y0 * prm.out[kind].cp + line[kind][j], scratch);
                    };
                    // input order `next` starts here: the decay pairs of the target order below it
                    if (k == order_at) {
                        if (next > 0 && prm.nclasses != 2 && prm.out[0].coef != nullptr && prm.out[1].coef != nullptr)
#pragma unroll
                            for (int kind = 0; kind < 2; ++kind) {
                                const long plane = (long)prm.out[kind].cp * prm.out[kind].ny;
                                const float* ca = prm.out[kind].coef + ((long)(next - 1) * 4 + 2 * prm.which) * plane;
                                warm(ca, kind);
                                warm(ca + plane, kind);
                            }
                        order_at += next <= prm.N ? nq_of(next) + (next & 1) : nst;
                        next += 2;
                    }
#pragma unroll
                    for (int kind = 0; kind < 2; ++kind) {
                        const int4 f = ld16i(base + prm.smem_rec_off[kind] + (k + 1) * S::REC_BYTES - 16);
                        if (__any_sync(0xffffffffu, (f.z | f.w) != 0)) warm(source_of(f), kind);
                    }
                }
                ++issued;
                if (++r == NR) { r = 0; ++u; }
            }
        };
        if (h == 1 && tl > 0 && prm.nclasses == 2) {
            // the decay pairs (and the source) of this tile (not the first: there
            // the consumers load them at once) into L2 while the consumers finish
            // the previous tiles; lane = (kind, class, plane a / b, half row of 32)
            issue(min(1, nst));
            const int kind = lane >> 4, c = (lane >> 3) & 1, ab = (lane >> 2) & 1, hx = lane & 1;
            const OutGrid& Gk = prm.out[kind];
            const int x = x0 + 32 * hx;
            if (x < Gk.nx) {
                const long plane = (long)Gk.cp * Gk.ny;
                // lanes with bit 1 clear: decay pairs; lanes 2 + 16 kind (+1): the kind's source
                const float* base = ((lane >> 1) & 1) == 0
                    ? (Gk.coef != nullptr ? Gk.coef + ((long)c * 4 + 2 * prm.which + ab) * plane + x : nullptr)
                    : ((lane & 12) == 0 && prm.pf_src[kind] != nullptr ? prm.pf_src[kind] + x : nullptr);
                if (base != nullptr)
                    for (int y = y0; y < y0 + S::TY && y < Gk.ny; ++y)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + (long)y * Gk.cp));
            }
            __syncwarp();
        }
        issue(nst);
    }
    if constexpr (WARM) asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok && lane == 0) drain(full, NR, abort_flag + 1, h, issued);
}

// Single-instance pass: a persistent grid; CTA b takes tiles b, b + gridDim.x,
// ... (raster order).  The CTAs then work on one contiguous band of tiles
// at any time, so the halo rows that vertically adjacent tiles share come
// from DRAM once, and each CTA's pipeline runs on across its tiles.
template <class S, bool WARM>
__global__ void __launch_bounds__(S::THREADS, S::MINB) k_tiled_pass(const __grid_constant__ Params prm,
                                                                                    int ntiles) {
    tiled_tiles<S, WARM>(prm, prm.maps, blockIdx.x, gridDim.x, ntiles, true);
}

// Batched pass: CTA b runs items[off[b]] .. items[off[b + 1] - 1], each a
// strided run of tiles of one instance, (instance, first tile, tile count,
// tile stride), streamed through one pipeline.  Instance i's
// parameters for parity P and coefficient set `which` are
// prms[(2 i + P) * 2 + which] in global memory; the CTA copies them to
// shared memory and hands TMA the tensor maps of the global copy.
template <class S>
__global__ void __launch_bounds__(S::THREADS, S::MINB) k_tiled_batch(const Params* __restrict__ prms,
                                                                                     const int4* __restrict__ items,
                                                                                     const int* __restrict__ off,
                                                                                     int P, int which) {
    __shared__ Params s_prm;
    const int begin = off[blockIdx.x], end = off[blockIdx.x + 1];
    for (int it = begin; it < end; ++it) {
        const int4 item = items[it];
        const Params* g = prms + (2 * item.x + P) * 2 + which;
        if (it != begin) __syncthreads();             // previous run done with s_prm and the barriers
        {
            const uint4* src = reinterpret_cast<const uint4*>(g);
            uint4* dst = reinterpret_cast<uint4*>(&s_prm);
            for (int i = threadIdx.x; i < (int)(sizeof(Params) / 16); i += blockDim.x) dst[i] = src[i];
        }
        __syncthreads();
        tiled_tiles<S, false>(s_prm, g->maps, item.y, item.w, item.y + (item.z - 1) * item.w + 1, it == begin);
    }
}

}  // namespace tiled
}  // namespace starmap
