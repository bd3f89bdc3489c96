// Tensor-core (tcgen05) likelihood kernel of libfg21 for sm_103a.
//
// Per channel f the reference-subtracted residual of every point is one small
// GEMM (Sec. 2.2 eq. fast_forward_model, rearranged about a per-request
// reference; see fg21_kernels.cu):
//
//   acc[p, t] = sum_k W[p, k] Bop[k, t],  k = 0..N+1
//     W[p, i]   = 2^sW expm1(-(beta_{p,i} - bbar_i) L_f)   (i < N)
//     W[p, N]   = 2^sW T21(nu_f; theta_p)                    (eq. t21model)
//     W[p, N+1] = -2^sW
//     Bop[i, t] = 2^sB wbar_{i,f} A[i,f,t],  Bop[N, t] = 2^sB,  Bop[N+1, t] = 2^sB dref[f,t]
//   so acc = -2^(sW+sB) (D - M)  and  chi2_p += sum_t acc^2 2^-2(sW+sB)   (eq. likelihood)
//
// The product runs as split precision on the tensor cores: both operands are
// split into hi + mid 16-bit values (FP16 or BF16) and three MMAs
// (hi*hi + hi*mid + mid*hi) accumulate in FP32 in tensor memory.
//
// One persistent CTA per SM walks a static list of work items (request, tile
// of 128 points, group of channels); a stage is one channel (one t-chunk) of
// the tile.  A CTA has two items in hand at once, one in each of two lanes with
// warps, rings and accumulators of their own that share nothing but the SM
// (20 warps; l = lane 0, 1):
//   warps 4l..4l+3       weight generators: warp w serves the 32 points of
//                        tensor-memory lane quadrant w%4; each thread evaluates
//                        its point's whole row of weights for the channel in
//                        registers, splits them into hi + mid and writes them
//                        straight into tensor memory (tcgen05.st), where the MMA
//                        reads its A operand;
//   warps 8+4l..8+4l+3   epilogue: tcgen05.ld of the accumulator rows of quadrant
//                        w%4; square-and-sum over t, unscale, compensated sum
//                        over channels, one partial chi2 per (point, item, half
//                        of the t-columns);
//   warp 16+l            TMA producer: cp.async.bulk.tensor loads of the
//                        channel's operand tile Bop (prepared per request in
//                        global memory);
//   warp 18+l            MMA issuer (the first is the tensor-memory owner).
// Shared memory carries only the operand tiles (the B side), so the tensor
// cores' shared-memory reads are one operand per MMA.  A lane's ring (1, 2 or 4
// stage slots) holds operand tiles in shared memory and weight blocks in tensor
// memory; its one accumulator is written, read and freed in two halves of the
// t-columns.  Barriers: `full` of a slot completes when the 4 generator warps
// have stored the weights and the TMA bytes have landed; `acc_free` of a half
// when the 4 epilogue warps have read it; `acc_done` and the slot's `done` take
// the tcgen05.commit after the first and after the second half's MMAs, the
// latter also telling the producers that the slot is free.
//
// What bounds it: instruction issue and latency in the sixteen arithmetic warps
// (FMA pipe about 54 % busy at 24 regions, 100 bins), so the stages are written
// to spend few instructions besides the arithmetic and to depend on nothing
// slow:
//  - every role runs its loops warp-uniformly, and the elected lane issues MMAs,
//    commits and copies under a predicate.  Issued from a branch that one lane
//    takes, a stage's six MMAs cost 677 cycles instead of the tensor pipe's 336;
//  - a stage is straight-line code for its number of region chunks (generators)
//    and column blocks (epilogue).  With loops over them inside the stage, the
//    epilogue alone took 1,580 cycles a stage;
//  - whole rows per warp and one item per lane, rather than two warps on halves
//    of each row, so that the waits, arrivals and sums of a stage are paid once;
//  - waits test the barrier before the suspending try_wait, which takes about
//    125 cycles even when the phase is complete.
// 16384 points, 24 regions, 301 channels, 100 bins: 97 us (prior draws) and 89 us
// (near the posterior), from 162 and 158 us with one item in hand, half rows and
// single-lane issue; 3001 points, 41 regions, 211 channels, 217 bins: 53 us from
// 71 us.
// Every wait is bounded (a few seconds of %globaltimer); on expiry the kernel
// sets a status bit, the roles stop, in-flight MMAs are drained with bounded
// waits and tensor memory is released before the CTA exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "fg21_internal.h"
#include "fg21_pdl.cuh"

namespace fg21 {

namespace {

constexpr int NUM_THREADS = 640;  // 20 warps: five share a scheduler's 16,384 registers, so 96 a thread
constexpr int LANES = 2;          // work items a CTA has in hand at once
constexpr int MAX_RING = 4;       // stage slots of a lane (the launch picks by tensor- and shared-memory room)
constexpr int FULL_ARRIVALS = 5;  // a lane's 4 generator warps + its TMA producer
constexpr int WARP_EPI = 8, WARP_TMA = 16, WARP_MMA = 18;
constexpr int EPI_NB = 4;         // accumulator blocks whose squares one set of chains sums
// TMA boxes are 64 x box_rows 16-bit values (128-byte rows); box_rows divides
// every request's tile height (a multiple of 8, at most 256)
constexpr uint64_t WAIT_LIMIT_NS = 4000000000ull;
// suspend-time hint of try_wait: a waiting thread sleeps (up to this long, or
// until the phase completes) instead of re-polling, leaving issue slots to the
// warps that compute
constexpr uint32_t TRY_WAIT_HINT_NS = 10000000u;
constexpr int WAIT_TRIES = 32;

struct __align__(8) Barriers {
    uint64_t full[LANES * MAX_RING];
    uint64_t done[LANES * MAX_RING];
    uint64_t acc_done[LANES];        // first half of the accumulator written
    uint64_t acc_free[LANES * 2];    // each half of the accumulator read
    uint64_t drain[LANES];
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
};

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// One arrival for the whole (converged) warp, made by an elected lane under a
// predicate rather than a branch.
__device__ __forceinline__ void mbar_arrive_warp(uint64_t *bar) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "@p mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n\t}" ::"r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "setp.ne.b32 e, %2, 0;\n\t"
        "@e mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
        "r"(bytes), "r"(elected)
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(TRY_WAIT_HINT_NS)
        : "memory");
    return ok != 0;
}
// Up to WAIT_TRIES tries: a waiting warp spends three instructions per try, and
// looks at the timer and the abort flag only between such runs.
__device__ __forceinline__ bool mbar_try_waits(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 n;\n\t"
        "mov.u32 n, 0;\n\t"
        "FG21_TRY:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "@p bra FG21_DONE;\n\t"
        "add.u32 n, n, 1;\n\t"
        "setp.lt.u32 q, n, %4;\n\t"
        "@q bra FG21_TRY;\n\t"
        "FG21_DONE:\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(TRY_WAIT_HINT_NS), "n"(WAIT_TRIES)
        : "memory");
    return ok != 0;
}
// Non-blocking test of a phase.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait of a converged warp: true when the phase completed; false on
// timeout or abort.  Votes make the outcome the same in every lane (and the
// branches on it warp-uniform).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, Barriers *S, unsigned *status,
                                          unsigned code, uint64_t limit_ns = WAIT_LIMIT_NS) {
    // (a try_wait takes about 125 cycles even on a phase that is complete)
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    if (__all_sync(0xffffffffu, mbar_try_waits(bar, parity))) return true;
    const uint64_t t0 = globaltimer();
    while (true) {
        if (__all_sync(0xffffffffu, mbar_try_waits(bar, parity))) return true;
        if (__any_sync(0xffffffffu, S->abort_flag != 0)) return false;
        if (__any_sync(0xffffffffu, globaltimer() - t0 > limit_ns)) {
            atomicOr(status, code);
            S->abort_flag = 1;
            return false;
        }
    }
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar,
                                            uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar)), "r"(elected)
        : "memory");
}
// Shared-memory matrix descriptor, K-major, no swizzle: core matrices of 8 rows
// x 16 bytes; lbo = byte distance between the two 8-element K chunks of an MMA
// step, sbo = byte distance between consecutive 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version of tcgen05
    return d;                 // base offset 0, relative LBO, swizzle none
}
// Instruction descriptor of kind::f16: D = F32, A = B = F16 (0) or BF16 (1),
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__device__ __forceinline__ uint32_t instr_desc(int M, int N, bool bf16) {
    const uint32_t fmt = bf16 ? 1u : 0u;
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// True in one lane of the (converged) warp.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(e));
    return e;
}
// D (+)= A B with A in tensor memory (128 lanes = rows, K packed two 16-bit
// values per 32-bit column) and B in shared memory.  Run by the whole converged
// warp and issued by its elected lane under a predicate: from a branch that only
// one lane takes, each tcgen05.mma costs about 107 cycles to issue (677 cycles
// for a stage's six, whatever N); issued this way the six take the 336 cycles
// the tensor pipe needs for them at N = 112 (105 at N = 16, 192 at N = 64), with
// the other warps' FMAs and tensor-memory traffic running or not.
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                           uint32_t accum, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(accum), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "setp.ne.b32 e, %1, 0;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)),
        "r"(elected)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {"
                 "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
                 "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr));
}
// Waits for this thread's tensor-memory loads.
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// This thread's lane, N consecutive 32-bit columns from taddr.
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3])
                 : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 2^e for integer e in the normal range (exact; the scale exponents here are
// clamped to +-40 each, so their sums stay within +-80).
__device__ __forceinline__ float exp2i(int e) {
    return __int_as_float((min(max(e, -126), 127) + 127) << 23);
}
__device__ __forceinline__ void kahan_add_dev(float &s, float &c, float x) {
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// ---------------------------------------------------------- work items
// A value that is the same in every lane of the (converged) warp, told to the
// compiler as such: loop bounds and slots made of it stay in uniform registers
// and its branches are warp-uniform.
__device__ __forceinline__ int uni(int v) { return __shfl_sync(0xffffffffu, v, 0); }

struct Item {
    int req, tile, g, f0, f1;
};
__device__ __forceinline__ int find_req(const ReqDesc *__restrict__ reqs, int n, int64_t item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (uni(reqs[mid].item_begin <= item)) lo = mid; else hi = mid - 1;
    }
    return lo;
}
// Called by a whole converged warp.
__device__ __forceinline__ Item decode_item(const ReqDesc *__restrict__ reqs, int n, int64_t item) {
    Item it;
    it.req = find_req(reqs, n, item);
    const ReqDesc &r = reqs[it.req];
    const int64_t lid = item - r.item_begin;
    const int tile = (lid >> 32) == 0 ? (int)((uint32_t)lid / (uint32_t)r.G) : (int)(lid / r.G);
    it.tile = uni(tile);
    it.g = uni((int)(lid - (int64_t)tile * r.G));
    const int f0 = it.g * r.ch_per_group;
    it.f0 = uni(f0);
    it.f1 = uni(min(r.F, f0 + r.ch_per_group));
    return it;
}

// ----------------------------------------------------- weight generation
// Packed FP32 pairs (fma/mul/sub .f32x2): one instruction for two lanes' worth
// of the Horner chains and splits.
__device__ __forceinline__ uint64_t pk2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// expm1 by its Taylor series on y = x / 2^s (|y| <= 0.55) and s squarings
// (1 + e)^2 - 1 = e (e + 2):  with y = d * nL / 2^s,
//   expm1(y) = sum_{j=1..D} e_j d^j,   e_j = (nL / 2^s)^j / j!,
// evaluated by Horner's rule in d (the per-point deviation) with the channel's
// coefficients e_j (2^sW folded into them when s = 0), on two arguments at
// once.  Relative truncation error |y|^D / (D+1)!: D = 3 for |y| <= 0.01,
// 5 for |y| <= 0.1, 8 for |y| <= 0.55; each squaring adds about two roundings.
// LO: the deviation is d + dlo (dlo2, its part below FP32); the last Horner
// step adds e_1 dlo, the first-order effect of dlo (its next term is about
// |y| times smaller and below FP32 resolution).
template <int D, int CH, bool LO>
__device__ __forceinline__ void em1_series2(uint64_t (&w)[CH], const uint64_t *d2, const uint64_t *e2,
                                            const uint64_t *dlo2) {
#pragma unroll
    for (int i = 0; i < CH; ++i) w[i] = fma2(e2[D], d2[i], e2[D - 1]);
#pragma unroll
    for (int j = D - 2; j >= 1; --j)
#pragma unroll
        for (int i = 0; i < CH; ++i) w[i] = fma2(w[i], d2[i], e2[j]);
#pragma unroll
    for (int i = 0; i < CH; ++i) w[i] = LO ? fma2(w[i], d2[i], mul2(e2[1], dlo2[i])) : mul2(w[i], d2[i]);
}

template <bool BF16>
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    if (BF16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    } else {
        __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}
// split a pair into hi (rounded) and mid (rounded remainder); the remainder
// a - hi by one mixed-precision FMA per value, exact
template <bool BF16>
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &mid) {
    hi = pack2<BF16>(a, b);
    float ra, rb;
    if (BF16)
        asm("{\n\t.reg .b16 l, h, m;\n\tmov.b32 {l, h}, %2;\n\tmov.b16 m, 0xBF80;\n\t"
            "fma.rn.f32.bf16 %0, l, m, %3;\n\tfma.rn.f32.bf16 %1, h, m, %4;\n\t}"
            : "=f"(ra), "=f"(rb)
            : "r"(hi), "f"(a), "f"(b));
    else
        asm("{\n\t.reg .b16 l, h, m;\n\tmov.b32 {l, h}, %2;\n\tmov.b16 m, 0xBC00;\n\t"
            "fma.rn.f32.f16 %0, l, m, %3;\n\tfma.rn.f32.f16 %1, h, m, %4;\n\t}"
            : "=f"(ra), "=f"(rb)
            : "r"(hi), "f"(a), "f"(b));
    mid = pack2<BF16>(ra, rb);
}

struct Params {
    const ReqDesc *reqs;
    int n_reqs;
    int64_t n_items;
    int b_stage_bytes;     // bytes of one operand-tile stage
    int acc_cols;          // tensor-memory columns of a lane's accumulator
    int half_col;          // ... and the first of its second half: the same for every request of a launch, so
                           // that the halves of two items with other column counts never overlap
    int ring_log2;         // a lane's stage slots (operand tile, weight block, barriers): 1, 2 or 4
    uint32_t tmem_cols;    // allocated tensor-memory columns
    unsigned *status;
    float *resid;          // validation mode: residuals [P][F][T] of request 0, else null
    int box_rows;          // rows per TMA box
};

// Slots of a lane's stage k: both rings are powers of two, so a role keeps one
// counter and masks it (phase parity flips each lap).
__device__ __forceinline__ uint32_t slot_of(uint32_t k, int ring_log2) { return k & ((1u << ring_log2) - 1u); }
__device__ __forceinline__ uint32_t phase_of(uint32_t k, int ring_log2) { return (k >> ring_log2) & 1u; }

// A CTA's items: lane l takes items blockIdx.x + gridDim.x (l + LANES j), j = 0, 1, ..
__device__ __forceinline__ int64_t first_item(int lane_id) { return blockIdx.x + (int64_t)gridDim.x * lane_id; }
__device__ __forceinline__ int64_t item_step() { return (int64_t)gridDim.x * LANES; }

// ------------------------------------------------------------ generators
// The weights of one item's stages by one warp (32 points).
// Per stage: wait until the weight slot is free (the MMAs of stage - ring are
// done), evaluate the series (the Horner chains of up to 8 region pairs advance
// together), split and store to tensor memory (hi at columns 0 .. Kr/2-1 of the
// slot's weight block, mid after them; one 32-bit column per pair, the lower K
// index in the low half), then one arrival on full[slot].  The last pair of the
// row is (trough, -1); pairs between the regions and it are zeros.  Returns
// false on a wait timeout.
//
// KR, NEV: the request's K and its chunks of 4 pairs that hold regions, ceil(N /
// 8), fixed at compile time so that a stage is straight-line code (a stage in a
// loop over chunks spends more issue slots on control than on the series); KR =
// 0 takes both at run time, for the forms that are not worth their own code.
// ALPHA (amplitude regions): the series runs on y = d nL + g with g = ln(alpha
// / abar) of each component; the coefficients 2^(-s j) / j! are then the same
// for every channel.  DF: the series degree (3, 5, 8, or 9: degree 8 of an
// argument halved s >= 1 times, and as many squarings).  With the short series
// (D = 3: a batch spread below ~0.007 in beta, as near a posterior) the
// deviations' low parts enter the weights.
template <int KP, bool BF16, int KR, int NEV, bool ALPHA, int DF>
__device__ __forceinline__ bool gen_item(const Params &prm, Barriers *S, uint32_t &stage, uint32_t slot0, const ReqDesc &r, const Item &it,
                                         SeriesPlan sp, uint32_t w_lane, int m) {
    constexpr bool FIXED = KR > 0;
    constexpr int UNITS = (FIXED ? KR : KP) / 16;          // K steps of the row: 8 pairs each
    constexpr int NP = FIXED ? NEV * 4 : KP / 2;           // pairs that may hold regions
    constexpr bool LO = DF == 3 && !ALPHA;
    constexpr int DEG = DF == 9 ? 8 : DF;
    constexpr bool X2 = LO || ALPHA;                       // a second operand per pair: the low part, or g
    constexpr bool X2_REGS = X2 && KP <= 32;               // ... kept in registers
    const int Kr = FIXED ? KR : uni(r.Kp), nch = uni(r.n_tchunks);
    const int nev = FIXED ? NEV : uni((r.N + 7) / 8);
    const float *pts = r.pts32 + (size_t)it.tile * r.pts_rows * 128 + m;
    uint64_t d2[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const bool in = 2 * i < Kr - 2;
        d2[i] = pk2(in ? pts[(size_t)(2 * i) * 128] : 0.0f, in ? pts[(size_t)(2 * i + 1) * 128] : 0.0f);
    }
    // pair-interleaved rows after the point operands: the components' g, or (no
    // amplitude regions) the deviations' low parts
    const float2 *pair2 = reinterpret_cast<const float2 *>(pts - m + (size_t)(Kr + 4) * 128) + m;
    uint64_t x2[X2_REGS ? NP : 1];
    if (X2_REGS) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 v = 2 * i < Kr ? __ldg(pair2 + (size_t)i * 128) : make_float2(0.0f, 0.0f);
            x2[i] = pk2(v.x, v.y);
        }
    }
    const float sW = exp2i(*r.scaleW);
    const float a21 = sW * pts[(size_t)(Kr - 2) * 128], nu21 = pts[(size_t)(Kr - 1) * 128];
    const float inv2s2 = pts[(size_t)Kr * 128];
    const float *nup = r.nu32;
    const float *nLp = r.nL32;
    const unsigned long long *coef = r.coef2;
    uint64_t e2[DEG + 1];
    e2[0] = 0;
    if (ALPHA) {
        const float ys = exp2i(-sp.s);
        float pw = sp.s ? 1.0f : sW, fact = 1.0f;
#pragma unroll
        for (int j = 1; j <= DEG; ++j) {
            pw *= ys;
            fact *= (float)j;
            const float e = pw * (1.0f / fact);
            e2[j] = pk2(e, e);
        }
    }
    for (int f = it.f0; f < it.f1; ++f) {
        const float dnu = __ldg(nup + f) - nu21;
        uint64_t nL2 = 0;
        if (ALPHA) {
            const float nL = __ldg(nLp + f);
            nL2 = pk2(nL, nL);
        } else {
            // the channel's coefficients e_j = (nL / 2^s)^j / j! (times 2^sW when s = 0), packed pairs
            const ulonglong2 *cf = reinterpret_cast<const ulonglong2 *>(coef + (size_t)f * 8);
#pragma unroll
            for (int j = 0; 2 * j < DEG; ++j) {
                const ulonglong2 v = __ldg(cf + j);
                e2[2 * j + 1] = v.x;
                if (2 * j + 2 <= DEG) e2[2 * j + 2] = v.y;
            }
        }
        const float s21 = a21 * __expf(-dnu * dnu * inv2s2);
        for (int c = 0; c < nch; ++c) {
        const uint32_t slot = slot0 + slot_of(stage, prm.ring_log2);
        if (!mbar_wait(&S->done[slot], phase_of(stage, prm.ring_log2) ^ 1u, S, prm.status, STATUS_TIMEOUT_GEN))
            return false;
        tc_fence_after();
        const uint32_t t_hi = w_lane + slot * KP, t_mid = t_hi + Kr / 2;
#pragma unroll
        for (int u = 0; u < UNITS; ++u) {
            if (!FIXED && 16 * u >= Kr) break;
            uint32_t H[8], M[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) H[i] = M[i] = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                constexpr int CH = 4;
                const int q = 2 * u + h;                   // chunk of 4 pairs
                if (FIXED ? q < NEV : q < nev) {
                    uint64_t w[CH], y2[CH], l2[CH];
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        y2[i] = d2[q * CH + i];
                        l2[i] = 0;
                        if (X2_REGS) {
                            l2[i] = x2[q * CH + i];
                        } else if (X2) {
                            const float2 v = __ldg(pair2 + (size_t)(q * CH + i) * 128);
                            l2[i] = pk2(v.x, v.y);
                        }
                        if (ALPHA) y2[i] = fma2(y2[i], nL2, l2[i]);
                    }
                    em1_series2<DEG, CH, LO>(w, y2, e2, l2);
                    if (DF == 9) {
                        const uint64_t two2 = pk2(2.0f, 2.0f), sW2 = pk2(sW, sW);
                        for (int k = 0; k < sp.s; ++k)
#pragma unroll
                            for (int i = 0; i < CH; ++i) w[i] = mul2(w[i], add2(w[i], two2));
#pragma unroll
                        for (int i = 0; i < CH; ++i) w[i] = mul2(w[i], sW2);
                    }
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        float a, b;
                        upk2(w[i], a, b);
                        split2<BF16>(a, b, H[h * CH + i], M[h * CH + i]);
                    }
                }
            }
            if (16 * (u + 1) == Kr) split2<BF16>(s21, -sW, H[7], M[7]);
            tmem_st8(t_hi + u * 8, H);
            tmem_st8(t_mid + u * 8, M);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        mbar_arrive_warp(&S->full[slot]);
        ++stage;
        }
    }
    return true;
}

// One item, K and chunk count at run time.
template <int KP, bool BF16, bool ALPHA>
__device__ __forceinline__ bool gen_item_any(const Params &prm, Barriers *S, uint32_t &stage, uint32_t slot0, const ReqDesc &r,
                                             const Item &it, uint32_t w_lane, int m) {
    const SeriesPlan sp{uni(r.scaleW[1]), uni(r.scaleW[2])};
    return sp.D == 3 ? gen_item<KP, BF16, 0, 0, ALPHA, 3>(prm, S, stage, slot0, r, it, sp, w_lane, m)
         : sp.D == 5 ? gen_item<KP, BF16, 0, 0, ALPHA, 5>(prm, S, stage, slot0, r, it, sp, w_lane, m)
         : sp.s == 0 ? gen_item<KP, BF16, 0, 0, ALPHA, 8>(prm, S, stage, slot0, r, it, sp, w_lane, m)
                     : gen_item<KP, BF16, 0, 0, ALPHA, 9>(prm, S, stage, slot0, r, it, sp, w_lane, m);
}

// One item by the code for its K and chunk count: NEV chunks of regions and
// the trough pair make K = 8 (NEV + 1) for an odd NEV, and 8 NEV or 8 (NEV + 2)
// for an even one.
template <int KP, bool BF16, int NEV, bool ALPHA>
__device__ __forceinline__ bool gen_item_nev(const Params &prm, Barriers *S, uint32_t &stage, uint32_t slot0,
                                             const ReqDesc &r, const Item &it, SeriesPlan sp, uint32_t w_lane, int m) {
    constexpr int K0 = NEV % 2 ? 8 * (NEV + 1) : 8 * NEV, K1 = NEV % 2 == 0 && 8 * (NEV + 2) <= KP ? 8 * (NEV + 2) : K0;
    if (K1 != K0 && uni(r.Kp == K1))
        return sp.D == 3 ? gen_item<KP, BF16, K1, NEV, ALPHA, 3>(prm, S, stage, slot0, r, it, sp, w_lane, m)
             : sp.D == 5 ? gen_item<KP, BF16, K1, NEV, ALPHA, 5>(prm, S, stage, slot0, r, it, sp, w_lane, m)
         : sp.s == 0 ? gen_item<KP, BF16, K1, NEV, ALPHA, 8>(prm, S, stage, slot0, r, it, sp, w_lane, m)
                     : gen_item<KP, BF16, K1, NEV, ALPHA, 9>(prm, S, stage, slot0, r, it, sp, w_lane, m);
    return sp.D == 3 ? gen_item<KP, BF16, K0, NEV, ALPHA, 3>(prm, S, stage, slot0, r, it, sp, w_lane, m)
         : sp.D == 5 ? gen_item<KP, BF16, K0, NEV, ALPHA, 5>(prm, S, stage, slot0, r, it, sp, w_lane, m)
     : sp.s == 0 ? gen_item<KP, BF16, K0, NEV, ALPHA, 8>(prm, S, stage, slot0, r, it, sp, w_lane, m)
                 : gen_item<KP, BF16, K0, NEV, ALPHA, 9>(prm, S, stage, slot0, r, it, sp, w_lane, m);
}
template <int KP, bool BF16, bool FIXED, bool ALPHA>
__device__ __forceinline__ bool gen_item_k(const Params &prm, Barriers *S, uint32_t &stage, uint32_t slot0,
                                           const ReqDesc &r, const Item &it, uint32_t w_lane, int m) {
    if constexpr (FIXED) {
        constexpr int MAX_NEV = KP / 8;
        const SeriesPlan sp{uni(r.scaleW[1]), uni(r.scaleW[2])};
#define FG21_NEV(n) \
    case n:         \
        if constexpr (n <= MAX_NEV) return gen_item_nev<KP, BF16, n, ALPHA>(prm, S, stage, slot0, r, it, sp, w_lane, m);
        switch (uni((r.N + 7) / 8)) {
            FG21_NEV(1)
            FG21_NEV(2)
            FG21_NEV(3)
            FG21_NEV(4)
            FG21_NEV(5)
            FG21_NEV(6)
            FG21_NEV(7)
            FG21_NEV(8)
        }
#undef FG21_NEV
    }
    return gen_item_any<KP, BF16, ALPHA>(prm, S, stage, slot0, r, it, w_lane, m);
}

// ------------------------------------------------------------- epilogue
// Sum of squares of 16-column accumulator blocks with packed FP32x2 FMAs:
// accumulator pair k sums columns 2k, 2k+8 (low half) and 2k+1, 2k+9 (high half)
// of every block, i.e. eight independent scalar chains in a fixed order,
// combined by a fixed tree after every EPI_NB blocks (half the instructions of
// scalar FMAs).
template <bool FIRST>
__device__ __forceinline__ void sq_block(uint64_t (&q)[4], const uint32_t *v) {
#pragma unroll
    for (int jj = 0; jj < 16; jj += 2) {
        const uint64_t x = pk2(__uint_as_float(v[jj]), __uint_as_float(v[jj + 1]));
        // the chains start with the bare square: x * x + 0
        q[(jj >> 1) & 3] = FIRST && jj < 8 ? mul2(x, x) : fma2(x, x, q[(jj >> 1) & 3]);
    }
}
__device__ __forceinline__ float sq_tree(uint64_t (&q)[4]) {
    float a[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        upk2(q[k], a[2 * k], a[2 * k + 1]);
    }
    return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}
// Loads NB (1 .. EPI_NB) blocks of this thread's accumulator row.
template <int NB>
__device__ __forceinline__ void acc_load(uint32_t taddr, uint32_t *v) {
    if (NB >= 2) tmem_ld32(taddr, v);
    else tmem_ld16(taddr, v);
    if (NB == 3) tmem_ld16(taddr + 32, v + 32);
    if (NB == 4) tmem_ld32(taddr + 32, v + 32);
}
template <int NB>
__device__ __forceinline__ float acc_sumsq(const uint32_t *v) {
    uint64_t q[4];
    sq_block<true>(q, v);
#pragma unroll
    for (int b = 1; b < NB; ++b) sq_block<false>(q, v + 16 * b);
    return sq_tree(q);
}
// Sum of squares of NB blocks of this thread's accumulator row, a set of chains
// for every EPI_NB of them; release() runs once they are in registers.
template <int NB, typename Release>
__device__ __forceinline__ float half_sumsq(uint32_t taddr, Release release) {
    constexpr int N0 = NB < EPI_NB ? NB : EPI_NB, N1 = NB - N0;
    float q = 0.0f;
    if constexpr (NB > 0) {
        uint32_t v[16 * EPI_NB];
        acc_load<N0>(taddr, v);
        tmem_ld_wait();
        if constexpr (N1 > 0) {
            q = acc_sumsq<N0>(v);
            acc_load<N1>(taddr + 16 * EPI_NB, v);
            tmem_ld_wait();
            release();
            q += acc_sumsq<N1>(v);
        } else {
            release();
            q = acc_sumsq<N0>(v);
        }
    } else {
        release();
    }
    return q;
}

// The epilogue of one item's stages by one warp (32 points): per stage wait for
// the MMAs, read the accumulator row, release its slot, square and sum; per
// item one compensated partial for each half of the t-blocks.
template <bool RESID, int NBLK>
__device__ __forceinline__ bool epi_item(const Params &prm, Barriers *S, uint32_t &stage, int lane_id,
                                         const ReqDesc &r, const Item &it, uint32_t acc_lane, int m) {
    const int64_t p = (int64_t)it.tile * 128 + m;
    const int sWexp = *r.scaleW;
    const int nch = uni(r.n_tchunks);
    const int *scaleB = r.scaleB + it.f0 * nch;
    const int n = (it.f1 - it.f0) * nch;
    float qs0 = 0.0f, qc0 = 0.0f, qs1 = 0.0f, qc1 = 0.0f, qf0 = 0.0f, qf1 = 0.0f;
    int sb_n = __ldg(scaleB), c = 0;
    for (int k = 0; k < n; ++k) {
        // 2^-(sW + sB), exponents within +-40 each
        const float unscale = __int_as_float((127 - sWexp - sb_n) << 23);
        sb_n = __ldg(scaleB + min(k + 1, n - 1));                  // next stage's scale, one ahead
        // the halves of the accumulator are written, read and freed one after the
        // other, so that the next stage's first half can start while this one's
        // second half is still read
        constexpr int HB = (NBLK + 1) / 2;
        float q0 = 0.0f, q1 = 0.0f;
        if (!mbar_wait(&S->acc_done[lane_id], stage & 1u, S, prm.status, STATUS_TIMEOUT_EPI)) return false;
        tc_fence_after();
        auto release = [&](int h) {
            tc_fence_before();
            __syncwarp();
            mbar_arrive_warp(&S->acc_free[2 * lane_id + h]);
        };
        if constexpr (!RESID) q0 = half_sumsq<HB>(acc_lane, [&] { release(0); });
        if (!mbar_wait(&S->done[(lane_id << prm.ring_log2) + slot_of(stage, prm.ring_log2)],
                       phase_of(stage, prm.ring_log2), S, prm.status, STATUS_TIMEOUT_EPI))
            return false;
        tc_fence_after();
        if constexpr (RESID) {
            const int Tc = r.Tc, T = r.T, F = r.F, nblk = r.Tc_pad / 16, hb = (nblk + 1) / 2;
            const int f = it.f0 + k / nch, t0 = (k % nch) * Tc, tn = min(Tc, T - t0);
            for (int b = 0; b < nblk; ++b) {
                uint32_t v[16];
                tmem_ld16(acc_lane + (b < hb ? b * 16 : prm.half_col + (b - hb) * 16), v);
                tmem_ld_wait();
                if (p < r.P)
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        const int t = b * 16 + jj;
                        if (t < tn) prm.resid[((size_t)p * F + f) * T + t0 + t] = -__uint_as_float(v[jj]) * unscale;
                    }
            }
            release(0);
            release(1);
        } else {
            q1 = half_sumsq<NBLK - HB>(acc_lane + prm.half_col, [&] { release(1); });
        }
        ++stage;
        qf0 += q0 * unscale * unscale;
        qf1 += q1 * unscale * unscale;
        if (++c == nch) {
            c = 0;
            kahan_add_dev(qs0, qc0, qf0);
            kahan_add_dev(qs1, qc1, qf1);
            qf0 = qf1 = 0.0f;
        }
    }
    if (!RESID && p < r.P)
        *reinterpret_cast<float4 *>(r.partials + (size_t)p * r.n_part + 2 * it.g) = make_float4(qs0, -qc0, qs1, -qc1);
    return true;
}
// ... by the code for its block count (1 .. 12).
template <bool RESID>
__device__ __forceinline__ bool epi_item_n(const Params &prm, Barriers *S, uint32_t &stage, int lane_id,
                                           const ReqDesc &r, const Item &it, uint32_t acc_lane, int m) {
    static_assert(TC_MAX / 16 == 12, "one case per block count");
    if constexpr (!RESID) {
#define FG21_NBLK(n) \
    case n: return epi_item<false, n>(prm, S, stage, lane_id, r, it, acc_lane, m);
        switch (uni(r.Tc_pad / 16)) {
            FG21_NBLK(2)
            FG21_NBLK(3)
            FG21_NBLK(4)
            FG21_NBLK(5)
            FG21_NBLK(6)
            FG21_NBLK(7)
            FG21_NBLK(8)
            FG21_NBLK(9)
            FG21_NBLK(10)
            FG21_NBLK(11)
            FG21_NBLK(12)
        }
#undef FG21_NBLK
    }
    return epi_item<RESID, 1>(prm, S, stage, lane_id, r, it, acc_lane, m);
}

// The stage's MMAs as straight-line code for KS k steps: the issuing thread
// shares its scheduler with ALU warps, and loop control between the MMAs
// measurably delays them.
//
// Each MMA rounds its sum toward zero in FP32 (measured on this part: the
// accumulator and the 16 products are aligned to the largest exponent E,
// truncated at 2^(E-25), added, and the sum truncated to FP32), so every MMA
// whose result is as large as the residual biases |D - M| low by about half an
// ulp.  The small correction products (hi*mid, mid*hi) of every k step go
// first, while the accumulator is still small, then the hi*hi products, last k
// step first: only the last MMA ends at the size of the residual, and the
// reduction adds back its expected half-ulp (chi2_scale).
template <int KS>
__device__ __forceinline__ void issue_mmas(uint32_t d_tmem, uint32_t w_hi, uint32_t w_mid, uint32_t b_addr,
                                           uint32_t b_lbo, uint32_t b_split, uint32_t idesc, uint32_t el) {
    // one descriptor for the stage's tile; each MMA adds its offset (16-byte
    // units) to the start-address field, which shared-memory addresses below
    // 256 KB never carry out of (building every descriptor afresh cost 3 % while one
    // lane issued from a branch of its own; the issuers now wait 60-70 % of the time)
    const uint64_t d0 = smem_desc(b_addr, b_lbo, 128);
    const uint32_t step = (2 * b_lbo) >> 4, split = b_split >> 4;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        mma_f16_ts(d_tmem, w_hi + ks * 8, d0 + split + ks * step, idesc, ks > 0 ? 1u : 0u, el);
        mma_f16_ts(d_tmem, w_mid + ks * 8, d0 + ks * step, idesc, 1u, el);
    }
#pragma unroll
    for (int ks = KS - 1; ks >= 0; --ks)
        mma_f16_ts(d_tmem, w_hi + ks * 8, d0 + ks * step, idesc, 1u, el);
}

// The MMAs and commits of every stage of one item (KS k steps).  The columns of
// a stage go in two halves (the epilogue's), each when its part of the
// accumulator has been read.
template <int KP, int KS, bool BF16>
__device__ __forceinline__ bool mma_item(const Params &prm, Barriers *S, uint32_t &stage, int lane_id, int n, int tc_pad,
                                         uint32_t tmem, uint32_t w_col0, uint32_t b_slots, uint32_t el) {
    const int n0 = (tc_pad / 16 + 1) / 2 * 16, n1 = tc_pad - n0;       // columns of the halves (n1 may be 0)
    const uint32_t idesc0 = instr_desc(128, n0, BF16), idesc1 = instr_desc(128, n1, BF16);
    const uint32_t b_lbo = (uint32_t)tc_pad * 16, b_split = 2 * KS * b_lbo;
    const uint32_t d = tmem + (uint32_t)(lane_id * prm.acc_cols), d1 = d + (uint32_t)prm.half_col;
    for (int k = 0; k < n; ++k) {
        const uint32_t slot = ((uint32_t)lane_id << prm.ring_log2) + slot_of(stage, prm.ring_log2);
        const uint32_t w_hi = tmem + w_col0 + slot * KP, b = b_slots + slot * prm.b_stage_bytes;
        if (!mbar_wait(&S->full[slot], phase_of(stage, prm.ring_log2), S, prm.status, STATUS_TIMEOUT_MMA) ||
            !mbar_wait(&S->acc_free[2 * lane_id], (stage & 1u) ^ 1u, S, prm.status, STATUS_TIMEOUT_MMA))
            return false;
        tc_fence_after();
        issue_mmas<KS>(d, w_hi, w_hi + 8 * KS, b, b_lbo, b_split, idesc0, el);
        mma_commit(&S->acc_done[lane_id], el);
        if (!mbar_wait(&S->acc_free[2 * lane_id + 1], (stage & 1u) ^ 1u, S, prm.status, STATUS_TIMEOUT_MMA))
            return false;
        tc_fence_after();
        if (n1) issue_mmas<KS>(d1, w_hi, w_hi + 8 * KS, b + n0 * 16, b_lbo, b_split, idesc1, el);
        mma_commit(&S->done[slot], el);
        ++stage;
    }
    return true;
}

// Tensor-memory columns: accumulator of lane l at l * acc_cols; weights of slot
// s after the accumulators, at s * KP (hi: Kr/2 columns, then mid: Kr/2).
// RESID: validation mode (residuals of request 0 to prm.resid instead of the
// chi2 partials); a separate instantiation keeps that code out of the
// production kernel.  ALPHA: some request of the launch has amplitude regions.
template <int KP, bool BF16, bool RESID, bool ALPHA>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    tc_loglike_kernel(const __grid_constant__ CUtensorMap tmap, const Params prm) {
    extern __shared__ __align__(1024) char smem_raw[];
    char *smem = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int ring = LANES << prm.ring_log2;
    char *b_slots = smem;                                             // [ring] x b_stage_bytes
    Barriers *S = reinterpret_cast<Barriers *>(b_slots + ring * prm.b_stage_bytes);

    // broadcast, so that the compiler knows the role branches to be warp-uniform
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ring; ++s) {
            mbar_init(&S->full[s], FULL_ARRIVALS);
            mbar_init(&S->done[s], 1);
        }
        for (int l = 0; l < LANES; ++l) {
            mbar_init(&S->acc_done[l], 1);
            mbar_init(&S->acc_free[2 * l], 4);       // the lane's epilogue warps
            mbar_init(&S->acc_free[2 * l + 1], 4);
            mbar_init(&S->drain[l], 1);
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S->tmem_base)),
                     "r"(prm.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    // the set-up above touches only this CTA's shared and tensor memory; from
    // here on the kernel reads what the operand pass wrote
    pdl_wait();
    const uint32_t tmem = __shfl_sync(0xffffffffu, S->tmem_base, 0);
    const uint32_t w_col0 = (uint32_t)(LANES * prm.acc_cols);
    const ReqDesc *reqs = prm.reqs;

    if (warp < WARP_EPI) {
        // ================================================ weight generators
        const int quad = warp & 3, lane_id = warp >> 2, m = quad * 32 + lane;
        const uint32_t w_lane = tmem + ((uint32_t)(quad * 32) << 16) + w_col0;
        const uint32_t slot0 = (uint32_t)lane_id << prm.ring_log2;
        uint32_t stage = 0;
        bool ok = true;
        for (int64_t item = first_item(lane_id); item < prm.n_items && ok; item += item_step()) {
            const Item it = decode_item(reqs, prm.n_reqs, item);
            const ReqDesc &r = reqs[it.req];
            if (ALPHA && r.Na) ok = gen_item_k<KP, BF16, !BF16 && !RESID && KP <= 32, true>(prm, S, stage, slot0, r, it, w_lane, m);
            else ok = gen_item_k<KP, BF16, !BF16 && !RESID && !ALPHA, false>(prm, S, stage, slot0, r, it, w_lane, m);
        }
    } else if (warp < WARP_TMA) {
        // ========================================================= epilogue
        const int quad = warp & 3, lane_id = (warp - WARP_EPI) >> 2, m = quad * 32 + lane;
        const uint32_t acc_lane = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(lane_id * prm.acc_cols);
        uint32_t stage = 0;
        bool ok = true;
        for (int64_t item = first_item(lane_id); item < prm.n_items && ok; item += item_step()) {
            const Item it = decode_item(reqs, prm.n_reqs, item);
            ok = epi_item_n<RESID>(prm, S, stage, lane_id, reqs[it.req], it, acc_lane, m);
        }
    } else if (warp < WARP_MMA) {
        // ====================================================== TMA producer
        // (the whole warp walks the lane's stages; its elected lane issues)
        const int lane_id = warp - WARP_TMA;
        const uint32_t el = elect_one(), slot0 = (uint32_t)lane_id << prm.ring_log2;
        bool ok = true;
        uint32_t stage = 0;
        for (int64_t item = first_item(lane_id); item < prm.n_items && ok; item += item_step()) {
            const Item it = decode_item(reqs, prm.n_reqs, item);
            const ReqDesc &r = reqs[it.req];
            const int rows = uni((int)r.tile_rows), n = (it.f1 - it.f0) * uni(r.n_tchunks);
            int row = uni((int)(r.tile_row0 + (int64_t)it.f0 * r.n_tchunks * r.tile_rows));
            for (int k = 0; k < n; ++k) {
                const uint32_t slot = slot0 + slot_of(stage, prm.ring_log2);
                // the operand slot is free once the MMAs of stage - ring are done
                if (!mbar_wait(&S->done[slot], phase_of(stage, prm.ring_log2) ^ 1u, S, prm.status,
                               STATUS_TIMEOUT_TMA)) {
                    ok = false;
                    break;
                }
                mbar_arrive_expect_tx(&S->full[slot], (uint32_t)(rows * 128), el);
                char *dst = b_slots + slot * prm.b_stage_bytes;
                for (int jr = 0; jr < rows; jr += prm.box_rows)
                    tma_load_2d(dst + jr * 128, &tmap, 0, row + jr, &S->full[slot], el);
                row += rows;
                ++stage;
            }
        }
        if (!ok) {
            // copies already issued land within microseconds; give them time
            // before the CTA (and its shared memory) goes away
            const uint64_t t0 = globaltimer();
            while (globaltimer() - t0 < 200000ull) {
            }
        }
        __syncwarp();
    } else {
        // ========================================================= MMA issuer
        // (the whole warp walks the lane's stages; its elected lane issues)
        const int lane_id = warp - WARP_MMA;
        const uint32_t el = elect_one(), b_addr = smem_u32(b_slots);
        bool ok = true;
        uint32_t stage = 0;
        for (int64_t item = first_item(lane_id); item < prm.n_items && ok; item += item_step()) {
            const Item it = decode_item(reqs, prm.n_reqs, item);
            const ReqDesc &r = reqs[it.req];
            const int n = (it.f1 - it.f0) * uni(r.n_tchunks), tc_pad = uni(r.Tc_pad), ks = uni(r.Kp / 16);
            if (KP == 16 || ks == 1)
                ok = mma_item<KP, 1, BF16>(prm, S, stage, lane_id, n, tc_pad, tmem, w_col0, b_addr, el);
            else if (KP == 32 || ks == 2)
                ok = mma_item<KP, 2, BF16>(prm, S, stage, lane_id, n, tc_pad, tmem, w_col0, b_addr, el);
            else if (ks == 3)
                ok = mma_item<KP, 3, BF16>(prm, S, stage, lane_id, n, tc_pad, tmem, w_col0, b_addr, el);
            else ok = mma_item<KP, 4, BF16>(prm, S, stage, lane_id, n, tc_pad, tmem, w_col0, b_addr, el);
        }
        // drain: every MMA issued so far completes before tensor memory is freed
        mma_commit(&S->drain[lane_id], el);
        const uint64_t t0 = globaltimer();
        while (!mbar_try_wait(&S->drain[lane_id], 0)) {
            if (globaltimer() - t0 > WAIT_LIMIT_NS) {
                atomicOr(prm.status, STATUS_TIMEOUT_DRAIN);
                break;
            }
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(prm.tmem_cols)
                     : "memory");
    }
}

// ------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
std::once_flag g_encode_once;
int g_encode_rc = FG21_OK;

size_t smem_bytes(int ring, int b_stage_bytes) {
    return 1024 + (size_t)ring * b_stage_bytes + sizeof(Barriers) + 64;
}

template <int KP, bool BF16, bool RESID, bool ALPHA>
cudaError_t launch_kpr(const CUtensorMap &map, const Params &prm, int grid, size_t sm, cudaStream_t stream) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(tc_loglike_kernel<KP, BF16, RESID, ALPHA>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    cudaError_t e = launch_dependent(tc_loglike_kernel<KP, BF16, RESID, ALPHA>, dim3(grid), dim3(NUM_THREADS), sm,
                                     stream, map, prm);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int KP, bool BF16>
cudaError_t launch_kp(const CUtensorMap &map, const Params &prm, int grid, size_t sm, bool alpha,
                      cudaStream_t stream) {
    if (prm.resid) return launch_kpr<KP, BF16, true, true>(map, prm, grid, sm, stream);
    if (alpha) return launch_kpr<KP, BF16, false, true>(map, prm, grid, sm, stream);
    return launch_kpr<KP, BF16, false, false>(map, prm, grid, sm, stream);
}

cudaError_t launch_common(const ReqDesc *d_reqs, int n_reqs, int64_t n_items, int kp_max, int tc_pad_max,
                          int precision, void *arena, int64_t arena_rows, unsigned *status, float *resid,
                          int box_rows, int num_sms, bool alpha, cudaStream_t stream) {
    if (n_items == 0) return cudaSuccess;
    if (tc_map_init() != FG21_OK) return cudaErrorNotSupported;
    CUtensorMap map;
    cuuint64_t gdim[2] = {64, (cuuint64_t)arena_rows};
    cuuint64_t gstride[1] = {128};
    if (box_rows < 8 || box_rows > 256 || box_rows % 8) return cudaErrorInvalidValue;
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estride[2] = {1, 1};
    CUresult cr = g_encode(&map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, arena, gdim, gstride, box, estride,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) return cudaErrorInvalidValue;
    const int kp = tc_launch_kp(kp_max);
    if (tc_pad_max < 16 || tc_pad_max > TC_MAX || tc_pad_max % 16) return cudaErrorInvalidValue;
    Params prm;
    prm.reqs = d_reqs;
    prm.n_reqs = n_reqs;
    prm.n_items = n_items;
    prm.b_stage_bytes = ((4 * kp_max * tc_pad_max) + 1023) & ~1023;
    prm.acc_cols = tc_pad_max;
    prm.half_col = (tc_pad_max / 16 + 1) / 2 * 16;
    // Tensor memory, for each of the two lanes: an accumulator (used in halves),
    // and 4, 2 or 1 stage slots as the rest and shared memory (operand tiles,
    // barriers) hold.
    prm.ring_log2 = 2;
    while (prm.ring_log2 > 0 && (LANES * tc_pad_max + ((LANES * kp) << prm.ring_log2) > 512 ||
                                 smem_bytes(LANES << prm.ring_log2, prm.b_stage_bytes) > 227 * 1024))
        --prm.ring_log2;
    const int ring = LANES << prm.ring_log2;
    uint32_t cols = 32;
    while (cols < (uint32_t)(LANES * tc_pad_max + ring * kp)) cols *= 2;
    if (cols > 512) return cudaErrorInvalidValue;
    prm.tmem_cols = cols;
    prm.status = status;
    prm.resid = resid;
    prm.box_rows = box_rows;
    // at least ~120 KB so that a single CTA (and its tensor memory) owns each SM
    size_t sm = smem_bytes(ring, prm.b_stage_bytes);
    if (sm < 120 * 1024) sm = 120 * 1024;
    if (sm > 227 * 1024) return cudaErrorInvalidValue;
    const int grid = (int)(n_items < num_sms ? n_items : num_sms);
    const bool bf16 = precision == FG21_PREC_BF16X3;
    if (kp == 16)
        return bf16 ? launch_kp<16, true>(map, prm, grid, sm, alpha, stream)
                    : launch_kp<16, false>(map, prm, grid, sm, alpha, stream);
    if (kp == 32)
        return bf16 ? launch_kp<32, true>(map, prm, grid, sm, alpha, stream)
                    : launch_kp<32, false>(map, prm, grid, sm, alpha, stream);
    return bf16 ? launch_kp<64, true>(map, prm, grid, sm, alpha, stream)
                : launch_kp<64, false>(map, prm, grid, sm, alpha, stream);
}

// Self-test of the bounded waits, on barriers that nothing ever arrives on.
// Warp 0 waits with the kernel's limit: it gives up first, sets
// STATUS_TIMEOUT_TMA and raises the abort flag.  Warps 1-3 wait with twice
// that limit and must come back through the abort flag, as the other roles of
// a stalled likelihood launch do, without a status bit of their own.
// elapsed[w] = nanoseconds warp w waited (all ones if its barrier completed).
__global__ void __launch_bounds__(128) wait_selftest_kernel(unsigned *status, unsigned long long *elapsed) {
    __shared__ Barriers S;
    if (threadIdx.x == 0) {
        mbar_init(&S.full[0], 1);
        mbar_init(&S.full[1], 1);
        S.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    const uint64_t t0 = globaltimer();
    const bool ok = warp == 0 ? mbar_wait(&S.full[0], 0, &S, status, STATUS_TIMEOUT_TMA)
                              : mbar_wait(&S.full[1], 0, &S, status, STATUS_TIMEOUT_GEN, 2 * WAIT_LIMIT_NS);
    const uint64_t dt = globaltimer() - t0;
    if ((threadIdx.x & 31) == 0) elapsed[warp] = ok ? ~0ull : dt;
}

// One MMA exactly as the likelihood kernel issues it (kind::f16, F16
// operands, F32 accumulator, M = 128, N = 16, K = 16, A in tensor memory, B
// from shared memory by descriptor): d = c + a b for caller-given operands, so
// that a host can check the accumulator's rounding.  a [128][16] and b
// [16 n][16 k] are F16 bit patterns, c and d [128][16] FP32.  One CTA of 128
// threads; the completion wait is bounded (status bit STATUS_TIMEOUT_MMA).
__global__ void __launch_bounds__(128, 1) mma_probe_kernel(const uint16_t *__restrict__ a,
                                                            const uint16_t *__restrict__ b,
                                                            const float *__restrict__ c, float *__restrict__ d,
                                                            unsigned *status) {
    __shared__ __align__(1024) uint16_t sb[2][16][8];      // [k chunk][n][8 values of k]
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tbase;
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tbase)),
                     "r"(32)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < 256; i += 128) sb[(i & 15) >> 3][i >> 4][i & 7] = b[i];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tbase, lane_base = tm + ((uint32_t)(warp * 32) << 16);
    uint32_t v[16];
#pragma unroll
    for (int n = 0; n < 16; ++n) v[n] = __float_as_uint(c[tid * 16 + n]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            lane_base),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = (uint32_t)a[tid * 16 + 2 * j] | ((uint32_t)a[tid * 16 + 2 * j + 1] << 16);
    tmem_st4(lane_base + 16, w);
    tmem_st4(lane_base + 20, w + 4);
    tmem_st_wait();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        const uint32_t el = elect_one();
        mma_f16_ts(tm, tm + 16, smem_desc(smem_u32(&sb[0][0][0]), 16 * 16, 128), instr_desc(128, 16, false), 1u, el);
        mma_commit(&bar, el);
    }
    const uint64_t t0 = globaltimer();
    bool ok = true;
    while (!mbar_try_wait(&bar, 0)) {
        if (globaltimer() - t0 > WAIT_LIMIT_NS) {
            if (tid == 0) atomicOr(status, STATUS_TIMEOUT_MMA);
            ok = false;
            break;
        }
    }
    tc_fence_after();
    uint32_t r[16];
    tmem_ld16(lane_base, r);
    tmem_ld_wait();
#pragma unroll
    for (int n = 0; n < 16; ++n) d[tid * 16 + n] = ok ? __uint_as_float(r[n]) : __int_as_float(0x7FC00000);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(32) : "memory");
    }
}

}  // namespace

cudaError_t launch_mma_probe(const uint16_t *a, const uint16_t *b, const float *c, float *d, unsigned *status,
                             cudaStream_t stream) {
    mma_probe_kernel<<<1, 128, 0, stream>>>(a, b, c, d, status);
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(unsigned *status, unsigned long long *elapsed, cudaStream_t stream) {
    wait_selftest_kernel<<<1, 128, 0, stream>>>(status, elapsed);
    return cudaGetLastError();
}

int tc_map_init() {
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
            cudaGetLastError();
            g_encode_rc = set_error(FG21_E_CUDA, "cuTensorMapEncodeTiled is not available");
            return;
        }
        g_encode = (EncodeTiledFn)fn;
    });
    return g_encode_rc;
}

int tc_box_rows(const int64_t *tile_rows, int n) {
    int64_t g = 0;
    for (int k = 0; k < n; ++k) {
        int64_t a = tile_rows[k], b = g;
        while (b) {
            int64_t t = a % b;
            a = b;
            b = t;
        }
        g = a;
    }
    int64_t box = 8;
    for (int64_t c = 256; c >= 8; c -= 8)
        if (g % c == 0) {
            box = c;
            break;
        }
    return (int)box;
}

cudaError_t launch_tc(const TcLaunch &L, int num_sms, cudaStream_t stream) {
    return launch_common(L.d_reqs, L.n_reqs, L.n_items, L.kp_max, L.tc_pad_max, L.precision, L.arena,
                         L.arena_rows, L.status, nullptr, L.box_rows, num_sms, L.alpha, stream);
}

cudaError_t launch_tc_residuals(const ReqDesc *h_req, const ReqDesc *d_req, int precision, float *resid,
                                cudaStream_t stream) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int sms = 1;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    char *arena = h_req->tiles - h_req->tile_row0 * 128;
    const int64_t rows = h_req->tile_row0 + (int64_t)h_req->F * h_req->n_tchunks * h_req->tile_rows;
    const int64_t items = (int64_t)h_req->n_tiles * h_req->G;
    return launch_common(d_req, 1, items, h_req->Kp, h_req->Tc_pad, precision, arena, rows, h_req->status, resid,
                         tc_box_rows(&h_req->tile_rows, 1), sms, true, stream);
}

}  // namespace fg21
