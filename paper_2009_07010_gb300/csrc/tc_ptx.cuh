// Inline-PTX building blocks for the tcgen05 kernels (sm_100 family, sm_103a):
// mbarriers with bounded waits, bulk and tensor (TMA) async copies, TMEM
// allocation and access, UMMA descriptors and issue, FP16/BF16 packing and the
// MUFU unit phasor.  Shared by k_tc.cu and k_kr.cu.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace psf {
namespace tc {

constexpr unsigned long long kTimeoutNs = 2000000000ull;

static __device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

static __device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static __device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
                 : "memory");
}

// try_wait; with a nonzero suspend-time hint the waiting thread is parked (no issue
// slots) until the phase completes or about `hint_ns` elapse.  Measured on GB300,
// parked waits beat polling for every role of this kernel (polling warps take
// issue slots from the generators).
static __device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity, uint32_t hint_ns) {
    uint32_t ok;
    if (hint_ns) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    }
    return ok != 0;
}
static constexpr uint32_t kSleepNs = 1000000u;

static __device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for the phase of `bar` with the given parity.  Returns false if the CTA is
// aborting or the wall-clock limit expired (then the abort flag and the global
// error flag are raised).
static __device__ __forceinline__ bool wait_bounded(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                             int *err, uint32_t hint_ns = kSleepNs) {
    if (mbar_try_wait(bar, parity, hint_ns)) return true;
    const unsigned long long t0 = globaltimer();
    for (;;) {
        if (mbar_try_wait(bar, parity, hint_ns)) return true;
        if (*abort_flag) return false;
        if (globaltimer() - t0 > kTimeoutNs) {
            *abort_flag = 1;
            if (err) atomicExch(err, 1);
            return false;
        }
    }
}

// wait_bounded by a converged warp, with a warp-uniform result.  The first look decides in
// one vote; the loop with its clock and flag reads is out of the way of the issue path.
static __device__ __forceinline__ bool wait_uniform(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int *err) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity, kSleepNs))) return true;
    return __all_sync(0xffffffffu, wait_bounded(bar, parity, abort_flag, err));
}

static __device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// Bulk (non-tensor) async copy global -> shared, completing `bytes` on `bar`.
// Both addresses 16-byte aligned, size a multiple of 16.
static __device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// The same bytes into L2 only.
static __device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

static __device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
static __device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
static __device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

static __device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)),
                 "r"(ncols)
                 : "memory");
}
static __device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
static __device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16, one CTA.
static __device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Issue path of an MMA warp.  The whole warp runs the issuing loop with warp-uniform
// control flow and one elected lane executes the tcgen05 instructions under a predicate:
// descriptors, TMEM address and instruction descriptor then stay in uniform registers and
// the four K steps of a stage leave back to back.  A loop under `if (lane == 0)` moves
// every operand to the uniform registers per instruction, one dependent move after
// another, and among busy generator warps that serial path, not the tensor core, set the
// stage time (GB300, 16 warps of FP32 and store work beside one issuer: 804 clock cycles
// per 128 x 256 x 64 stage; 604 in this form; the tensor core alone takes 512.  At
// 128 x 128 x 64 with idle generators 472 and 300).
static __device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}
// A value that is the same in every lane, marked as such for the compiler.
static __device__ __forceinline__ uint32_t warp_uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

// Low and high words of desc_sw128; the address field (16-byte units) is in the low word,
// and shared addresses below 256 KB cannot carry out of it.
static __device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }
static constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);

// The four K = 16 steps (32 bytes of the 128-byte rows each) of one 64-deep operand stage:
// D (+)= A B^T, the first step accumulating if `accumulate`.  Called by the whole warp;
// the lane with elected != 0 issues.
static __device__ __forceinline__ void umma_f16_x4(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc,
                                                   uint32_t accumulate, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred p, q, t;\n\t.reg .b32 x, y;\n\t.reg .b64 a, b;\n\t"
        "setp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %5, 0;\n\tsetp.eq.u32 t, %6, %6;\n\t"
        "mov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\t"
        "@p tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, q;\n\t"
        "add.u32 x, %1, 2;\n\tadd.u32 y, %2, 2;\n\tmov.b64 a, {x, %3};\n\tmov.b64 b, {y, %3};\n\t"
        "@p tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
        "add.u32 x, %1, 4;\n\tadd.u32 y, %2, 4;\n\tmov.b64 a, {x, %3};\n\tmov.b64 b, {y, %3};\n\t"
        "@p tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
        "add.u32 x, %1, 6;\n\tadd.u32 y, %2, 6;\n\tmov.b64 a, {x, %3};\n\tmov.b64 b, {y, %3};\n\t"
        "@p tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(kDescHi), "r"(idesc), "r"(accumulate), "r"(elected)
        : "memory");
}

// umma_commit by the elected lane of a converged warp.
static __device__ __forceinline__ void umma_commit_elected(uint64_t *bar, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t"
        "@p tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)),
        "r"(elected)
        : "memory");
}

// Arrive on `bar` once all previously issued tcgen05.mma of this thread complete.
static __device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

// 32 TMEM lanes x 16 consecutive 32-bit columns -> 16 registers per thread.
static __device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), version 1 (sm_100 family).
static __device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::f16: FP32 accumulator, FP16 (0) or BF16 (1)
// operands, both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
static __host__ __device__ constexpr uint32_t idesc_f16(int M, int N, int bf16) {
    return (1u << 4) | ((uint32_t)bf16 << 7) | ((uint32_t)bf16 << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// Byte offset of the 32-bit (re, im) pair `kp` (0..31) of row `row` in a K-major
// 128-byte-swizzled tile: 16-byte chunk index XOR (row mod 8).
static __device__ __forceinline__ uint32_t sw128_pair_offset(int row, int kp) {
    return (uint32_t)row * 128u + ((uint32_t)(((kp >> 2) ^ (row & 7))) << 4) + ((uint32_t)(kp & 3) << 2);
}

template <int BF16>
static __device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    if (BF16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    } else {
        __half2 h = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}

template <int BF16>
static __device__ __forceinline__ float2 unpack2(uint32_t v) {
    if (BF16) {
        const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162 *>(&v);
        return __bfloat1622float2(h);
    } else {
        const __half2 h = *reinterpret_cast<const __half2 *>(&v);
        return __half22float2(h);
    }
}

// Low parts of a pair packed by pack2 (split precision): each value minus its 16-bit
// rounding (exact in FP32), rounded to 16 bits again.
template <int BF16>
static __device__ __forceinline__ uint32_t pack2_lo(float lo, float hi, uint32_t packed) {
    const float2 r = unpack2<BF16>(packed);
    return pack2<BF16>(lo - r.x, hi - r.y);
}

static __device__ __forceinline__ uint32_t pow2_cols(int n) {
    uint32_t c = 32;
    while ((int)c < n) c <<= 1;
    return c;
}

// exp(2 pi i x) via the MUFU sine/cosine of the reduced argument (|error| ~ 1e-6).
static __device__ __forceinline__ float2 cis_turns(float x) {
    const float f = x - rintf(x);
    float s, c;
    __sincosf(6.28318530717958647f * f, &s, &c);
    return make_float2(c, s);
}

static __device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}


// Nearest integer by adding 1.5 * 2^23 (|x| < 2^22; the conversion unit's rounding
// instruction runs at a quarter of the FP32 rate).
static __device__ __forceinline__ float nearest(float x) { return __fadd_rn(__fadd_rn(x, 12582912.0f), -12582912.0f); }

// exp(2 pi i x) as cis_turns, without the conversion unit.
static __device__ __forceinline__ float2 cis_fast(float x) {
    float2 z;
    __sincosf(6.28318530717958647f * (x - nearest(x)), &z.y, &z.x);
    return z;
}

// cos and sin of the step 2 pi x from the half angle: the recurrence x_{n+1} = 2 cos(step) x_n
// - x_{n-1} amplifies an error of cos(step) by up to the square of its length where the step
// is small, and 1 - 2 sin^2 (2 cos^2 - 1 beyond a quarter turn) keeps that error at the
// rounding of 1.
static __device__ __forceinline__ void step_phasor(float x, float &re, float &im) {
    const float f = x - nearest(x);
    float s, c;
    __sincosf(3.14159265358979324f * f, &s, &c);
    re = fabsf(f) < 0.25f ? fmaf(-2.0f * s, s, 1.0f) : fmaf(2.0f * c, c, -1.0f);
    im = 2.0f * s * c;
}

static __device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// Sign with which the recurrences carry row r of an operand tile (pieces of 8 or 16 rows
// seeded at their middle): + - - + repeated; the output applies it.
static __host__ __device__ __forceinline__ constexpr float row_sign(int r) { return ((r + 1) & 2) ? -1.0f : 1.0f; }

// Four 8x8 b16 matrices from registers to shared memory.  Lane t holds, per matrix,
// the 32-bit pair at matrix row t/4, columns 2(t%4), 2(t%4)+1; lanes 8m..8m+7 give
// the 16-byte row addresses of matrix m.  With one K-major 128-byte operand row per
// matrix, lane t's pair is K' elements (2t, 2t+1) of that row: one instruction
// stores four operand rows of one 32-visibility stage.
template <int OFF>
static __device__ __forceinline__ void stmatrix_x4_at(uint32_t saddr, uint32_t v0, uint32_t v1, uint32_t v2,
                                                      uint32_t v3) {   // at saddr + OFF bytes
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0 + %5], {%1, %2, %3, %4};" ::"r"(saddr), "r"(v0),
                 "r"(v1), "r"(v2), "r"(v3), "n"(OFF)
                 : "memory");
}

// 2-D tiled TMA load of one box into shared memory, completing on `bar`.
static __device__ __forceinline__ void tma_load_2d(void *dst, const void *tmap, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// 16 consecutive 32-bit TMEM columns of 32 lanes <- 16 registers per thread.
static __device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 columns at a time, loads without their wait so that several can be in flight:
// tmem_ld32_issue ... tmem_wait_ld before the registers are read.
static __device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
static __device__ __forceinline__ void tmem_wait_ld(uint32_t (&a)[32], uint32_t (&b)[32]) {
    // the registers pass through the wait so that no use is scheduled ahead of it
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(a[i]), "+r"(b[i]));
}
static __device__ __forceinline__ void tmem_st32_issue(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
static __device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

}  // namespace tc
}  // namespace psf
