// tcgen05 (5th-generation tensor core) contraction of the smeared PSF, sm_103a.
//
// One CTA computes one 128 x ncols output tile of one cutout over a contiguous
// range of visibilities (split-K), as the real GEMM of Eqs. 21-22 in separable form:
//   P[j][i] = sum_k Re( c_k[j] a_k[i] ),   c_k[j] = w_k exp(2 pi i v_k dm_j),
//                                          a_k[i] = exp(2 pi i u_k dl_i),
//   A'[j][2k] = Re c, A'[j][2k+1] = Im c,  B'[i][2k] = Re a, B'[i][2k+1] = -Im a,
//   P = A' B'^T  with K' = 2K (FP16 or BF16 operands, FP32 accumulation in TMEM).
//
// Warp roles (TcShape; numbers for the 16 generator warps of most instances):
//   warps 0-15  operand generators (groups on stages s mod groups): per pipeline stage of
//               32 visibilities each lane owns one visibility and generates 32 or 64
//               twiddle rows (tw_rows), writing FP16/BF16 pairs straight into the
//               128-byte-swizzled K-major shared-memory layout the MMA reads;
//   warps 16-19 drain: every kDrainStages stages the issuers switch to their second
//               TMEM accumulator while these warps read the first ones (tcgen05.ld),
//               add them and add the sum into the CTA's FP32 partial tile in global
//               memory.  Short TMEM accumulation runs bound the tensor-core rounding
//               growth.  In split precision each add into the running sum is an
//               error-free TwoSum whose rounding error goes back into the drained
//               accumulator, on which the issuer's next range in that buffer
//               accumulates (compensated summation, the correction carried by the
//               tensor core);
//   warps 20, 22  TMEM allocation and the tcgen05.mma issue: with NISS = 2 (tiles of at
//               most 128 columns) one issues the even stages and one the odd ones, each
//               into accumulators of its own, so that one issuer's barrier wait overlaps
//               the other issuer's MMAs; with NISS = 1 one issues every stage;
//   warp 21     the uv/w input ring: one bulk copy pair per stage, refilled when the
//               generator group of the stage has written it (`in_empty`).
// Stages are handed over with mbarriers (input copies -> generators: `in_full`,
// generators -> input warp: `in_empty`, generators -> MMA: `full`, MMA commit ->
// generators: `empty`, MMA commit -> drain: `acc_full`, drain -> MMA: `acc_empty`).
// An issuing warp does nothing per stage but wait, issue and commit: MMA issue blocks it,
// so its serial latency bounds the stage rate.  Every wait is bounded by a wall-clock limit; on
// expiry the CTA raises the plan's error flag, stops all roles, waits (bounded) for
// its bulk copies and issued MMAs and frees TMEM.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "psf_internal.cuh"
#include "tc_ptx.cuh"

namespace psf {
namespace {
using namespace tc;

constexpr int kInStages = 16;      // per-visibility input (uv, w) ring depth
constexpr int kKS = 32;            // complex visibilities per stage (K' = 64 = one 128 B row)
// Warp roles of an instance.  Group g of the generator warps writes the stages s = g (mod
// groups).  A group waiting for slot reuse (stage s - S consumed) must find the slot's
// previous phase (stage s - 2S) already consumed, or the parity test of the barrier aliases;
// that holds when the group's previous stage s - groups waited for stage s - groups - S >=
// s - 2S, i.e. groups <= S.  With two issuers the group count must also be even: each issuer
// commits in order, but the two do not order each other, so both stages have to belong to
// the same issuer (an instance with five groups aliased and gave up its bounded waits).
//
// The generators bound the kernel (4 h MeerKAT cutout, exact: 3.72 ms without the MMAs, 2.50 ms
// without the twiddle rows, 3.78 ms together, before the last two of the following).  Seeds,
// barrier waits and loop code are about 130 of a warp's 290-350 instructions per stage, so
// the instances of the 128-pixel cutout give a warp 64 rows: with complex weights two warps
// take A, two the conjugate-symmetric B, the roles rotating with the group so that each
// falls on every scheduler (warp mod 4); in the fused form one takes A and two take B, one
// per weight.  Exact 4.39 -> 3.56 ms, fused 5.95 -> 4.60 ms.  24 warps of 64 registers were
// slower (recomputed addresses: 312 M -> 395 M instructions; fused 5.6 ms), as were six
// groups of two (3.85 ms) or three warps (3.69 ms) for the exact form.
template <int kStages, int NISS, int MIR, int SPLIT>
struct TcShape {
    static constexpr bool kTall = !SPLIT && ((MIR == 0 && kStages == 6) || (MIR == 4 && kStages == 4));
    static constexpr int kGroupWarps = kTall && MIR == 4 ? 3 : 4;
    static constexpr int kGroups0 = kStages < 4 ? kStages : 4;
    static constexpr int kGroups = NISS == 2 ? (kGroups0 & ~1) : kGroups0;
    static constexpr int kGen = kGroups * kGroupWarps;
    static constexpr int kDrainWarp0 = (kGen + 3) / 4 * 4;   // lane quarter = warp mod 4
    static constexpr int kMmaWarp = kDrainWarp0 + 4;
    static constexpr int kInWarp = kMmaWarp + 1;
    static constexpr int kMma2Warp = kMmaWarp + 2;
    static constexpr int kThreads = (kMmaWarp + 3) * 32;
    static_assert(NISS == 1 || kGroups % 2 == 0, "two issuers need an even number of generator groups");
    static_assert(kGroups <= kStages && kGroups <= kInStages, "generator groups exceed a ring depth");
};
constexpr int kDrainStages = 64;   // stages accumulated in TMEM between drains
// Split precision: the tensor core's FP32 accumulation loses about 2^-24.5 of the running
// value per added MMA (measured: the error of a cutout grows with the MMAs accumulated
// between drains, 64-stage runs of 12 MMAs left ~1e-5), so the runs are 8 stages and the
// drain warps keep the running sum in TMEM.
//
// Running sums of nearly equal terms (a coherent pixel such as the PSF peak, where every
// range adds about the same value) do not round at random: the sum sits on its own ulp
// grid and each add rounds the same way, so plain FP32 adds drift by up to ulp/2 per
// range (about 1.5e-5 of the peak over 1500 ranges).  Every add is therefore a TwoSum,
// s + v = t + e exactly, and e is written into the drained accumulator; the issuer's first
// MMA of the next range in that buffer keeps it (accumulate) instead of clearing it.
constexpr int kDrainStagesSplit = 8;

// t = fl(a + b) and the exact rounding error e (a + b = t + e), any magnitudes (Knuth).
__device__ __forceinline__ void two_sum(float a, float b, float &t, float &e) {
    t = a + b;
    const float bp = t - a;
    e = (a - (t - bp)) + (b - bp);
}
// *p += v without reading the old value back.
__device__ __forceinline__ void red_add(float *p, float v) {
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
constexpr int kATileBytes = 128 * 128;
// Twiddle rows of one visibility (this lane): value(r) = [w] exp(2 pi i theta (n0 + r)),
// written as an FP16/BF16 (re, im) pair at the lane's K-major swizzled slot, four rows (one
// of each of four pieces of PIECE = 8 or 16 rows) per stmatrix.  Each piece is seeded at its
// two middle rows and runs outwards by x_{n+1} = C x_n - x_{n-1}, C = 2 cos(step): one packed
// FMA per row, where the complex step of a phasor recurrence takes two (and its seeds every
// fourth row more): 888 M warp instructions of the exact launch on the 1 h MeerKAT cutout
// became 638 M.  The subtraction is left to the output: the rows are carried with the signs
// of row_sign, for which every step is y = (+-C) y + y.
// Seeds: sine/cosine evaluations for the middle row of the first piece, the step and the
// stride between pieces; three squarings and products give the rest.
struct TwSeeds {
    float2 xa[4], xb[4];   // rows PIECE/2 - 1 and PIECE/2 of the four pieces
    float2 C;              // (2 cos(step), 2 cos(step))
};

template <int PIECE>
__device__ __forceinline__ TwSeeds tw_seeds(float theta, int n0, float2 wk, bool weighted) {
    TwSeeds S;
    float2 st;
    step_phasor(theta, st.x, st.y);
    const float f = theta - nearest(theta);
    const float2 s1 = cis_fast((float)PIECE * f), s2 = cmulf(s1, s1);
    float2 z = cis_fast(theta * (float)(n0 + PIECE / 2 - 1));
    if (weighted) z = cmulf(z, wk);
    S.xa[0] = z;
    S.xa[1] = cmulf(z, s1);
    S.xa[2] = cmulf(z, s2);
    S.xa[3] = cmulf(S.xa[1], s2);
#pragma unroll
    for (int m = 0; m < 4; ++m) S.xb[m] = cmulf(S.xa[m], st);
    S.C = make_float2(2.0f * st.x, 2.0f * st.x);
    return S;
}

// Store of one row of each piece.  at: the lane's address of row 0 (piece lane / 8, chunk
// lane % 8 of its tile); MIRROR: the conjugates (a sign-bit XOR of the imaginary half) go to
// the rows R0 - r, mat being the lane's address of row R0; CPLX: (-Im z, Re z) at the same rows
// cplx_off bytes further on; SPLIT: the low parts (value minus its rounding, rounded again)
// lo_off bytes further on.
template <int BF16, int ROW, bool MIRROR, bool CPLX, bool SPLIT>
__device__ __forceinline__ void tw_row(uint32_t at, uint32_t mat, uint32_t cplx_off, uint32_t lo_off,
                                       const float2 (&x)[4]) {
    constexpr uint32_t kConj = 0x80000000u;
    constexpr uint32_t kSw = (uint32_t)(ROW & 7) << 4, kMsw = (uint32_t)((8 - (ROW & 7)) & 7) << 4;
    uint32_t v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = pack2<BF16>(x[m].x, x[m].y);
    const uint32_t addr = at ^ kSw, maddr = mat ^ kMsw;
    stmatrix_x4_at<ROW * 128>(addr, v[0], v[1], v[2], v[3]);
    if (MIRROR) stmatrix_x4_at<-ROW * 128>(maddr, v[0] ^ kConj, v[1] ^ kConj, v[2] ^ kConj, v[3] ^ kConj);
    if (CPLX)
        stmatrix_x4_at<ROW * 128>(addr + cplx_off, pack2<BF16>(-x[0].y, x[0].x), pack2<BF16>(-x[1].y, x[1].x),
                                  pack2<BF16>(-x[2].y, x[2].x), pack2<BF16>(-x[3].y, x[3].x));
    if (SPLIT) {
        uint32_t l[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) l[m] = pack2_lo<BF16>(x[m].x, x[m].y, v[m]);
        stmatrix_x4_at<ROW * 128>(addr + lo_off, l[0], l[1], l[2], l[3]);
        if (MIRROR)
            stmatrix_x4_at<-ROW * 128>(maddr + lo_off, l[0] ^ kConj, l[1] ^ kConj, l[2] ^ kConj, l[3] ^ kConj);
    }
}

// The 4 PIECE rows from the tile row at `base` (a multiple of 8 rows).  MIRROR:
// conjugates at the rows R0 - r, mbase = the address of row R0 (a multiple of 8); with
// `tail` the conjugate of the value one step past the last row at `tail_addr` (row 0).
template <int BF16, int PIECE, bool MIRROR = false, bool CPLX = false, bool SPLIT = false>
__device__ __forceinline__ void tw_rows(const TwSeeds &S, uint32_t base, uint32_t mbase = 0, bool tail = false,
                                        uint32_t tail_addr = 0, uint32_t cplx_off = 0, uint32_t lo_off = 0) {
    static_assert(PIECE == 8 || PIECE == 16, "piece");
    const uint32_t piece = (threadIdx.x >> 3) & 3u, chunk = (threadIdx.x & 7u) << 4;
    const uint32_t at = base + piece * (PIECE * 128u) + chunk, mat = mbase - piece * (PIECE * 128u) + chunk;
    const float2 nC = neg2(S.C);
    float2 fp[4], fc[4], bp[4], bc[4];
#define TW_ROW(R, X) tw_row<BF16, R, MIRROR, CPLX, SPLIT>(at, mat, cplx_off, lo_off, X)
    TW_ROW(PIECE / 2 - 1, S.xa);
    TW_ROW(PIECE / 2, S.xb);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        fp[m] = bc[m] = S.xa[m];
        fc[m] = bp[m] = S.xb[m];
    }
#define TW_STEP(K)                                                                      \
    {                                                                                   \
        _Pragma("unroll") for (int m = 0; m < 4; ++m) {                                 \
            const float2 c = ((K) & 1) ? nC : S.C;                                      \
            const float2 f = __ffma2_rn(c, fc[m], fp[m]), b = __ffma2_rn(c, bc[m], bp[m]); \
            fp[m] = fc[m];                                                              \
            fc[m] = f;                                                                  \
            bp[m] = bc[m];                                                              \
            bc[m] = b;                                                                  \
        }                                                                               \
        TW_ROW(PIECE / 2 + (K), fc);                                                    \
        TW_ROW(PIECE / 2 - 1 - (K), bc);                                                \
    }
    TW_STEP(1)
    TW_STEP(2)
    TW_STEP(3)
    if constexpr (PIECE == 16) {
        TW_STEP(4)
        TW_STEP(5)
        TW_STEP(6)
        TW_STEP(7)
    }
#undef TW_STEP
#undef TW_ROW
    if (MIRROR && tail) {   // row 4 PIECE: one more step of the last piece (sign +)
        const float2 x = __ffma2_rn(S.C, fc[3], fp[3]);
        const uint32_t lane = threadIdx.x & 31u;
        const uint32_t h = pack2<BF16>(x.x, -x.y);   // row 0: chunk lane / 4 (unswizzled), pair lane mod 4
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(tail_addr + lane * 4u), "r"(h) : "memory");
        if (SPLIT)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(tail_addr + lo_off + lane * 4u),
                         "r"(pack2_lo<BF16>(x.x, -x.y, h))
                         : "memory");
    }
}

struct SmemLayout {
    uint32_t a_off, b_off, in_off, bar_off, bytes;
};

constexpr uint32_t kInSlotBytes = kKS * 16;   // uv (8 B) + w (8 B) per visibility

// Operand ring depth for a tile width: as many 128-row A + ncols-row B stages as fit
// in ~192 KB (4 at 256 columns, 6 at 128, 8 at <= 64); split precision stages hold hi
// and lo tiles of both operands (3 at 128 columns, 4 at <= 64; tiles of at most 128
// columns).
__host__ __device__ constexpr int stages_for(int ncols_max, int split = 0) {
    return split ? (ncols_max > 64 ? 3 : 4) : (ncols_max > 128 ? 4 : (ncols_max > 64 ? 6 : 8));
}

__host__ __device__ inline SmemLayout smem_layout(int ncols_max, int kStages, uint32_t in_slot = kInSlotBytes,
                                                  int split = 0) {
    SmemLayout L;
    const uint32_t bt = (uint32_t)ncols_max * 128u;
    L.a_off = 0;
    L.b_off = kStages * kATileBytes * (1 + split);
    L.in_off = L.b_off + kStages * ((bt + 1023u) / 1024u * 1024u) * (1 + split);
    L.bar_off = L.in_off + kInStages * in_slot;
    L.bytes = L.bar_off + 512;   // 2 S + 2 kInStages + 8 barriers (<= 56 x 8 B), TMEM address, abort flag
    return L;
}

// MIR: 1 = the weights of the launch are real, so whole-cutout tiles may use the
// conjugate-symmetric generation (a separate instance keeps its register pressure out
// of the complex-weight kernel); 2 = real weights and every tile of the launch spans
// a whole 64- or 128-pixel cutout (no unmirrored path compiled in); 4 = the fused uv +
// image-plane form on such tiles: the A operand holds the unweighted column twiddles,
// the B operand (2 N rows) the row twiddles times the Method 1 weights (rows 0 .. N-1)
// and times the Method 2 weights (rows N .. 2N-1), so one N = 2 ncols MMA yields both
// cutouts side by side in TMEM (w2: second weight rows; part2: offset of the second
// cutout's partial sums from `partial`); 5 = complex output: A as in mode 0, B of 2 ncols
// rows = the conjugated row twiddles (a_r, -a_i) and then (a_i, a_r), so the two halves
// of the accumulator are the real and the imaginary parts of the cutout.
//
// SPLIT = 1 (split precision, MIR 0-2, tiles of at most 128 columns): every operand
// value x is held as hi = rnd16(x) and lo = rnd16(x - hi) in two tiles of the stage, and
// each stage issues A_hi B_hi + A_hi B_lo + A_lo B_hi into the same accumulator (the
// lo x lo term is below the 16-bit rounding of the lo parts).  The stages are twice as
// large, so the ring holds 3 or 4 of them and as many generator groups run.
template <int MIR>
__device__ __forceinline__ bool whole_cutout(const TcItem &it) {   // conjugate-symmetric generation
    return MIR == 2 || MIR == 4 ||
           (MIR == 1 && it.j0 == 0 && it.i0 == 0 && it.ncols == it.N && it.N <= 128 && (it.N & 63) == 0);
}

template <int BF16, int kStages, int NISS, int MIR, int SPLIT = 0>
__global__ void __launch_bounds__(TcShape<kStages, NISS, MIR, SPLIT>::kThreads, 1)
    k_psf_tc(const float2 *__restrict__ uv, const float2 *__restrict__ w, int64_t ldw,
             const TcItem *__restrict__ items, int ncols_max, float cell, float *__restrict__ partial,
             int64_t split_stride, int *err, const float2 *__restrict__ w2, int64_t part2) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1024-byte alignment of the operand tiles (swizzle atoms)
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr int kBMul = (MIR == 4 || MIR == 5) ? 2 : 1;           // B rows per output column
    constexpr uint32_t kSlot = (MIR == 4) ? kKS * 24 : kInSlotBytes;   // uv, w (, w2) per visibility
    using Sh = TcShape<kStages, NISS, MIR, SPLIT>;
    constexpr int kGrp = Sh::kGroups, kGroupWarps = Sh::kGroupWarps;
    constexpr int kDrainWarp0 = Sh::kDrainWarp0, kMmaWarp = Sh::kMmaWarp, kInWarp = Sh::kInWarp;
    constexpr int kMma2Warp = Sh::kMma2Warp;
    static_assert(!SPLIT || MIR <= 2, "split precision covers the plain and mirrored real-weight forms");
    // Two issuers take alternate stages; with an even ring depth every slot (and its release
    // barrier) then belongs to one issuer.  An odd depth makes the two issuing threads commit
    // alternately to the same release barrier, and such launches (3 stages, two issuers)
    // gave up bounded waits in about one launch in eight on GB300 with the protocol reading
    // correctly; two issuers are therefore only used with even depths.
    static_assert(NISS == 1 || kStages % 2 == 0, "two MMA issuers need an even operand ring depth");
    constexpr int kRange = SPLIT ? kDrainStagesSplit : kDrainStages;   // stages per accumulation run
    const SmemLayout L = smem_layout(kBMul * ncols_max, kStages, kSlot, SPLIT);
    uint64_t *full = (uint64_t *)(smem + L.bar_off);
    uint64_t *empty = full + kStages;
    uint64_t *in_full = empty + kStages;
    uint64_t *in_empty = in_full + kInStages;
    uint64_t *acc_full = in_empty + kInStages;   // [issuer][buffer]
    uint64_t *acc_empty = acc_full + 4;          // [buffer], shared by the issuers
    uint64_t *done_bar = acc_empty + 2;          // [issuer]
    uint32_t *s_tmem = (uint32_t *)(done_bar + 2);
    volatile int *s_abort = (volatile int *)(s_tmem + 1);
    volatile int no_abort = 0;   // teardown waits ignore the abort flag

    const TcItem it = items[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ncols = it.ncols;
    const uint32_t bt_stride = ((uint32_t)(kBMul * ncols_max) * 128u + 1023u) / 1024u * 1024u;   // one B tile
    const uint32_t b_stage = bt_stride * (1 + SPLIT);                  // hi (and lo) B tiles of a stage
    constexpr uint32_t kAStage = kATileBytes * (1 + SPLIT);
    const uint32_t acc_cols = pow2_cols(kBMul * ncols_max);
    const int nst = (it.k1 - it.k0 + kKS - 1) / kKS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], kGroupWarps);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kInStages; ++s) {
            mbar_init(&in_full[s], 1);
            mbar_init(&in_empty[s], kGroupWarps);
        }
        for (int a = 0; a < 4; ++a) mbar_init(&acc_full[a], 1);
        for (int a = 0; a < 2; ++a) mbar_init(&acc_empty[a], 4);
        for (int a = 0; a < 2; ++a) mbar_init(&done_bar[a], 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // accumulator (issuer q, buffer b) at TMEM column (2 q + b) acc_cols
    // accumulators (issuer, buffer) and, with split precision, the running sum
    const uint32_t tmem_cols = pow2_cols((2 * NISS + SPLIT) * (int)acc_cols);
    if (warp == kMmaWarp) {
        tmem_alloc(s_tmem, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;

    if (warp < Sh::kGen) {
        // ------------------------------------------------------------ generators
        const int grp = warp / kGroupWarps, gw = warp % kGroupWarps;
        const int half = it.N / 2;
        // Conjugate symmetry about the cutout centre (pixel offsets (r - N/2) cell):
        // row N - r of the row twiddles holds the conjugate of row r, and so do the
        // column twiddles when the weights are real (uv and image-plane methods).  For
        // a tile that spans a whole cutout of 64 or 128 pixels only rows N/2 .. N-1 are
        // generated; rows 1 .. N/2 are their conjugates and row 0 the conjugate of the
        // value one step past row N-1.
        const bool mirror = whole_cutout<MIR>(it);
        // 32-row chains of the A (128 rows) and B tiles (complex output: A rows past the
        // cutout are skipped)
        const int nA = mirror ? it.N / 64 : (MIR == 5 ? min(4, (it.N - it.j0 + 31) / 32) : 4);
        const int nB = mirror ? it.N / 64 : ncols / 32;
        for (int s_i = grp; s_i < nst; s_i += kGrp) {
            const int slot = s_i % kStages;
            const uint32_t ph = (uint32_t)(s_i / kStages) & 1u;
            const int islot = s_i % kInStages;
            if (!wait_uniform(&in_full[islot], (uint32_t)(s_i / kInStages) & 1u, s_abort, err)) break;
            const float2 *in_uv = (const float2 *)(smem + L.in_off + islot * kSlot);
            const float2 uvk = in_uv[lane];
            const bool kin = it.k0 + s_i * kKS + lane < it.k1;
            const float2 wk = kin ? in_uv[kKS + lane] : make_float2(0.f, 0.f);
            const float w2k = (MIR == 4 && kin) ? in_uv[2 * kKS + lane].x : 0.f;
            const uint32_t a_tile = smem_u32(smem + L.a_off + slot * kAStage);
            const uint32_t b_tile = smem_u32(smem + L.b_off + slot * b_stage);
            const float tv = uvk.y * cell, tu = -uvk.x * cell;
            auto slot_free = [&]() { return s_i < kStages || wait_uniform(&empty[slot], ph ^ 1u, s_abort, err); };
            // seeds before the wait for the operand slot, rows after it
            if (Sh::kTall && MIR == 0 && nA == 4 && nB == 4) {
                // complex weights on a full 128 x 128 tile: A (weighted column twiddles) in warps 0-1,
                // 64 rows each; B (conjugated row twiddles) in warps 2-3, conjugate-symmetric where the
                // tile is a whole cutout (32 generated rows each), else 64 rows each
                const int role = (gw + grp) & 3;   // each role on every scheduler (warp mod 4)
                const bool isA = role < 2;
                if (!isA && it.N == 128) {
                    const int c = role - 2;
                    const TwSeeds S = tw_seeds<8>(tu, 32 * c, wk, false);
                    if (!slot_free()) break;
                    tw_rows<BF16, 8, true>(S, b_tile + (uint32_t)(64 + 32 * c) * 128u, b_tile + (uint32_t)(64 - 32 * c) * 128u,
                                           c == 1, b_tile);
                } else {
                    const int r0 = 64 * (role & 1);
                    const TwSeeds S = tw_seeds<16>(isA ? tv : tu, (isA ? it.j0 : it.i0) + r0 - half, wk, isA);
                    if (!slot_free()) break;
                    tw_rows<BF16, 16>(S, (isA ? a_tile : b_tile) + (uint32_t)r0 * 128u);
                }
            } else if (Sh::kTall && MIR == 4 && it.N == 128) {
                // fused form on a 128-pixel cutout: A in warp 0, B with the Method 1 weights in warp 1,
                // with the Method 2 weights in warp 2; rows 64 .. 127 and their mirrors
                const TwSeeds S = tw_seeds<16>(gw ? tu : tv, 0, make_float2(gw == 2 ? w2k : wk.x, 0.f), gw > 0);
                if (!slot_free()) break;
                const uint32_t t0 = (gw ? b_tile : a_tile) + (gw == 2 ? 128u * 128u : 0u);
                tw_rows<BF16, 16, true>(S, t0 + 64 * 128, t0 + 64 * 128, true, t0);
            } else {
                bool free = false;
                // units: the 32-row chains of A, then those of B (in the fused form once per weight)
                constexpr int kBW = MIR == 4 ? 2 : 1;
                for (int ch = gw; ch < nA + kBW * nB; ch += kGroupWarps) {
                    const bool isA = ch < nA;
                    const int c = isA ? ch : (ch - nA) / kBW;
                    const uint32_t tile = isA ? a_tile : b_tile;
                    if (MIR == 4 || mirror) {
                        // rows R0 .. R0 + 31 (R0 = N/2 + 32 c) and their mirrors N - R0 - r; the fused form
                        // weights the row twiddles (both halves of B), the others the column twiddles
                        const int R0 = half + 32 * c;
                        const bool second = MIR == 4 && !isA && ((ch - nA) & 1);
                        const float2 wv = MIR == 4 ? make_float2(second ? w2k : wk.x, 0.f) : wk;
                        const TwSeeds S = tw_seeds<8>(isA ? tv : tu, 32 * c, wv, isA != (MIR == 4));
                        if (!free && !(free = slot_free())) break;
                        const uint32_t t0 = tile + (second ? (uint32_t)it.N * 128u : 0u);
                        tw_rows<BF16, 8, true, false, SPLIT>(S, t0 + (uint32_t)R0 * 128u,
                                                             t0 + (uint32_t)(it.N - R0) * 128u, c == it.N / 64 - 1, t0, 0,
                                                             isA ? (uint32_t)kATileBytes : bt_stride);
                    } else {   // weighted column twiddles c_k[j] (A) or conjugated row twiddles (a_r, -a_i) (B)
                        const TwSeeds S = tw_seeds<8>(isA ? tv : tu, (isA ? it.j0 : it.i0) + 32 * c - half, wk, isA);
                        if (!free && !(free = slot_free())) break;
                        if (MIR == 5 && !isA)
                            tw_rows<BF16, 8, false, true>(S, tile + c * 32 * 128, 0, false, 0, (uint32_t)ncols * 128u);
                        else
                            tw_rows<BF16, 8, false, false, SPLIT>(S, tile + c * 32 * 128, 0, false, 0, 0,
                                                                  isA ? (uint32_t)kATileBytes : bt_stride);
                    }
                }
                if (!free && !slot_free()) break;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&full[slot]);
                // the input slot is released only after the stores that depend on its values
                mbar_arrive(&in_empty[islot]);
            }
        }
    } else if (warp == kMmaWarp || (NISS == 2 && warp == kMma2Warp)) {
        // ------------------------------------------------------------ MMA issue
        // Issuer q takes the stages s = q (mod NISS); with an even ring depth every
        // slot belongs to one issuer.  Accumulation range d covers stages
        // [d kRange, (d + 1) kRange) and uses buffer b = d mod 2.
        {
            const int q = (warp == kMmaWarp) ? 0 : 1;
            // The issue path is short and warp-uniform (umma_f16_x4); among the generators its
            // instructions count more than the tensor core's time.
            const uint32_t el = elect_one();
            const uint32_t idesc = warp_uniform(idesc_f16(128, kBMul * ncols, BF16));
            const uint32_t ad0 = warp_uniform(desc_lo(smem_u32(smem + L.a_off)));
            const uint32_t bd0 = warp_uniform(desc_lo(smem_u32(smem + L.b_off)));
            const uint32_t b_units = warp_uniform(b_stage >> 4), tm0 = warp_uniform(tmem);
            const uint32_t cols = warp_uniform(acc_cols);
            // one ring round per outer iteration, unrolled over this issuer's slots
            const uint32_t adq = ad0 + (uint32_t)q * (kAStage >> 4), bdq = bd0 + (uint32_t)q * b_units;
            int r = q, d = 0;
            uint32_t ph = 0;
            bool stop = false;
            for (int s0 = q; s0 < nst && !stop; s0 += kStages, ph ^= 1u) {
#pragma unroll
                for (int i = 0; i < kStages / NISS; ++i) {
                    const int s_i = s0 + NISS * i;
                    if (s_i >= nst || stop) break;
                    const int b = d & 1;
                    if (r == q && d >= 2 &&   // first own stage of a range: the buffer's last drain is done
                        !wait_uniform(&acc_empty[b], (uint32_t)((d >> 1) - 1) & 1u, s_abort, err)) {
                        stop = true;
                        break;
                    }
                    if (!wait_uniform(&full[q + NISS * i], ph, s_abort, err)) { stop = true; break; }
                    tc_fence_after();
                    const uint32_t ad = adq + (uint32_t)(NISS * i) * (kAStage >> 4);
                    const uint32_t bd = bdq + (uint32_t)(NISS * i) * b_units;
                    const uint32_t dt = tm0 + (uint32_t)(2 * q + b) * cols;
                    // a range's first MMA clears the buffer, except issuer 0's from range 2 on:
                    // the drain has left the compensation of the running sum there
                    umma_f16_x4(dt, ad, bd, idesc, (r != q || (SPLIT && q == 0 && d >= 2)) ? 1u : 0u, el);
                    if (SPLIT) {   // A_hi B_lo, then A_lo B_hi
                        umma_f16_x4(dt, ad, bd + (bt_stride >> 4), idesc, 1u, el);
                        umma_f16_x4(dt, ad + (kATileBytes >> 4), bd, idesc, 1u, el);
                    }
                    umma_commit_elected(&empty[q + NISS * i], el);
                    r += NISS;
                    if (r >= kRange || s_i + NISS >= nst) umma_commit_elected(&acc_full[2 * q + b], el);
                    if (r >= kRange) {
                        r -= kRange;
                        ++d;
                    }
                }
            }
            // all issued MMAs complete before TMEM is released (waited for even after
            // an abort; the wait is still time-limited)
            umma_commit_elected(&done_bar[q], el);
            wait_bounded(&done_bar[q], 0, &no_abort, err);
        }
        __syncwarp();
    } else if (warp == kInWarp) {
        // ------------------------------------------------------------ input ring
        // stage s's uv and w (256 B each) into slot s % kInStages, once the generator
        // group of stage s - kInStages has read that slot
        if (lane == 0) {
            const float2 *wp = w + (int64_t)it.slot * ldw;
            int issued = 0;
            for (int s_i = 0; s_i < nst; ++s_i) {
                const int islot = s_i % kInStages;
                if (s_i >= kInStages &&
                    !wait_bounded(&in_empty[islot], (uint32_t)(s_i / kInStages - 1) & 1u, s_abort, err))
                    break;
                uint8_t *dst = smem + L.in_off + islot * kSlot;
                const int32_t kb = it.k0 + s_i * kKS;
                mbar_arrive_expect_tx(&in_full[islot], kSlot);
                bulk_g2s(dst, uv + kb, kKS * 8, &in_full[islot]);
                bulk_g2s(dst + kKS * 8, wp + kb, kKS * 8, &in_full[islot]);
                if (MIR == 4) bulk_g2s(dst + kKS * 16, w2 + (int64_t)it.slot * ldw + kb, kKS * 8, &in_full[islot]);
                issued = s_i + 1;
            }
            // every copy has landed before the CTA exits (the last use of each slot)
            for (int s_i = max(0, issued - kInStages); s_i < issued; ++s_i)
                wait_bounded(&in_full[s_i % kInStages], (uint32_t)(s_i / kInStages) & 1u, &no_abort, err);
        }
        __syncwarp();
    } else if (warp < kDrainWarp0) {
        // fills the generator warps up to a multiple of four: idle
    } else if (warp == kMma2Warp) {
        // second issuer, idle with one issuer (NISS == 1): it must not join the drain
        // warps (lane quarters 0-3, four arrivals per accumulator release)
    } else {
        // ------------------------------------------------------------ drain
        // The partial cutout is stored transposed (element (j, i) at i N + j), so the 32
        // lanes of a warp (32 consecutive rows j, one column per access) touch one
        // contiguous 128-byte line.
        const int q = warp - kDrainWarp0;          // TMEM lane quarter (warp % 4)
        const int j = it.j0 + q * 32 + lane;       // output row (m offset index)
        float *dst = partial + (int64_t)it.split * split_stride + it.out_off + (int64_t)it.i0 * it.N + j;
        const int64_t cstride = it.N;
        const bool row_ok = j < it.N;
        const int ncol_valid = min(ncols, it.N - it.i0);
        float *dst2 = dst + part2;   // second cutout of the fused form
        // signs of the operand rows (row_sign; mirrored tiles count from the cutout's centre)
        const bool mirror = whole_cutout<MIR>(it);
        const bool mirror_b = mirror || (Sh::kTall && MIR == 0 && it.N == 128);
        auto sign_of = [&](int r, bool m) { return row_sign(m ? abs(r - it.N / 2) : r); };
        const float rs = sign_of(q * 32 + lane, mirror);
        if (nst == 0) {
            if (row_ok)
                for (int c = 0; c < ncol_valid; ++c) {
                    dst[c * cstride] = 0.f;
                    if (kBMul == 2) dst2[c * cstride] = 0.f;
                }
        }
        const int ndrain = (nst + kRange - 1) / kRange;
        // split precision: running sum of the drained ranges in TMEM columns after the
        // accumulators
        const uint32_t tsum = tmem + ((uint32_t)(q * 32) << 16) + 2u * NISS * acc_cols;
        for (int d = 0; d < ndrain; ++d) {
            const int b = d & 1;
            // issuer 1 has a stage in range d unless the range holds a single stage
            const bool two = (NISS == 2) && (min(nst, (d + 1) * kRange) - d * kRange > 1);
            bool ok = wait_bounded(&acc_full[b], (uint32_t)(d >> 1) & 1u, s_abort, err);
            if (two && ok) ok = wait_bounded(&acc_full[2 + b], (uint32_t)(d >> 1) & 1u, s_abort, err);
            if (!__all_sync(0xffffffffu, ok)) break;   // warp-uniform exit
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * acc_cols;
            for (int c0 = 0; c0 < kBMul * ncols; c0 += 16) {
                // fused form: columns ncols .. 2 ncols - 1 are the second cutout
                float *const dd = (kBMul == 2 && c0 >= ncols) ? dst2 : dst;
                const int cb = (kBMul == 2 && c0 >= ncols) ? c0 - ncols : c0;
                float v[16];
                tmem_ld16(ta + (uint32_t)c0, v);
                if (two) {
                    float v2[16];
                    tmem_ld16(ta + 2u * acc_cols + (uint32_t)c0, v2);
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] += v2[e];
                }
                float sg[4];   // row sign times the sign of columns c0 + e (e mod 4)
#pragma unroll
                for (int e = 0; e < 4; ++e) sg[e] = rs * sign_of(cb + e, mirror_b);
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] *= sg[e & 3];
                if (SPLIT) {
                    float sv[16], cv[16];   // running sum; compensation for the buffer's next range
#pragma unroll
                    for (int e = 0; e < 16; ++e) sv[e] = 0.f;
                    if (d > 0) tmem_ld16(tsum + (uint32_t)c0, sv);
#pragma unroll
                    for (int e = 0; e < 16; ++e) two_sum(sv[e], v[e], v[e], cv[e]);
                    if (d < ndrain - 1) {
                        tmem_st16(tsum + (uint32_t)c0, v);
                    } else if (row_ok) {   // last range: the CTA's sum goes out once
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            if (cb + e < ncol_valid) dd[(cb + e) * cstride] = v[e];
                    }
                    // issuer 0's buffer b is accumulated on again by range d + 2
                    if (d + 2 < ndrain) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) cv[e] *= sg[e & 3];
                        tmem_st16(ta + (uint32_t)c0, cv);
                    }
                    continue;
                }
                // The first range stores, later ones add by reductions, which return nothing
                // (one thread owns each element, so the sum has a fixed order): a load, an add and
                // a store per element took an L2 round trip per eight.
                if (row_ok) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (cb + e < ncol_valid) {
                            if (d == 0) dd[(cb + e) * cstride] = v[e];
                            else red_add(dd + (cb + e) * cstride, v[e]);
                        }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMmaWarp) tmem_dealloc(tmem, tmem_cols);
}

// Self-test: one 128 x n x 64 FP16 GEMM through the same layout, descriptors,
// instruction descriptor and TMEM read-out as the contraction kernel.
__global__ void __launch_bounds__(128, 1)
    k_selftest(const __half *__restrict__ A, const __half *__restrict__ B, float *__restrict__ D, int n,
               int *err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *a_tile = smem;
    uint8_t *b_tile = smem + kATileBytes;
    uint64_t *bar = (uint64_t *)(smem + kATileBytes + 256 * 128);
    uint32_t *s_tmem = (uint32_t *)(bar + 1);
    volatile int *s_abort = (volatile int *)(s_tmem + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cols = pow2_cols(n);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        tmem_alloc(s_tmem, cols);
        tmem_relinquish();
    }
    // operands: pairs of FP16 (k' = 2 kp, 2 kp + 1) into the swizzled K-major tiles
    for (int idx = threadIdx.x; idx < 128 * 32; idx += blockDim.x) {
        const int row = idx >> 5, kp = idx & 31;
        *reinterpret_cast<uint32_t *>(a_tile + sw128_pair_offset(row, kp)) =
            *reinterpret_cast<const uint32_t *>(A + row * 64 + 2 * kp);
    }
    for (int idx = threadIdx.x; idx < n * 32; idx += blockDim.x) {
        const int row = idx >> 5, kp = idx & 31;
        *reinterpret_cast<uint32_t *>(b_tile + sw128_pair_offset(row, kp)) =
            *reinterpret_cast<const uint32_t *>(B + row * 64 + 2 * kp);
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    if (threadIdx.x == 0) {
        const uint32_t idesc = idesc_f16(128, n, 0);
        const uint64_t ad = desc_sw128(smem_u32(a_tile)), bd = desc_sw128(smem_u32(b_tile));
        for (int kk = 0; kk < 4; ++kk) umma_f16(tmem, ad + 2 * kk, bd + 2 * kk, idesc, kk > 0 ? 1u : 0u);
        umma_commit(bar);
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, wait_bounded(bar, 0, s_abort, err));
    tc_fence_after();
    if (ok) {
        const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16);
        for (int c0 = 0; c0 < n; c0 += 16) {
            float v[16];
            tmem_ld16(ta + (uint32_t)c0, v);
            for (int e = 0; e < 16; ++e) D[(warp * 32 + lane) * n + c0 + e] = v[e];
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, cols);
}

// A wait that nothing completes: the bounded-wait path with a caller-given limit.
__global__ void k_wait_timeout(unsigned long long limit_ns, int *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long t0 = globaltimer();
        for (;;) {
            if (mbar_try_wait(&bar, 0, 100000u)) return;   // never completes
            if (globaltimer() - t0 > limit_ns) {
                atomicExch(err, 1);
                return;
            }
        }
    }
}

}  // namespace

int selftest_timeout(int limit_ms) {
    int *err = nullptr;
    if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return PSF_ENOMEM; }
    cudaError_t e = cudaMemset(err, 0, sizeof(int));
    if (e == cudaSuccess) {
        k_wait_timeout<<<1, 32>>>((unsigned long long)limit_ms * 1000000ull, err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    int flag = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&flag, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (e != cudaSuccess) { cudaGetLastError(); return PSF_ECUDA; }
    return flag ? PSF_ETIMEOUT : PSF_OK;
}

template <int BF16, int S, int NISS, int MIR, int SPLIT = 0>
static cudaError_t launch_tc_t(const DevObs &o, const float2 *w, int64_t ldw, const TcItem *items, int nitems,
                               int ncols_max, float cell, float *partial, int64_t split_stride, int *err,
                               cudaStream_t st, const float2 *w2 = nullptr, int64_t part2 = 0) {
    const SmemLayout L =
        smem_layout((MIR == 4 || MIR == 5 ? 2 : 1) * ncols_max, S, MIR == 4 ? kKS * 24 : kInSlotBytes, SPLIT);
    const size_t bytes = L.bytes + 1024;
    cudaError_t e = cudaFuncSetAttribute(k_psf_tc<BF16, S, NISS, MIR, SPLIT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    k_psf_tc<BF16, S, NISS, MIR, SPLIT><<<nitems, TcShape<S, NISS, MIR, SPLIT>::kThreads, bytes, st>>>(o.uv, w, ldw, items, ncols_max, cell,
                                                                          partial, split_stride, err, w2, part2);
    return cudaGetLastError();
}

cudaError_t launch_psf_tc(const DevObs &o, const float2 *w, int64_t ldw, const TcItem *items, int nitems,
                          int ncols_max, int bf16, float cell, int wreal, float *partial, int64_t split_stride,
                          int *err, cudaStream_t st, int split) {
    if (nitems <= 0) return cudaSuccess;
    if (split) {   // tiles of at most 128 columns
        if (ncols_max > 128) return cudaErrorInvalidValue;
        // 3 stages (128 columns): one issuer (twelve MMAs per stage hide its barrier round
        // trip; two issuers need an even depth); 4 stages (<= 64 columns): two issuers
#define PSF_TC_SPLIT(B, SS)                                                                                    \
    if (bf16 == B && stages_for(ncols_max, 1) == SS) {                                                         \
        constexpr int NI = SS % 2 == 0 ? 2 : 1;                                                                \
        if (wreal == 2)                                                                                        \
            return launch_tc_t<B, SS, NI, 2, 1>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, \
                                                err, st);                                                      \
        return wreal ? launch_tc_t<B, SS, NI, 1, 1>(o, w, ldw, items, nitems, ncols_max, cell, partial,        \
                                                    split_stride, err, st)                                     \
                     : launch_tc_t<B, SS, NI, 0, 1>(o, w, ldw, items, nitems, ncols_max, cell, partial,        \
                                                    split_stride, err, st);                                    \
    }
        PSF_TC_SPLIT(0, 3) PSF_TC_SPLIT(0, 4) PSF_TC_SPLIT(1, 3) PSF_TC_SPLIT(1, 4)
#undef PSF_TC_SPLIT
        return cudaErrorInvalidValue;
    }
    const int S = stages_for(ncols_max);
    // two issuers while both double-buffered accumulator pairs fit in TMEM (<= 128 columns)
#define PSF_TC_CASE(B, SS)                                                                                  \
    if (bf16 == B && S == SS) {                                                                             \
        constexpr int NI = SS == 4 ? 1 : 2;                                                                 \
        if (wreal == 2)                                                                                     \
            return launch_tc_t<B, SS, NI, 2>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, \
                                             err, st);                                                      \
        return wreal ? launch_tc_t<B, SS, NI, 1>(o, w, ldw, items, nitems, ncols_max, cell, partial,         \
                                                 split_stride, err, st)                                      \
                     : launch_tc_t<B, SS, NI, 0>(o, w, ldw, items, nitems, ncols_max, cell, partial,         \
                                                 split_stride, err, st);                                     \
    }
    PSF_TC_CASE(0, 4) PSF_TC_CASE(0, 6) PSF_TC_CASE(0, 8) PSF_TC_CASE(1, 4) PSF_TC_CASE(1, 6) PSF_TC_CASE(1, 8)
#undef PSF_TC_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_psf_tc_uvimg(const DevObs &o, const float2 *w_uv, const float2 *w_img, int64_t ldw,
                                const TcItem *items, int nitems, int ncols_max, int bf16, float cell, float *partial,
                                int64_t split_stride, int64_t part2, int *err, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    if (ncols_max != 64 && ncols_max != 128) return cudaErrorInvalidValue;
    // B tiles of 2 ncols rows: 128 rows -> 6 stages, two issuers; 256 rows -> 4 stages, one
    if (ncols_max == 64)
        return bf16 ? launch_tc_t<1, 6, 2, 4>(o, w_uv, ldw, items, nitems, 64, cell, partial, split_stride, err, st,
                                              w_img, part2)
                    : launch_tc_t<0, 6, 2, 4>(o, w_uv, ldw, items, nitems, 64, cell, partial, split_stride, err, st,
                                              w_img, part2);
    return bf16 ? launch_tc_t<1, 4, 1, 4>(o, w_uv, ldw, items, nitems, 128, cell, partial, split_stride, err, st,
                                          w_img, part2)
                : launch_tc_t<0, 4, 1, 4>(o, w_uv, ldw, items, nitems, 128, cell, partial, split_stride, err, st,
                                          w_img, part2);
}

cudaError_t launch_psf_tc_cplx(const DevObs &o, const float2 *w, int64_t ldw, const TcItem *items, int nitems,
                               int ncols_max, int bf16, float cell, float *partial, int64_t split_stride,
                               int64_t part2, int *err, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    if (ncols_max > 128) return cudaErrorInvalidValue;
    // B tiles of 2 ncols rows: <= 128 rows -> 6 stages, two issuers; up to 256 -> 4, one
    if (2 * ncols_max <= 128)
        return bf16 ? launch_tc_t<1, 6, 2, 5>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, err,
                                              st, nullptr, part2)
                    : launch_tc_t<0, 6, 2, 5>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, err,
                                              st, nullptr, part2);
    return bf16 ? launch_tc_t<1, 4, 1, 5>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, err, st,
                                          nullptr, part2)
                : launch_tc_t<0, 4, 1, 5>(o, w, ldw, items, nitems, ncols_max, cell, partial, split_stride, err, st,
                                          nullptr, part2);
}

int selftest_umma(const void *a, const void *b, float *d, int n) {
    int *err = nullptr;
    if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return PSF_ENOMEM; }
    cudaMemset(err, 0, sizeof(int));
    const size_t bytes = kATileBytes + 256 * 128 + 256 + 1024;
    cudaError_t e = cudaFuncSetAttribute(k_selftest, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) {
        k_selftest<<<1, 128, bytes>>>((const __half *)a, (const __half *)b, d, n, err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    int flag = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&flag, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (e != cudaSuccess) { cudaGetLastError(); return PSF_ECUDA; }
    return flag ? PSF_ETIMEOUT : PSF_OK;
}

}  // namespace psf
