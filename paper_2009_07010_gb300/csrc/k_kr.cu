// Batched (Khatri-Rao) tcgen05 contraction: many positions with the same cutout size.
//
//   X[p][q] = sum_k Re( w_{p,k} KR_k[q] ),   KR_k[q] = exp(2 pi i (u_k dl_i + v_k dm_j)),
//   pixel q = j N + i,  w_{p,k} = W_k D_k(l0_p)                         (Eqs. 21-22)
//
// Point reflection.  KR_k at the pixel offset (-dl, -dm) is the conjugate of KR_k at
// (dl, dm), so with
//   E[p][q] = sum_k Re w_{p,k} cos(phase_k(q)),   O[p][q] = sum_k -Im w_{p,k} sin(phase_k(q))
// the two pixels are E + O and E - O.  Only a half plane of pixels is contracted (rows
// j >= N/2, plus row 0 and the lower half of column 0, whose reflections lie outside the
// cutout): two real GEMMs with K' = K each (one for real weights, O = 0) instead of one
// with K' = 2K over all pixels, which is half the tensor work and half the twiddles per
// cutout.  256 x 64^2 on 14.1 M visibilities, exact: contraction 49.8 ms -> 21.9 ms;
// 512 mixed cutouts on 7.1 M visibilities, Method 1 (real): 167.5 ms -> 54.4 ms
// (both with the contiguous weight stages and the unrolled issue loop below).
//
// One CTA computes a 128-position tile of 128 representative pixels (256 for real
// weights) over a range of visibilities, in 64-visibility stages:
//   A  the weights, 128 positions x 64 visibilities, FP16/BF16 (Re w, and a second tile of
//      -Im w), precomputed per chunk of visibilities, stage after stage in the swizzled
//      layout (w16_offset), so that a stage is one contiguous bulk copy.  (As rows of the
//      chunk, loaded by 2-D TMA, the 128 segments of a stage lay megabytes, often a power
//      of two, apart, and L2 delivered 4.5-5.5 TB/s in all: with the point reflection that
//      left the stages of 512 tensor cycles at 1100 (real) and 1750 (complex).)
//   B  cos (and sin) of the pixel phases, pixels x 64 visibilities, generated on chip.
// Warp roles:
//   generators   one group of four warps per operand slot (warps 0-15, or 0-11 with complex
//                weights, whose 64 KB stages leave a ring of three): each lane owns two
//                visibilities of a stage and writes their twiddles of 32 or 64 pixels as
//                FP16/BF16 pairs into the swizzled layout (kr_seeds, kr_chain);
//   fold warps   (the others up to 19) every fold range add the active TMEM accumulators into
//                a running-sum region of TMEM (short FP32 accumulation runs); at the end they
//                add sum + active of each pixel and of its reflection into the output with
//                global atomics (the output is zeroed first; several visibility ranges of a
//                tile add up);
//   warp 20      bulk copies of the weight tiles of each stage;
//   warp 21      TMEM allocation and the tcgen05.mma issue (M = 128, K = 16, N = the tile's
//                pixels).  Among the generators its instructions, not the tensor core, set
//                the stage time (without generators a real stage takes 585 cycles, without
//                MMAs 730, together 812), so its loop is unrolled over the ring slots;
//   warp 22      the uv input ring (bulk copies), refilled when the generator group
//                of a stage has read its slot.
// An item starts in operand slot 0; barrier phases are kept per slot.
// Every barrier wait is bounded (2 s); on expiry the CTA raises the error flag, stops,
// waits (bounded) for its copies in flight and issued MMAs and frees TMEM.
#include "psf_internal.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>

#include <algorithm>

namespace psf {
namespace {
using namespace tc;

constexpr int kKrIn = 16;             // uv input ring depth (stages)
constexpr int kKrKS = 64;             // visibilities per stage (K' = 64 = one 128 B row)
constexpr int kKrGroupWarps = 4;
constexpr int kKrTmaWarp = 20;
constexpr int kKrMmaWarp = 21;
constexpr int kKrInWarp = 22;
constexpr int kKrThreads = 23 * 32;
constexpr int kKrAhead = 12;          // stages between an L2 prefetch and its copy
constexpr uint32_t kKrATile = 128 * 128;   // 128 positions x 64 visibilities x 2 B
constexpr uint32_t kKrBTile = 256 * 128;   // 256 twiddle rows x 64 visibilities x 2 B
constexpr uint32_t kKrInSlot = kKrKS * 8;  // uv per stage

// Real weights: one A tile, 256 cosine rows (48 KB stages, 4 deep).  Complex weights: A
// tiles of Re w and -Im w, 128 cosine and 128 sine rows (64 KB stages, 3 deep).
template <int REAL>
struct KrShape {
    static constexpr int kStages = REAL ? 4 : 3;    // one generator group per slot
    static constexpr int kFoldWarp0 = kStages * kKrGroupWarps;
    static constexpr int kFoldWarps = kKrTmaWarp - kFoldWarp0;   // 4 or 8
    // stages per accumulation run, a multiple of the ring depth: about 4096 visibilities
    // with real and 2048 with complex weights.  The tensor core's FP32 accumulation loses
    // some 2^-24.5 of the running value per MMA, and runs of twice that length doubled the
    // error of the exact cutouts (1.0e-5 -> 1.8e-5 of their 2-norm).
    static constexpr int kFoldStages = (REAL ? 64 : 32) / kStages * kStages;
    static constexpr uint32_t kA = REAL ? kKrATile : 2 * kKrATile;
    static constexpr int kRuns = REAL ? 8 : 4;   // 32-pixel runs per tile
    // roles that read each item index from the ring: the generator and fold warps, the MMA
    // issuer and the uv ring (one arrival each)
    static constexpr int kReaders = kKrTmaWarp + 1 + 1;
    static constexpr uint32_t kSmem = kStages * (kA + kKrBTile) + kKrIn * kKrInSlot + 512 + 1024;
    static_assert(kStages <= kKrIn && kFoldWarp0 % 4 == 0 && kFoldWarps % 4 == 0, "warp roles");
    static_assert((2 * kStages + 2 * kKrIn + 3 + 5) * 8 + 2 * 4 + 8 <= 512, "barrier block exceeds its reserve");
};

// Representative pixels of an N x N cutout (N a multiple of 32), in 32-pixel runs: the rows
// j >= N/2 (N^2/64 runs along l), row 0 (N/32 runs along l), and column 0 (runs along m
// from j = 0; of these only 1 <= j < N/2 are written).
struct KrRun {
    int i0, j0, along_m;
};
__device__ __forceinline__ KrRun kr_run(int r, int N) {
    const int per_row = N / 32, main_runs = (N / 2) * per_row;
    if (r < main_runs) return KrRun{32 * (r % per_row), N / 2 + r / per_row, 0};
    r -= main_runs;
    if (r < per_row) return KrRun{32 * r, 0, 0};
    return KrRun{0, 32 * (r - per_row), 1};
}

__device__ __forceinline__ void cis2(float2 x, float2 &re, float2 &im) {   // exp(2 pi i x) of two phases in turns
    __sincosf(6.28318530717958647f * (x.x - nearest(x.x)), &im.x, &re.x);
    __sincosf(6.28318530717958647f * (x.y - nearest(x.y)), &im.y, &re.y);
}

// (ar + i ai)(br + i bi) for two visibilities at a time; nbi = -bi.
__device__ __forceinline__ float2 mul_re(float2 ar, float2 ai, float2 br, float2 nbi) {
    return __ffma2_rn(ar, br, __fmul2_rn(ai, nbi));
}
__device__ __forceinline__ float2 mul_im(float2 ar, float2 ai, float2 br, float2 bi) {
    return __ffma2_rn(ar, bi, __fmul2_rn(ai, br));
}

// Step phasor and 16-pixel stride of a run's direction, visibilities (a, b) of the lane.
struct KrSteps {
    float2 sr, si, tr, ti;
};
__device__ __forceinline__ KrSteps kr_steps(float2 th) {
    KrSteps S;
    step_phasor(th.x, S.sr.x, S.si.x);
    step_phasor(th.y, S.sr.y, S.si.y);
    const float2 f = make_float2(th.x - nearest(th.x), th.y - nearest(th.y));
    cis2(make_float2(16.0f * f.x, 16.0f * f.y), S.tr, S.ti);
    return S;
}

template <int BF16, int ROW>
__device__ __forceinline__ void kr_row(const uint32_t (&addr)[8], const float2 (&x)[4]) {
    const uint32_t v0 = pack2<BF16>(x[0].x, x[0].y), v1 = pack2<BF16>(x[1].x, x[1].y);
    const uint32_t v2 = pack2<BF16>(x[2].x, x[2].y), v3 = pack2<BF16>(x[3].x, x[3].y);
    stmatrix_x4_at<ROW * 128>(addr[ROW & 7], v0, v1, v2, v3);
}

// Rows 0 .. 15 of four 16-pixel pieces (one stream per stmatrix matrix), from their rows 7
// and 8 outwards: x_{n+1} = C x_n - x_{n-1}, C = 2 cos(step), one packed FMA per pixel and
// two visibilities (a complex step takes four), at most eight steps from a seed, so that
// rounding grows by less than ten.  The subtraction is left to the output: the rows are
// carried as y = +-x with the signs + - - + + - - + ... (row_sign), for which every step is
// y = (+-C) y + y.
template <int BF16>
__device__ __forceinline__ void kr_chain(const uint32_t (&addr)[8], const float2 (&x7)[4], const float2 (&x8)[4],
                                         const float2 (&C)[4]) {
    float2 fp[4], fc[4], bp[4], bc[4];
    kr_row<BF16, 7>(addr, x7);
    kr_row<BF16, 8>(addr, x8);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        fp[m] = x7[m];
        fc[m] = x8[m];
        bp[m] = x8[m];
        bc[m] = x7[m];
    }
#define KR_STEP(F, B, SGN)                                                          \
    {                                                                               \
        _Pragma("unroll") for (int m = 0; m < 4; ++m) {                             \
            const float2 c = SGN ? C[m] : neg2(C[m]);                               \
            const float2 f = __ffma2_rn(c, fc[m], fp[m]);                           \
            const float2 b = __ffma2_rn(c, bc[m], bp[m]);                           \
            fp[m] = fc[m];                                                          \
            fc[m] = f;                                                              \
            bp[m] = bc[m];                                                          \
            bc[m] = b;                                                              \
        }                                                                           \
        kr_row<BF16, F>(addr, fc);                                                  \
        kr_row<BF16, B>(addr, bc);                                                  \
    }
    KR_STEP(9, 6, 0)
    KR_STEP(10, 5, 1)
    KR_STEP(11, 4, 0)
    KR_STEP(12, 3, 1)
    KR_STEP(13, 2, 0)
    KR_STEP(14, 1, 1)
#undef KR_STEP
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        fc[m] = __ffma2_rn(neg2(C[m]), fc[m], fp[m]);
        bc[m] = __ffma2_rn(neg2(C[m]), bc[m], bp[m]);
    }
    kr_row<BF16, 15>(addr, fc);
    kr_row<BF16, 0>(addr, bc);
}

// A run's constants: the phase of its row 7 is tu cu + tv cv (turns), its step tu or tv.
struct KrRunC {
    float cu, cv;
    bool along_m;
};
__device__ __forceinline__ KrRunC kr_run_const(int r, int N) {
    const KrRun run = kr_run(r, N);
    return KrRunC{(float)(run.i0 - N / 2 + (run.along_m ? 0 : 7)), (float)(run.j0 - N / 2 + (run.along_m ? 7 : 0)),
                  run.along_m != 0};
}

// Seeds of this warp's four streams for one stage.  Real weights: the 64 cosine rows of two
// runs, two pieces each; complex weights: the two pieces of one run's 32 cosine rows and of
// its sine rows.  uv = (u, v) of the lane's two visibilities.
template <int REAL>
__device__ __forceinline__ void kr_seeds(float4 uv, float cell, const KrRunC (&run)[2], float2 (&x7)[4],
                                         float2 (&x8)[4], float2 (&C)[4]) {
    const float2 tu = make_float2(uv.x * cell, uv.z * cell), tv = make_float2(uv.y * cell, uv.w * cell);
    KrSteps S = kr_steps(run[0].along_m ? tv : tu);
#pragma unroll
    for (int h = 0; h < (REAL ? 2 : 1); ++h) {
        if (h == 1 && run[1].along_m != run[0].along_m) S = kr_steps(run[1].along_m ? tv : tu);
        float2 zr, zi;
        cis2(make_float2(fmaf(tu.x, run[h].cu, tv.x * run[h].cv), fmaf(tu.y, run[h].cu, tv.y * run[h].cv)), zr, zi);
        const float2 nsi = neg2(S.si), nti = neg2(S.ti);
        const float2 yr = mul_re(zr, zi, S.tr, nti), yi = mul_im(zr, zi, S.tr, S.ti);   // second piece
        const float2 c2 = make_float2(2.0f * S.sr.x, 2.0f * S.sr.y);
        x7[2 * h] = zr;
        x7[2 * h + 1] = yr;
        x8[2 * h] = mul_re(zr, zi, S.sr, nsi);
        x8[2 * h + 1] = mul_re(yr, yi, S.sr, nsi);
        C[2 * h] = C[2 * h + 1] = c2;
        if (!REAL) {
            x7[2] = zi;
            x7[3] = yi;
            x8[2] = mul_im(zr, zi, S.sr, S.si);
            x8[3] = mul_im(yr, yi, S.sr, S.si);
            C[2] = C[3] = c2;
        }
    }
}

template <int BF16, int REAL>
__global__ void __launch_bounds__(kKrThreads, 1)
    k_psf_kr(const uint8_t *__restrict__ wblocks, int64_t nblk, const KrItem *__restrict__ items, int nitems,
             int *__restrict__ queue, const float2 *__restrict__ uv, int32_t kchunk0, float cell,
             const int64_t *__restrict__ out_off, float *__restrict__ out, int *err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    using Sh = KrShape<REAL>;
    constexpr int kStages = Sh::kStages;
    uint8_t *a_base = smem;
    uint8_t *b_base = smem + kStages * Sh::kA;
    uint8_t *in_base = b_base + kStages * kKrBTile;
    uint64_t *full = (uint64_t *)(in_base + kKrIn * kKrInSlot);
    uint64_t *empty = full + kStages;
    uint64_t *in_full = empty + kStages;
    uint64_t *in_empty = in_full + kKrIn;
    uint64_t *acc_full = in_empty + kKrIn;
    uint64_t *acc_empty = acc_full + 1;
    uint64_t *done_bar = acc_empty + 1;
    uint64_t *item_full = done_bar + 1;    // [2]: the item index of ring slot written
    uint64_t *item_empty = item_full + 2;  // [2]: every role has read it
    uint64_t *item_done = item_empty + 2;  // the fold warps have finished an item
    int *s_item = (int *)(item_done + 1);   // [2]
    uint32_t *s_tmem = (uint32_t *)(s_item + 2);
    volatile int *s_abort = (volatile int *)(s_tmem + 1);
    volatile int no_abort = 0;   // teardown waits ignore the abort flag

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int KS = kKrKS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], kKrGroupWarps + 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kKrIn; ++s) {
            mbar_init(&in_full[s], 1);
            mbar_init(&in_empty[s], kKrGroupWarps);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, Sh::kFoldWarps);
        mbar_init(done_bar, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&item_full[b], 1);
            mbar_init(&item_empty[b], Sh::kReaders);
        }
        mbar_init(item_done, Sh::kFoldWarps);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kKrMmaWarp) {
        tmem_alloc(s_tmem, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;   // columns [0, 256): active accumulators, [256, 512): running sums

    // Every role walks the same item sequence from the two-slot ring: the li-th item of
    // this CTA is in slot li & 1; a role reads it, acknowledges (item_empty) and keeps the
    // index in registers.  item < 0 ends the sequence.
    auto next_item = [&](int li, bool ack) -> int {
        const int slot = li & 1;
        if (!wait_bounded(&item_full[slot], (uint32_t)(li >> 1) & 1u, s_abort, err)) return -2;
        const int item = *(volatile int *)&s_item[slot];
        if (ack) mbar_arrive(&item_empty[slot]);
        return item;
    };
    auto item_stages = [&](const KrItem &it) { return (it.ke - it.kb + KS - 1) / KS; };

    if (warp < Sh::kFoldWarp0) {
        // ------------------------------------------------------------ pixel twiddles
        const int grp = warp / kKrGroupWarps, gw = warp % kKrGroupWarps;   // group = operand slot
        // stmatrix lane address: matrix m = lane / 8 is stream m (piece m of the warp's 64
        // rows, or with complex weights the two pieces of 32 cosine rows and of the sine rows
        // 128 further), 16-byte chunk lane % 8; row n of a piece adds n * 128 and swaps the
        // chunk by n mod 8
        const uint32_t lane_off =
            (REAL ? (uint32_t)(gw * 64 + 16 * (lane >> 3))
                  : (uint32_t)(gw * 32 + 16 * ((lane >> 3) & 1) + 128 * (lane >> 4))) * 128u + ((uint32_t)(lane & 7) << 4);
        const uint32_t dst = smem_u32(b_base + grp * kKrBTile) + lane_off;
        int g0 = 0;          // global index of the current item's first stage
        uint32_t uses = 0;   // stages this group has written
        bool ok = true;
        for (int li = 0; ok; ++li) {
            int item = -2;
            if (lane == 0) item = next_item(li, true);
            item = __shfl_sync(0xffffffffu, item, 0);
            if (item < 0) { ok = item == -1; break; }
            const KrItem it = items[item];
            const int nst = item_stages(it);
            const int r0 = it.q0 / 32 + gw * (REAL ? 2 : 1);   // this warp's first run
            const KrRunC run[2] = {kr_run_const(r0, it.N), kr_run_const(r0 + 1, it.N)};
            for (int s = grp; s < nst; s += kStages, ++uses) {
                const int g = g0 + s;
                const int islot = g % kKrIn;
                if (!wait_uniform(&in_full[islot], (uint32_t)(g / kKrIn) & 1u, s_abort, err)) { ok = false; break; }
                const float4 uv2 = reinterpret_cast<const float4 *>(in_base + islot * kKrInSlot)[lane];
                float2 x7[4], x8[4], C[4];
                kr_seeds<REAL>(uv2, cell, run, x7, x8, C);
                if (uses > 0 && !wait_uniform(&empty[grp], (uses - 1) & 1u, s_abort, err)) { ok = false; break; }
                uint32_t addr[8];
#pragma unroll
                for (int n = 0; n < 8; ++n) addr[n] = dst ^ ((uint32_t)n << 4);
                kr_chain<BF16>(addr, x7, x8, C);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&full[grp]);
                    // The uv slot is released only now, behind the proxy fence above: its refill is a
                    // write of the async proxy, and that fence is what orders the generic reads of the
                    // slot before it.  Released right after the reads, with no fence between, one
                    // 32-pixel run of one stage was wrong in up to half of the calls with many short
                    // items; none of 2000 such calls since.
                    mbar_arrive(&in_empty[islot]);
                }
            }
            g0 += nst;
        }
    } else if (warp == kKrTmaWarp) {
        // ------------------------------------------------------------ items and weight tiles
        if (lane == 0) {
            uint32_t used_bits = 0, phase_bits = 0;   // per slot: used before; parity of its last release
            for (int li = 0;; ++li) {
                const int islot = li & 1;
                if (li >= 2 && !wait_bounded(&item_empty[islot], (uint32_t)((li >> 1) - 1) & 1u, s_abort, err)) break;
                // Items do not overlap in the pipeline: the next one is published once the
                // fold warps have written the previous one out (a ring refill per item, counted
                // in kr_ranges' item cost).
                if (li >= 1 && !wait_bounded(item_done, (uint32_t)(li - 1) & 1u, s_abort, err)) break;
                const int idx = atomicAdd(queue, 1);   // largest items first (host order)
                const int item = idx < nitems ? idx : -1;
                s_item[islot] = item;
                mbar_arrive(&item_full[islot]);   // release: the index is visible to the waiters
                if (item < 0) break;
                const KrItem it = items[item];
                const int nst = item_stages(it);
                const uint8_t *src = wblocks + ((int64_t)(it.wrow / 128) * nblk + (it.kb - kchunk0) / KS) * Sh::kA;
                bool stop = false;
                for (int s = 0; s < nst; ++s) {
                    const int slot = s % kStages;
                    const uint32_t used = (used_bits >> slot) & 1u, ph = (phase_bits >> slot) & 1u;
                    if (used && !wait_bounded(&empty[slot], ph, s_abort, err)) { stop = true; break; }
                    if (used) phase_bits ^= 1u << slot;
                    used_bits |= 1u << slot;
                    mbar_arrive_expect_tx(&full[slot], Sh::kA);
                    // With complex weights (three slots, twice the bytes) the copies' latency shows: one CTA
                    // per tile row brings later stages into L2 (contraction of 256 x 64^2 exact 22.6 ->
                    // 21.7 ms; with real weights 57.5 -> 61 ms, so not there).
                    if (!REAL && it.q0 == 0 && s + kKrAhead < nst) bulk_prefetch_l2(src + (int64_t)(s + kKrAhead) * Sh::kA, Sh::kA);
                    bulk_g2s(a_base + slot * Sh::kA, src + (int64_t)s * Sh::kA, Sh::kA, &full[slot]);
                }
                if (stop) break;
            }
        }
        __syncwarp();
    } else if (warp == kKrMmaWarp) {
        // ------------------------------------------------------------ MMA issue
        {
            // warp-uniform issue path (umma_f16_x4): slot and phase by increment, descriptors
            // by adding the slot offset to the address field
            const uint32_t el = elect_one();
            const uint32_t ad0 = warp_uniform(desc_lo(smem_u32(a_base)));
            const uint32_t bd0 = warp_uniform(desc_lo(smem_u32(b_base)));
            const uint32_t tm0 = warp_uniform(tmem);
            uint32_t phase_bits = 0, folds = 0;   // per slot: parity of its next full phase
            bool stop = false;
            for (int li = 0; !stop; ++li) {
                int item = next_item(li, lane == 0);
                __syncwarp();
                item = __shfl_sync(0xffffffffu, item, 0);
                if (item < 0) break;
                const KrItem it = items[item];
                const int nst = (int)warp_uniform((uint32_t)item_stages(it));
                const uint32_t idesc = warp_uniform(idesc_f16(128, it.npx, BF16));
                for (int s0 = 0, in_acc = 0; s0 < nst && !stop; s0 += kStages) {
                    if (in_acc == 0 && folds > 0 && !wait_uniform(acc_empty, (folds - 1) & 1u, s_abort, err)) {
                        stop = true;
                        break;
                    }
#pragma unroll
                    for (int j = 0; j < kStages; ++j) {
                        if (s0 + j >= nst || stop) break;
                        if (!wait_uniform(&full[j], (phase_bits >> j) & 1u, s_abort, err)) { stop = true; break; }
                        tc_fence_after();
                        const uint32_t ad = ad0 + (uint32_t)j * (Sh::kA >> 4), bd = bd0 + (uint32_t)j * (kKrBTile >> 4);
                        const uint32_t acc = j ? 1u : (in_acc ? 1u : 0u);
                        umma_f16_x4(tm0, ad, bd, idesc, acc, el);
                        if (!REAL)   // -Im w against the sine rows, columns 128 ..
                            umma_f16_x4(tm0 + 128u, ad + (kKrATile >> 4), bd + (128u * 128u >> 4), idesc, acc, el);
                        umma_commit_elected(&empty[j], el);
                    }
                    phase_bits ^= (1u << min(kStages, nst - s0)) - 1u;
                    in_acc += kStages;
                    if (in_acc == Sh::kFoldStages || s0 + kStages >= nst) {
                        umma_commit_elected(acc_full, el);
                        ++folds;
                        in_acc = 0;
                    }
                }
            }
            umma_commit_elected(done_bar, el);
            wait_bounded(done_bar, 0, &no_abort, err);   // even after an abort (time-limited)
        }
        __syncwarp();
    } else if (warp == kKrInWarp) {
        // ------------------------------------------------------------ uv input ring
        if (lane == 0) {
            int g = 0, issued = 0;
            bool stop = false;
            for (int li = 0; !stop; ++li) {
                const int item = next_item(li, true);
                if (item < 0) break;
                const KrItem it = items[item];
                const int nst = item_stages(it);
                for (int s = 0; s < nst; ++s, ++g) {
                    const int islot = g % kKrIn;
                    if (g >= kKrIn && !wait_bounded(&in_empty[islot], (uint32_t)(g / kKrIn - 1) & 1u, s_abort, err)) {
                        stop = true;
                        break;
                    }
                    mbar_arrive_expect_tx(&in_full[islot], KS * 8);
                    bulk_g2s(in_base + islot * kKrInSlot, uv + it.kb + s * KS, KS * 8, &in_full[islot]);
                    issued = g + 1;
                }
            }
            // every copy has landed before the CTA exits (the last use of each slot)
            for (int q = max(0, issued - kKrIn); q < issued; ++q)
                wait_bounded(&in_full[q % kKrIn], (uint32_t)(q / kKrIn) & 1u, &no_abort, err);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ fold / output
        const int qw = warp & 3;                                // TMEM lane quarter
        constexpr int kParts = Sh::kFoldWarps / 4;              // the tile's pixels, in this many parts
        constexpr int kPart = 32 * Sh::kRuns / kParts;
        const int p0 = (warp - Sh::kFoldWarp0) / 4 * kPart;     // this warp's first pixel
        const int row = qw * 32 + lane;              // position row of the tile
        const uint32_t ta = tmem + ((uint32_t)(qw * 32) << 16);
        int F = 0;   // global fold range index
        bool ok = true;
        for (int li = 0; ok; ++li) {
            int item = -2;
            if (lane == 0) item = next_item(li, true);
            item = __shfl_sync(0xffffffffu, item, 0);
            if (item < 0) break;
            const KrItem it = items[item];
            const int nfold = (item_stages(it) + Sh::kFoldStages - 1) / Sh::kFoldStages;
            const bool row_ok = row < it.npos;
            const int N = it.N;
            float *dst = out + (row_ok ? out_off[it.slot0 + row] : 0);
            for (int f = 0; f < nfold; ++f, ++F) {
                const bool w = wait_bounded(acc_full, (uint32_t)F & 1u, s_abort, err);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                tc_fence_after();
                const bool last = (f == nfold - 1);
                if (!last) {   // running sum (+)= accumulator, 32 columns at a time
                    const int c_end = min(it.npx, p0 + kPart);
#pragma unroll 1
                    for (int h = 0; h < (REAL ? 1 : 2); ++h)
#pragma unroll 1
                        for (int c0 = p0; c0 < c_end; c0 += 32) {
                            const uint32_t tc0 = ta + (uint32_t)(c0 + 128 * h);
                            uint32_t v[32], u[32];
                            tmem_ld32_issue(tc0, v);
                            if (f > 0) {
                                tmem_ld32_issue(tc0 + 256u, u);
                                tmem_wait_ld(v, u);
#pragma unroll
                                for (int e = 0; e < 32; ++e)
                                    v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(u[e]));
                            } else {
                                tmem_wait_ld(v, v);
                            }
                            tmem_st32_issue(tc0 + 256u, v);
                        }
                    tmem_wait_st();
                }
                // the end: columns c0 .. c0 + 15 (E) and, with complex weights, 128 + c0 .. (O)
                for (int c0 = p0; last && c0 < min(it.npx, p0 + kPart); c0 += 16) {
                    float v[REAL ? 1 : 2][16];
#pragma unroll
                    for (int h = 0; h < (REAL ? 1 : 2); ++h) {
                        const uint32_t tc0 = ta + (uint32_t)(c0 + 128 * h);
                        tmem_ld16(tc0, v[h]);
                        if (f > 0) {
                            float sacc[16];
                            tmem_ld16(tc0 + 256u, sacc);
#pragma unroll
                            for (int e = 0; e < 16; ++e) v[h][e] += sacc[e];
                        }
                    }
                    if (!row_ok) continue;
                    // pixel E + O, reflected pixel E - O (kr_run's order of pixels; a chunk of 16
                    // lies in one run)
                    const int q = it.q0 + c0;
                    const KrRun run = kr_run(q / 32, N);
                    const int t0 = q & 31;
                    const int pix = run.j0 * N + run.i0 + (run.along_m ? t0 * N : t0);
                    const int pstep = run.along_m ? N : 1;
                    const bool mirrored = !run.along_m && run.j0 > N / 2;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float E = row_sign(e) * v[0][e], O = REAL ? 0.f : row_sign(e) * v[REAL ? 0 : 1][e];
                        const int j = run.j0 + t0 + e;
                        if (!run.along_m || (j >= 1 && j < N / 2)) atomicAdd(dst + pix + e * pstep, E + O);
                        if (mirrored && run.i0 + t0 + e >= 1) atomicAdd(dst + N * N + N - pix - e, E - O);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty);
            }
            __syncwarp();
            if (ok && lane == 0) mbar_arrive(item_done);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kKrMmaWarp) tmem_dealloc(tmem, 512);
}

}  // namespace

template <int BF16, int REAL>
static cudaError_t launch_kr_t(const void *w16, int64_t nblk, const KrItem *items, int nitems, int *queue, int nctas,
                               const float2 *uv, int32_t kchunk0, float cell, const int64_t *out_off, float *out,
                               int *err, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_psf_kr<BF16, REAL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)KrShape<REAL>::kSmem);
    if (e != cudaSuccess) return e;
    k_psf_kr<BF16, REAL><<<nctas, kKrThreads, KrShape<REAL>::kSmem, st>>>((const uint8_t *)w16, nblk, items, nitems, queue, uv, kchunk0, cell,
                                                                   out_off, out, err);
    return cudaGetLastError();
}

cudaError_t launch_psf_kr(const void *w16, int64_t nblk, const KrItem *items, int nitems, int *queue, int nctas, const float2 *uv,
                          int32_t kchunk0, float cell, const int64_t *out_off, float *out, int bf16, int real, int *err,
                          cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    nctas = std::max(1, std::min(nctas, nitems));
    cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    if (bf16)
        return real ? launch_kr_t<1, 1>(w16, nblk, items, nitems, queue, nctas, uv, kchunk0, cell, out_off, out, err, st)
                    : launch_kr_t<1, 0>(w16, nblk, items, nitems, queue, nctas, uv, kchunk0, cell, out_off, out, err, st);
    return real ? launch_kr_t<0, 1>(w16, nblk, items, nitems, queue, nctas, uv, kchunk0, cell, out_off, out, err, st)
                : launch_kr_t<0, 0>(w16, nblk, items, nitems, queue, nctas, uv, kchunk0, cell, out_off, out, err, st);
}

// 2-D tensor map over a FP16/BF16 matrix: dim0 = pitch elements, dim1 = rows; box 64 x 128
// elements (one 128-byte-swizzled stage of 128 rows).
int make_weight_map(void *map_out, void *w16, int bf16, int64_t pitch_elems, int64_t rows) {
    typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !ptr) {
            cudaGetLastError();
            return PSF_ECUDA;
        }
        fn = (EncodeFn)ptr;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)pitch_elems, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)pitch_elems * 2};
    const cuuint32_t box[2] = {64, 128};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = fn((CUtensorMap *)map_out, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                    w16, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? PSF_OK : PSF_ECUDA;
}

int kr_tile_pixels(int real) { return 32 * (real ? KrShape<1>::kRuns : KrShape<0>::kRuns); }

// Representative pixels of an N x N cutout in the order of kr_run (a multiple of 32).
int kr_pixels(int N) { return N * N / 2 + N + (N / 2 + 31) / 32 * 32; }

}  // namespace psf
