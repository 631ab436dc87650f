// Adjoint (vector-Jacobian product) of the cutout map of Eqs. 21-22 on the tensor cores.
//
// For a cotangent R = dL/dP (packed like the forward output) and positions p of one
// cutout size N, the adjoint needs per (position, visibility)
//   H_pk = sum_q R_p[q] exp(2 pi i (u_k dl_i + v_k dm_j)),   pixel q = j N + i,
// and then dL/dW_k = sum_p Re(D_k(l0_p) H_pk), dL/dl0_p = sum_k W_k Re(dD_k/dl0 H_pk)
// (likewise m0).  H is a GEMM: M = positions, N = visibilities (real and imaginary
// parts), K = pixels, with the pixel twiddles KR_k[q] generated on chip.
//
//   k_adj_r16   R (FP32, packed cutouts) -> a FP16/BF16 matrix [position row][pixel] of
//               one size group (rows padded to 128 with zeros): the TMA-loaded A operand;
//   k_adj_tc    one CTA per SM, looping over (128-position tile, 128-visibility tile)
//               items of a visibility chunk; per item the K loop runs over the N^2
//               pixels in 64-pixel stages.  Warps 0-15 (four groups on stages s mod 4):
//               each lane of a group owns one visibility of the item and writes its
//               twiddles for the stage's 64 pixels -- two 32-pixel runs along a cutout
//               row, phasor recurrences from a MUFU seed per run -- as the B operand rows
//               (Re KR_k: rows 0-127, Im KR_k: rows 128-255; K-major, 128-byte swizzle);
//               warp 20 loads the R tile of each stage by 2-D TMA; warp 21 issues
//               tcgen05.mma (M = 128, N = 256, K = 16) into one of two TMEM accumulators
//               (items alternate); warps 16-19 write the finished accumulator as
//               H[row][k] = (Re, Im) float32 pairs while the next item accumulates;
//   k_adj_fold  grid-stride over the visibilities of the chunk, one thread per visibility
//               at a time: D and its gradient for every position (the decorrelation of
//               the plan's method), dL/dW_k summed over positions (one write per
//               visibility), dL/d(l0, m0) summed per warp in shared memory, then per block;
//   k_adj_sum   the per-block position sums added in float64 (and over chunks).
// Every barrier wait is bounded (2 s); on expiry the CTA raises the error flag, stops,
// waits (bounded) for its copies in flight and issued MMAs and frees TMEM.
#include "decorr.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>

#include <algorithm>

namespace psf {
namespace {
using namespace tc;

constexpr int kAdjS = 4;              // operand ring depth
constexpr int kAdjGroups = 4;         // generator groups (stages s mod 4)
constexpr int kAdjGroupWarps = 4;     // one lane per visibility of the 128-visibility tile
constexpr int kAdjEpiWarp0 = 16;
constexpr int kAdjTmaWarp = 20;
constexpr int kAdjMmaWarp = 21;
constexpr int kAdjThreads = 22 * 32;
static_assert(kAdjGroups == kAdjS, "one generator group per operand slot");
constexpr uint32_t kAdjATile = 128 * 128;   // 128 positions x 64 pixels x 2 B
constexpr uint32_t kAdjBTile = 256 * 128;   // 256 rows (Re, Im of 128 visibilities) x 64 pixels x 2 B
constexpr uint32_t kAdjSmem = kAdjS * (kAdjATile + kAdjBTile) + 256 + 1024;

// 32 pixels of one cutout row for this lane's visibility, pixel offsets i = i0 .. i0+31:
// z(i) = exp(2 pi i (tu (i0 - N/2 + i') + tv (j - N/2))), written as FP16/BF16 into the
// lane's real row (re_row) and imaginary row (im_row) at the 16-byte chunks c0 .. c0+3
// (8 pixels per chunk).  Four 8-pixel pieces from one MUFU seed, two at a time.
template <int BF16>
__device__ __forceinline__ void adj_run32(uint32_t re_row, uint32_t im_row, int row, int c0, float tu, float tv,
                                          int i0, int j, int half, float2 st, float2 st8, float2 st16) {
    const float2 z0 = cis_turns(fmaf(tu, (float)(i0 - half), tv * (float)(j - half)));
    const float2 sr = make_float2(st.x, st.x), si = make_float2(st.y, st.y), nsi = make_float2(-st.y, -st.y);
    const uint32_t sw = (uint32_t)(row & 7);
    // pieces p = 0..3 start at pixels 8p; pieces (0, 1) and then (2, 3) run packed for FFMA2
#pragma unroll
    for (int pp = 0; pp < 2; ++pp) {
        const float2 za = pp ? cmulf(z0, st16) : z0;
        const float2 zb = cmulf(za, st8);
        float2 re = make_float2(za.x, zb.x), im = make_float2(za.y, zb.y), pre, pim;
        uint32_t wre[2][4], wim[2][4];   // [piece][word]
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (q & 1) {
                wre[0][q >> 1] = pack2<BF16>(pre.x, re.x);
                wre[1][q >> 1] = pack2<BF16>(pre.y, re.y);
                wim[0][q >> 1] = pack2<BF16>(pim.x, im.x);
                wim[1][q >> 1] = pack2<BF16>(pim.y, im.y);
            } else {
                pre = re;
                pim = im;
            }
            if (q < 7) {
                const float2 t = __fmul2_rn(im, nsi), u = __fmul2_rn(im, sr);
                im = __ffma2_rn(re, si, u);
                re = __ffma2_rn(re, sr, t);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t off = ((uint32_t)(c0 + 2 * pp + e) ^ sw) << 4;
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(re_row + off), "r"(wre[e][0]),
                         "r"(wre[e][1]), "r"(wre[e][2]), "r"(wre[e][3])
                         : "memory");
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(im_row + off), "r"(wim[e][0]),
                         "r"(wim[e][1]), "r"(wim[e][2]), "r"(wim[e][3])
                         : "memory");
        }
    }
}

template <int BF16>
__global__ void __launch_bounds__(kAdjThreads, 1)
    k_adj_tc(const __grid_constant__ CUtensorMap rmap, int ntile_pos, int ntile_vis, int N, const float2 *__restrict__ uv,
             int32_t kc0, int32_t kcn, float cell, float2 *__restrict__ H, int64_t ldh, int *err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *a_base = smem;
    uint8_t *b_base = smem + kAdjS * kAdjATile;
    uint64_t *full = (uint64_t *)(b_base + kAdjS * kAdjBTile);
    uint64_t *empty = full + kAdjS;
    uint64_t *acc_full = empty + kAdjS;     // [buffer]
    uint64_t *acc_empty = acc_full + 2;     // [buffer]
    uint64_t *done_bar = acc_empty + 2;
    uint32_t *s_tmem = (uint32_t *)(done_bar + 1);
    volatile int *s_abort = (volatile int *)(s_tmem + 1);
    volatile int no_abort = 0;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nitems = ntile_pos * ntile_vis;
    const int nst = N * N / 64;   // 64-pixel stages per item (N a multiple of 32: a multiple of 16)
    // this CTA's items: blockIdx.x, blockIdx.x + gridDim.x, ...
    const int my_items = blockIdx.x < nitems ? (nitems - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kAdjS; ++s) {
            mbar_init(&full[s], kAdjGroupWarps + 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        mbar_init(done_bar, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kAdjMmaWarp) {
        tmem_alloc(s_tmem, 512);   // two 256-column accumulators
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    const int half = N / 2;

    if (warp < kAdjGroups * kAdjGroupWarps) {
        // ------------------------------------------------------------ pixel twiddles
        const int grp = warp / kAdjGroupWarps;
        const int vrow = (warp % kAdjGroupWarps) * 32 + lane;   // visibility row of the tile
        const uint32_t bt = smem_u32(b_base + grp * kAdjBTile);   // the group's slot
        const uint32_t re_row = bt + (uint32_t)vrow * 128u, im_row = bt + (uint32_t)(128 + vrow) * 128u;
        const int dj = 64 * kAdjS / N, di = 64 * kAdjS % N;   // pixels between a group's stages
        uint32_t uses = 0;
        bool ok = true;
        for (int li = 0; li < my_items && ok; ++li) {
            const int vt = (blockIdx.x + li * gridDim.x) % ntile_vis;
            const int kk = vt * 128 + vrow;   // this lane's visibility and its pixel step
            const float2 uvk = kk < kcn ? uv[kc0 + kk] : make_float2(0.f, 0.f);
            const float tu = uvk.x * cell, tv = uvk.y * cell;
            const float2 st = cis_turns(tu);
            const float2 s2 = cmulf(st, st), s4 = cmulf(s2, s2);
            const float2 st8 = cmulf(s4, s4), st16 = cmulf(st8, st8);
            int j[2], i0[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                j[r] = (grp * 64 + r * 32) / N;
                i0[r] = grp * 64 + r * 32 - j[r] * N;
            }
            for (int s = grp; s < nst; s += kAdjS, ++uses) {
                if (uses > 0 && !wait_uniform(&empty[grp], (uses - 1) & 1u, s_abort, err)) { ok = false; break; }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    adj_run32<BF16>(re_row, im_row, vrow, 4 * r, tu, tv, i0[r], j[r], half, st, st8, st16);
                    j[r] += dj;
                    i0[r] += di;
                    if (i0[r] >= N) {
                        i0[r] -= N;
                        ++j[r];
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[grp]);
            }
        }
    } else if (warp == kAdjTmaWarp) {
        // ------------------------------------------------------------ R tiles
        if (lane == 0) {
            for (int g = 0; g < my_items * nst; ++g) {
                const int li = g / nst, s = g - li * nst;
                const int slot = g % kAdjS;
                if (g >= kAdjS && !wait_bounded(&empty[slot], (uint32_t)((g / kAdjS) & 1) ^ 1u, s_abort, err)) break;
                const int item = blockIdx.x + li * gridDim.x;
                const int pt = item / ntile_vis;
                mbar_arrive_expect_tx(&full[slot], kAdjATile);
                tma_load_2d(a_base + slot * kAdjATile, &rmap, s * 64, pt * 128, &full[slot]);
            }
        }
        __syncwarp();
    } else if (warp == kAdjMmaWarp) {
        // ------------------------------------------------------------ MMA issue
        {
            const uint32_t el = elect_one();
            const uint32_t idesc = idesc_f16(128, 256, BF16);
            const uint32_t ad0 = warp_uniform(desc_lo(smem_u32(a_base)));
            const uint32_t bd0 = warp_uniform(desc_lo(smem_u32(b_base)));
            const uint32_t tm0 = warp_uniform(tmem);
            // an item's stages are a multiple of the ring depth: one round per outer iteration,
            // unrolled over the slots (the issue path's instructions count, see k_kr.cu)
            uint32_t ph = 0;
            bool stop = false;
            for (int li = 0; li < my_items && !stop; ++li) {
                const int b = li & 1;
                // the epilogue has read this buffer's previous item (li - 2)
                if (li >= 2 && !wait_uniform(&acc_empty[b], (uint32_t)((li >> 1) - 1) & 1u, s_abort, err)) break;
                const uint32_t dt = tm0 + (uint32_t)b * 256u;
                for (int s0 = 0; s0 < nst && !stop; s0 += kAdjS, ph ^= 1u) {
#pragma unroll
                    for (int j = 0; j < kAdjS; ++j) {
                        if (!wait_uniform(&full[j], ph, s_abort, err)) { stop = true; break; }
                        tc_fence_after();
                        umma_f16_x4(dt, ad0 + (uint32_t)j * (kAdjATile >> 4), bd0 + (uint32_t)j * (kAdjBTile >> 4), idesc,
                                    (s0 | j) ? 1u : 0u, el);
                        umma_commit_elected(&empty[j], el);
                    }
                }
                if (!stop) umma_commit_elected(&acc_full[b], el);
            }
            umma_commit_elected(done_bar, el);
            wait_bounded(done_bar, 0, &no_abort, err);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue: TMEM -> H
        const int qw = warp - kAdjEpiWarp0;   // TMEM lane quarter
        const int row = qw * 32 + lane;       // position row of the tile
        for (int li = 0; li < my_items; ++li) {
            const int b = li & 1;
            const bool ok = wait_bounded(&acc_full[b], (uint32_t)(li >> 1) & 1u, s_abort, err);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            const int item = blockIdx.x + li * gridDim.x;
            const int pt = item / ntile_vis, vt = item - pt * ntile_vis;
            float2 *dst = H + (int64_t)(pt * 128 + row) * ldh + (int64_t)vt * 128;
            const uint32_t ta = tmem + ((uint32_t)(qw * 32) << 16) + (uint32_t)b * 256u;
            for (int c0 = 0; c0 < 128; c0 += 16) {
                float vr[16], vi[16];
                tmem_ld16(ta + (uint32_t)c0, vr);
                tmem_ld16(ta + 128u + (uint32_t)c0, vi);
#pragma unroll
                for (int e = 0; e < 16; e += 2)
                    *reinterpret_cast<float4 *>(dst + c0 + e) = make_float4(vr[e], vi[e], vr[e + 1], vi[e + 1]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kAdjMmaWarp) tmem_dealloc(tmem, 512);
}

// R of a size group -> FP16/BF16 rows: r16[row][q] = R[offs[row] + q] for row < npos,
// zero for the padding rows up to `rows`.
template <int BF16>
__global__ void __launch_bounds__(256) k_adj_r16(const float *__restrict__ R, const int64_t *__restrict__ offs,
                                                 int npos, int rows, int n2, uint16_t *__restrict__ r16) {
    const int row = blockIdx.y;
    for (int q = 2 * (blockIdx.x * blockDim.x + threadIdx.x); q < n2; q += 2 * gridDim.x * blockDim.x) {
        float a = 0.f, b = 0.f;
        if (row < npos) {
            a = R[offs[row] + q];
            b = R[offs[row] + q + 1];
        }
        *reinterpret_cast<uint32_t *>(r16 + (int64_t)row * n2 + q) = pack2<BF16>(a, b);
    }
    (void)rows;
}

struct AdjPosT {
    float4 L, dLl, dLm;   // direction (l0, m0, n0-1) and its derivatives
};

constexpr int kFoldThreads = 256;
constexpr int kFoldWarps = kFoldThreads / 32;

// Grid-stride over the visibilities k = kc0 + t of the chunk, one thread per visibility
// at a time: D_k(l0_p) and its gradient for every position p of the group,
// dL/dW_k (+)= sum_p Re(D H_pk) (one write per visibility), and per warp the sums of
// W_k Re(dD/dl0 H_pk), W_k Re(dD/dm0 H_pk) in shared memory [warp][p][2]; each block
// writes its per-position totals to partial[block][p][2].
template <bool FAST>
__global__ void __launch_bounds__(kFoldThreads) k_adj_fold(DevObs o, int method, uint32_t flags,
                                                           const AdjPosT *__restrict__ pos, int npos,
                                                           const float2 *__restrict__ H, int64_t ldh, int32_t kc0,
                                                           int32_t kcn, float *__restrict__ gW, int accumulate_gW,
                                                           double *__restrict__ partial) {
    extern __shared__ float red[];   // [kFoldWarps][npos][2]
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < kFoldWarps * npos * 2; e += kFoldThreads) red[e] = 0.f;
    __syncthreads();
    float *myred = red + (int64_t)wid * npos * 2;
    for (int64_t base = (int64_t)blockIdx.x * kFoldThreads; base < kcn; base += (int64_t)gridDim.x * kFoldThreads) {
        const int64_t t = base + threadIdx.x;
        const bool valid = t < kcn;
        const int32_t k = kc0 + (int32_t)(valid ? t : 0);
        const int bin = k / o.nout, r = k - bin * o.nout;
        const float Wk = valid ? o.W[k] : 0.f;
        float gw = 0.f;
        for (int p = 0; p < npos; ++p) {
            float gl = 0.f, gm = 0.f;
            if (valid) {
                const AdjPosT P = pos[p];
                float4 g;
                const float2 D = decorr<true, FAST>(o, method, flags, bin, r, P.L, P.dLl, P.dLm, &g);
                const float2 h = H[(int64_t)p * ldh + t];
                gw += D.x * h.x - D.y * h.y;
                gl = Wk * (g.x * h.x - g.y * h.y);
                gm = Wk * (g.z * h.x - g.w * h.y);
            }
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) {
                gl += __shfl_xor_sync(0xffffffffu, gl, sh);
                gm += __shfl_xor_sync(0xffffffffu, gm, sh);
            }
            if (lane == 0) {   // the warp's only writer of its row
                myred[2 * p] += gl;
                myred[2 * p + 1] += gm;
            }
        }
        if (valid && gW) gW[k] = accumulate_gW ? gW[k] + gw : gw;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < npos * 2; e += kFoldThreads) {
        double s = 0.0;
        for (int w = 0; w < kFoldWarps; ++w) s += red[(int64_t)w * npos * 2 + e];
        partial[(int64_t)blockIdx.x * npos * 2 + e] = s;
    }
}

// sinc_pi and its derivative together: for |y| <= 1/2 the Taylor series to order 12 in pi y
// and its derivative (truncation below 2e-8), else the general forms.
__device__ __forceinline__ void sinc_pair(float y, float *v, float *dv) {
    if (fabsf(y) <= 0.5f) {
        const float z = y * y;
        float q = fmaf(z, 1.4842879e-4f, -2.3460810e-3f), d = fmaf(z, 6.0f * 1.4842879e-4f, 5.0f * -2.3460810e-3f);
        q = fmaf(z, q, 2.6147848e-2f);
        d = fmaf(z, d, 4.0f * 2.6147848e-2f);
        q = fmaf(z, q, -1.9075182e-1f);
        d = fmaf(z, d, 3.0f * -1.9075182e-1f);
        q = fmaf(z, q, 8.1174243e-1f);
        d = fmaf(z, d, 2.0f * 8.1174243e-1f);
        q = fmaf(z, q, -1.6449341f);
        d = fmaf(z, d, -1.6449341f);
        *v = fmaf(z, q, 1.0f);
        *dv = 2.0f * y * d;
    } else {
        *v = sincpi_poly(y);
        *dv = dsincpi(y);
    }
}

// The exact method's fold with affine output channels (nu_r = nu_0 + r dnu, the boxcar):
// a thread owns one bin and eight consecutive channels (visibilities k0 .. k0 + 7).  Per raw
// sample s the channel-independent factor f = Dirichlet x sinc of X_s = uvw_s . L0, its
// derivative and the phasor e_s of the middle of the channels are evaluated once; with
// x_j = j - 7/2, r_s = -2 pi dnu ds / c, p_s the derivative of the middle phase, q_s that of r_s,
//   D_j       = (1/n) sum_s e^{i r x_j} e f
//   dD_j/dl0  = (1/n) sum_s e^{i r x_j} [e (df/dX X_l + i p f) + i x_j e f q]
// and with |r_s| <= kMomentMax for every sample (the limit of the exact weights) the moments
// in r of e f, of the bracket's first term (both to r^3) and of e f q (to r^2) give every
// channel; their product with the channels' W_k H_k needs only h_m = sum_j W_j H_j x_j^m / m!.
// Otherwise the channels are summed sample by sample (fold_general).  A bin's samples are
// kept in shared memory across the positions, one column per thread.  As eight channel
// recurrences per sample, records reread per position and the derivative of the sinc from
// sincospi, the fold took 4.9 ms for 96 positions x 3.5 M visibilities; 3.4 ms now.
constexpr int kFoldCap = 12;   // samples of a bin kept in shared memory
constexpr float kFoldMomentMax = 0.0143f;

struct FoldBin {
    float4 ub, ch;
    int2 sm;
    float inv;
};

// Sample by sample: D_j H_j, and this bin's share of dL/dl0, dL/dm0.
__device__ __noinline__ void fold_general(const DevObs &o, const FoldBin &B, const AdjPosT &P, const float4 *hp,
                                          const float *Wk, float *gw, float *gl_out, float *gm_out) {
    const float nu0 = B.ch.x, dnu = o.dnu_ch;
    const float Xbar = dot3(B.ub, P.L), Xbl = dot3(B.ub, P.dLl), Xbm = dot3(B.ub, P.dLm);
    float Dr[8], Di[8], Lr[8], Li[8], Mr[8], Mi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { Dr[j] = Di[j] = Lr[j] = Li[j] = Mr[j] = Mi[j] = 0.f; }
    for (int s = 0; s < B.sm.y; ++s) {
        const float4 d = o.samp[B.sm.x + s];
        const float ds = dot3(d, P.L), dsl = dot3(d, P.dLl), dsm = dot3(d, P.dLm);
        const float Xs = Xbar + ds, Xl = Xbl + dsl, Xm = Xbm + dsm;
        const float a = B.ch.z * Xs * kInvC, y = B.ch.w * Xs * kInvC;
        const float dir = dirichlet_fast(o.favg, a), sc = sincpi_fast(y);
        const float f = dir * sc;
        const float df = (ddirichlet(o.favg, a) * B.ch.z * sc + dir * dsincpi(y) * B.ch.w) * kInvC;
        const float al = df * Xl, am = df * Xm;                           // real parts
        const float pl0 = -2.0f * kPiF * nu0 * dsl * kInvC * f, pdl = -2.0f * kPiF * dnu * dsl * kInvC * f;
        const float pm0 = -2.0f * kPiF * nu0 * dsm * kInvC * f, pdm = -2.0f * kPiF * dnu * dsm * kInvC * f;
        float es, ec, rs, rc;
        sincospi2_fast(-nu0 * ds * kInvC, &es, &ec);
        sincospi2_fast(-dnu * ds * kInvC, &rs, &rc);
        float er = ec, ei = es;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            Dr[j] = fmaf(er, f, Dr[j]);
            Di[j] = fmaf(ei, f, Di[j]);
            const float bl = fmaf((float)j, pdl, pl0), bm = fmaf((float)j, pdm, pm0);   // imaginary parts
            Lr[j] += er * al - ei * bl;
            Li[j] += er * bl + ei * al;
            Mr[j] += er * am - ei * bm;
            Mi[j] += er * bm + ei * am;
            const float tr = er * rc - ei * rs;
            ei = er * rs + ei * rc;
            er = tr;
        }
    }
    float gl = 0.f, gm = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float4 h4 = hp[j >> 1];
        const float hr = (j & 1) ? h4.z : h4.x, hi = (j & 1) ? h4.w : h4.y;
        gw[j] += (Dr[j] * hr - Di[j] * hi) * B.inv;
        gl += Wk[j] * (Lr[j] * hr - Li[j] * hi) * B.inv;
        gm += Wk[j] * (Mr[j] * hr - Mi[j] * hi) * B.inv;
    }
    *gl_out = gl;
    *gm_out = gm;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 scale2(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
__device__ __forceinline__ float2 fma2(float2 a, float s, float2 c) { return __ffma2_rn(a, make_float2(s, s), c); }
__device__ __forceinline__ float re_mul(float2 a, float2 b) { return a.x * b.x - a.y * b.y; }   // Re(a b)
__device__ __forceinline__ float im_mul(float2 a, float2 b) { return a.x * b.y + a.y * b.x; }   // Im(a b)

__global__ void __launch_bounds__(kFoldThreads, 2)
    k_adj_fold_exact8(DevObs o, const AdjPosT *__restrict__ pos, int npos, const float2 *__restrict__ H, int64_t ldh,
                      int32_t kc0, int32_t kcn, float *__restrict__ gW, int accumulate_gW, double *__restrict__ partial) {
    extern __shared__ __align__(16) float4 fold_smem[];   // [kFoldCap][threads] samples, then [kFoldWarps][npos][2]
    float *const red = reinterpret_cast<float *>(fold_smem + kFoldCap * kFoldThreads);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < kFoldWarps * npos * 2; e += kFoldThreads) red[e] = 0.f;
    __syncthreads();
    float *myred = red + (int64_t)wid * npos * 2;
    float4 *const mys = fold_smem + threadIdx.x;
    const int64_t ngrp = (kcn + 7) / 8;
    for (int64_t base = (int64_t)blockIdx.x * kFoldThreads; base < ngrp; base += (int64_t)gridDim.x * kFoldThreads) {
        const int64_t gi = base + threadIdx.x;
        const bool valid = gi < ngrp;
        const int32_t t0 = (int32_t)(valid ? gi * 8 : 0);     // chunk-relative first visibility
        const int32_t k0 = kc0 + t0;                          // kc0 and nout are multiples of 8
        const int bin = k0 / o.nout, r0 = k0 - bin * o.nout;
        FoldBin B;
        B.ub = o.bin_ubar[bin];
        B.sm = o.bin_samp[bin];
        B.ch = o.chan[r0];
        B.inv = 1.0f / (float)B.sm.y;
        const float nu_mid = -(B.ch.x + 3.5f * o.dnu_ch) * kInvC, two_pi = 2.0f * kPiF;
        const float r1 = -two_pi * o.dnu_ch * kInvC, wy = B.ch.w * kInvC, wa = B.ch.z * kInvC;
        const bool cached = B.sm.y <= kFoldCap;
        if (cached)
            for (int s = 0; s < B.sm.y; ++s) mys[s * kFoldThreads] = o.samp[B.sm.x + s];   // read by this thread only
        float Wk[8], gw[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            Wk[j] = (valid && t0 + j < kcn) ? o.W[k0 + j] : 0.f;
            gw[j] = 0.f;
        }
        for (int p = 0; p < npos; ++p) {
            float gl = 0.f, gm = 0.f;
            if (valid) {
                const AdjPosT P = pos[p];
                const float Xbar = dot3(B.ub, P.L), Xbl = dot3(B.ub, P.dLl), Xbm = dot3(B.ub, P.dLm);
                const float2 zero = make_float2(0.f, 0.f);
                float2 M0 = zero, M1 = zero, M2 = zero, M3 = zero;                // of e f
                float2 A0 = zero, A1 = zero, A2 = zero, A3 = zero;                // of e (df/dX X_l + i p_l f)
                float2 C0 = zero, C1 = zero, C2 = zero, C3 = zero;                // the same for m0
                float2 B0 = zero, B1 = zero, B2 = zero, E0 = zero, E1 = zero, E2 = zero;   // of e f q_l, e f q_m
                float far = 0.f;
                for (int s = 0; s < B.sm.y; ++s) {
                    const float4 d = cached ? mys[s * kFoldThreads] : o.samp[B.sm.x + s];
                    const float ds = dot3(d, P.L), dsl = dot3(d, P.dLl), dsm = dot3(d, P.dLm);
                    const float Xs = Xbar + ds;
                    float f, df;
                    sinc_pair(wy * Xs, &f, &df);
                    df *= wy;
                    if (o.favg > 1) {
                        const float a = wa * Xs, dir = dirichlet_fast(o.favg, a);
                        df = dir * df + ddirichlet(o.favg, a) * wa * f;
                        f *= dir;
                    }
                    float es, ec;
                    cis_mufu(nu_mid * ds, &es, &ec);
                    const float r = r1 * ds, pf = two_pi * nu_mid * f;
                    far = fmaxf(far, fabsf(r));
                    float2 e = make_float2(ec * f, es * f);
                    float2 bl = scale2(e, r1 * dsl), bm = scale2(e, r1 * dsm);
                    M0 = add2(M0, e);
                    e = scale2(e, r);
                    M1 = add2(M1, e);
                    e = scale2(e, r);
                    M2 = add2(M2, e);
                    M3 = fma2(e, r, M3);
                    const float ul = df * (Xbl + dsl), vl = pf * dsl, um = df * (Xbm + dsm), vm = pf * dsm;
                    float2 al = make_float2(ec * ul - es * vl, ec * vl + es * ul);
                    float2 am = make_float2(ec * um - es * vm, ec * vm + es * um);
                    A0 = add2(A0, al);
                    C0 = add2(C0, am);
                    B0 = add2(B0, bl);
                    E0 = add2(E0, bm);
                    al = scale2(al, r);
                    am = scale2(am, r);
                    bl = scale2(bl, r);
                    bm = scale2(bm, r);
                    A1 = add2(A1, al);
                    C1 = add2(C1, am);
                    B1 = add2(B1, bl);
                    E1 = add2(E1, bm);
                    al = scale2(al, r);
                    am = scale2(am, r);
                    B2 = fma2(bl, r, B2);
                    E2 = fma2(bm, r, E2);
                    A2 = add2(A2, al);
                    C2 = add2(C2, am);
                    A3 = fma2(al, r, A3);
                    C3 = fma2(am, r, C3);
                }
                const float4 *hp = reinterpret_cast<const float4 *>(H + (int64_t)p * ldh + t0);
                if (far <= kFoldMomentMax) {
                    float2 h0 = zero, h1 = zero, h2 = zero, h3 = zero;   // sum_j W_j H_j x_j^m / m!
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float x = (float)j - 3.5f, x2 = 0.5f * x * x, x3 = x * x * x / 6.0f;
                        const float4 h4 = hp[j >> 1];
                        const float2 h = (j & 1) ? make_float2(h4.z, h4.w) : make_float2(h4.x, h4.y);
                        const float Dr = M0.x - x * M1.y - x2 * M2.x + x3 * M3.y;
                        const float Di = M0.y + x * M1.x - x2 * M2.y - x3 * M3.x;
                        gw[j] = fmaf(Dr * h.x - Di * h.y, B.inv, gw[j]);
                        const float2 wh = scale2(h, Wk[j]);
                        h0 = add2(h0, wh);
                        h1 = fma2(wh, x, h1);
                        h2 = fma2(wh, x2, h2);
                        h3 = fma2(wh, x3, h3);
                    }
                    // Re(sum_m i^m A_m h_m + i sum_m i^m (m + 1) B_m h_{m+1})
                    gl = B.inv * (re_mul(A0, h0) - im_mul(A1, h1) - re_mul(A2, h2) + im_mul(A3, h3) - im_mul(B0, h1) -
                                  2.0f * re_mul(B1, h2) + 3.0f * im_mul(B2, h3));
                    gm = B.inv * (re_mul(C0, h0) - im_mul(C1, h1) - re_mul(C2, h2) + im_mul(C3, h3) - im_mul(E0, h1) -
                                  2.0f * re_mul(E1, h2) + 3.0f * im_mul(E2, h3));
                } else {   // (fmaxf drops a NaN: such a sample is in the moments above, which are then NaN)
                    float wk[8], g8[8];   // copies: the arrays of the common path stay in registers
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        wk[j] = Wk[j];
                        g8[j] = gw[j];
                    }
                    float a, b;
                    fold_general(o, B, P, hp, wk, g8, &a, &b);
                    gl = a;
                    gm = b;
#pragma unroll
                    for (int j = 0; j < 8; ++j) gw[j] = g8[j];
                }
            }
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) {
                gl += __shfl_xor_sync(0xffffffffu, gl, sh);
                gm += __shfl_xor_sync(0xffffffffu, gm, sh);
            }
            if (lane == 0) {
                myred[2 * p] += gl;
                myred[2 * p + 1] += gm;
            }
        }
        if (valid && gW) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (t0 + j < kcn) gW[k0 + j] = accumulate_gW ? gW[k0 + j] + gw[j] : gw[j];
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < npos * 2; e += kFoldThreads) {
        double s = 0.0;
        for (int w = 0; w < kFoldWarps; ++w) s += red[(int64_t)w * npos * 2 + e];
        partial[(int64_t)blockIdx.x * npos * 2 + e] = s;
    }
}

// g_lm[2 idx[p] + d] (+)= sum over blocks of partial[block][p][d], in float64.
__global__ void __launch_bounds__(256) k_adj_sum(const double *__restrict__ partial, int nblk, int npos,
                                                 const int32_t *__restrict__ idx, int accumulate,
                                                 double *__restrict__ g_lm) {
    const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;   // one warp per element
    if (e >= npos * 2) return;
    double s = 0.0;
    for (int c = lane; c < nblk; c += 32) s += partial[(int64_t)c * npos * 2 + e];
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) s += __shfl_down_sync(0xffffffffu, s, sh);
    if (lane) return;
    const int64_t o = 2 * (int64_t)idx[e >> 1] + (e & 1);
    g_lm[o] = accumulate ? g_lm[o] + s : s;
}

}  // namespace

int adj_tc_smem_bytes() { return (int)kAdjSmem; }

cudaError_t launch_adj_r16(const float *R, const int64_t *offs, int npos, int rows, int n2, int bf16, void *r16,
                           cudaStream_t st) {
    dim3 grid((unsigned)std::max(1, std::min(64, (n2 / 2 + 255) / 256)), (unsigned)rows);
    if (bf16) k_adj_r16<1><<<grid, 256, 0, st>>>(R, offs, npos, rows, n2, (uint16_t *)r16);
    else k_adj_r16<0><<<grid, 256, 0, st>>>(R, offs, npos, rows, n2, (uint16_t *)r16);
    return cudaGetLastError();
}

cudaError_t launch_adj_tc(const void *rmap, int ntile_pos, int ntile_vis, int N, const float2 *uv, int32_t kc0,
                          int32_t kcn, float cell, float2 *H, int64_t ldh, int bf16, int nsm, int *err,
                          cudaStream_t st) {
    const int nitems = ntile_pos * ntile_vis;
    if (nitems <= 0) return cudaSuccess;
    const int grid = std::min(nitems, nsm);
    const CUtensorMap *m = (const CUtensorMap *)rmap;
    cudaError_t e;
    if (bf16) {
        e = cudaFuncSetAttribute(k_adj_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdjSmem);
        if (e != cudaSuccess) return e;
        k_adj_tc<1><<<grid, kAdjThreads, kAdjSmem, st>>>(*m, ntile_pos, ntile_vis, N, uv, kc0, kcn, cell, H, ldh, err);
    } else {
        e = cudaFuncSetAttribute(k_adj_tc<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdjSmem);
        if (e != cudaSuccess) return e;
        k_adj_tc<0><<<grid, kAdjThreads, kAdjSmem, st>>>(*m, ntile_pos, ntile_vis, N, uv, kc0, kcn, cell, H, ldh, err);
    }
    return cudaGetLastError();
}

int adj_fold_max_pos() { return 1024; }
int adj_fold_blocks(int nsm) { return 4 * nsm; }

cudaError_t launch_adj_fold(const DevObs &o, int method, uint32_t flags, const void *pos, int npos, const float2 *H,
                            int64_t ldh, int32_t kc0, int32_t kcn, float *gW, int accumulate_gW, double *partial,
                            const int32_t *idx, double *g_lm, int accumulate_lm, int fast, int nsm, cudaStream_t st) {
    if (npos <= 0 || npos > adj_fold_max_pos()) return cudaErrorInvalidValue;
    const int nblk = adj_fold_blocks(nsm);
    const size_t smem = (size_t)kFoldWarps * npos * 2 * sizeof(float);
    cudaError_t e;
    // H rows of 8-visibility groups read as float4 pairs: ldh, kc0 multiples of 8
    if (fast && method == kExact && o.chan_affine && o.nout % 8 == 0 && kc0 % 8 == 0 && ldh % 8 == 0) {
        const size_t smem8 = smem + (size_t)kFoldCap * kFoldThreads * sizeof(float4);
        e = cudaFuncSetAttribute(k_adj_fold_exact8, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem8);
        if (e != cudaSuccess) return e;
        k_adj_fold_exact8<<<nblk, kFoldThreads, smem8, st>>>(o, (const AdjPosT *)pos, npos, H, ldh, kc0, kcn, gW,
                                                           accumulate_gW, partial);
    } else if (fast) {
        e = cudaFuncSetAttribute(k_adj_fold<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_adj_fold<true><<<nblk, kFoldThreads, smem, st>>>(o, method, flags, (const AdjPosT *)pos, npos, H, ldh, kc0,
                                                          kcn, gW, accumulate_gW, partial);
    } else {
        e = cudaFuncSetAttribute(k_adj_fold<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_adj_fold<false><<<nblk, kFoldThreads, smem, st>>>(o, method, flags, (const AdjPosT *)pos, npos, H, ldh,
                                                           kc0, kcn, gW, accumulate_gW, partial);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_adj_sum<<<(npos * 2 + 7) / 8, 256, 0, st>>>(partial, nblk, npos, idx, accumulate_lm, g_lm);
    return cudaGetLastError();
}

}  // namespace psf
