// Smearing weights w_{p,k} = W_k D_k(l0_p), the FP32 CUDA-core contraction and the
// float64 reduction of split-K partial cutouts.
//
// Weights (Eqs. 13, 35, 44): one thread per (position, visibility), streamed over
// visibilities with coalesced 16-byte loads of the bin records.
//
// FP32 contraction (Eqs. 21-22 as a separable DFT): a CTA owns a pixel tile of one cutout
// and a contiguous range of visibilities; the tile body (twiddle chains from float-float
// seed phases, packed FMAs, compensated FP32 sums) is fp32t::tile_block, and split-K
// partials are added in float64, so the path meets 1e-6 relative.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "decorr.cuh"
#include "fp32_tile.cuh"

namespace psf {

// --------------------------------------------------------------- weights
template <bool FAST>
__global__ void __launch_bounds__(256) k_weights(DevObs o, int method, uint32_t flags,
                                                 const float4 *__restrict__ pos, int32_t k0,
                                                 int32_t kn, float2 *__restrict__ w, int64_t ldw) {
    // grid-stride over the visibilities (a few waves of blocks rather than one thread
    // per visibility: the per-visibility work is a handful of loads and sines)
    const int p = blockIdx.y;
    const float4 L = pos[p];
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int32_t kk = blockIdx.x * blockDim.x + threadIdx.x; kk < kn; kk += gridDim.x * blockDim.x) {
        const int32_t k = k0 + kk;
        const int bin = k / o.nout;
        const int r = k - bin * o.nout;
        float2 D = decorr<false, FAST>(o, method, flags, bin, r, L, z, z, nullptr);
        const float Wk = o.W[k];
        w[(int64_t)p * ldw + kk] = make_float2(Wk * D.x, Wk * D.y);
    }
}

// Sums over the raw samples of one bin for the eight affine channels r0 .. r0 + 7 of a
// thread and R positions: S_j = sum_s f_s exp(-2 pi i (nu_r0 + j dnu) ds_s / c), f_s the
// channel-independent factor (the raw channels' Dirichlet kernel times their sinc, Eq. 13
// with a boxcar).  A sample's record is loaded once for the R positions (the records of a
// warp's bins lie a bin apart, so a load touches up to 32 lines).
//
// The channels' phases about the middle of the eight differ by r_s x_j, r_s = -2 pi dnu ds_s / c,
// x_j = j - 7/2, which is small where the averaging is worth anything: with |r_s| <= kMomentMax
// for every sample the moments M_m = sum_s f_s e_s r_s^m, m = 0 .. 3, give
//   S_j = M_0 + i x_j M_1 - x_j^2/2 M_2 - i x_j^3/6 M_3     (truncation (3.5 r)^4 / 24 < 3e-7),
// seven packed operations per sample instead of a phasor recurrence over the channels
// (14, and a second sine and cosine); otherwise the recurrence is run.  256 positions x
// 14.1 M visibilities: 14.4 ms with a recurrence from three sine/cosine pairs and one
// position at a time, 13.3 ms with four positions and the two-term recurrence, 8.7 ms with
// moments.
constexpr float kMomentMax = 0.0143f;

template <int R>
__device__ __forceinline__ void exact8_sums(const DevObs &o, float4 ub, int2 sm, float4 ch, const float4 (&L)[R],
                                            float2 (&S)[R][8]) {
    const float nu_mid = -(ch.x + 3.5f * o.dnu_ch) * kInvC, wy = ch.w * kInvC, wa = ch.z * kInvC;
    const float r1 = -2.0f * kPiF * o.dnu_ch * kInvC;   // r per metre
    float Xbar[R], far[R];
    float2 M[R][4];
#pragma unroll
    for (int p = 0; p < R; ++p) {
        Xbar[p] = dot3(ub, L[p]);
        far[p] = 0.f;
#pragma unroll
        for (int m = 0; m < 4; ++m) M[p][m] = make_float2(0.f, 0.f);
    }
    for (int s = 0; s < sm.y; ++s) {
        const float4 d = __ldg(o.samp + sm.x + s);
#pragma unroll
        for (int p = 0; p < R; ++p) {
            const float ds = dot3(d, L[p]);
            const float Xs = Xbar[p] + ds;
            float f = sincpi_poly(wy * Xs);
            if (o.favg > 1) f *= dirichlet_poly(o.favg, wa * Xs);
            float es, ec;
            cis_mufu(nu_mid * ds, &es, &ec);
            const float r = r1 * ds;
            far[p] = fmaxf(far[p], fabsf(r));
            const float2 rr = make_float2(r, r);
            float2 e = make_float2(ec * f, es * f);
            M[p][0] = __fadd2_rn(M[p][0], e);
            e = __fmul2_rn(e, rr);
            M[p][1] = __fadd2_rn(M[p][1], e);
            e = __fmul2_rn(e, rr);
            M[p][2] = __fadd2_rn(M[p][2], e);
            M[p][3] = __ffma2_rn(e, rr, M[p][3]);
        }
    }
#pragma unroll
    for (int p = 0; p < R; ++p) {
        if (far[p] <= kMomentMax) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float x = (float)j - 3.5f;
                S[p][j] = make_float2(M[p][0].x - x * M[p][1].y - 0.5f * x * x * M[p][2].x + x * x * x / 6.0f * M[p][3].y,
                                      M[p][0].y + x * M[p][1].x - 0.5f * x * x * M[p][2].y - x * x * x / 6.0f * M[p][3].x);
            }
        } else {   // (fmaxf drops a NaN: such a sample is in the moments above, which are then NaN)
            // from the phasors of channels 3 and 4 outwards, e_{j+1} = 2 cos(step) e_j - e_{j-1}
#pragma unroll
            for (int j = 0; j < 8; ++j) S[p][j] = make_float2(0.f, 0.f);
            for (int s = 0; s < sm.y; ++s) {
                const float ds = dot3(__ldg(o.samp + sm.x + s), L[p]);
                const float Xs = Xbar[p] + ds;
                float f = sincpi_poly(wy * Xs);
                if (o.favg > 1) f *= dirichlet_poly(o.favg, wa * Xs);
                float es, ec, rs, rc;
                cis_mufu(-(ch.x + 3.0f * o.dnu_ch) * kInvC * ds, &es, &ec);
                cis_small(-o.dnu_ch * kInvC * ds, &rs, &rc);
                float2 e[8];
                e[3] = make_float2(ec * f, es * f);
                e[4] = make_float2(e[3].x * rc - e[3].y * rs, e[3].x * rs + e[3].y * rc);
                const float C = 2.0f * rc;
#pragma unroll
                for (int j = 5; j < 8; ++j) {
                    e[j] = make_float2(C * e[j - 1].x - e[j - 2].x, C * e[j - 1].y - e[j - 2].y);
                    e[7 - j] = make_float2(C * e[8 - j].x - e[9 - j].x, C * e[8 - j].y - e[9 - j].y);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) S[p][j] = __fadd2_rn(S[p][j], e[j]);
            }
        }
    }
}

// Exact-method weights of the tensor-core paths (FP32 (Re w, Im w) per position row) from
// exact8_sums: a thread owns eight consecutive channels of one
// bin (k0 and nout multiples of 8).
__global__ void __launch_bounds__(256) k_weights_exact8(DevObs o, const float4 *__restrict__ pos, int32_t k0,
                                                        int32_t kn, float2 *__restrict__ w, int64_t ldw) {
    const int p = blockIdx.y;
    const float4 L[1] = {pos[p]};
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; (int64_t)g * 8 < kn; g += gridDim.x * blockDim.x) {
        const int32_t kk0 = 8 * g;
        const int32_t kb = k0 + kk0;   // k0 and nout are multiples of 8: one bin per group
        const int bin = kb / o.nout;
        const int r0 = kb - bin * o.nout;
        float2 S[1][8];
        exact8_sums<1>(o, o.bin_ubar[bin], o.bin_samp[bin], o.chan[r0], L, S);
        const float inv = 1.0f / (float)o.bin_samp[bin].y;
        float2 *dst = w + (int64_t)p * ldw + kk0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (kk0 + j < kn) {
                const float Wk = o.W[kb + j] * inv;
                dst[j] = make_float2(Wk * S[0][j].x, Wk * S[0][j].y);
            }
    }
}

// Methods 1 and 2 (real weights, no windows) for affine channels: a thread owns eight
// consecutive channels of one bin.  Per bin the frequency sinc is the same for every channel
// (Method 1: ubar . L Dnu / c; Method 2: (Dnu / nu) |u| |l0| = |ubar| Dnu / c |l0|, with equal
// Dnu), and the time sinc's argument is linear in nu_r.  One visibility per thread, each with
// its own integer division, records and two MUFU sincs, took 376 us per method for 58.1 M
// visibilities; now 200 us, and 319 us for both methods in one pass (METHODS bit 0: Method 1
// into w, bit 1: Method 2 into w2).
template <int METHODS>
__global__ void __launch_bounds__(256) k_weights_real8(DevObs o, uint32_t flags, const float4 *__restrict__ pos,
                                                       int32_t k0, int32_t kn, float2 *__restrict__ w,
                                                       float2 *__restrict__ w2, int64_t ldw) {
    const int p = blockIdx.y;
    const float4 L = pos[p];
    const float rho = sqrtf(L.x * L.x + L.y * L.y);
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; (int64_t)g * 8 < kn; g += gridDim.x * blockDim.x) {
        const int32_t kk0 = 8 * g, kb = k0 + kk0;
        const int bin = kb / o.nout, r0 = kb - bin * o.nout;
        const float4 ub = o.bin_ubar[bin], ch = o.chan[r0];
        float Wk[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) Wk[j] = kk0 + j < kn ? o.W[kb + j] : 0.f;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if (!(METHODS & (1 << m))) continue;
            float a, B;   // time sinc argument per frequency, frequency sinc argument
            if (m == 0) {
                a = dot3(o.bin_edge[bin], L) * kInvC;
                B = dot3(ub, L) * ch.y * kInvC;
            } else {
                const float len = sqrtf(ub.x * ub.x + ub.y * ub.y);
                float udot = -ub.y, vdot = ub.x;
                if (flags & PSF_IMG_LITERAL_THETA) {
                    const float th = (ub.y != 0.0f) ? atanf(ub.x / ub.y) : (ub.x >= 0.0f ? 0.5f * kPiF : -0.5f * kPiF);
                    float st, ct;
                    sincosf(th, &st, &ct);
                    udot = -len * st;
                    vdot = len * ct;
                }
                a = (float)kOmegaE * ub.w * (udot * L.x + vdot * L.y) * kInvC;
                B = ch.y * kInvC * len * rho;
            }
            const float sB = sincpi_poly(B);
            float2 *dst = (m == 0 ? w : w2) + (int64_t)p * ldw + kk0;
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const float v0 = Wk[j] * sB * sincpi_poly(a * fmaf((float)j, o.dnu_ch, ch.x));
                const float v1 = Wk[j + 1] * sB * sincpi_poly(a * fmaf((float)(j + 1), o.dnu_ch, ch.x));
                if (kk0 + j + 1 < kn)   // ldw and kk0 + j are even: 16-byte aligned
                    *reinterpret_cast<float4 *>(dst + j) = make_float4(v0, 0.f, v1, 0.f);
                else if (kk0 + j < kn)
                    dst[j] = make_float2(v0, 0.f);
            }
        }
    }
}

// Channels shared by eight-channel groups aligned with the range.
static bool groups_of_8(const DevObs &o, int32_t k0) { return o.chan_affine && o.nout % 8 == 0 && k0 % 8 == 0; }

static int weight_sms() {   // SM count of the first device used (only sizes the grids)
    static int nsm = 0;
    if (nsm == 0 && cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, 0) != cudaSuccess) {
        cudaGetLastError();
        nsm = 152;
    }
    return nsm;
}
static dim3 grid_of_8(int32_t kn, int npos) {
    const int64_t b = std::min<int64_t>((kn / 8 + 255) / 256 + 1,
                                        (int64_t)weight_sms() * 16 / std::max(1, std::min(npos, 16)));
    return dim3((unsigned)std::max<int64_t>(1, b), npos);
}

cudaError_t launch_weights_uvimg(const DevObs &o, uint32_t flags, const float4 *pos, int npos, int32_t nvis,
                                 float2 *w_uv, float2 *w_img, int64_t ldw, int *nkernels, cudaStream_t st) {
    *nkernels = 0;
    if (npos <= 0 || nvis <= 0) return cudaSuccess;
    if (!o.win && groups_of_8(o, 0)) {
        *nkernels = 1;
        k_weights_real8<3><<<grid_of_8(nvis, npos), 256, 0, st>>>(o, flags, pos, 0, nvis, w_uv, w_img, ldw);
        return cudaGetLastError();
    }
    *nkernels = 2;
    const cudaError_t e = launch_weights(o, kUV, flags, pos, npos, 0, nvis, w_uv, ldw, 1, st);
    return e != cudaSuccess ? e : launch_weights(o, kImg, flags, pos, npos, 0, nvis, w_img, ldw, 1, st);
}

cudaError_t launch_weights(const DevObs &o, int method, uint32_t flags, const float4 *pos, int npos,
                           int32_t k0, int32_t kn, float2 *w, int64_t ldw, int fast, cudaStream_t st) {
    if (npos <= 0 || kn <= 0) return cudaSuccess;
    const int64_t blocks =
        std::min<int64_t>((kn + 255) / 256, (int64_t)weight_sms() * 16 / std::max(1, std::min(npos, 16)));
    dim3 grid((unsigned)std::max<int64_t>(1, blocks), npos);
    if (fast && !o.win && groups_of_8(o, k0)) {
        const dim3 g8 = grid_of_8(kn, npos);
        if (method == kExact) k_weights_exact8<<<g8, 256, 0, st>>>(o, pos, k0, kn, w, ldw);
        else if (method == kUV) k_weights_real8<1><<<g8, 256, 0, st>>>(o, flags, pos, k0, kn, w, nullptr, ldw);
        else k_weights_real8<2><<<g8, 256, 0, st>>>(o, flags, pos, k0, kn, nullptr, w, ldw);
        return cudaGetLastError();
    }
    if (fast) k_weights<true><<<grid, 256, 0, st>>>(o, method, flags, pos, k0, kn, w, ldw);
    else k_weights<false><<<grid, 256, 0, st>>>(o, method, flags, pos, k0, kn, w, ldw);
    return cudaGetLastError();
}

// --------------------------------------------------------------- FP16/BF16 weights
// Weights of a position chunk for the batched tensor-core contraction: row r holds
// position slot_of_row[r] (padding rows, slot < 0, are left as they are), Re w and -Im w in
// two planes (w16_offset); columns (k - kc0) at or beyond kcn are zero.  The weights are
// rounded to 16 bits, so the fast sine/cosine forms are used.
// One thread per visibility (column) and a block of kRowsPerBlock position rows: the
// visibility's records (bin, channel, weight, raw samples) are loaded once and reused
// for every row; each warp writes 32 consecutive columns of one row at a time.
constexpr int kRowsPerBlock = 32;

// Rounding of the weights to 16 bits.  Round-to-nearest is biased on these data: with
// natural weights most values W_k D_k sit just below the power of two W_k (small
// decorrelation), where every one rounds up, and a PSF peak sums them coherently (a bias
// of ~1e-5 of the peak over 2e8 visibilities).  Stochastic rounding (cvt.rs) is unbiased:
// the random bits, a hash of (position, visibility), make the rounding errors average out
// like independent ones.  The hash is deterministic, so a call is reproducible.
__device__ __forceinline__ uint32_t sr_bits(uint32_t slot, uint32_t k) {
    uint32_t h = k * 0x9E3779B1u ^ (slot + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 16;
    h *= 0x7FEB352Du;
    h ^= h >> 15;
    h *= 0x846CA68Bu;
    h ^= h >> 16;
    return h;
}

// (x, y) -> packed 16-bit pair, x in the low half (the layout of __floats2half2_rn)
template <int BF16>
__device__ __forceinline__ uint32_t pack_sr(float x, float y, uint32_t rbits) {
    uint32_t d;
    if (BF16) asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(y), "f"(x), "r"(rbits));
    else asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(y), "f"(x), "r"(rbits));
    return d;
}

template <int BF16>
__global__ void __launch_bounds__(256) k_weights16(DevObs o, int method, uint32_t flags,
                                                   const float4 *__restrict__ pos,
                                                   const int32_t *__restrict__ slot_of_row, int rows, int32_t kc0,
                                                   int32_t kcn, int64_t kpitch, uint32_t *__restrict__ w16) {
    const int32_t kk = blockIdx.x * blockDim.x + threadIdx.x;
    if (kk >= kpitch) return;   // kpitch is a multiple of 64: whole warps leave
    const int row0 = blockIdx.y * kRowsPerBlock;
    const bool valid = kk < kcn;
    const int32_t k = kc0 + (valid ? kk : 0);
    const int bin = k / o.nout;
    const int r = k - bin * o.nout;
    const float Wk = valid ? o.W[k] : 0.f;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const int odd = threadIdx.x & 1;
    for (int row = row0; row < min(rows, row0 + kRowsPerBlock); ++row) {
        const int slot = slot_of_row[row];
        if (slot < 0) continue;   // padding rows: their sums are not used, whatever they hold
        float2 w = make_float2(0.f, 0.f);
        if (valid) {
            const float2 D = decorr<false, true>(o, method, flags, bin, r, pos[slot], z, z, nullptr);
            w = make_float2(Wk * D.x, Wk * D.y);
        }
        // even lanes store the pair's real parts, odd lanes its imaginary parts
        const uint32_t own = pack_sr<BF16>(w.x, -w.y, sr_bits((uint32_t)slot, (uint32_t)k));
        const uint32_t nbr = __shfl_xor_sync(0xffffffffu, own, 1);
        const uint32_t v = odd ? __byte_perm(nbr, own, 0x7632) : __byte_perm(own, nbr, 0x5410);
        w16[w16_offset(row, kk & ~1, kpitch >> 6, 2, odd) >> 1] = v;
    }
}

// Real weights (Methods 1 and 2, no windows): one FP16/BF16 value W_k D_k per
// visibility; a thread owns the visibility pair (2 kp, 2 kp + 1) of a row (kpitch2 pairs
// per row).  Both methods are D = sinc(A) sinc(B) with arguments that are, per
// visibility, fixed forms in the position: Method 1 (Eq. 35) A = a . L and B = b . L
// with a = (uvw(t_e) - uvw(t_s)) nu_r / c and b = ubar Dnu_r / c; Method 2 (Eqs. 38-44)
// A = a . L with a = omega_E Dt (udot, vdot, 0) and B = f |(l0, m0)| with
// f = (Dnu_r / nu_r) |(u, v)|.  The thread forms a, b, f once for its two visibilities
// (decorr_uv / decorr_img do the same per call) and each position costs two dot
// products and two sincs.
template <int BF16>
__global__ void __launch_bounds__(256) k_weights16_real(DevObs o, int method, uint32_t flags,
                                                        const float4 *__restrict__ pos,
                                                        const int32_t *__restrict__ slot_of_row, int rows,
                                                        int32_t kc0, int32_t kcn, int64_t kpitch2,
                                                        uint32_t *__restrict__ w16) {
    const int32_t kp = blockIdx.x * blockDim.x + threadIdx.x;
    if (kp >= kpitch2) return;
    const int row0 = blockIdx.y * kRowsPerBlock;
    float4 a[2], b[2];   // A = a . L; B = b . L (Method 1) or b.x |(l0, m0)| (Method 2)
    float Wk[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int32_t kk = 2 * kp + e;
        const bool valid = kk < kcn;
        const int32_t k = kc0 + (valid ? kk : 0);
        const int bin = k / o.nout;
        const int r = k - bin * o.nout;
        Wk[e] = valid ? o.W[k] : 0.f;
        const float4 ub = o.bin_ubar[bin];
        const float4 ch = o.chan[r];
        if (method == kUV) {
            const float4 ed = o.bin_edge[bin];
            const float sa = ch.x * kInvC, sb = ch.y * kInvC;
            a[e] = make_float4(ed.x * sa, ed.y * sa, ed.z * sa, 0.f);
            b[e] = make_float4(ub.x * sb, ub.y * sb, ub.z * sb, 0.f);
        } else {
            const float sc = ch.x * kInvC;
            const float u = ub.x * sc, v = ub.y * sc;
            const float uvlen = sqrtf(u * u + v * v);
            float udot = -v, vdot = u;
            if (flags & PSF_IMG_LITERAL_THETA) {
                const float th = (v != 0.0f) ? atanf(u / v) : (u >= 0.0f ? 0.5f * kPiF : -0.5f * kPiF);
                float st, ct;
                sincosf(th, &st, &ct);
                udot = -uvlen * st;
                vdot = uvlen * ct;
            }
            const float wdt = (float)kOmegaE * ub.w;
            a[e] = make_float4(wdt * udot, wdt * vdot, 0.f, 0.f);
            b[e] = make_float4(ch.y / ch.x * uvlen, 0.f, 0.f, 0.f);
        }
    }
    // two channels of one bin have the same frequency sinc (equal Dnu): evaluated once
    const bool same = b[0].x == b[1].x && b[0].y == b[1].y && b[0].z == b[1].z;
    // the block's rows lie in one position tile: block base, then 32-bit row offsets
    uint32_t *const base = w16 + (w16_offset(row0 & ~127, 2 * (int64_t)(kp & ~31), kpitch2 >> 5, 1, 0) >> 1);
    const int chunk = (kp & 31) >> 2, word = kp & 3;
    for (int row = row0; row < min(rows, row0 + kRowsPerBlock); ++row) {
        const int slot = slot_of_row[row];
        if (slot < 0) continue;   // padding rows: their sums are not used, whatever they hold
        const float4 P = pos[slot];
        const float rho = method == kUV ? 0.f : sqrtf(P.x * P.x + P.y * P.y);
        float wv[2], sB[2];
        sB[0] = sincpi_poly((method == kUV) ? dot3(b[0], P) : b[0].x * rho);
        sB[1] = same ? sB[0] : sincpi_poly((method == kUV) ? dot3(b[1], P) : b[1].x * rho);
#pragma unroll
        for (int e = 0; e < 2; ++e) wv[e] = Wk[e] == 0.f ? 0.f : Wk[e] * sincpi_poly(dot3(a[e], P)) * sB[e];
        const int r = row & 127;
        base[(r << 5) + ((chunk ^ (r & 7)) << 2) + word] = pack_sr<BF16>(wv[0], wv[1], sr_bits((uint32_t)slot, (uint32_t)(kc0 + 2 * kp)));
    }
}

// Exact weights with affine channels (boxcar): a thread owns up to eight channels of one bin
// (group gr of the bin's ceil(nout / 8)) and kRows4 position rows at a time (exact8_sums).
// A bin may lie across the chunk's ends, and with nout not a multiple of 8 the groups are
// not aligned to 8 columns: EVEN8 (nout, kc0 multiples of 8) stores 16 bytes per plane and
// row, otherwise single values; the threads after the last bin zero the columns from kcn to the
// end of its 64-column stage.  (Bins of 6 channels took the general kernel before, with the
// Dirichlet kernel, sinc and phasor per channel: 73 positions x 8.7 M visibilities, 20 raw
// channels per output channel, 16.8 ms; 4.2 ms now.)
constexpr int kRows4 = 4;

template <int BF16, bool EVEN8>
__global__ void __launch_bounds__(128, 4) k_weights16_exact8(DevObs o, const float4 *__restrict__ pos,
                                                          const int32_t *__restrict__ slot_of_row, int rows,
                                                          int32_t kc0, int32_t kcn, int64_t kpitch, int32_t bin0,
                                                          int64_t ngroups, uint32_t *__restrict__ w16) {
    const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int row0 = blockIdx.y * kRowsPerBlock, row1 = min(rows, row0 + kRowsPerBlock);
    uint16_t *const w = reinterpret_cast<uint16_t *>(w16);
    const int64_t nblk = kpitch >> 6;
    if (gi >= ngroups) {   // zero columns kcn .. of the last stage
        const int64_t kk = kcn + (gi - ngroups);
        if (kk < ((int64_t)kcn + 63) / 64 * 64)
            for (int row = row0; row < row1; ++row)
                w[w16_offset(row, kk, nblk, 2, 0)] = w[w16_offset(row, kk, nblk, 2, 1)] = 0;
        return;
    }
    const int ng = (o.nout + 7) / 8;
    const int bin = bin0 + (int)(gi / ng), r0 = 8 * (int)(gi % ng);
    const int nch = min(8, o.nout - r0);
    const float4 ub = o.bin_ubar[bin];
    const int2 sm = o.bin_samp[bin];
    const float4 ch = o.chan[r0];
    const int32_t k0 = bin * o.nout + r0, kk0 = k0 - kc0;   // column of the first channel (may be negative)
    if (kk0 + nch <= 0 || kk0 >= kcn) return;
    float Wk[8];
    const float inv = 1.0f / (float)sm.y;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        Wk[j] = (j < nch && kk0 + j >= 0 && kk0 + j < kcn) ? o.W[k0 + j] * inv : 0.f;
    // aligned groups: the block's rows lie in one position tile; the -Im w block follows (4096 words)
    uint32_t *const base = w16 + (w16_offset(row0 & ~127, max(kk0, 0) & ~63, nblk, 2, 0) >> 1);
    const int chunk = (kk0 >> 3) & 7;
    for (int rb = row0; rb < row1; rb += kRows4) {
        int slot[kRows4];
        float4 L[kRows4];
        bool any = false;
#pragma unroll
        for (int p = 0; p < kRows4; ++p) {
            slot[p] = rb + p < row1 ? slot_of_row[rb + p] : -1;
            any = any || slot[p] >= 0;
            L[p] = slot[p] >= 0 ? pos[slot[p]] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (!any) continue;   // padding rows: their sums are not used, whatever they hold
        float2 S[kRows4][8];
        exact8_sums<kRows4>(o, ub, sm, ch, L, S);
#pragma unroll
        for (int p = 0; p < kRows4; ++p) {
            if (slot[p] < 0) continue;
            uint32_t packed[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                packed[j] = pack_sr<BF16>(Wk[j] * S[p][j].x, -Wk[j] * S[p][j].y,
                                          sr_bits((uint32_t)slot[p], (uint32_t)(k0 + j)));
            if (EVEN8) {
                uint32_t pr[4], pi[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    pr[j] = __byte_perm(packed[2 * j], packed[2 * j + 1], 0x5410);
                    pi[j] = __byte_perm(packed[2 * j], packed[2 * j + 1], 0x7632);
                }
                const int r = (rb + p) & 127;
                uint32_t *const at = base + (r << 5) + ((chunk ^ (r & 7)) << 2);
                *reinterpret_cast<uint4 *>(at) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
                *reinterpret_cast<uint4 *>(at + 4096) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j < nch && kk0 + j >= 0 && kk0 + j < kcn) {
                        const int64_t at = w16_offset(rb + p, kk0 + j, nblk, 2, 0);
                        w[at] = (uint16_t)(packed[j] & 0xffffu);
                        w[at + 8192] = (uint16_t)(packed[j] >> 16);
                    }
            }
        }
    }
}

cudaError_t launch_weights16(const DevObs &o, int method, uint32_t flags, const float4 *pos,
                             const int32_t *slot_of_row, int rows, int32_t kc0, int32_t kcn, int64_t kpitch,
                             int bf16, void *w16, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    if (method == kExact && o.chan_affine && kcn > 0) {   // chan_affine excludes windows
        const unsigned gy = (unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock);
        const int ng = (o.nout + 7) / 8;
        const int32_t bin0 = kc0 / o.nout, bin1 = (int32_t)(((int64_t)kc0 + kcn - 1) / o.nout);
        const int64_t ngroups = (int64_t)(bin1 - bin0 + 1) * ng;
        dim3 grid((unsigned)((ngroups + 63 + 127) / 128), gy);
        const bool even8 = o.nout % 8 == 0 && kc0 % 8 == 0 && kcn % 8 == 0;
#define PSF_W16E(B, E)                                                                                            \
    k_weights16_exact8<B, E><<<grid, 128, 0, st>>>(o, pos, slot_of_row, rows, kc0, kcn, kpitch, bin0, ngroups,    \
                                                   (uint32_t *)w16)
        if (bf16) {
            if (even8) PSF_W16E(1, true);
            else PSF_W16E(1, false);
        } else {
            if (even8) PSF_W16E(0, true);
            else PSF_W16E(0, false);
        }
#undef PSF_W16E
        return cudaGetLastError();
    }
    const unsigned gy = (unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock);
    if (method != kExact && !o.win) {   // real weights: kpitch pairs per row hold 2 kpitch visibilities
        const int64_t kp2 = kpitch / 2;
        dim3 grid((unsigned)((kp2 + 255) / 256), gy);
        if (bf16)
            k_weights16_real<1><<<grid, 256, 0, st>>>(o, method, flags, pos, slot_of_row, rows, kc0, kcn, kp2,
                                                      (uint32_t *)w16);
        else
            k_weights16_real<0><<<grid, 256, 0, st>>>(o, method, flags, pos, slot_of_row, rows, kc0, kcn, kp2,
                                                      (uint32_t *)w16);
        return cudaGetLastError();
    }
    dim3 grid((unsigned)((kpitch + 255) / 256), gy);
    if (bf16)
        k_weights16<1><<<grid, 256, 0, st>>>(o, method, flags, pos, slot_of_row, rows, kc0, kcn, kpitch,
                                             (uint32_t *)w16);
    else
        k_weights16<0><<<grid, 256, 0, st>>>(o, method, flags, pos, slot_of_row, rows, kc0, kcn, kpitch,
                                             (uint32_t *)w16);
    return cudaGetLastError();
}

// Zero the listed cutouts (outputs that are accumulated with atomics).
__global__ void __launch_bounds__(256) k_zero_cutouts(float *__restrict__ out, const int64_t *__restrict__ offs,
                                                      const int32_t *__restrict__ npix) {
    const int p = blockIdx.y;
    const int64_t n2 = (int64_t)npix[p] * npix[p];
    float *dst = out + offs[p];
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n2; q += (int64_t)gridDim.x * blockDim.x)
        dst[q] = 0.f;
}

cudaError_t launch_zero_cutouts(float *out, const int64_t *offs, const int32_t *npix, int npos, cudaStream_t st) {
    if (npos <= 0) return cudaSuccess;
    k_zero_cutouts<<<dim3(16, npos), 256, 0, st>>>(out, offs, npix);
    return cudaGetLastError();
}

// --------------------------------------------------------------- FP32 contraction
// One CTA per (tile, visibility range); the tile body is fp32t::tile_block.
template <int A, int B>
__global__ void __launch_bounds__(256, 1)
    k_psf_fp32(const float2 *__restrict__ uv, const float2 *__restrict__ uv_lo, const float2 *__restrict__ w, int64_t ldw,
               int32_t nvis, const Tile *__restrict__ tiles, int32_t kper, float2 cell, float *__restrict__ partial,
               int64_t split_stride) {
    extern __shared__ __align__(16) float fp32_smem[];
    const Tile t = tiles[blockIdx.x];
    const int32_t kbeg = blockIdx.y * kper;
    fp32t::tile_block<A, B>(fp32_smem, uv, uv_lo, w + (int64_t)t.slot * ldw, kbeg, min(nvis, kbeg + kper), t.N, t.i0, t.j0,
                            cell, partial + (int64_t)blockIdx.y * split_stride + t.out_off);
}

// Tile shapes (8 A x 8 B pixels) and their relative cost per pixel-visibility term (larger
// blocks per thread load fewer operands per FMA): a call takes the shape with the least
// padded work over its cutouts.
static const struct { int A, B; double cost; } kFp32Shapes[] = {{8, 8, 1.0}, {10, 5, 1.1}, {6, 6, 1.15}, {4, 4, 1.5}};

int fp32_shape(const int32_t *npix, int npos, int *ti, int *tj) {
    int best = 0;
    double best_cost = 0.0;
    for (int s = 0; s < 4; ++s) {
        const int Ti = 8 * kFp32Shapes[s].A, Tj = 8 * kFp32Shapes[s].B;
        double c = 0.0;
        for (int p = 0; p < npos; ++p)
            c += (double)((npix[p] + Ti - 1) / Ti * Ti) * ((npix[p] + Tj - 1) / Tj * Tj) * kFp32Shapes[s].cost;
        if (s == 0 || c < best_cost) { best = s; best_cost = c; }
    }
    *ti = 8 * kFp32Shapes[best].A;
    *tj = 8 * kFp32Shapes[best].B;
    return best;
}

template <int A, int B>
static cudaError_t launch_fp32_t(const DevObs &o, const float2 *w, int64_t ldw, const Tile *tiles, int ntiles, int nsplit,
                                 int32_t kper, double cell, float *partial, int64_t split_stride, cudaStream_t st) {
    constexpr size_t smem = fp32t::Block<A, B>::kSmem;
    cudaError_t e = cudaFuncSetAttribute(k_psf_fp32<A, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_psf_fp32<A, B><<<dim3(ntiles, nsplit), 256, smem, st>>>(o.uv, o.uv_lo, w, ldw, o.nvis, tiles, kper,
                                                              fp32t::cell_pair(cell), partial, split_stride);
    return cudaGetLastError();
}

cudaError_t launch_psf_fp32(const DevObs &o, const float2 *w, int64_t ldw, const Tile *tiles, int ntiles,
                            int nsplit, int32_t kper, double cell, float *partial, int64_t split_stride, int shape,
                            cudaStream_t st) {
    if (ntiles <= 0) return cudaSuccess;
    switch (shape) {
        case 0: return launch_fp32_t<8, 8>(o, w, ldw, tiles, ntiles, nsplit, kper, cell, partial, split_stride, st);
        case 1: return launch_fp32_t<10, 5>(o, w, ldw, tiles, ntiles, nsplit, kper, cell, partial, split_stride, st);
        case 2: return launch_fp32_t<6, 6>(o, w, ldw, tiles, ntiles, nsplit, kper, cell, partial, split_stride, st);
        case 3: return launch_fp32_t<4, 4>(o, w, ldw, tiles, ntiles, nsplit, kper, cell, partial, split_stride, st);
        default: return cudaErrorInvalidValue;
    }
}

// --------------------------------------------------------------- FP32 FMA rate
// Denominator of the FP32 path's roofline: every thread runs kFmaChains independent
// chains x <- x c + b (|c| < 1, so the values stay bounded), as scalar FMAs or as packed
// pairs (fma.rn.f32x2, one instruction for two FMAs).  The last values are written so
// that nothing is optimised away.
constexpr int kFmaChains = 16;

template <int PACKED>
__global__ void __launch_bounds__(256) k_fma_rate(int iters, float seed, float *__restrict__ out) {
    const float b = seed * 1e-3f + 1e-9f * threadIdx.x, c = 0.999f - 1e-7f * blockIdx.x;
    float r = 0.f;
    if (PACKED) {
        unsigned long long x[kFmaChains], bb, cc;
        asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(b));
        asm("mov.b64 %0, {%1, %1};" : "=l"(cc) : "f"(c));
#pragma unroll
        for (int j = 0; j < kFmaChains; ++j) {
            const float v = seed + j;
            asm("mov.b64 %0, {%1, %2};" : "=l"(x[j]) : "f"(v), "f"(-v));
        }
#pragma unroll 4
        for (int it = 0; it < iters; ++it)
#pragma unroll
            for (int j = 0; j < kFmaChains; ++j) asm volatile("fma.rn.f32x2 %0, %0, %1, %2;" : "+l"(x[j]) : "l"(cc), "l"(bb));
#pragma unroll
        for (int j = 0; j < kFmaChains; ++j) {
            float lo, hi;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x[j]));
            r += lo + hi;
        }
    } else {
        float x[kFmaChains];
#pragma unroll
        for (int j = 0; j < kFmaChains; ++j) x[j] = seed + j;
#pragma unroll 8
        for (int it = 0; it < iters; ++it)
#pragma unroll
            for (int j = 0; j < kFmaChains; ++j) x[j] = fmaf(x[j], c, b);
#pragma unroll
        for (int j = 0; j < kFmaChains; ++j) r += x[j];
    }
    out[(int64_t)blockIdx.x * blockDim.x + threadIdx.x] = r;
}

int selftest_fma_rate(int packed, double *flops_per_s) {
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PSF_ECUDA;
    const int blocks = nsm * 8, threads = 256, iters = 1 << 15;
    float *out = nullptr;
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = PSF_OK;
    double best = 0.0;
    if (cudaMalloc(&out, sizeof(float) * blocks * threads) != cudaSuccess) return PSF_ENOMEM;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
        cudaEventCreate(&e1) != cudaSuccess) {
        rc = PSF_ECUDA;
    } else {
        for (int rep = 0; rep < 4 && rc == PSF_OK; ++rep) {   // the first launch is warm-up
            cudaEventRecord(e0, st);
            if (packed) k_fma_rate<1><<<blocks, threads, 0, st>>>(iters, 1.0f + rep, out);
            else k_fma_rate<0><<<blocks, threads, 0, st>>>(iters, 1.0f + rep, out);
            cudaEventRecord(e1, st);
            float ms = 0.f;
            if (cudaGetLastError() != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
                rc = PSF_ECUDA;
                break;
            }
            const double flops = 2.0 * (packed ? 2 : 1) * kFmaChains * (double)iters * blocks * threads;
            if (rep > 0 && ms > 0.f) best = std::max(best, flops / (ms * 1e-3));
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    cudaFree(out);
    if (rc == PSF_OK) *flops_per_s = best;
    return rc;
}

// --------------------------------------------------------------- split reduction
// One block row per position; 32 pixels per block, the splits of a pixel shared by eight
// threads (splits s mod 8, four loads in flight each) and their float64 sums added in a
// fixed order (deterministic).  One thread per pixel walked up to 152 splits one L2 round
// trip after another (24 us per cutout).  Partials use chunk-local packed offsets, the
// output the caller's offsets.
__global__ void __launch_bounds__(256) k_reduce(const float *__restrict__ partial, int nsplit,
                                                int64_t stride, const int64_t *__restrict__ loc_offs,
                                                const int64_t *__restrict__ out_offs,
                                                const int32_t *__restrict__ npix, int transposed,
                                                float *__restrict__ out, const float *__restrict__ partial2,
                                                float *__restrict__ out2) {
    if (blockIdx.z) {
        partial = partial2;
        out = out2;
    }
    __shared__ double sum[8][32];
    const int p = blockIdx.y;
    const int N = npix[p];
    const int64_t n2 = (int64_t)N * N;
    const float *src = partial + loc_offs[p];
    float *dst = out + out_offs[p];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int64_t q0 = (int64_t)blockIdx.x * 32; q0 < n2; q0 += (int64_t)gridDim.x * 32) {
        const int64_t q = q0 + tx;
        double s = 0.0;
        if (q < n2) {
            int sp = ty;
            for (; sp + 24 < nsplit; sp += 32) {
                float v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = src[(int64_t)(sp + 8 * u) * stride + q];
#pragma unroll
                for (int u = 0; u < 4; ++u) s += (double)v[u];
            }
            for (; sp < nsplit; sp += 8) s += (double)src[(int64_t)sp * stride + q];
        }
        sum[ty][tx] = s;
        __syncthreads();
        if (ty == 0 && q < n2) {
#pragma unroll
            for (int u = 1; u < 8; ++u) s += sum[u][tx];
            // transposed partials hold (j, i) at q = i N + j
            const int64_t o = transposed ? (q % N) * N + q / N : q;
            dst[o] = (float)s;
        }
        __syncthreads();
    }
}

cudaError_t launch_reduce(const float *partial, int nsplit, int64_t stride, const int64_t *loc_offs,
                          const int64_t *out_offs, const int32_t *npix, int npos, int transposed, float *out,
                          cudaStream_t st, const float *partial2, float *out2) {
    if (npos <= 0) return cudaSuccess;
    dim3 grid((unsigned)std::max(16, 512 / npos), npos, partial2 ? 2 : 1);
    k_reduce<<<grid, 256, 0, st>>>(partial, nsplit, stride, loc_offs, out_offs, npix, transposed, out, partial2, out2);
    return cudaGetLastError();
}

// --------------------------------------------------------------- binning (plan build)
// One thread per averaging bin: baseline b (binary search in bin_first), bin tau of its
// tavg[b] raw samples s0 = tau tavg[b] ...  Eq. 12's bin centre is the mean of the raw
// uvw, summed in sample order in float64 and divided by n; the edge delta (Eq. 33) is
// uvw(last) - uvw(first) scaled by n / (n - 1) (the bin's full width), or for a single
// sample the central difference of the neighbouring samples; the raw samples are kept as
// float32 offsets from the centre.  The same float64 operations in the same order as a
// host loop, so the records are bit-identical to host binning.
__global__ void __launch_bounds__(256) k_bin(const double *__restrict__ uvw, int ntime, int nbl,
                                             const int32_t *__restrict__ tavg, const int32_t *__restrict__ bin_first,
                                             const int64_t *__restrict__ samp_first, double dt_raw,
                                             float4 *__restrict__ bin_ubar, double2 *__restrict__ bin_uv64,
                                             float4 *__restrict__ bin_edge, int2 *__restrict__ bin_samp,
                                             float4 *__restrict__ samp) {
    const int32_t bin = blockIdx.x * blockDim.x + threadIdx.x;
    if (bin >= bin_first[nbl]) return;
    int lo = 0, hi = nbl;   // bin_first[lo] <= bin < bin_first[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (bin_first[mid] <= bin) lo = mid; else hi = mid;
    }
    const int b = lo, n = tavg[b];
    const int64_t tau = bin - bin_first[b];
    const int64_t s0 = tau * n;
    const double *ub = uvw + (size_t)b * ntime * 3;
    double mean[3] = {0, 0, 0}, edge[3] = {0, 0, 0};
    for (int64_t s = s0; s < s0 + n; ++s)
        for (int d = 0; d < 3; ++d) mean[d] += ub[s * 3 + d];
    for (int d = 0; d < 3; ++d) mean[d] /= n;
    if (n >= 2) {
        for (int d = 0; d < 3; ++d) edge[d] = __dmul_rn(ub[(s0 + n - 1) * 3 + d] - ub[s0 * 3 + d], (double)n) / (double)(n - 1);
    } else if (ntime >= 2) {
        const int64_t sa = s0 > 0 ? s0 - 1 : s0, sb = s0 < ntime - 1 ? s0 + 1 : s0;
        for (int d = 0; d < 3; ++d) edge[d] = (ub[sb * 3 + d] - ub[sa * 3 + d]) / (double)(sb - sa);
    }
    const int64_t rec = samp_first[b] + tau * n;
    bin_ubar[bin] = make_float4((float)mean[0], (float)mean[1], (float)mean[2], (float)(n * dt_raw));
    bin_uv64[bin] = make_double2(mean[0], mean[1]);
    bin_edge[bin] = make_float4((float)edge[0], (float)edge[1], (float)edge[2], 0.f);
    bin_samp[bin] = make_int2((int)rec, n);
    for (int s = 0; s < n; ++s) {
        const double *u = ub + (s0 + s) * 3;
        samp[rec + s] = make_float4((float)(u[0] - mean[0]), (float)(u[1] - mean[1]), (float)(u[2] - mean[2]), 0.f);
    }
}

cudaError_t launch_bin(const double *uvw, int ntime, int nbl, const int32_t *tavg, const int32_t *bin_first,
                       const int64_t *samp_first, int64_t nbin, double dt_raw, float4 *bin_ubar, double2 *bin_uv64,
                       float4 *bin_edge, int2 *bin_samp, float4 *samp, cudaStream_t st) {
    if (nbin <= 0) return cudaSuccess;
    k_bin<<<(unsigned)((nbin + 255) / 256), 256, 0, st>>>(uvw, ntime, nbl, tavg, bin_first, samp_first, dt_raw,
                                                           bin_ubar, bin_uv64, bin_edge, bin_samp, samp);
    return cudaGetLastError();
}

// --------------------------------------------------------------- per-visibility tables
// uv[k] + uv_lo[k] = ubar (x, y) nu_r / c in wavelengths, formed in float64 from the bin
// means and channel frequencies and split into a rounded float pair; W[k] = tavg * favg
// when no weights are given.
__global__ void __launch_bounds__(256) k_fill_vis(DevObs o, const double2 *__restrict__ bin_uv64,
                                                  const double2 *__restrict__ chan64, float2 *__restrict__ uv,
                                                  float2 *__restrict__ uv_lo, float *__restrict__ W, int natural) {
    const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= o.nvis) return;
    const int bin = k / o.nout;
    const int r = k - bin * o.nout;
    const double2 ub = bin_uv64[bin];
    const double nu = chan64[r].x;
    const double u = ub.x * nu / kCLight, v = ub.y * nu / kCLight;
    const float uh = (float)u, vh = (float)v;
    uv[k] = make_float2(uh, vh);
    uv_lo[k] = make_float2((float)(u - (double)uh), (float)(v - (double)vh));
    if (natural) W[k] = (float)(o.bin_samp[bin].y * o.favg);
}

cudaError_t launch_fill_vis(const DevObs &o, const double2 *bin_uv64, const double2 *chan64, float2 *uv,
                            float2 *uv_lo, float *W, int natural, cudaStream_t st) {
    k_fill_vis<<<(o.nvis + 255) / 256, 256, 0, st>>>(o, bin_uv64, chan64, uv, uv_lo, W, natural);
    return cudaGetLastError();
}

}  // namespace psf
