// FP32 CUDA-core contraction of one tile of a cutout over a range of visibilities (Eqs.
// 21-22 as a separable DFT): row twiddles a_k[i] = exp(2 pi i u_k dl_i) and weighted column
// twiddles c_k[j] = w_k exp(2 pi i v_k dm_j) are staged in shared memory chunk by chunk, and
// every thread accumulates a block of pixels of Re(c a), two FMAs per term.  Sums stay short
// in FP32 (32 visibilities) and are folded into a compensated (Kahan) total.
//   tile_block  the FP32 path (weights read from a buffer): packed FMAs on 4 x 4 to 8 x 8
//               blocks per thread, double-buffered chunks
//   tile_sum    the allocation-free entry point (weights evaluated inline), whose launch
//               keeps to statically sized shared memory
//
// Phase accuracy.  A pixel phase u_k (i - N/2) cell reaches tens of turns, so forming it
// in FP32 leaves ~2^-24 relative, i.e. several 1e-6 rad, of error in every term -- more
// than the 1e-6 bound allows when a cutout sums only tens of visibilities.  The phase is
// therefore carried as a float-float pair: u_k = u_hi + u_lo (both rounded from the
// float64 bin centre), cell = cell_hi + cell_lo, the product by the exact-error FMA
// identity, and the whole turns are removed exactly (x - rint(x)) before anything is
// rounded; each visibility's chains of twiddles start from such seeds every 8 pixels.
#pragma once

#include "decorr.cuh"

namespace psf {
namespace fp32t {

constexpr int kT = 64;     // tile edge (pixels) of tile_sum
// row pitch: 32 lanes write one column of 32 rows; with a pitch of 64 all of them hit one bank
constexpr int kTP = kT + 2;
constexpr int kKC = 32;    // visibilities per shared-memory chunk
constexpr int kSeg = 16;   // twiddles per generator thread (two chains of 8)
constexpr int kChain = 8;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// (x_hi + x_lo) (c_hi + c_lo) as an unevaluated pair (hi, lo): hi = fl(x_hi c_hi), lo its
// rounding error (exact by FMA) plus the cross terms (the lo x lo term is below 2^-48).
__device__ __forceinline__ float2 ff_mul(float xh, float xl, float ch, float cl) {
    const float p = xh * ch;
    const float e = fmaf(xh, ch, -p);
    return make_float2(p, fmaf(xh, cl, fmaf(xl, ch, e)));
}

// Fractional part of th * n in turns, in [-1/2, 1/2] up to one rounding (|n| < 2^24): the
// product's high part loses its whole turns exactly before the low parts are added.
__device__ __forceinline__ float ff_turns(float2 th, int n) {
    const float fn = (float)n;
    const float p = th.x * fn;
    const float e = fmaf(th.x, fn, -p);
    const float r = p - rintf(p);   // exact: |p - rint(p)| <= 1/2 with p's spacing
    return r + fmaf(th.y, fn, e);
}

// exp(2 pi i t), t in turns
__device__ __forceinline__ float2 cis_acc(float t) {
    float s, c;
    sincospif(2.0f * t, &s, &c);
    return make_float2(c, s);
}

// Adds to tot[b][a] the sum over k in [kbeg, kend) of Re(c_k[j] a_k[i]) for the pixel
// block of this thread (rows j = j0 + 4 ty + b, columns i = i0 + 4 tx + a, 16 x 16
// threads), with w_k = wfn(k).  Called by all 256 threads of the block.
template <class WFn>
__device__ __forceinline__ void tile_sum(const float2 *__restrict__ uv, const float2 *__restrict__ uv_lo,
                                         int32_t kbeg, int32_t kend, int N, int i0, int j0, float2 cell, WFn wfn,
                                         float2 (&sa)[kKC][kTP], float2 (&sc)[kKC][kTP], float (&tot)[4][4]) {
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    // generator role: visibility lane gk of the chunk, 16-twiddle segment gs (0-3 rows, 4-7 cols)
    const int gk = tid & 31, gs = tid >> 5;
    const int half = N / 2;
    const int seg_first = (gs & 3) * kSeg;
    const int n_first = (gs < 4 ? i0 : j0) + seg_first - half;   // pixel offset index of the chain start

    float acc[4][4], cmp[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) { acc[b][a] = 0.f; cmp[b][a] = 0.f; }

    for (int32_t kc = kbeg; kc < kend; kc += kKC) {
        const int32_t k = kc + gk;
        float2 s0 = make_float2(0.f, 0.f), s1 = s0, step = make_float2(1.f, 0.f);
        if (k < kend) {
            const float2 uh = uv[k], ul = uv_lo[k];
            const float2 th = gs < 4 ? ff_mul(uh.x, ul.x, cell.x, cell.y) : ff_mul(uh.y, ul.y, cell.x, cell.y);
            s0 = cis_acc(ff_turns(th, n_first));
            s1 = cis_acc(ff_turns(th, n_first + kChain));
            step = cis_acc(ff_turns(th, 1));
            if (gs >= 4) {
                const float2 wk = wfn(k);
                s0 = cmul(s0, wk);
                s1 = cmul(s1, wk);
            }
        }
        __syncthreads();   // previous chunk consumed
        float2 *dst = (gs < 4 ? &sa[gk][seg_first] : &sc[gk][seg_first]);
#pragma unroll
        for (int q = 0; q < kChain; ++q) {
            dst[q] = s0;
            dst[q + kChain] = s1;
            s0 = cmul(s0, step);
            s1 = cmul(s1, step);
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < kKC; ++kk) {
            const float4 a01 = *reinterpret_cast<const float4 *>(&sa[kk][tx * 4]);
            const float4 a23 = *reinterpret_cast<const float4 *>(&sa[kk][tx * 4 + 2]);
            const float4 c01 = *reinterpret_cast<const float4 *>(&sc[kk][ty * 4]);
            const float4 c23 = *reinterpret_cast<const float4 *>(&sc[kk][ty * 4 + 2]);
            const float ar[4] = {a01.x, a01.z, a23.x, a23.z}, ai[4] = {a01.y, a01.w, a23.y, a23.w};
            const float cr[4] = {c01.x, c01.z, c23.x, c23.z}, ci[4] = {c01.y, c01.w, c23.y, c23.w};
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[b][a] = fmaf(cr[b], ar[a], fmaf(-ci[b], ai[a], acc[b][a]));
        }
        // fold the chunk sum into the compensated total
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float y = acc[b][a] - cmp[b][a];
                const float s = tot[b][a] + y;
                cmp[b][a] = (s - tot[b][a]) - y;
                tot[b][a] = s;
                acc[b][a] = 0.f;
            }
    }
}

// Writes this thread's 4 x 4 block to dst[j * N + i] (pixels inside the cutout only).
__device__ __forceinline__ void tile_store(float *dst, int N, int i0, int j0, const float (&tot)[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int j = j0 + ty * 4 + b;
        if (j >= N) continue;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = i0 + tx * 4 + a;
            if (i < N) dst[(int64_t)j * N + i] = tot[b][a];
        }
    }
}

// ---------------------------------------------------------------- the FP32 path's tile
// A tile of 8 A x 8 B pixels (columns i, rows j; A even) by 256 threads: 64 threads hold the
// tile, A x B pixels each (pixel pairs i = 2 (tx + 8 q) + (0, 1), rows j = ty + 8 r), four
// times over, each taking every fourth visibility of a 64-visibility chunk.  Per visibility a
// thread loads A/2 + B operands and issues A B packed FMAs (a 4 x 4 block of scalar FMAs, as
// in tile_sum, spends as many shared-memory cycles as FMA cycles), and the next chunk's
// twiddles are generated while this one is summed.  What it was bound by before: the twiddle
// stores, 32 lanes to one bank (32-way conflicts, twice the time of the FMAs).
template <int A, int B>
struct Block {
    static constexpr int kTi = 8 * A, kTj = 8 * B;
    static constexpr int kChunk = 64;
    // floats per visibility: (ar, ar', ai, ai') per pixel pair; (cr, -ci) per row; the pads
    // spread 32 visibilities' stores over the banks
    static constexpr int kPa = 2 * kTi + 4, kPc = 2 * kTj + 2;
    static constexpr int kBuf = kChunk * (kPa + kPc);
    static constexpr size_t kSmem = 2 * kBuf * sizeof(float);
    static_assert(A % 2 == 0 && kTi % 16 == 0, "pixel pairs, chains of 8");
    static_assert((size_t)3 * kTi * kTj * sizeof(double) <= kSmem, "slice sums fit the buffers");
};

// Twiddles of visibility k (this thread's lane of the chunk) for half of the tile's columns
// (part 0, 1) or rows (part 2, 3): chains of at most 8 from float-float seed phases.
template <int A, int B>
__device__ __forceinline__ void block_generate(float *buf, int gk, int part, int32_t k, int32_t kend,
                                               const float2 *__restrict__ uv, const float2 *__restrict__ uv_lo,
                                               const float2 *__restrict__ w, int i0, int j0, int half, float2 cell) {
    using S = Block<A, B>;
    const bool ok = k < kend, cols = part < 2;
    const float2 uh = ok ? uv[k] : make_float2(0.f, 0.f), ul = ok ? uv_lo[k] : make_float2(0.f, 0.f);
    const float2 wk = cols ? make_float2(1.f, 0.f) : (ok ? w[k] : make_float2(0.f, 0.f));
    const float2 th = cols ? ff_mul(uh.x, ul.x, cell.x, cell.y) : ff_mul(uh.y, ul.y, cell.x, cell.y);
    const float2 step = cis_acc(ff_turns(th, 1));
    const int len = cols ? S::kTi / 2 : S::kTj / 2, first = (part & 1) * len;
    const int n0 = (cols ? i0 : j0) + first - half;
    float *const da = buf + gk * S::kPa + 2 * first;
    float *const dc = buf + S::kChunk * S::kPa + gk * S::kPc + 2 * first;
#pragma unroll 1
    for (int c = 0; c < len; c += kChain) {
        float2 z = cis_acc(ff_turns(th, n0 + c));
        if (!cols) z = cmul(z, wk);
#pragma unroll
        for (int q = 0; q < kChain; q += 2) {
            const float2 y = cmul(z, step);
            if (cols) {
                *reinterpret_cast<float4 *>(da + 2 * (c + q)) = make_float4(z.x, y.x, z.y, y.y);
            } else if (c + q < len) {
                *reinterpret_cast<float2 *>(dc + 2 * (c + q)) = make_float2(z.x, -z.y);
                *reinterpret_cast<float2 *>(dc + 2 * (c + q) + 2) = make_float2(y.x, -y.y);
            }
            z = cmul(y, step);
        }
    }
}

// Sum over k in [kbeg, kend) of Re(c_k[j] a_k[i]) for the tile at (i0, j0), written to
// dst[j N + i] (pixels inside the cutout).  Called by all 256 threads; smem: Block::kSmem bytes.
template <int A, int B>
__device__ __forceinline__ void tile_block(float *smem, const float2 *__restrict__ uv, const float2 *__restrict__ uv_lo,
                                           const float2 *__restrict__ w, int32_t kbeg, int32_t kend, int N, int i0,
                                           int j0, float2 cell, float *dst) {
    using S = Block<A, B>;
    const int tid = threadIdx.x, slice = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
    float2 acc[B][A / 2], tot[B][A / 2], ncmp[B][A / 2];
    const float2 zero = make_float2(0.f, 0.f), minus1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int r = 0; r < B; ++r)
#pragma unroll
        for (int q = 0; q < A / 2; ++q) acc[r][q] = tot[r][q] = ncmp[r][q] = zero;
    block_generate<A, B>(smem, tid & 63, slice, kbeg + (tid & 63), kend, uv, uv_lo, w, i0, j0, N / 2, cell);
    __syncthreads();
    int b = 0, n = 0;
    for (int32_t kc = kbeg; kc < kend; kc += S::kChunk, b ^= 1, ++n) {
        if (kc + S::kChunk < kend)
            block_generate<A, B>(smem + (b ^ 1) * S::kBuf, tid & 63, slice, kc + S::kChunk + (tid & 63), kend, uv, uv_lo,
                                 w, i0, j0, N / 2, cell);
        const float *pa = smem + b * S::kBuf + slice * S::kPa + 4 * tx;
        const float *pc = smem + b * S::kBuf + S::kChunk * S::kPa + slice * S::kPc + 2 * ty;
#pragma unroll 2
        for (int kk = 0; kk < S::kChunk / 4; ++kk) {
            float4 a[A / 2];
#pragma unroll
            for (int q = 0; q < A / 2; ++q) a[q] = *reinterpret_cast<const float4 *>(pa + 32 * q);
#pragma unroll
            for (int r = 0; r < B; ++r) {
                const float2 c = *reinterpret_cast<const float2 *>(pc + 16 * r);
                const float2 cr = make_float2(c.x, c.x), ci = make_float2(c.y, c.y);
#pragma unroll
                for (int q = 0; q < A / 2; ++q) {
                    acc[r][q] = __ffma2_rn(ci, make_float2(a[q].z, a[q].w), acc[r][q]);
                    acc[r][q] = __ffma2_rn(cr, make_float2(a[q].x, a[q].y), acc[r][q]);
                }
            }
            pa += 4 * S::kPa;
            pc += 4 * S::kPc;
        }
        if ((n & 1) || kc + S::kChunk >= kend) {   // 32 visibilities of this slice: Kahan, ncmp = -(compensation)
#pragma unroll
            for (int r = 0; r < B; ++r)
#pragma unroll
                for (int q = 0; q < A / 2; ++q) {
                    const float2 y = __fadd2_rn(acc[r][q], ncmp[r][q]);
                    const float2 s = __fadd2_rn(tot[r][q], y);
                    ncmp[r][q] = __fadd2_rn(__ffma2_rn(s, minus1, tot[r][q]), y);
                    tot[r][q] = s;
                    acc[r][q] = zero;
                }
        }
        __syncthreads();
    }
    // the four slices' totals, in float64 and in a fixed order
    double *red = reinterpret_cast<double *>(smem);
    if (slice)
#pragma unroll
        for (int r = 0; r < B; ++r)
#pragma unroll
            for (int q = 0; q < A / 2; ++q) {
                double *d = red + (((slice - 1) * B + r) * (A / 2) + q) * 128 + 2 * (tid & 63);
                d[0] = (double)tot[r][q].x + (double)ncmp[r][q].x;
                d[1] = (double)tot[r][q].y + (double)ncmp[r][q].y;
            }
    __syncthreads();
    if (slice) return;
#pragma unroll
    for (int r = 0; r < B; ++r) {
        const int j = j0 + ty + 8 * r;
#pragma unroll
        for (int q = 0; q < A / 2; ++q) {
            double v[2] = {(double)tot[r][q].x + (double)ncmp[r][q].x, (double)tot[r][q].y + (double)ncmp[r][q].y};
#pragma unroll
            for (int sl = 0; sl < 3; ++sl) {
                const double *d = red + ((sl * B + r) * (A / 2) + q) * 128 + 2 * tid;
                v[0] += d[0];
                v[1] += d[1];
            }
            const int i = i0 + 2 * (tx + 8 * q);
            if (j < N && i < N) {   // N is even: both pixels of a pair are inside or outside
                dst[(int64_t)j * N + i] = (float)v[0];
                dst[(int64_t)j * N + i + 1] = (float)v[1];
            }
        }
    }
}

// Pixel size as a float pair (hi, lo) with hi + lo = cell to ~2^-48.
inline float2 cell_pair(double cell) {
    const float hi = (float)cell;
    return make_float2(hi, (float)(cell - (double)hi));
}

}  // namespace fp32t
}  // namespace psf
