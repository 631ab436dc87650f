// Gridded image-plane approximation: Eq. 45 with Algorithm 1 on the cutout's uv grid.
//
// Eq. 45 writes the image-plane approximation as F^-1{F{P} . D}: the effective PSF P
// is transformed once, and per source position only the distortion D of Algorithm 1
// is evaluated on the uv cells before one inverse transform.  Here the grid is the
// N x N Fourier grid of an N x N cutout of pixel size cell: cells du = dv = 1/(N cell),
// cell (a, b) at u = (a - N/2) du, v = (b - N/2) dv, so that the transform pair is the
// N x N DFT of the cutout's pixel grid.
//
// Position independent, once per (N, cell, precision) and kept by the plan:
//   P  the effective PSF, the cutout at the phase centre where every decorrelation
//      is 1 (computed by the visibility-level path of the plan's precision),
//   S  = F{P} / N^2 (k_grid_dft_rows / k_grid_dft_cols, FP64),
//   per cell the W-weighted means of dt_k and dnu_r / nu_r over the visibilities whose
//      nearest cell is this cell or its mirror, modulo N; cells that receive none take
//      the means over all visibilities (k_grid_cells, FP64 sums); the nearest-cell
//      decision a' = floor(u_k N cell + 0.5), u_k = ubar nu_r / c, is taken in FP64
//      with IEEE round-to-nearest operations in exactly that order,
//   the table G[b][a] = (Re S, Im S, alpha, beta), alpha = omega_E dt_c du and
//      beta = (dnu/nu)_c |u_c|, so that Algorithm 1's half phase changes are
//      A = alpha (a' m0 - b' l0) (theta = atan2(v, u); (b' m0 - a' l0) for the literal
//      arctan(u/v)) and B = beta rho (k_grid_table).
// Per position (k_img_grid): D = sinc(A) sinc(B) on the cells and the real part of
// F^-1{S D}.  With S Hermitian, that real part is F^-1{S D'} where D' averages D over
// each cell and its mirror modulo N; D' differs from D only on the Nyquist row and
// column (a' or b' = -N/2, their own mirrors).  S D' is Hermitian, so the transform runs
// on half the cells: column transforms over b, then per row a real-output transform
// built from one complex transform of half the length, all in shared memory with the
// small DFTs in registers.
#include <cuda_runtime.h>

#include "psf_internal.cuh"

namespace psf {
namespace {

__device__ __forceinline__ int mod_n(int64_t x, int n) {
    const int64_t r = x % n;
    return (int)(r < 0 ? r + n : r);
}

// ------------------------------------------------------------------ table build

__device__ __forceinline__ void cell_flush(double *acc, int c1, int c2, double sw, double sdt, double sr) {
    if (c1 < 0) return;
    atomicAdd(acc + 3 * c1, sw);
    atomicAdd(acc + 3 * c1 + 1, sdt);
    atomicAdd(acc + 3 * c1 + 2, sr);
    atomicAdd(acc + 3 * c2, sw);
    atomicAdd(acc + 3 * c2 + 1, sdt);
    atomicAdd(acc + 3 * c2 + 2, sr);
}

// One thread per (baseline, output channel): walks the baseline's time bins, whose uv
// track stays in one cell for many consecutive bins, and adds its running sums to the
// cell and its mirror whenever the cell changes.  acc[3 q + (0, 1, 2)] = sum W,
// sum W dt, sum W dnu/nu of cell q = b N + a; glob = the same sums over all visibilities.
__global__ void k_grid_cells(const double2 *__restrict__ bin_uv, const int2 *__restrict__ bin_samp,
                             const int32_t *__restrict__ bin_first, const double2 *__restrict__ chan,
                             const float *__restrict__ W, int nbl, int nout, double dt_raw, int N, double ncell,
                             double *__restrict__ acc, double *__restrict__ glob) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double gw = 0, gdt = 0, gr = 0;
    if (t < (int64_t)nbl * nout) {
        const int b = (int)(t / nout), r = (int)(t % nout);
        const double nu = chan[r].x, rr = __ddiv_rn(chan[r].y, nu);
        int c1 = -1, c2 = -1;
        double sw = 0, sdt = 0, sr = 0;
        const int e = bin_first[b + 1];
        for (int bin = bin_first[b]; bin < e; ++bin) {
            const double2 ub = bin_uv[bin];
            const double u = __ddiv_rn(__dmul_rn(ub.x, nu), kCLight);
            const double v = __ddiv_rn(__dmul_rn(ub.y, nu), kCLight);
            const int64_t ia = (int64_t)floor(__dadd_rn(__dmul_rn(u, ncell), 0.5));
            const int64_t ib = (int64_t)floor(__dadd_rn(__dmul_rn(v, ncell), 0.5));
            const int n1 = mod_n(ib + N / 2, N) * N + mod_n(ia + N / 2, N);
            const double w = (double)W[(int64_t)bin * nout + r];
            const double dt = __dmul_rn((double)bin_samp[bin].y, dt_raw);
            if (n1 != c1) {
                cell_flush(acc, c1, c2, sw, sdt, sr);
                c1 = n1;
                c2 = mod_n(-ib + N / 2, N) * N + mod_n(-ia + N / 2, N);
                sw = sdt = sr = 0;
            }
            sw += w;
            sdt += w * dt;
            sr += w * rr;
            gw += w;
            gdt += w * dt;
            gr += w * rr;
        }
        cell_flush(acc, c1, c2, sw, sdt, sr);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        gw += __shfl_xor_sync(0xffffffffu, gw, o);
        gdt += __shfl_xor_sync(0xffffffffu, gdt, o);
        gr += __shfl_xor_sync(0xffffffffu, gr, o);
    }
    if ((threadIdx.x & 31) == 0 && gw != 0.0) {
        atomicAdd(glob, gw);
        atomicAdd(glob + 1, gdt);
        atomicAdd(glob + 2, gr);
    }
}

// exp(-2 pi i m / N) for m in [0, N), in shared memory.
__device__ __forceinline__ void dft_table(double2 *tw, int N) {
    for (int m = threadIdx.x; m < N; m += blockDim.x) {
        double s, c;
        sincospi(2.0 * m / N, &s, &c);
        tw[m] = make_double2(c, -s);
    }
    __syncthreads();
}

__device__ __forceinline__ int twiddle_index(int x, int y, int N) {
    return mod_n((int64_t)(x - N / 2) * (int64_t)(y - N / 2), N);
}

// Y[j][a] = sum_i P[j][i] exp(-2 pi i (a - N/2)(i - N/2) / N); block j, thread a.
__global__ void k_grid_dft_rows(const float *__restrict__ P, double2 *__restrict__ Y, int N) {
    extern __shared__ double2 tw[];
    dft_table(tw, N);
    const int j = blockIdx.x;
    for (int a = threadIdx.x; a < N; a += blockDim.x) {
        double re = 0, im = 0;
        for (int i = 0; i < N; ++i) {
            const double2 w = tw[twiddle_index(a, i, N)];
            const double p = (double)P[(int64_t)j * N + i];
            re += p * w.x;
            im += p * w.y;
        }
        Y[(int64_t)j * N + a] = make_double2(re, im);
    }
}

// S[b][a] = sum_j Y[j][a] exp(-2 pi i (b - N/2)(j - N/2) / N); block b, thread a.
__global__ void k_grid_dft_cols(const double2 *__restrict__ Y, double2 *__restrict__ S, int N) {
    extern __shared__ double2 tw[];
    dft_table(tw, N);
    const int b = blockIdx.x;
    for (int a = threadIdx.x; a < N; a += blockDim.x) {
        double re = 0, im = 0;
        for (int j = 0; j < N; ++j) {
            const double2 w = tw[twiddle_index(b, j, N)];
            const double2 y = Y[(int64_t)j * N + a];
            re += y.x * w.x - y.y * w.y;
            im += y.x * w.y + y.y * w.x;
        }
        S[(int64_t)b * N + a] = make_double2(re, im);
    }
}

// G[b N + a] = (Re S / N^2, Im S / N^2, omega_E dt_c du, (dnu/nu)_c |u_c|) for cell (a, b).
__global__ void k_grid_table(const double2 *__restrict__ S, const double *__restrict__ acc,
                             const double *__restrict__ glob, int N, double du, float4 *__restrict__ G) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (int64_t)N * N) return;
    const int a = (int)(q % N), b = (int)(q / N);
    const double sw = acc[3 * q];
    const double gw = glob[0];
    const double dt = sw > 0 ? acc[3 * q + 1] / sw : (gw > 0 ? glob[1] / gw : 0.0);
    const double r = sw > 0 ? acc[3 * q + 2] / sw : (gw > 0 ? glob[2] / gw : 0.0);
    const double ua = (a - N / 2) * du, vb = (b - N / 2) * du;
    const double inv = 1.0 / ((double)N * N);
    G[q] = make_float4((float)(S[q].x * inv), (float)(S[q].y * inv), (float)(kOmegaE * dt * du),
                                        (float)(r * sqrt(ua * ua + vb * vb)));
}

// ------------------------------------------------------------------ per-position transform

// sinc_pi(x) = sin(pi x) / (pi x) = (-1)^n [sin(pi f) / (pi f)] (f / x), x = n + f, |f| <= 1/2.
// n comes from adding 1.5 * 2^23 (|x| < 2^22), which rounds x to the nearest integer and
// leaves the parity of n in the lowest mantissa bit; the bracket is its Taylor series in
// (pi f)^2 to order 10 (truncation error < 4e-8).  f / x is left as a fraction.
struct SincParts {
    float q, f;
    int parity;
};

__device__ __forceinline__ SincParts sinc_parts(float x) {
    const float t = x + 12582912.0f;
    const float n = t - 12582912.0f;
    const float f = x - n;
    const float z = f * f;
    float q = fmaf(z, -2.3460810e-3f, 2.6147848e-2f);
    q = fmaf(z, q, -1.9075182e-1f);
    q = fmaf(z, q, 8.1174243e-1f);
    q = fmaf(z, q, -1.6449341f);
    q = fmaf(z, q, 1.0f);
    return {q, f, __float_as_int(t)};
}

// (-1)^par sinc_pi(x) sinc_pi(y) for x, y > 0 with one quotient.
__device__ __forceinline__ float sinc2_fast(float x, float y, int par) {
    const SincParts a = sinc_parts(x), b = sinc_parts(y);
    const float v = (a.q * b.q) * __fdividef(a.f * b.f, x * y);
    return __int_as_float(__float_as_int(v) ^ ((a.parity ^ b.parity ^ par) << 31));
}

// (-1)^par D' of a cell (offsets af, bf from the grid's centre): its smearing factor, averaged
// with that of the mirror cell modulo N on the Nyquist row and column.  1e-18 keeps the sincs'
// arguments (their magnitudes; g.z, g.w, rho >= 0) off zero, where f / x = 1, without a select.
__device__ __forceinline__ float cell_factor(const float4 &g, float af, float bf, float lin0, float cx, float cb,
                                             float rho, bool a0, bool b0, int par) {
    const float y = fmaf(g.w, rho, 1e-18f);
    float d = sinc2_fast(fabsf(g.z * fmaf(bf, cb, lin0)) + 1e-18f, y, par);
    if (a0 || b0) {
        const float ma = a0 ? af : -af, mb = b0 ? bf : -bf;
        d = 0.5f * (d + sinc2_fast(fabsf(g.z * fmaf(ma, cx, mb * cb)) + 1e-18f, y, par));
    }
    return d;
}

__host__ __device__ constexpr int ilog2(int r) { return r <= 1 ? 0 : 1 + ilog2(r / 2); }

__host__ __device__ constexpr int bitrev(int i, int r) {
    int o = 0;
    for (int b = 1; b < r; b <<= 1) {
        o = (o << 1) | (i & 1);
        i >>= 1;
    }
    return o;
}

// cos and sin of 2 pi e / 16.
__host__ __device__ constexpr float cos16(int e) {
    return e == 0 ? 1.f : e == 1 ? 0.92387953f : e == 2 ? 0.70710678f : e == 3 ? 0.38268343f
         : e == 4 ? 0.f : e == 5 ? -0.38268343f : e == 6 ? -0.70710678f : -0.92387953f;
}
__host__ __device__ constexpr float sin16(int e) {
    return e == 0 ? 0.f : e == 1 ? 0.38268343f : e == 2 ? 0.70710678f : e == 3 ? 0.92387953f
         : e == 4 ? 1.f : e == 5 ? 0.92387953f : e == 6 ? 0.70710678f : 0.38268343f;
}

// v exp(+2 pi i e / R), 0 <= e < R / 2 (a compile-time constant once unrolled).
template <int R>
__device__ __forceinline__ float2 rot(float2 v, int e) {
    const int e16 = e * (16 / R);
    if (e16 == 0) return v;
    if (e16 == 4) return make_float2(-v.y, v.x);
    const float c = cos16(e16), s = sin16(e16);
    return make_float2(v.x * c - v.y * s, v.x * s + v.y * c);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// In-register inverse DFT y[k] = sum_n x[n] exp(+2 pi i n k / R), R in {2, 4, 8, 16}:
// radix-2 decimation in time, natural order in and out.
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&x)[R]) {
    static_assert(R == 2 || R == 4 || R == 8 || R == 16, "radix");
    float2 t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) t[bitrev(i, R)] = x[i];
#pragma unroll
    for (int st = 0; st < ilog2(R); ++st) {
        const int m = 1 << st;
#pragma unroll
        for (int s = 0; s < R; s += 2 * m)
#pragma unroll
            for (int k = 0; k < m; ++k) {
                const float2 u = t[s + k];
                const float2 v = rot<R>(t[s + k + m], k * (R / (2 * m)));
                t[s + k] = make_float2(u.x + v.x, u.y + v.y);
                t[s + k + m] = make_float2(u.x - v.x, u.y - v.y);
            }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) x[i] = t[i];
}

// Shapes: the column transforms (length N over b) run as R1 x R2 Cooley-Tukey, the row
// transforms (length M = N/2, the complex core of each real row) as Q1 x Q2; T threads.
template <int N>
struct GridFft;
template <>
struct GridFft<16> { static constexpr int R1 = 4, R2 = 4, Q1 = 4, Q2 = 2, T = 64; };
template <>
struct GridFft<32> { static constexpr int R1 = 8, R2 = 4, Q1 = 4, Q2 = 4, T = 128; };
template <>
struct GridFft<64> { static constexpr int R1 = 8, R2 = 8, Q1 = 8, Q2 = 4, T = 128; };
template <>
struct GridFft<128> { static constexpr int R1 = 16, R2 = 8, Q1 = 8, Q2 = 8, T = 256; };

// Row stride of Z in k_img_grid: Q2 past the M columns, so that the rows a half warp works on
// (16 / Q2 of them, Q2 lanes each) fall on different banks.
template <int N>
__host__ __device__ constexpr int grid_ld() { return N / 2 + GridFft<N>::Q2; }

template <int N>
constexpr int grid_smem_bytes() { return (N * grid_ld<N>() + N) * (int)sizeof(float2); }

template <int N>
constexpr int grid_min_blocks() { return N == 128 ? 3 : N == 64 ? 6 : 8; }

// One CTA per position (grid-stride).  X = (-1)^(a+b) S D' is Hermitian, so only the
// cells a in [0, N/2] are formed, with the N twiddles exp(+2 pi i m / N) in shared memory.
// Z [N rows][LD] holds what passes between the stages: row c = b + N/2 modulo N (this rotation
// is the sign (-1)^j of the outputs), later output row j.
//   (0) the columns a = 0 and a = N/2 of X into Z's columns M and M + 1
//   (1) columns: length-N inverse DFT over b for a in [0, N/2), the first stage on cells that
//       the thread forms itself; column 0 carries X[.][0] + i X[.][N/2], whose transforms are
//       both real, and is unpacked into them
//   (2) rows: each row j is Hermitian in a, and its real inverse DFT x is obtained from
//       one length-N/2 complex DFT of C[k] = E[k] + i O[k], E[k] = Z[k] + conj Z[N/2 - k],
//       O[k] = (Z[k] - conj Z[N/2 - k]) exp(2 pi i k / N): it returns x[2n] + i x[2n+1];
//       out[j][i] = (-1)^i x[i], two floats per store.
// Cell and pixel index origins are at N/2: exp(2 pi i (a - N/2)(i - N/2) / N) =
// (-1)^(a + i) exp(2 pi i a i / N) for N % 4 == 0.
//
// Bound by instruction issue (268 MB written for 4096 positions of 128 pixels take 40 us).  With
// X written to Z before the first stage, block-wide exchanges between all stages and the result
// once more through Z those took 250 us; 201 us now.  The first stage works on its own cells,
// the second stage of the columns in place (stage one stores (n2, k1) as row k1 + R1 n2, from
// where the thread that takes k1 reads and to where it writes), a row stays within one warp
// (these: 212 us), the two sincs of a cell share a quotient, signs are integer operations on
// the sinc's and rotations of the rows, and a lane keeps its twiddles of the row pass.
template <int N>
__global__ void __launch_bounds__(GridFft<N>::T, grid_min_blocks<N>())
    k_img_grid(const float4 *__restrict__ G, const GridPos *__restrict__ pos, int npos, float *__restrict__ out) {
    using F = GridFft<N>;
    constexpr int M = N / 2, LD = grid_ld<N>(), T = F::T, R1 = F::R1, R2 = F::R2, Q1 = F::Q1, Q2 = F::Q2;
    constexpr int RW = 32 / Q2;   // rows of a warp at a time
    static_assert(R1 * R2 == N && Q1 * Q2 == M && Q1 % Q2 == 0 && R2 % 2 == 0 && N % RW == 0, "shape");
    extern __shared__ float2 smem[];
    float2 *Z = smem;
    float2 *tw = smem + N * LD;
    for (int m = threadIdx.x; m < N; m += T) {
        float s, c;
        sincospif(2.0f * (float)m / (float)N, &s, &c);
        tw[m] = make_float2(c, s);
    }
    const int lane = threadIdx.x & 31;
    for (int p = blockIdx.x; p < npos; p += gridDim.x) {
        const GridPos gp = pos[p];
        const float cx = gp.c.x, cb = gp.c.y, rho = gp.c.z;
        // (0)
        for (int it = threadIdx.x; it < 2 * N; it += T) {
            const int b = it % N, h = it / N;   // column a = h M
            const float4 g = __ldg(G + b * N + h * M);
            const float af = h ? 0.f : (float)(-M), bf = (float)(b - M);
            // on column M the mirror cell (a' = 0, -b') has the same D (D is even)
            const float d = cell_factor(g, af, bf, af * cx, cx, cb, rho, h == 0, h == 0 && b == 0, b);
            Z[(b ^ M) * LD + M + h] = make_float2(g.x * d, g.y * d);
        }
        __syncthreads();
        // (1a) R1-point DFT over c = n2 + R2 n1, twiddle exp(2 pi i n2 k1 / N), to row k1 + R1 n2
#pragma unroll 1
        for (int it = threadIdx.x; it < M * R2; it += T) {
            const int a = it % M, n2 = it / M;
            const float af = (float)(a - M), lin0 = af * cx, c0 = (float)n2;
            const float4 *g0 = G + n2 * N + a;
            float2 x[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1) {
                const int off = R2 * n1 < M ? R2 * n1 : R2 * n1 - N;   // b - M = n2 + off
                const float4 g = __ldg(g0 + (off + M) * N);
                const float d = cell_factor(g, af, c0 + (float)off, lin0, cx, cb, rho, false, off == -M && n2 == 0,
                                            a + n2);   // R2 and M are even
                x[n1] = make_float2(g.x * d, g.y * d);
            }
            if (a == 0) {
#pragma unroll
                for (int n1 = 0; n1 < R1; ++n1) {
                    const float2 *z = Z + (n2 + R2 * n1) * LD + M;
                    x[n1] = make_float2(z[0].x - z[1].y, z[0].y + z[1].x);
                }
            }
            dft_reg<R1>(x);
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1) Z[(k1 + R1 * n2) * LD + a] = cmul(x[k1], tw[n2 * k1]);
        }
        __syncthreads();
        // (1b) R2-point DFT over n2 for each (a, k1), in place: output rows j = k1 + R1 k2
#pragma unroll 2
        for (int it = threadIdx.x; it < M * R1; it += T) {
            const int a = it % M, k1 = it / M;
            float2 *z = Z + k1 * LD;
            float2 y[R2];
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2) y[n2] = z[R1 * n2 * LD + a];
            dft_reg<R2>(y);
            if (a == 0) {
#pragma unroll
                for (int k2 = 0; k2 < R2; ++k2) {
                    z[R1 * k2 * LD] = make_float2(y[k2].x, 0.f);
                    z[R1 * k2 * LD + M] = make_float2(y[k2].y, 0.f);
                }
            } else {
#pragma unroll
                for (int k2 = 0; k2 < R2; ++k2) z[R1 * k2 * LD + a] = y[k2];
            }
        }
        __syncthreads();
        // (2) RW rows per warp and turn.  (2a) C[k] for k = n2 + Q2 n1, Q1-point DFT over n1, twiddle
        // exp(2 pi i n2 k1 / M) = tw[2 n2 k1]; exchanged within the row at k1 Q2 + (n2 + k1) % Q2
        // (banks).  (2b) Q2-point DFT over n2 for each k1: y[k1 + Q1 k2] = x[2n] + i x[2n+1].
        const int n2 = lane % Q2;
        float2 ta[Q1], tb[Q1];   // the lane's twiddles
#pragma unroll
        for (int n1 = 0; n1 < Q1; ++n1) {
            ta[n1] = tw[n2 + Q2 * n1];
            tb[n1] = tw[2 * n2 * n1];
        }
        float *o = out + gp.off;
        const bool wide = (reinterpret_cast<uintptr_t>(o) & 7) == 0;   // the caller's buffer may start at any float
#pragma unroll 1
        for (int j0 = (threadIdx.x / 32) * RW; j0 < N; j0 += (T / 32) * RW) {
            float2 *z = Z + (j0 + lane / Q2) * LD;
            float2 c[Q1];
#pragma unroll
            for (int n1 = 0; n1 < Q1; ++n1) {
                const int k = n2 + Q2 * n1;
                const float2 zk = z[k], zm = z[M - k];
                const float2 e = make_float2(zk.x + zm.x, zk.y - zm.y);
                const float2 od = cmul(make_float2(zk.x - zm.x, zk.y + zm.y), ta[n1]);
                c[n1] = make_float2(e.x - od.y, e.y + od.x);
            }
            dft_reg<Q1>(c);
            __syncwarp();
#pragma unroll
            for (int k1 = 0; k1 < Q1; ++k1) z[k1 * Q2 + (n2 + k1) % Q2] = cmul(c[k1], tb[k1]);
            __syncwarp();
#pragma unroll
            for (int h = 0; h < Q1 / Q2; ++h) {
                const int q = h * 32 + lane, k1 = q % Q1, j = j0 + q / Q1;
                const float2 *zr = Z + j * LD + k1 * Q2;
                float2 y[Q2];
#pragma unroll
                for (int i = 0; i < Q2; ++i) y[i] = zr[(i + k1) % Q2];
                dft_reg<Q2>(y);
                float *oj = o + j * N + 2 * k1;
#pragma unroll
                for (int k2 = 0; k2 < Q2; ++k2) {
                    const float2 v = make_float2(y[k2].x, -y[k2].y);
                    if (wide) {
                        __stcs(reinterpret_cast<float2 *>(oj + 2 * Q1 * k2), v);
                    } else {
                        __stcs(oj + 2 * Q1 * k2, v.x);
                        __stcs(oj + 2 * Q1 * k2 + 1, v.y);
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <int N>
cudaError_t launch_img_grid_n(const float4 *G, const GridPos *pos, int npos, float *out, int nsm, cudaStream_t st) {
    constexpr int smem = grid_smem_bytes<N>();
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_img_grid<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    int per_sm = 1;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_img_grid<N>, GridFft<N>::T, smem);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<int64_t>(npos, (int64_t)nsm * std::max(1, per_sm) * 4);
    k_img_grid<N><<<grid, GridFft<N>::T, smem, st>>>(G, pos, npos, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ CLEAN loop
// Algorithm 2's loop on one cluster of eight CTAs, many iterations per launch.  As separate
// kernels an iteration took 27.6 us on a 2048^2 image with N = 128: the argmax read the whole
// image (5.7 us), one CTA evaluated the PSF (15 us), and four launches followed one another.
// Here
//   * the peak is found from per-row maxima: the window of an iteration changes N rows, and
//     each CTA renews the maxima of its own N/8 of them (per 64-pixel segment, then per row);
//   * the PSF's columns, then its rows, are shared by the CTAs, exchanged through distributed
//     shared memory, with k_img_grid's cells and transforms;
//   * cluster barriers order everything.  Gridded: (1) the columns' results lie in the row
//     owners' shared memory, (2) the rows are done (their centre is read remotely), (3) residual
//     and keys are renewed; no CTA renews keys before (1) and (2), which follow everyone's
//     reading of them.  One given PSF: a barrier between the reading and the renewal, and (3).
// 10.9 us per iteration.  FACET: one given PSF (P, any even N) instead of the gridded one.
// Maxima are 64-bit keys as k_clean_argmax forms them (value, then the first pixel).
constexpr int kClCtas = 8, kClThreads = 256, kClSeg = 64;

__device__ __forceinline__ unsigned long long clean_key(float v, int64_t pix) {
    const unsigned int u = __float_as_uint(v);
    const unsigned int o = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)o << 32) | (unsigned long long)(0xffffffffu - (unsigned int)pix);
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long k) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, k, o);
        k = x > k ? x : k;
    }
    return k;
}
// Keys of the segments s0 .. s1 of row y, then of the row, by one warp.  Residual and keys
// are read past L1: other CTAs of the cluster write them.
__device__ __forceinline__ void clean_row_keys(const float *res, int y, int nl, int nseg, int s0, int s1,
                                               unsigned long long *seg, unsigned long long *row) {
    const int lane = threadIdx.x & 31;
    for (int s = s0; s <= s1; ++s) {
        unsigned long long k = 0;
#pragma unroll
        for (int h = 0; h < kClSeg; h += 32) {
            const int x = s * kClSeg + h + lane;
            if (x < nl) {
                const int64_t pix = (int64_t)y * nl + x;
                const unsigned long long q = clean_key(__ldcg(res + pix), pix);
                k = q > k ? q : k;
            }
        }
        k = warp_max(k);
        if (lane == 0) seg[(int64_t)y * nseg + s] = k;
    }
    __syncwarp();
    unsigned long long k = 0;
    for (int s = lane; s < nseg; s += 32) {
        const unsigned long long q = __ldcg(seg + (int64_t)y * nseg + s);
        k = q > k ? q : k;
    }
    k = warp_max(k);
    if (lane == 0) row[y] = k;
}

__global__ void __launch_bounds__(256) k_clean_keys(const float *__restrict__ res, int nl, int nm, int nseg,
                                                    unsigned long long *__restrict__ seg,
                                                    unsigned long long *__restrict__ row) {
    for (int y = blockIdx.x * 8 + (threadIdx.x >> 5); y < nm; y += gridDim.x * 8)
        clean_row_keys(res, y, nl, nseg, 0, nseg - 1, seg, row);
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {   // p's address in CTA `rank`
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ float cluster_load(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int N, bool FACET>
__global__ void __launch_bounds__(kClThreads) __cluster_dims__(kClCtas, 1, 1)
    k_clean_loop(const float4 *__restrict__ G, const float *__restrict__ Pf, int nf, float *res, float *__restrict__ model,
                 CleanState *st, int nl, int nm, double cell, double lc, double mc, float gain, float threshold, int max_iter,
                 int chunk, int literal, int32_t *__restrict__ comp_pix, float *__restrict__ comp_flux,
                 unsigned long long *seg, unsigned long long *row) {
    using F = GridFft<N>;
    constexpr int M = N / 2, LD = M + 1, R1 = F::R1, R2 = F::R2, Q1 = F::Q1, Q2 = F::Q2, T = kClThreads;
    constexpr int CA = M / kClCtas, LC = CA + 1, NR = N / kClCtas;   // columns and rows of a CTA
    static_assert(M % kClCtas == 0 && NR * Q2 <= T && NR * Q1 <= T, "cluster shape");
    __shared__ float4 Gc[FACET ? 1 : N * CA + N];   // this CTA's cells (and column M in CTA 0)
    __shared__ float2 Zc[FACET ? 1 : N * LC];       // its columns
    __shared__ float2 Zr[FACET ? 1 : NR * LD];      // its rows
    __shared__ float2 tw[FACET ? 1 : N];
    __shared__ unsigned long long wbest[T / 32];
    __shared__ float gpos[3];
    const int c = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nseg = (nl + kClSeg - 1) / kClSeg;
    const int np = FACET ? nf : N, half = np / 2;             // window size
    const int rows = (np + kClCtas - 1) / kClCtas;            // window rows of a CTA
    if (!FACET) {
        for (int m = tid; m < N; m += T) {
            float s, cc;
            sincospif(2.0f * (float)m / (float)N, &s, &cc);
            tw[m] = make_float2(cc, s);
        }
        for (int it = tid; it < N * CA; it += T) Gc[it] = G[(it / CA) * N + c * CA + it % CA];
        if (c == 0)
            for (int b = tid; b < N; b += T) Gc[N * CA + b] = G[b * N + M];
    }
    int iter = st->iter;
    const int stop_at = min(max_iter, iter + chunk);
    bool done = st->done != 0;
    // every CTA of the cluster runs before its shared memory is written by another (and this
    // CTA's tables are filled)
    cluster_barrier();
    while (!done && iter < stop_at) {
        // peak: every CTA takes the maximum of all row keys
        unsigned long long k = 0;
        for (int y = tid; y < nm; y += T) {
            const unsigned long long q = __ldcg(row + y);
            k = q > k ? q : k;
        }
        k = warp_max(k);
        if (lane == 0) wbest[warp] = k;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < T / 32; ++w) k = wbest[w] > k ? wbest[w] : k;
        const int pix = (int)(0xffffffffu - (unsigned int)(k & 0xffffffffull));
        const unsigned int ob = (unsigned int)(k >> 32);
        const float peak = __uint_as_float((ob & 0x80000000u) ? (ob & 0x7fffffffu) : ~ob);
        if (iter > 0 && !(peak > threshold)) {   // the same decision in every thread of the cluster
            done = true;
            break;
        }
        const int px = pix % nl, py = pix / nl;
        const float g = gain * peak;
        float scale;
        if (FACET) {
            scale = g / Pf[half * np + half];
            cluster_barrier();   // every CTA has read the row keys before one renews its own
        } else {
            if (tid == 0) {
                const double l0 = lc + (px - nl / 2) * cell, m0 = mc + (py - nm / 2) * cell;
                gpos[0] = literal ? (float)-l0 : (float)m0;
                gpos[1] = literal ? (float)m0 : (float)-l0;
                gpos[2] = (float)sqrt(l0 * l0 + m0 * m0);
            }
            __syncthreads();
            const float cx = gpos[0], cb = gpos[1], rho = gpos[2];
            // (0) X on this CTA's cells (k_img_grid)
#pragma unroll 4
            for (int it = tid; it < N * CA; it += T) {
                const int al = it % CA, b = it / CA, a = c * CA + al;
                const float4 q = Gc[it];
                const float af = (float)(a - M), lin0 = af * cx, bf = (float)(b - M);
                const float d = cell_factor(q, af, bf, lin0, cx, cb, rho, a == 0, b == 0, a + b);
                Zc[b * LC + al] = make_float2(q.x * d, q.y * d);
            }
            if (c == 0)
                for (int b = tid; b < N; b += T) {
                    const float4 q = Gc[N * CA + b];
                    const float bf = (float)(b - M);
                    const float d = cell_factor(q, 0.f, bf, 0.f, cx, cb, rho, false, false, b);   // M is even
                    Zc[b * LC + CA] = make_float2(q.x * d, q.y * d);
                }
            __syncthreads();
            // (1a), (1b) columns; the results go to the CTAs that own the rows
            for (int it = tid; it < CA * R2; it += T) {
                const int al = it % CA, n2 = it / CA;
                float2 x[R1];
#pragma unroll
                for (int n1 = 0; n1 < R1; ++n1) {
                    const int r = (n2 + R2 * n1) * LC;
                    float2 v = Zc[r + al];
                    if (c == 0 && al == 0) {
                        const float2 w = Zc[r + CA];
                        v = make_float2(v.x - w.y, v.y + w.x);
                    }
                    x[n1] = v;
                }
                dft_reg<R1>(x);
#pragma unroll
                for (int k1 = 0; k1 < R1; ++k1) Zc[(n2 + R2 * k1) * LC + al] = cmul(x[k1], tw[n2 * k1]);
            }
            __syncthreads();
            for (int it = tid; it < CA * R1; it += T) {
                const int al = it % CA, k1 = it / CA, a = c * CA + al;
                float2 y[R2];
#pragma unroll
                for (int n2 = 0; n2 < R2; ++n2) y[n2] = Zc[(R2 * k1 + n2) * LC + al];
                dft_reg<R2>(y);
#pragma unroll
                for (int k2 = 0; k2 < R2; ++k2) {
                    const int r = k1 + R1 * k2, own = r / NR;
                    float2 *z = Zr + (r % NR) * LD;
                    if (a == 0) {
                        cluster_store(cluster_addr(z, own), make_float2(y[k2].x, 0.f));
                        cluster_store(cluster_addr(z + M, own), make_float2(y[k2].y, 0.f));
                    } else {
                        cluster_store(cluster_addr(z + a, own), y[k2]);
                    }
                }
            }
            cluster_barrier();
            // (2a), (2b) rows
            {
                float2 v[Q1];
                const int j = tid % NR, n2 = tid / NR;
                const bool on = tid < NR * Q2;
                if (on) {
#pragma unroll
                    for (int n1 = 0; n1 < Q1; ++n1) {
                        const int kk = n2 + Q2 * n1;
                        const float2 zk = Zr[j * LD + kk], zm = Zr[j * LD + M - kk];
                        const float2 e = make_float2(zk.x + zm.x, zk.y - zm.y);
                        const float2 o = cmul(make_float2(zk.x - zm.x, zk.y + zm.y), tw[kk]);
                        v[n1] = make_float2(e.x - o.y, e.y + o.x);
                    }
                }
                __syncthreads();
                if (on) {
                    dft_reg<Q1>(v);
#pragma unroll
                    for (int k1 = 0; k1 < Q1; ++k1) Zr[j * LD + n2 + Q2 * k1] = cmul(v[k1], tw[2 * n2 * k1]);
                }
            }
            __syncthreads();
            {
                float2 v[Q2];
                const int j = tid % NR, k1 = tid / NR;
                const bool on = tid < NR * Q1;
                if (on) {
#pragma unroll
                    for (int n2 = 0; n2 < Q2; ++n2) v[n2] = Zr[j * LD + Q2 * k1 + n2];
                }
                __syncthreads();
                if (on) {
                    dft_reg<Q2>(v);
#pragma unroll
                    for (int k2 = 0; k2 < Q2; ++k2) Zr[j * LD + k1 + Q1 * k2] = v[k2];
                }
            }
            cluster_barrier();
            // centre pixel (row N/2, sign +)
            scale = g / cluster_load(cluster_addr(Zr + ((N / 2) % NR) * LD + N / 4, (N / 2) / NR));
        }
        // subtract on this CTA's window rows, then renew the rows' maxima
        const int x0 = max(0, px - half), x1 = min(nl, px - half + np);
        for (int e = tid; e < rows * np; e += T) {
            const int jl = e / np, i = e - jl * np, j = c * rows + jl;
            const int x = px + i - half, y = py + j - half;
            if (j >= np || x < 0 || x >= nl || y < 0 || y >= nm) continue;
            float P;
            if (FACET) {
                P = Pf[(int64_t)j * np + i];
            } else {
                const float2 v = Zr[jl * LD + (i >> 1)];
                const float sg = (j & 1) ? -1.f : 1.f;
                P = (i & 1) ? -sg * v.y : sg * v.x;
            }
            float *r = res + (int64_t)y * nl + x;
            *r = __ldcg(r) - scale * P;
        }
        if (c == 0 && tid == 0) {
            if (model) model[pix] += g;
            if (comp_pix) comp_pix[iter] = pix;
            if (comp_flux) comp_flux[iter] = g;
        }
        __syncthreads();
        for (int jl = warp; jl < rows; jl += T / 32) {
            const int j = c * rows + jl, y = py + j - half;
            if (j < np && y >= 0 && y < nm && x1 > x0)
                clean_row_keys(res, y, nl, nseg, x0 / kClSeg, (x1 - 1) / kClSeg, seg, row);
        }
        ++iter;
        cluster_barrier();
    }
    cluster_barrier();   // no CTA leaves while its shared memory or the record may be read
    if (c == 0 && tid == 0) {
        st->iter = iter;
        st->done = done || iter >= max_iter;
    }
}

template <int N, bool FACET>
cudaError_t launch_clean_loop_t(const float4 *G, const float *P, int nf, float *res, float *model, CleanState *st, int nl,
                                int nm, double cell, double lc, double mc, float gain, float threshold, int max_iter,
                                int chunk, int literal, int32_t *cpix, float *cflux, unsigned long long *seg,
                                unsigned long long *row, cudaStream_t s) {
    k_clean_loop<N, FACET><<<kClCtas, kClThreads, 0, s>>>(G, P, nf, res, model, st, nl, nm, cell, lc, mc, gain, threshold,
                                                          max_iter, chunk, literal, cpix, cflux, seg, row);
    return cudaGetLastError();
}

}  // namespace

bool img_grid_supported(int N) { return N == 16 || N == 32 || N == 64 || N == 128; }

cudaError_t launch_grid_cells(const double2 *bin_uv, const int2 *bin_samp, const int32_t *bin_first,
                              const double2 *chan, const float *W, int nbl, int nout, double dt_raw, int N,
                              double ncell, double *acc, double *glob, cudaStream_t st) {
    const int64_t n = (int64_t)nbl * nout;
    const int threads = 256;
    k_grid_cells<<<(unsigned)((n + threads - 1) / threads), threads, 0, st>>>(bin_uv, bin_samp, bin_first, chan, W,
                                                                             nbl, nout, dt_raw, N, ncell, acc, glob);
    return cudaGetLastError();
}

cudaError_t launch_grid_dft(const float *P, double2 *Y, double2 *S, int N, cudaStream_t st) {
    const int threads = std::min(N, 256);
    const size_t smem = (size_t)N * sizeof(double2);
    k_grid_dft_rows<<<N, threads, smem, st>>>(P, Y, N);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_grid_dft_cols<<<N, threads, smem, st>>>(Y, S, N);
    return cudaGetLastError();
}

cudaError_t launch_grid_table(const double2 *S, const double *acc, const double *glob, int N, double du,
                              float4 *G, cudaStream_t st) {
    const int64_t n = (int64_t)N * N;
    k_grid_table<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(S, acc, glob, N, du, G);
    return cudaGetLastError();
}

size_t clean_keys_bytes(int nl, int nm) {
    return ((size_t)nm * ((nl + kClSeg - 1) / kClSeg) + nm) * sizeof(unsigned long long);
}

cudaError_t launch_clean_keys(const float *res, int nl, int nm, void *keys, int nsm, cudaStream_t s) {
    const int nseg = (nl + kClSeg - 1) / kClSeg;
    unsigned long long *row = (unsigned long long *)keys, *seg = row + nm;
    k_clean_keys<<<std::min((nm + 7) / 8, 8 * nsm), 256, 0, s>>>(res, nl, nm, nseg, seg, row);
    return cudaGetLastError();
}

cudaError_t launch_clean_loop(const float4 *G, const float *P, int N, float *res, float *model, CleanState *st, int nl,
                              int nm, double cell, double lc, double mc, float gain, float threshold, int max_iter,
                              int chunk, int literal, int32_t *cpix, float *cflux, void *keys, cudaStream_t s) {
    unsigned long long *row = (unsigned long long *)keys, *seg = row + nm;
#define PSF_CLEAN_LOOP(NN, FACET)                                                                                      \
    return launch_clean_loop_t<NN, FACET>(G, P, N, res, model, st, nl, nm, cell, lc, mc, gain, threshold, max_iter, chunk, \
                                          literal, cpix, cflux, seg, row, s)
    if (P) PSF_CLEAN_LOOP(16, true);
    switch (N) {
        case 16: PSF_CLEAN_LOOP(16, false);
        case 32: PSF_CLEAN_LOOP(32, false);
        case 64: PSF_CLEAN_LOOP(64, false);
        case 128: PSF_CLEAN_LOOP(128, false);
        default: return cudaErrorInvalidValue;
    }
#undef PSF_CLEAN_LOOP
}

cudaError_t launch_img_grid(const float4 *G, const GridPos *pos, int npos, int N, float *out, int nsm,
                            cudaStream_t st) {
    if (npos <= 0) return cudaSuccess;
    switch (N) {
        case 16: return launch_img_grid_n<16>(G, pos, npos, out, nsm, st);
        case 32: return launch_img_grid_n<32>(G, pos, npos, out, nsm, st);
        case 64: return launch_img_grid_n<64>(G, pos, npos, out, nsm, st);
        case 128: return launch_img_grid_n<128>(G, pos, npos, out, nsm, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace psf
