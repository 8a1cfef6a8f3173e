// Projection basis of one compression (Section 3.3, Eq. 2-3 with the transforms of
// Appendix A).  DCT-II of length N, truncation to L components, L-point inverse DCT and the
// sqrt(L/N) rescale are one linear map Y = P X with
//
//   P[m][n] = (1/N) * [ 1 + 2 * sum_{t=1}^{L-1} cos(pi t (2m+1)/(2L)) * cos(pi t (2n+1)/(2N)) ].
//
// Its entries are evaluated in closed form (basis.cuh), accurate to a few fp64 ulps, and rounded once to fp32 and once to bf16.
#include <algorithm>

#include "basis.cuh"
#include "common.cuh"

namespace freqkv {
namespace {

__global__ void build_basis_kernel(float* __restrict__ p_f32, __nv_bfloat16* __restrict__ p_bf16, int32_t n_in,
                                   int32_t n_keep, int32_t first, int32_t ld, int32_t rows_pad)
{
    const int64_t total = (int64_t)rows_pad * ld;
    const int64_t N = n_in, L = n_keep;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t m = i / ld, n = i % ld;
        double p = 0.0;
        if (m < L && n < N) p = basis_entry(m, n, N, L, first);
        if (p_f32) p_f32[i] = (float)p;
        if (p_bf16) p_bf16[i] = __double2bfloat16(p);
    }
}

// Folded basis for the tensor-core path.  The cosines of the DCT are symmetric or antisymmetric
// under n -> N-1-n and m -> L-1-m according to the parity of the frequency index t, so
// P[m][N-1-n] = Pe[m][n] - Po[m][n] and P[L-1-m][n] = Pe[m][n] - Po[m][n], where Pe (Po) is the part
// of the sum over even (odd) t:  Pe = (P[m][n] + P[m][N-1-n]) / 2,  Po = (P[m][n] - P[m][N-1-n]) / 2.
// Only m < ceil(L/2), n < ceil(N/2) are stored: plane 0 = Pe, plane 1 = Po, each rows_pad x ld,
// zero padded.  For odd N the middle column of Po is zero and that of Pe is P itself, for odd L the
// middle row of Po is zero: the formulas above give exactly that.
// When a band starting at an odd component t0 is retained, the parity of the inverse's index t'
// is opposite to that of t = t0 + t': Pe is then antisymmetric and Po symmetric under m -> L-1-m,
// which only changes a sign in the tensor-core kernel's epilogue.
__global__ void build_folded_basis_kernel(__nv_bfloat16* __restrict__ out, int32_t n_in, int32_t n_keep, int32_t first,
                                          int32_t ld, int32_t rows_pad)
{
    const int64_t plane = (int64_t)rows_pad * ld;
    const int64_t N = n_in, L = n_keep;
    const int64_t Nh = (N + 1) / 2, Lh = (L + 1) / 2;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < plane; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t m = i / ld, n = i % ld;
        double pe = 0.0, po = 0.0;
        if (m < Lh && n < Nh) {
            const double a = basis_entry(m, n, N, L, first), b = basis_entry(m, N - 1 - n, N, L, first);
            pe = 0.5 * (a + b);
            po = 0.5 * (a - b);
        }
        out[i] = __double2bfloat16(pe);
        out[plane + i] = __double2bfloat16(po);
    }
}

// Four blocks.  For even L the even-t part Pe is, up to a factor, the basis of the compression of
// N/2 rows to L/2 (t = 2t': cos(pi t' (2m+1) / (2 (L/2))) cos(pi t' (2n+1) / (2 (N/2)))), so it has the same
// symmetries one level down: with N' = N/2, L' = L/2, n < N'/2, m < ceil(L'/2)
//     Pee[m][n] = (Pe[m][n] + Pe[m][N'-1-n]) / 2,   Peo[m][n] = (Pe[m][n] - Pe[m][N'-1-n]) / 2,
//     s_m = Pee uu + Peo uv,   s_{L'-1-m} = Pee uu - Peo uv,     uu_n = u_n + u_{N'-1-n},  uv_n = u_n - u_{N'-1-n}.
// The odd-t part, t = 2t'+1, has the frequencies of a DCT-IV, z_t' = sum_n v_n cos((2t'+1)(2n+1) phi), phi = pi / (4N').
// Neighbours t' = 2k and 2k - 1 are the cosine of a sum and of a difference of (2n+1) 4k phi and (2n+1) phi, so
//     z_2k = C_k - S_k,  z_{2k-1} = C_k + S_k,   C_k = sum_n cos((2n+1) phi) v_n cos(pi k (2n+1) / N'),  S_k with sines,
// and under n -> N'-1-n the first factor changes cosine and sine while the second keeps (changes) its sign:
//     C_k = sum_{n < N'/2} p_n cos(pi k (2n+1) / N'),  p_n = cos(theta_n) v_n + sin(theta_n) v_{N'-1-n},
//     S_k = sum_{n < N'/2} q_n sin(pi k (2n+1) / N'),  q_n = sin(theta_n) v_n - cos(theta_n) v_{N'-1-n},  theta_n = (2n+1) phi.
// (The splitting of a DCT-IV into two transforms of half its length by plane rotations: Wang, "Fast algorithms for
// the discrete W transform and for the discrete Fourier transform", 1984.)  The inverse of length L' is the transpose
// of the same: with theta'_m = pi (2m+1) / (4L'), d_m = cos(theta'_m) A_m + sin(theta'_m) B_m and
// d_{L'-1-m} = sin(theta'_m) A_m - cos(theta'_m) B_m,
//     A = PA p,  PA[m][n] = (1/N) [D(a+) + D(a-)],   B = PB q,  PB[m][n] = (1/N) [D(a-) - D(a+)],
//     a± = (2m+1) N' ± (2n+1) L',   D(a) = sin((2K+1) pi a / (2N'L')) / sin(pi a / (2N'L')),   K = floor((L'-1) / 2),
// because the retained t' < L' pair up.  For even L' the last one, t' = L'-1 = 2K' - 1 with K' = L'/2, has lost its
// partner: z = C_K' + S_K' both go to B, with weight (2/N) (-1)^m.
// Planes: 0 = Pee, 1 = Peo, 2 = PA, 3 = PB in columns n < N'/2 and, for even L', the weights of p in B behind them.
// The entries of the four planes at (m, n), n < N/2 (planes 0 to 2 end at N/4).
__device__ inline void quad_entries(int64_t m, int64_t n, int64_t N, int64_t L, double (&e)[4])
{
    const int64_t Nh = N / 2, Lh = L / 2, Nq = Nh / 2, Lq = (Lh + 1) / 2;
    const int64_t K1 = 2 * ((Lh - 1) / 2) + 1, unit = 2 * Nh * Lh;  // 2K+1; angles are integer multiples of pi / unit
    auto pe = [&](int64_t c) { return 0.5 * (basis_entry(m, c, N, L, 0) + basis_entry(m, N - 1 - c, N, L, 0)); };
    auto series = [&](int64_t a) {
        if (a == 0) return (double)K1;
        return sinpi((double)((K1 * a) % (2 * unit)) / (double)unit) / sinpi((double)a / (double)unit);
    };
    e[0] = e[1] = e[2] = e[3] = 0.0;
    if (m < Lq && n < Nq) {
        const double a = pe(n), b = pe(Nh - 1 - n);
        e[0] = 0.5 * (a + b);
        e[1] = 0.5 * (a - b);
        const int64_t u = (2 * m + 1) * Nh, w = (2 * n + 1) * Lh;
        const double plus = series(u + w), minus = series(u - w);
        e[2] = (plus + minus) / (double)N;
        e[3] = (minus - plus) / (double)N;
    }
    if (m < Lq && n < 2 * Nq && Lh % 2 == 0) {  // the component without a partner
        const int64_t k = (Lh / 2 * (2 * (n % Nq) + 1)) % (2 * Nh);
        const double x = (double)k / (double)Nh, weight = (m % 2 ? -2.0 : 2.0) / (double)N;
        e[3] += weight * (n < Nq ? sinpi(x) : cospi(x));
    }
}

__device__ inline void store_turns(float2* turns, int64_t n_in, int64_t i0, int64_t step)
{
    for (int64_t n = i0; n < n_in / 4; n += step) {
        double sn, cs;
        sincospi((double)(2 * n + 1) / (double)(2 * n_in), &sn, &cs);  // theta_n
        turns[n] = make_float2((float)cs, (float)sn);
    }
}

// The same blocks, or the two of one level, in fp32 and transposed: [blocks][k_pad][m_pad], zero past the ends.
__global__ void build_fold_f32_kernel(float* __restrict__ out, float2* __restrict__ turns, int32_t n_in, int32_t n_keep, int32_t blocks,
                                      int32_t k_pad, int32_t m_pad)
{
    const int64_t plane = (int64_t)k_pad * m_pad, N = n_in, L = n_keep;
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < plane; i += step) {
        const int64_t n = i / m_pad, m = i % m_pad;
        if (blocks == 4) {
            double e[4];
            quad_entries(m, n, N, L, e);
#pragma unroll
            for (int b = 0; b < 4; ++b) out[b * plane + i] = (float)e[b];
        } else {
            double a = 0.0, b = 0.0;
            if (m < (L + 1) / 2 && n < (N + 1) / 2) {
                a = basis_entry(m, n, N, L, 0);
                b = basis_entry(m, N - 1 - n, N, L, 0);
            }
            out[i] = (float)(0.5 * (a + b));
            out[plane + i] = (float)(0.5 * (a - b));
        }
    }
    if (blocks == 4) store_turns(turns, n_in, i0, step);
}

// The plain orthonormal DCT-II of length N, folded the same way (power-spectrum analysis): plane 0
// holds the even rows C[2m][n], plane 1 the odd rows C[2m+1][n], n < ceil(N/2); applied to
// u_n = x_n + x_{N-1-n} and v_n = x_n - x_{N-1-n} they give the components z_2m and z_2m+1 (for odd N the
// middle column meets u = x once; the odd rows vanish there).  C[t][n] = alpha_t cos(pi t (2n+1) / (2N)),
// the phase t (2n+1) reduced exactly modulo 4N.
__global__ void build_dct_folded_kernel(__nv_bfloat16* __restrict__ out, int32_t n_in, int32_t ld, int32_t rows_pad)
{
    const int64_t plane = (int64_t)rows_pad * ld;
    const int64_t N = n_in, Nh = (N + 1) / 2;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * plane; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t eo = i / plane, j = i % plane, m = j / ld, n = j % ld, t = 2 * m + eo;
        double c = 0.0;
        if (t < N && n < Nh) {
            const int64_t k = (t * (2 * n + 1)) % (4 * N);
            c = (t == 0 ? sqrt(1.0 / (double)N) : sqrt(2.0 / (double)N)) * cospi((double)k / (double)(2 * N));
        }
        out[i] = __double2bfloat16(c);
    }
}

}  // namespace

cudaError_t launch_build_dct_folded(__nv_bfloat16* out, int32_t n_in, int32_t ld, int32_t rows_pad, cudaStream_t stream)
{
    const int64_t total = (int64_t)2 * rows_pad * ld;
    int64_t blocks = std::min<int64_t>((total + 255) / 256, 148 * 32);
    build_dct_folded_kernel<<<(unsigned)std::max<int64_t>(blocks, 1), 256, 0, stream>>>(out, n_in, ld, rows_pad);
    return cudaGetLastError();
}

cudaError_t launch_build_fold_f32(float* out, float2* turns, int32_t n_in, int32_t n_keep, int32_t blocks, int32_t k_pad,
                                  int32_t m_pad, cudaStream_t stream)
{
    const int64_t total = (int64_t)k_pad * m_pad;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 148 * 32));
    build_fold_f32_kernel<<<(unsigned)grid, 256, 0, stream>>>(out, turns, n_in, n_keep, blocks, k_pad, m_pad);
    return cudaGetLastError();
}

cudaError_t launch_build_folded_basis(__nv_bfloat16* out, int32_t n_in, int32_t n_keep, int32_t first, int32_t ld,
                                      int32_t rows_pad, cudaStream_t stream)
{
    const int64_t total = (int64_t)rows_pad * ld;
    const int threads = 256;
    int64_t blocks = (total + threads - 1) / threads;
    if (blocks > 148 * 32) blocks = 148 * 32;
    if (blocks < 1) blocks = 1;
    build_folded_basis_kernel<<<(unsigned)blocks, threads, 0, stream>>>(out, n_in, n_keep, first, ld, rows_pad);
    return cudaGetLastError();
}

cudaError_t launch_build_basis(float* p_f32, __nv_bfloat16* p_bf16, int32_t n_in, int32_t n_keep, int32_t first,
                               int32_t ld, int32_t rows_pad, cudaStream_t stream)
{
    const int64_t total = (int64_t)rows_pad * ld;
    const int threads = 256;
    int64_t blocks = (total + threads - 1) / threads;
    if (blocks > 148 * 32) blocks = 148 * 32;
    if (blocks < 1) blocks = 1;
    build_basis_kernel<<<(unsigned)blocks, threads, 0, stream>>>(p_f32, p_bf16, n_in, n_keep, first, ld, rows_pad);
    return cudaGetLastError();
}

}  // namespace freqkv
