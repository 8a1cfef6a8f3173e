// fp32 caches whose lengths are no powers of two: the projection Y = P X on the CUDA cores (Section 3.3,
// Eq. 2-3 with the transforms of Appendix A folded into P), with the symmetries of the basis taken out first.
//
// One level (any lengths): u, v = x_n +- x_{N-1-n} and S = Pe u, D = Po v, y_m = S + D, y_{L-1-m} = S - D: half the
// multiply-adds of the plain product.  Four blocks (N a multiple of 4, L even): uu, uv, p, q and Pee, Peo, PA, PB of
// a quarter of each length (derived in basis.cu): a quarter of them.  All of it stays in fp32; the sums are two
// and four times shorter than the plain product's.
//
//   fold_f32_kernel      reads every non-sink row once and writes the 2 or 4 folded planes to scratch; HBM- or L2-bound.
//   product_f32_kernel   one CTA computes TM rows x TN channels of one block of one matrix; slices of 16 folded rows come
//                        through a ring of cp.async stages (the basis is stored transposed, so both operands arrive in
//                        the order they are read in).  Bound by FFMA issue: a thread owns 8 x 8 products, 64 FFMA for
//                        four 16-byte shared-memory loads, and a warp reads 4 x 8 distinct vectors of each operand.
//   unfold_f32_kernel    combines the blocks and stores the 2 or 4 output rows of each folded row into the cache.
// Only the last kernel writes the cache, and the ones before it are done reading it by then: safe in place.
//
// Large values.  An infinite element is infinite in every folded row it enters, so sums and differences of these would be NaN where
// the plain product has an infinity, and values near the end of the range would overflow in a sum of four.  The fold therefore looks at
// the magnitudes that pass through it (free: it waits for memory), and a matrix with an element of 2^100 or more takes the
// plain product after all, with its entries evaluated on the spot.  Below that nothing overflows: entries are below 1, |p|, |q| and
// a sum of four below 2^102, and four sums of 2^23 of these below the end of the range.  What the look at the flags costs: 64
// matrices 2044 -> 1022 nothing (229 us with the append), few kept rows in tiles of one warp up to a tenth (4000 -> 16 161 -> 183 us, the
// plain product 281; 66 -> 64 of 2048 matrices 50 -> 55, 62).
//
// Measured against the plain product (64 matrices of 128 channels unless said): 2044 -> 1022 959 -> 212 us, odd lengths
// 2043 -> 1021 959 -> 387 us, 4000 -> 2000 3655 -> 1040 us, 2 matrices 2044 -> 1022 107 -> 23 us; error against 64 bits
// 5.7e-7 -> 2.8e-7.  (All blocks of a tile in one CTA, combined in registers without a third kernel, left a thread 4 x 4
// products of each and took 253 us.)
#include <algorithm>

#include "basis.cuh"
#include "common.cuh"

namespace freqkv {
namespace {

constexpr int TK = 16, STAGES = 3;
constexpr int MOST_SHARES = 64;                 // blocks per matrix of the first and the last kernel
constexpr float LARGE = 1.2676506002282294e30f;  // 2^100

__device__ __forceinline__ float largest(float m, const float4& v)
{
    return fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));  // a NaN is no obstacle to folding
}

// Has a block of the fold seen a large value of this matrix?  The same answer for all threads of the block.
__device__ __forceinline__ bool any_large(const int32_t* flags, int32_t mat, int32_t shares)
{
    int32_t f = 0;
    for (int32_t i = threadIdx.x; i < shares; i += blockDim.x) f |= __ldg(flags + (size_t)mat * MOST_SHARES + i);
    return __syncthreads_or(f);
}

// Planes of one matrix: [blocks][rows of a plane][head_dim]; rows = ceil(n_in / blocks).
template <int BLOCKS>
__global__ void __launch_bounds__(256) fold_f32_kernel(const CacheView view, int32_t first, int32_t n_in, int32_t sink,
                                                       const float2* __restrict__ turns, float4* __restrict__ planes,
                                                       int32_t* __restrict__ flags)
{
    const uint32_t vecs = (uint32_t)view.head_dim / 4;
    const uint32_t rows = (uint32_t)(n_in + BLOCKS - 1) / BLOCKS, plane = rows * vecs;
    const int32_t mat = first + (int32_t)blockIdx.x, tensor = mat / view.mats_per_tensor;
    const float* x = static_cast<const float*>(tensor_base(view, tensor)) + matrix_offset(view, mat % view.mats_per_tensor) +
                     (int64_t)sink * view.stride_token;
    float4* out = planes + (size_t)blockIdx.x * BLOCKS * plane;
    auto row = [&](int32_t n, uint32_t vec) { return __ldg(reinterpret_cast<const float4*>(x + (int64_t)n * view.stride_token) + vec); };
    float most = 0.f;
    for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < plane; i += gridDim.y * blockDim.x) {
        const int32_t n = (int32_t)(i / vecs);
        const uint32_t vec = i - (uint32_t)n * vecs;
        const float4 a = row(n, vec), b = row(n_in - 1 - n, vec);
        most = largest(largest(most, a), b);
        const float4 u = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        const float4 v = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
        if constexpr (BLOCKS == 2) {
            const bool middle = n_in - 1 - n == n;  // the middle row of an odd length enters u once and v as zero (a - a)
            out[i] = middle ? a : u;
            out[plane + i] = v;
        } else {
            const float4 c = row(n_in / 2 - 1 - n, vec), d = row(n_in / 2 + n, vec);
            most = largest(largest(most, c), d);
            const float4 u2 = make_float4(c.x + d.x, c.y + d.y, c.z + d.z, c.w + d.w);
            const float4 v2 = make_float4(c.x - d.x, c.y - d.y, c.z - d.z, c.w - d.w);
            const float2 t = __ldg(turns + n);
            out[i] = make_float4(u.x + u2.x, u.y + u2.y, u.z + u2.z, u.w + u2.w);
            out[plane + i] = make_float4(u.x - u2.x, u.y - u2.y, u.z - u2.z, u.w - u2.w);
            out[2 * plane + i] = make_float4(fmaf(t.y, v.x, -t.x * v2.x), fmaf(t.y, v.y, -t.x * v2.y), fmaf(t.y, v.z, -t.x * v2.z),
                                             fmaf(t.y, v.w, -t.x * v2.w));  // q
            out[3 * plane + i] = make_float4(fmaf(t.x, v.x, t.y * v2.x), fmaf(t.x, v.y, t.y * v2.y), fmaf(t.x, v.z, t.y * v2.z),
                                             fmaf(t.x, v.w, t.y * v2.w));   // p
        }
    }
    const int32_t large = __syncthreads_or(most >= LARGE);
    if (threadIdx.x == 0) flags[(size_t)blockIdx.x * MOST_SHARES + blockIdx.y] = large;
}

struct ProductParams {
    const float* basis;      // [blocks][basis_k][m_pad]: transposed, zero past the ends
    const float* planes;     // [matrix][blocks][rows][head_dim]
    float* out;              // [matrix][blocks][rows_out][head_dim]
    int32_t head_dim, blocks, m_pad, basis_k;
    int32_t rows, rows_last, rows_out;  // folded rows of a plane; rows the last block's product runs over (q, or q and then p)
    const int32_t* flags;    // [matrix][MOST_SHARES]: large values seen by the fold's blocks, of which there are `shares`
    int32_t shares;
    // the plain product of a matrix with large values
    CacheView view;
    int32_t first, n_in, n_keep, sink;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid)
{
    const int bytes = valid ? 16 : 0;  // 0 source bytes: the destination is zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// The plain product for this CTA's share of a matrix with large values: of the blocks * rows_out rows that the matrix has in `out`,
// the first n_keep are its output rows as they are.  Entries, order of the sums and rounding are project_simt_kernel's.
template <int TM, int TN, int M, int N>
__device__ __noinline__ void plain_product(const ProductParams& p, float (*As)[TM], float (*Bs)[TN], int32_t mat, int32_t block, int32_t m0, int32_t c0,
                                           int ty, int tx)
{
    constexpr int THREADS = TM / M * TN / N;
    const int32_t index = p.first + mat, tensor = index / p.view.mats_per_tensor;
    const float* x = static_cast<const float*>(tensor_base(p.view, tensor)) + matrix_offset(p.view, index % p.view.mats_per_tensor) +
                     (int64_t)p.sink * p.view.stride_token;
    const int32_t row0 = block * p.rows_out + m0;
    float acc[M][N] = {};
#pragma unroll 1
    for (int32_t k0 = 0; k0 < p.n_in; k0 += TK) {
        __syncthreads();
#pragma unroll 1
        for (int idx = threadIdx.x; idx < TK * TM; idx += THREADS) {
            const int k = idx / TM, m = idx % TM;
            const bool ok = k0 + k < p.n_in && m0 + m < p.rows_out && row0 + m < p.n_keep;
            As[k][m] = ok ? (float)basis_entry(row0 + m, k0 + k, p.n_in, p.n_keep, 0) : 0.f;
        }
#pragma unroll 1
        for (int idx = threadIdx.x; idx < TK * TN / 4; idx += THREADS) {
            const int k = idx / (TN / 4), c = idx % (TN / 4) * 4;
            const bool ok = k0 + k < p.n_in && c0 + c < p.head_dim;
            *reinterpret_cast<float4*>(&Bs[k][c]) =
                ok ? *reinterpret_cast<const float4*>(x + (int64_t)(k0 + k) * p.view.stride_token + c0 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
#pragma unroll 1
        for (int k = 0; k < min(TK, p.n_in - k0); ++k) {
#pragma unroll
            for (int i = 0; i < M; ++i)
#pragma unroll
                for (int j = 0; j < N; ++j) acc[i][j] = fmaf(As[k][ty + i / 4 * 16 + i % 4], Bs[k][tx + j / 4 * 32 + j % 4], acc[i][j]);
        }
    }
    float* out = p.out + (size_t)(mat * p.blocks + block) * p.rows_out * p.head_dim;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const int32_t m = m0 + ty + i / 4 * 16 + i % 4;
        if (m >= p.rows_out) continue;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int32_t c = c0 + tx + j / 4 * 32 + j % 4;
            if (c < p.head_dim) out[(size_t)m * p.head_dim + c] = acc[i][j];
        }
    }
}

// grid: x = matrix * blocks + block, y = TM folded output rows, z = TN channels.  A warp covers 4 M x 8 N products: lane
// (ly, lx) has rows ly * 4 + 16 i and channels lx * 4 + 32 j, four of each.
template <int TM, int TN, int M, int N>
__global__ void __launch_bounds__(TM / M * TN / N) product_f32_kernel(const __grid_constant__ ProductParams p)
{
    constexpr int THREADS = TM / M * TN / N, WARPS_N = TN / (8 * N);
    constexpr int A_VECS = TK * TM / 4, B_VECS = TK * TN / 4;  // 16-byte vectors of a stage
    __shared__ __align__(16) float As[STAGES][TK][TM];
    __shared__ __align__(16) float Bs[STAGES][TK][TN];

    const int tid = threadIdx.x, warp = tid / 32, ly = tid % 32 / 8, lx = tid % 8;
    const int ty = warp / WARPS_N * 4 * M + ly * 4, tx = warp % WARPS_N * 8 * N + lx * 4;
    const int32_t m0 = blockIdx.y * TM, c0 = blockIdx.z * TN;
    const int32_t block = blockIdx.x % p.blocks, mat = blockIdx.x / p.blocks;
    // the four blocks' inputs lie in the order uu, uv, q, p: block 2 (PA) reads p, block 3 (PB) q and, where it runs on, p
    const int32_t plane = p.blocks == 4 && block >= 2 ? 5 - block : block;
    const int32_t limit = block == p.blocks - 1 ? p.rows_last : p.rows, steps = (limit + TK - 1) / TK;
    const float* a_src = p.basis + (size_t)block * p.basis_k * p.m_pad + m0;
    const float* b_src = p.planes + ((size_t)mat * p.blocks + plane) * p.rows * p.head_dim + c0;

    int32_t next = 0;
    auto fetch = [&](int stage) {
        if (next < steps) {
            const int32_t k0 = next * TK;
#pragma unroll
            for (int i = 0; i < (A_VECS + THREADS - 1) / THREADS; ++i) {
                const int idx = tid + i * THREADS, k = idx / (TM / 4), m = idx % (TM / 4) * 4;
                if (A_VECS % THREADS == 0 || idx < A_VECS)
                    cp_async16((uint32_t)__cvta_generic_to_shared(&As[stage][k][m]), a_src + (size_t)(k0 + k) * p.m_pad + m, true);
            }
#pragma unroll
            for (int i = 0; i < (B_VECS + THREADS - 1) / THREADS; ++i) {
                const int idx = tid + i * THREADS, k = idx / (TN / 4), c = idx % (TN / 4) * 4;
                const bool ok = k0 + k < limit && c0 + c < p.head_dim;
                if (B_VECS % THREADS == 0 || idx < B_VECS)
                    cp_async16((uint32_t)__cvta_generic_to_shared(&Bs[stage][k][c]), ok ? b_src + (size_t)(k0 + k) * p.head_dim + c : p.planes, ok);
            }
        }
        ++next;
        asm volatile("cp.async.commit_group;" ::: "memory");  // empty past the end: the count of groups stays in step
    };

    float acc[M][N] = {};
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) fetch(s);
    if (any_large(p.flags, mat, p.shares)) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        plain_product<TM, TN, M, N>(p, As[0], Bs[0], mat, block, m0, c0, ty, tx);
        return;
    }
    int stage = 0;
#pragma unroll 1
    for (int32_t st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();  // this stage has landed for every thread, and every thread is done with the one refilled next
        fetch(stage == 0 ? STAGES - 1 : stage - 1);
#pragma unroll
        for (int k = 0; k < TK; ++k) {
            float a[M], b[N];
#pragma unroll
            for (int i = 0; i < M; i += 4) *reinterpret_cast<float4*>(&a[i]) = *reinterpret_cast<const float4*>(&As[stage][k][ty + i * 4]);
#pragma unroll
            for (int j = 0; j < N; j += 4) *reinterpret_cast<float4*>(&b[j]) = *reinterpret_cast<const float4*>(&Bs[stage][k][tx + j * 8]);
#pragma unroll
            for (int i = 0; i < M; ++i)
#pragma unroll
                for (int j = 0; j < N; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        stage = stage + 1 == STAGES ? 0 : stage + 1;
    }
    float* out = p.out + (size_t)blockIdx.x * p.rows_out * p.head_dim;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const int32_t m = m0 + ty + (i / 4) * 16 + i % 4;
        if (m >= p.rows_out) continue;
#pragma unroll
        for (int j = 0; j < N; j += 4) {
            const int32_t c = c0 + tx + j * 8;
            if (c < p.head_dim)
                *reinterpret_cast<float4*>(out + (size_t)m * p.head_dim + c) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
        }
    }
}

// One thread per folded row and four channels; grid as fold_f32_kernel's.
template <int BLOCKS>
__global__ void __launch_bounds__(256) unfold_f32_kernel(const CacheView view, int32_t first, int32_t n_keep, int32_t sink,
                                                         const float4* __restrict__ sums, const int32_t* __restrict__ flags, int32_t shares)
{
    const uint32_t vecs = (uint32_t)view.head_dim / 4;
    const int32_t rows_half = (n_keep + 1) / 2, rows_out = BLOCKS == 2 ? rows_half : (rows_half + 1) / 2;
    const uint32_t plane = (uint32_t)rows_out * vecs;
    const int32_t mat = first + (int32_t)blockIdx.x, tensor = mat / view.mats_per_tensor;
    float* y = static_cast<float*>(tensor_base(view, tensor)) + matrix_offset(view, mat % view.mats_per_tensor) +
               (int64_t)sink * view.stride_token;
    const float4* in = sums + (size_t)blockIdx.x * BLOCKS * plane;
    if (any_large(flags, (int32_t)blockIdx.x, shares)) {  // the output rows themselves
        const uint32_t total = (uint32_t)n_keep * vecs;
        for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < total; i += gridDim.y * blockDim.x) {
            const uint32_t m = i / vecs;
            reinterpret_cast<float4*>(y + (int64_t)m * view.stride_token)[i - m * vecs] = __ldg(in + i);
        }
        return;
    }
    for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < plane; i += gridDim.y * blockDim.x) {
        const int32_t m = (int32_t)(i / vecs);
        const uint32_t vec = i - (uint32_t)m * vecs;
        auto store = [&](int32_t r, const float4& v) { reinterpret_cast<float4*>(y + (int64_t)r * view.stride_token)[vec] = v; };
        const float4 a = __ldg(in + i), b = __ldg(in + plane + i);
        const float4 s = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        const float4 t = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
        if constexpr (BLOCKS == 2) {
            store(m, s);
            if (n_keep - 1 - m != m) store(n_keep - 1 - m, t);
        } else {
            const float4 A = __ldg(in + 2 * plane + i), B = __ldg(in + 3 * plane + i);
            float cs, sn;  // theta'_m = pi (2m+1) / (2L)
            sincospif((float)(2 * m + 1) / (float)(2 * n_keep), &sn, &cs);
            const float4 d = make_float4(fmaf(cs, A.x, sn * B.x), fmaf(cs, A.y, sn * B.y), fmaf(cs, A.z, sn * B.z), fmaf(cs, A.w, sn * B.w));
            const float4 e = make_float4(fmaf(sn, A.x, -cs * B.x), fmaf(sn, A.y, -cs * B.y), fmaf(sn, A.z, -cs * B.z), fmaf(sn, A.w, -cs * B.w));
            store(m, make_float4(s.x + d.x, s.y + d.y, s.z + d.z, s.w + d.w));
            store(n_keep - 1 - m, make_float4(s.x - d.x, s.y - d.y, s.z - d.z, s.w - d.w));
            const int32_t mh = rows_half - 1 - m;
            if (mh != m) {  // the middle row of an odd L/2 is its own mirror
                store(mh, make_float4(t.x + e.x, t.y + e.y, t.z + e.z, t.w + e.w));
                store(rows_half + m, make_float4(t.x - e.x, t.y - e.y, t.z - e.z, t.w - e.w));
            }
        }
    }
}

template <int TM, int TN, int M, int N>
void launch_product(const ProductParams& p, int32_t count, cudaStream_t stream)
{
    const dim3 grid((unsigned)(count * p.blocks), (unsigned)((p.rows_out + TM - 1) / TM), (unsigned)((p.head_dim + TN - 1) / TN));
    product_f32_kernel<TM, TN, M, N><<<grid, TM / M * TN / N, 0, stream>>>(p);
}

template <int BLOCKS>
cudaError_t launch_blocks(const CacheView& view, int32_t first, int32_t count, const Basis& basis, int32_t sink, float* scratch,
                          int sm_count, cudaStream_t stream)
{
    const int32_t rows_half = (basis.n_keep + 1) / 2;
    ProductParams p;
    p.basis = basis.f32_fold;
    p.planes = scratch;
    p.head_dim = view.head_dim;
    p.blocks = BLOCKS;
    p.m_pad = basis.f32_fold_m;
    p.basis_k = basis.f32_fold_k;
    p.rows = (basis.n_in + BLOCKS - 1) / BLOCKS;
    p.rows_last = BLOCKS == 4 && basis.n_keep / 2 % 2 == 0 ? 2 * p.rows : p.rows;
    p.rows_out = BLOCKS == 2 ? rows_half : (rows_half + 1) / 2;
    p.out = scratch + (size_t)count * BLOCKS * p.rows * view.head_dim;
    auto share = [&](int32_t rows) { return (unsigned)std::min<int64_t>(((int64_t)rows * (view.head_dim / 4) + 255) / 256, MOST_SHARES); };
    int32_t* flags = reinterpret_cast<int32_t*>(p.out + (size_t)count * BLOCKS * p.rows_out * view.head_dim);
    p.flags = flags;
    p.shares = (int32_t)share(p.rows);
    p.view = view;
    p.first = first;
    p.n_in = basis.n_in;
    p.n_keep = basis.n_keep;
    p.sink = sink;
    fold_f32_kernel<BLOCKS><<<dim3((unsigned)count, share(p.rows)), 256, 0, stream>>>(view, first, basis.n_in, sink, basis.f32_turns,
                                                                                    reinterpret_cast<float4*>(scratch), flags);
    // 8 x 8 products a thread take the fewest shared-memory loads, 4 x 4 spread few matrices over more SMs (2 matrices of
    // 2044 -> 1022: 41 and 23 us).  Tiles of 128 rows read the folded inputs least often; where they would leave much of
    // the last one empty, tiles of 32 (64 matrices of 256 rows a block 212 and 222 us, 16 of 281 rows 75 and 58 us).
    const int64_t rows128 = (p.rows_out + 127) / 128 * 128, rows32 = (p.rows_out + 31) / 32 * 32;
    const int64_t large = (int64_t)count * BLOCKS * ((p.rows_out + 127) / 128) * ((view.head_dim + 63) / 64);
    if (large < 2 * sm_count)
        launch_product<32, 32, 4, 4>(p, count, stream);
    else if (rows128 * 10 <= rows32 * 11)
        launch_product<128, 64, 8, 8>(p, count, stream);
    else
        launch_product<32, 64, 8, 8>(p, count, stream);
    unfold_f32_kernel<BLOCKS><<<dim3((unsigned)count, share(p.rows_out)), 256, 0, stream>>>(view, first, basis.n_keep, sink,
                                                                                         reinterpret_cast<const float4*>(p.out), flags, p.shares);
    return cudaGetLastError();
}

}  // namespace

// Blocks of the folded fp32 product: 4 where the lengths allow it, else 2.
int32_t fold_f32_blocks(int32_t n_in, int32_t n_keep) { return n_in % 4 == 0 && n_keep % 2 == 0 ? 4 : 2; }

size_t fold_f32_scratch_bytes(int32_t n_in, int32_t n_keep, int32_t head_dim)
{
    const int32_t blocks = fold_f32_blocks(n_in, n_keep), rows_half = (n_keep + 1) / 2;
    const int32_t rows = (n_in + blocks - 1) / blocks, rows_out = blocks == 2 ? rows_half : (rows_half + 1) / 2;
    // the folded inputs, the blocks' products, the fold's flags
    return (size_t)blocks * (rows + rows_out) * head_dim * sizeof(float) + MOST_SHARES * sizeof(int32_t);
}

cudaError_t launch_fold_f32(const CacheView& view, int32_t first, int32_t count, const Basis& basis, int32_t sink, void* scratch,
                            int sm_count, cudaStream_t stream)
{
    if (count <= 0) return cudaSuccess;
    float* planes = static_cast<float*>(scratch);
    return fold_f32_blocks(basis.n_in, basis.n_keep) == 4 ? launch_blocks<4>(view, first, count, basis, sink, planes, sm_count, stream)
                                                          : launch_blocks<2>(view, first, count, basis, sink, planes, sm_count, stream);
}

}  // namespace freqkv
