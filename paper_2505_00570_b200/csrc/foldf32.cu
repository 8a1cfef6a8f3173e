// fp32 caches whose lengths are no powers of two: the projection Y = P X on the CUDA cores (Section 3.3,
// Eq. 2-3 with the transforms of Appendix A folded into P), with the symmetries of the basis taken out first.
//
// One level (any lengths): u, v = x_n +- x_{N-1-n} and S = Pe u, D = Po v, y_m = S + D, y_{L-1-m} = S - D: half the
// multiply-adds of the plain product.  Four blocks (N a multiple of 4, L even): uu, uv, p, q and Pee, Peo, PA, PB of
// a quarter of each length (derived in basis.cu): a quarter of them.  All of it stays in fp32; the sums are two
// and four times shorter than the plain product's.
//
//   fold_f32_kernel      reads every non-sink row once and writes the 2 or 4 folded planes to scratch; HBM- or L2-bound.
//   product_f32_kernel   one CTA computes TM rows x TN channels of every block of one matrix, one block after the
//                        other (accumulators of all of them stay in registers), then combines them and stores the
//                        2 or 4 output rows of each folded row straight into the cache: it reads only scratch and
//                        basis, so that is safe in place, and nothing is copied back.  A thread owns 4 rows x 4
//                        channels of every block; slices of 16 folded rows come through a ring of cp.async stages (the
//                        basis is stored transposed, so both operands arrive in the order they are read in).
//                        Bound by FFMA issue: 16 FFMA for two 16-byte shared-memory loads.
//
// Measured against the plain product (64 matrices of 128 channels unless said): 2044 -> 1022 959 -> 253 us, odd lengths
// 2043 -> 1021 959 -> 443 us, 4000 -> 2000 3655 -> 1131 us, one head 2044 -> 1022 (2 matrices) 107 -> 49 us; error against
// 64 bits 5.7e-7 -> 2.8e-7.
#include <algorithm>

#include "common.cuh"

namespace freqkv {
namespace {

constexpr int TK = 16, STAGES = 3;

// Planes of one matrix: [blocks][rows of a plane][head_dim]; rows = ceil(n_in / blocks).
template <int BLOCKS>
__global__ void __launch_bounds__(256) fold_f32_kernel(const CacheView view, int32_t first, int32_t n_in, int32_t sink,
                                                       const float2* __restrict__ turns, float4* __restrict__ planes)
{
    const uint32_t vecs = (uint32_t)view.head_dim / 4;
    const uint32_t rows = (uint32_t)(n_in + BLOCKS - 1) / BLOCKS, plane = rows * vecs;
    const int32_t mat = first + (int32_t)blockIdx.x, tensor = mat / view.mats_per_tensor;
    const float* x = static_cast<const float*>(tensor_base(view, tensor)) + matrix_offset(view, mat % view.mats_per_tensor) +
                     (int64_t)sink * view.stride_token;
    float4* out = planes + (size_t)blockIdx.x * BLOCKS * plane;
    auto row = [&](int32_t n, uint32_t vec) { return __ldg(reinterpret_cast<const float4*>(x + (int64_t)n * view.stride_token) + vec); };
    for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < plane; i += gridDim.y * blockDim.x) {
        const int32_t n = (int32_t)(i / vecs);
        const uint32_t vec = i - (uint32_t)n * vecs;
        const float4 a = row(n, vec), b = row(n_in - 1 - n, vec);
        const float4 u = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        const float4 v = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
        if constexpr (BLOCKS == 2) {
            const bool middle = n_in - 1 - n == n;  // the middle row of an odd length enters u once and v as zero (a - a)
            out[i] = middle ? a : u;
            out[plane + i] = v;
        } else {
            const float4 c = row(n_in / 2 - 1 - n, vec), d = row(n_in / 2 + n, vec);
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
}

struct ProductParams {
    const float* basis;      // [blocks][basis_k][m_pad]: transposed, zero past the ends
    const float* planes;     // [matrix][blocks][rows][head_dim]
    int32_t first, n_in, n_keep, sink;
    int32_t m_pad, basis_k;
    int32_t rows, rows_last;  // folded rows of a plane; rows the last block's product runs over (q, or q and then p)
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid)
{
    const int bytes = valid ? 16 : 0;  // 0 source bytes: the destination is zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// grid: x = matrix, y = TM folded output rows, z = TN channels.
template <int BLOCKS, int TM, int TN>
__global__ void __launch_bounds__((TM / 4) * (TN / 4)) product_f32_kernel(const CacheView view, const ProductParams p)
{
    constexpr int THREADS = (TM / 4) * (TN / 4);
    constexpr int A_VECS = TK * TM / 4, B_VECS = TK * TN / 4;  // 16-byte vectors of a stage
    __shared__ __align__(16) float As[STAGES][TK][TM];
    __shared__ __align__(16) float Bs[STAGES][TK][TN];

    const int tid = threadIdx.x, ty = tid / (TN / 4), tx = tid % (TN / 4);
    const int32_t m0 = blockIdx.y * TM, c0 = blockIdx.z * TN;
    const float* planes = p.planes + (size_t)blockIdx.x * BLOCKS * p.rows * view.head_dim;

    // The product's slices in one sequence over all blocks, so that the ring runs on from block to block.
    const int32_t steps = (p.rows + TK - 1) / TK, steps_last = (p.rows_last + TK - 1) / TK;
    // fetch cursor: block and slice of the next stage to fill
    int32_t f_block = 0, f_step = 0;
    auto fetch = [&](int stage) {
        if (f_block < BLOCKS) {
            const int32_t k0 = f_step * TK;
            // the four blocks' inputs lie in the order uu, uv, q, p: block 2 (PA) reads p, block 3 (PB) q and, where it runs on, p
            const int32_t plane = BLOCKS == 4 && f_block >= 2 ? 5 - f_block : f_block;
            const int32_t limit = f_block == BLOCKS - 1 ? p.rows_last : p.rows;
            const float* a = p.basis + ((size_t)f_block * p.basis_k + k0) * p.m_pad + m0;
            const float* b = planes + ((size_t)plane * p.rows + k0) * view.head_dim;
#pragma unroll
            for (int i = 0; i < (A_VECS + THREADS - 1) / THREADS; ++i) {
                const int idx = tid + i * THREADS, k = idx / (TM / 4), m = idx % (TM / 4) * 4;
                if (A_VECS % THREADS == 0 || idx < A_VECS)
                    cp_async16((uint32_t)__cvta_generic_to_shared(&As[stage][k][m]), a + (size_t)k * p.m_pad + m, true);
            }
#pragma unroll
            for (int i = 0; i < (B_VECS + THREADS - 1) / THREADS; ++i) {
                const int idx = tid + i * THREADS, k = idx / (TN / 4), c = idx % (TN / 4) * 4;
                const bool ok = k0 + k < limit && c0 + c < view.head_dim;
                if (B_VECS % THREADS == 0 || idx < B_VECS)
                    cp_async16((uint32_t)__cvta_generic_to_shared(&Bs[stage][k][c]), ok ? b + (size_t)k * view.head_dim + c0 + c : planes, ok);
            }
            if (++f_step == (f_block == BLOCKS - 1 ? steps_last : steps)) {
                f_step = 0;
                ++f_block;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");  // empty past the end: the count of groups stays in step
    };

    float acc[BLOCKS][4][4] = {};
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) fetch(s);
    int stage = 0;
#pragma unroll
    for (int blk = 0; blk < BLOCKS; ++blk) {
        const int32_t n_steps = blk == BLOCKS - 1 ? steps_last : steps;
#pragma unroll 1
        for (int32_t st = 0; st < n_steps; ++st) {
            asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
            __syncthreads();  // this stage has landed for every thread, and every thread is done with the one refilled next
            fetch(stage == 0 ? STAGES - 1 : stage - 1);
#pragma unroll
            for (int k = 0; k < TK; ++k) {
                const float4 a = *reinterpret_cast<const float4*>(&As[stage][k][ty * 4]);
                const float4 b = *reinterpret_cast<const float4*>(&Bs[stage][k][tx * 4]);
                const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[blk][i][j] = fmaf(av[i], bv[j], acc[blk][i][j]);
            }
            stage = stage + 1 == STAGES ? 0 : stage + 1;
        }
    }

    const int32_t c = c0 + tx * 4;
    if (c >= view.head_dim) return;
    const int32_t mat = p.first + (int32_t)blockIdx.x, tensor = mat / view.mats_per_tensor;
    float* y = static_cast<float*>(tensor_base(view, tensor)) + matrix_offset(view, mat % view.mats_per_tensor) +
               (int64_t)p.sink * view.stride_token + c;
    auto store = [&](int32_t r, const float (&v)[4]) {
        *reinterpret_cast<float4*>(y + (int64_t)r * view.stride_token) = make_float4(v[0], v[1], v[2], v[3]);
    };
    const int32_t rows_half = (p.n_keep + 1) / 2, rows_out = BLOCKS == 2 ? rows_half : (rows_half + 1) / 2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int32_t m = m0 + ty * 4 + i;
        if (m >= rows_out) continue;
        float o0[4], o1[4];
        if constexpr (BLOCKS == 2) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                o0[j] = acc[0][i][j] + acc[1][i][j];
                o1[j] = acc[0][i][j] - acc[1][i][j];
            }
            store(m, o0);
            if (p.n_keep - 1 - m != m) store(p.n_keep - 1 - m, o1);
        } else {
            float ct, st;  // theta'_m = pi (2m+1) / (2L)
            sincospif((float)(2 * m + 1) / (float)(2 * p.n_keep), &st, &ct);
            const int32_t mh = rows_half - 1 - m;
            float o2[4], o3[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float s0 = acc[0][i][j] + acc[1][i][j], s1 = acc[0][i][j] - acc[1][i][j];
                const float d0 = fmaf(ct, acc[2][i][j], st * acc[3][i][j]), d1 = fmaf(st, acc[2][i][j], -ct * acc[3][i][j]);
                o0[j] = s0 + d0;
                o1[j] = s0 - d0;
                o2[j] = s1 + d1;
                o3[j] = s1 - d1;
            }
            store(m, o0);
            store(p.n_keep - 1 - m, o1);
            if (mh != m) {  // the middle row of an odd L/2 is its own mirror
                store(mh, o2);
                store(rows_half + m, o3);
            }
        }
    }
}

template <int BLOCKS, int TM, int TN>
void launch_product(const CacheView& view, const ProductParams& p, int32_t count, int32_t rows_out, cudaStream_t stream)
{
    const dim3 grid((unsigned)count, (unsigned)((rows_out + TM - 1) / TM), (unsigned)((view.head_dim + TN - 1) / TN));
    product_f32_kernel<BLOCKS, TM, TN><<<grid, (TM / 4) * (TN / 4), 0, stream>>>(view, p);
}

template <int BLOCKS>
cudaError_t launch_blocks(const CacheView& view, int32_t first, int32_t count, const Basis& basis, int32_t sink, float* scratch,
                          int sm_count, cudaStream_t stream)
{
    ProductParams p;
    p.basis = basis.f32_fold;
    p.planes = scratch;
    p.first = first;
    p.n_in = basis.n_in;
    p.n_keep = basis.n_keep;
    p.sink = sink;
    p.m_pad = basis.f32_fold_m;
    p.basis_k = basis.f32_fold_k;
    p.rows = (basis.n_in + BLOCKS - 1) / BLOCKS;
    p.rows_last = BLOCKS == 4 && basis.n_keep / 2 % 2 == 0 ? 2 * p.rows : p.rows;
    const int64_t vecs = (int64_t)p.rows * (view.head_dim / 4);
    const unsigned fold_y = (unsigned)std::min<int64_t>((vecs + 255) / 256, 64);
    fold_f32_kernel<BLOCKS><<<dim3((unsigned)count, fold_y), 256, 0, stream>>>(view, first, basis.n_in, sink, basis.f32_turns,
                                                                             reinterpret_cast<float4*>(scratch));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int32_t rows_half = (basis.n_keep + 1) / 2, rows_out = BLOCKS == 2 ? rows_half : (rows_half + 1) / 2;
    // Large tiles reuse a shared-memory operand twice as often; small ones spread few matrices over more SMs.
    const int64_t large = (int64_t)count * ((rows_out + 31) / 32) * ((view.head_dim + 63) / 64);
    if (large >= 2 * sm_count)
        launch_product<BLOCKS, 32, 64>(view, p, count, rows_out, stream);
    else
        launch_product<BLOCKS, 16, 32>(view, p, count, rows_out, stream);
    return cudaGetLastError();
}

}  // namespace

// Blocks of the folded fp32 product: 4 where the lengths allow it, else 2.
int32_t fold_f32_blocks(int32_t n_in, int32_t n_keep) { return n_in % 4 == 0 && n_keep % 2 == 0 ? 4 : 2; }

size_t fold_f32_scratch_bytes(int32_t n_in, int32_t n_keep, int32_t head_dim)
{
    const int32_t blocks = fold_f32_blocks(n_in, n_keep);
    return (size_t)blocks * ((n_in + blocks - 1) / blocks) * head_dim * sizeof(float);
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
