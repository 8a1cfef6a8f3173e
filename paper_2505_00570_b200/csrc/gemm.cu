// Tensor-core execution of the compression Y = P X (Section 3.3, Eq. 2-3 with the transforms
// of Appendix A folded into the basis P, see basis.cu) on the 5th-generation tensor cores of
// sm_100a: tcgen05.mma with accumulators in tensor memory, operands staged by TMA.
//
// Symmetry fold.  The DCT cosines are even or odd under n -> N-1-n (and m -> L-1-m) according to
// the parity of the frequency t, so with P = Pe + Po split into its even-t and odd-t parts
//     u_n = x_n + x_{N-1-n},   v_n = x_n - x_{N-1-n}            (n < ceil(N/2))
//     s_m = sum_n Pe[m][n] u_n,   d_m = sum_n Po[m][n] v_n      (m < ceil(L/2))
//     y_m = s_m + d_m,   y_{L-1-m} = s_m - d_m
// which is the same linear map with half the multiply-adds.  (For odd N the middle row enters u
// once and v as zero; for odd L the middle output row has d = 0 and is written once.)
// This folded form serves retained bands above the lowest component and the power spectrum; a plain compression of more than
// 256 kept rows runs in one pass over the cache (nearfar.cu), of fewer as one dense product (MODE_DIRECT).
//
// Two kernels per call:
//   fold_kernel         reads every non-sink cache row once and writes U and V (bf16) to a scratch
//                       buffer, one plane of ceil(N/2) x 128 per (matrix, u|v); HBM-bound.
//   freqkv_fold_gemm_kernel  persistent, one CTA per SM, CTAs paired into clusters of two that share
//                       every MMA (tcgen05 cta_group::2).  A cluster works on output tiles of 256
//                       folded rows x 256 columns (the K matrix and the V matrix of one (batch,
//                       layer, kv_head) side by side, so K and V share every instruction): CTA r
//                       of the pair holds rows 128 r .. 128 r + 127 of the basis slice and of the
//                       accumulators, and HALF of the input slice (r = 0: the K channels, r = 1: the
//                       V channels) -- the tensor cores of both SMs read both halves, so every
//                       byte of U / V is brought into shared memory once per 256 output rows.  Per
//                       tile the pair first accumulates S = Pe U, then D = Po V, in the two halves
//                       of tensor memory.  In each CTA:
//     warp 0      TMA producer: per 64-row slice of the contraction one box of Pe or Po (128 x 64)
//                 and 2 boxes of U or V (64 rows x 64 channels), 128-byte swizzled, into a ring
//                 of 6 stages of 32 KB; the bytes of both CTAs complete the leader's barrier;
//     warp 1      MMA issuer (leader CTA only): 4 tcgen05.mma (256 x 256 x 16) per stage, commits
//                 multicast to the barriers of both CTAs;
//     warps 4-11  epilogue: when S is complete they park it in registers (which frees that half
//                 of tensor memory for the next tile while D is still accumulating); when D is
//                 complete they form s + d and s - d, round to bf16 (nearest even) and store rows
//                 m and L-1-m straight into the cache.  Both steps overlap the MMAs of the
//                 neighbouring phases, so the tensor pipe never waits for the epilogue.
// The kernel reads only the scratch planes and the basis, so writing the cache in place is safe.
//
// Every wait on an mbarrier is bounded in time: a wait that runs out sets a bit in the status
// word, raises a CTA-wide abort flag that ends every other role's loop, the producer lets its
// copies in flight land, the two CTAs meet at a cluster barrier, tensor memory is freed and
// the kernel returns.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <vector>

#include "gemm.cuh"

namespace freqkv {
namespace {

constexpr int BM = 128;        // folded output rows per CTA and tile (the cluster's tile has 2 x 128); 256 columns: K | V
constexpr int BK = 64;         // contraction slice per stage (folded rows)
constexpr int STAGES = 6;
constexpr int A_BYTES = BM * BK * 2;               // 16 KB: 128 rows x 64 bf16, 128 B per row
constexpr int B_CHUNK_BYTES = BK * 128;            // 8 KB: 64 rows x 64 channels
constexpr int B_BYTES = 2 * B_CHUNK_BYTES;         // 16 KB: this CTA's 128 of the 256 columns
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;     // 32 KB per CTA
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* alignment slack */ + 256 /* barriers */;
constexpr int NUM_THREADS = 320;                   // direct and spectrum modes: 10 warps
// The kernel of the folded forms: three warpgroups (producer and MMA issuer | epilogue | epilogue) that share the
// registers unevenly.  The shares add up to what the block is launched with: 40 + 2 * 232 = 3 * 168.
constexpr int FOLD_THREADS = 384, FOLD_LAUNCH_REGS = 168, CONTROL_REGS = 40, EPILOGUE_REGS = 232;
static_assert(CONTROL_REGS + 2 * EPILOGUE_REGS <= 3 * FOLD_LAUNCH_REGS, "a larger sum would wait for registers for ever");
constexpr int EPI_WARPS = 8;
constexpr unsigned long long LANDING_NS = 1000000ull;        // 1 ms: far longer than any copy in flight needs

constexpr uint32_t ERR_FULL_WAIT = 1u, ERR_EMPTY_WAIT = 2u, ERR_ACC_FULL_WAIT = 4u, ERR_ACC_EMPTY_WAIT = 8u;

// One pass of a call: how its matrices fold and what their tiles are.
struct FoldParams {
    int32_t sink;
    int32_t mirror_sign;        // +1: y[L-1-m] = s - d;  -1: y[L-1-m] = d - s (a retained band that starts at an odd component)
    int32_t wide_rows;          // every row is 32-byte aligned
    int32_t total_tiles;
    int32_t pair0;              // first (batch, layer, kv_head) triple
    int32_t n_keep, rows_half;
    int32_t basis_rows_pad;     // row offset of the Po plane inside the basis tensor map
    int32_t k_steps;            // slices per phase
    int32_t m_pairs;            // tiles of 256 folded rows per triple
    int32_t* status;
    unsigned long long wait_limit_ns;  // bound of every mbarrier wait
};

struct GemmParams {
    int32_t n_keep;             // L
    int32_t basis_rows_pad;     // row offset of the Po plane inside the basis tensor map
    int32_t pair0, pair_count;  // (batch, layer, kv_head) triples covered by this launch
    int32_t m_pairs, k_steps;   // tiles of 256 folded rows per (batch, layer, kv_head); slices per phase
    int32_t sink;
    // power-spectrum mode only: per tensor [layers][kv_heads][n_in] sums, the weight of one squared value
    float* spectrum[2];
    float spectrum_scale;
    int32_t n_in;
    int32_t* status;
    unsigned long long wait_limit_ns;  // bound of every mbarrier wait
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Address of the same shared-memory location in CTA `rank` of this cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Acquire at cluster scope: some of the arrivals these waits observe come from the peer CTA.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete.  Gives up when another role has raised
// the abort flag or after `limit_ns`; in the second case it records `err_bit` and raises the
// flag itself.  Returns false when it gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                          uint32_t err_bit, unsigned long long limit_ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (global_timer_ns() - t0 > limit_ns) {
            atomicOr(status, (int32_t)err_bit);
            *abort_flag = 1;
            __threadfence_block();
            return false;
        }
    }
}

// TMA loads of a CTA pair: the data lands in this CTA's shared memory, the bytes are counted on
// the barrier `cluster_bar` of the leader CTA.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int32_t c0,
                                            int32_t c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int32_t c0,
                                            int32_t c1, int32_t c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int32_t c0,
                                            int32_t c1, int32_t c2, int32_t c3, int32_t c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

// Shared-memory matrix descriptor of tcgen05.mma: start address, leading and stride byte offsets
// (all in 16-byte units), descriptor version 1, 128-byte swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // version
    d |= (uint64_t)2 << 61;  // SWIZZLE_128B
    return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, A K-major, B MN-major, M = 256 (128 rows
// in each CTA of the pair), N = 256.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (0u << 15) | (1u << 16) | ((256u >> 3) << 17) |
                           ((256u >> 4) << 24);

// Issued by one thread of the leader CTA; both CTAs' tensor cores run it, each on its 128 rows of A
// and D, with B read from the shared memory of both.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(IDESC), "r"(accumulate)
        : "memory");
}

// When every MMA issued so far has finished, arrive on the barrier at this offset in BOTH CTAs.
__device__ __forceinline__ void umma_commit_both(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((uint16_t)3)
        : "memory");
}

// 32 lanes x 32 consecutive columns of tensor memory into registers r[OFF .. OFF+31].
template <int OFF, int NREG>
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[NREG])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[OFF + 0]), "=r"(r[OFF + 1]), "=r"(r[OFF + 2]), "=r"(r[OFF + 3]), "=r"(r[OFF + 4]), "=r"(r[OFF + 5]),
          "=r"(r[OFF + 6]), "=r"(r[OFF + 7]), "=r"(r[OFF + 8]), "=r"(r[OFF + 9]), "=r"(r[OFF + 10]), "=r"(r[OFF + 11]),
          "=r"(r[OFF + 12]), "=r"(r[OFF + 13]), "=r"(r[OFF + 14]), "=r"(r[OFF + 15]), "=r"(r[OFF + 16]),
          "=r"(r[OFF + 17]), "=r"(r[OFF + 18]), "=r"(r[OFF + 19]), "=r"(r[OFF + 20]), "=r"(r[OFF + 21]),
          "=r"(r[OFF + 22]), "=r"(r[OFF + 23]), "=r"(r[OFF + 24]), "=r"(r[OFF + 25]), "=r"(r[OFF + 26]),
          "=r"(r[OFF + 27]), "=r"(r[OFF + 28]), "=r"(r[OFF + 29]), "=r"(r[OFF + 30]), "=r"(r[OFF + 31])
        : "r"(taddr)
        : "memory");
}

// 32 lanes x 16 consecutive columns.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// ---- fold: U = X + reversed X, V = X - reversed X, one 16-byte vector (8 channels) per item ----

__device__ __forceinline__ void fold8(const uint4& a, const uint4& b, uint4* u, uint4* v)
{
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
    uint32_t uw[4], vw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float a0 = __uint_as_float(aw[i] << 16), a1 = __uint_as_float(aw[i] & 0xffff0000u);
        const float b0 = __uint_as_float(bw[i] << 16), b1 = __uint_as_float(bw[i] & 0xffff0000u);
        uw[i] = pack_bf16(a0 + b0, a1 + b1);
        vw[i] = pack_bf16(a0 - b0, a1 - b1);
    }
    *u = make_uint4(uw[0], uw[1], uw[2], uw[3]);
    *v = make_uint4(vw[0], vw[1], vw[2], vw[3]);
}

// One fold job: the non-sink rows of `pair_count` (batch, layer, kv_head) triples starting at
// pair0, K and V, into the planes ((pair_local * 2 + tensor) * 2 + (0 = U, 1 = V)) of `dst`, each
// n_half rows x 128 channels (16 vectors of 16 bytes per row).
struct FoldJob {
    int32_t pair0, pair_count, n_in, n_half, sink;
    uint4* dst;
};

// One level: matrix pt of the job (pair_local * 2 + tensor), the y-th of gridDim.y shares of its n_half * 16 vectors.
// The matrix arithmetic is done once per thread; each thread then folds four vectors per round,
// all eight loads first.  Reads and writes are streaming (each byte is touched once).
__device__ __forceinline__ void fold_one_level(const CacheView& view, const FoldJob& job, uint32_t pt)
{
    const char* x = static_cast<const char*>(tensor_base(view, pt & 1)) +
                    (matrix_offset(view, job.pair0 + (int32_t)(pt >> 1)) + (int64_t)job.sink * view.stride_token) * 2;
    const int64_t row_bytes = view.stride_token * 2;
    const uint32_t total = (uint32_t)job.n_half * 16u;
    uint4* u_plane = job.dst + (int64_t)pt * 2 * total;
    // a block works on chunks of 1024 consecutive vectors (64 rows and their 64 mirror rows)
    for (uint32_t c0 = blockIdx.y * 1024u; c0 < total; c0 += gridDim.y * 1024u) {
        uint4 a[4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t i = c0 + j * 256u + threadIdx.x;
            if (i < total) {
                const int32_t n = (int32_t)(i >> 4), nr = job.n_in - 1 - n;
                a[j] = __ldcs(reinterpret_cast<const uint4*>(x + n * row_bytes) + (i & 15u));
                b[j] = __ldcs(reinterpret_cast<const uint4*>(x + nr * row_bytes) + (i & 15u));
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t i = c0 + j * 256u + threadIdx.x;
            if (i < total) {
                const int32_t n = (int32_t)(i >> 4);
                uint4 u, v;
                fold8(a[j], b[j], &u, &v);
                if (job.n_in - 1 - n == n) {  // middle row of an odd-length signal: u = x, v = 0
                    u = a[j];
                    v = make_uint4(0u, 0u, 0u, 0u);
                }
                __stcs(u_plane + i, u);
                __stcs(u_plane + total + i, v);
            }
        }
    }
}

// Block x: matrix x of the job.
__global__ void __launch_bounds__(256) fold_kernel(const CacheView view, const FoldJob job) { fold_one_level(view, job, blockIdx.x); }

// The other two uses of the same tiles:
// MODE_SPECTRUM: the basis holds the even and the odd rows of the plain N-point DCT-II instead of
//   Pe and Po, so S and D are the components z_2m and z_2m+1 themselves; the epilogue squares them,
//   sums over the 128 channels of its tensor and adds the sum to the power spectrum of its
//   (layer, kv head).  Nothing is written to the cache.
// MODE_DIRECT: for at most 256 kept rows (small retaining ratios) the fold would cost more
//   than it saves: the basis is the plain L x N matrix P, the input slices come straight from the
//   cache (map_x = K tensor, map_v = V tensor, 5-D maps over the non-sink rows), there is one
//   accumulator and one tile per (batch, layer, kv_head).  The tile's rows are stored only after
//   every slice of its matrices has been read, so writing in place is safe here too.
constexpr int MODE_SPECTRUM = 1, MODE_DIRECT = 2;

// Registers of the calling warpgroup from here on (every warp of it executes this).
template <int REGS, bool MORE>
__device__ __forceinline__ void set_registers()
{
    if constexpr (MORE)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS));
    else
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS));
}

// 16 channels of one output row: one 32-byte store where every row is 32-byte aligned, else two of 16 bytes.
__device__ __forceinline__ void store_row16(__nv_bfloat16* dst, const uint32_t (&v)[8], bool wide)
{
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                     "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    } else {
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

// ---- the product of the folded forms ----

__global__ void __launch_bounds__(FOLD_THREADS, 1)
freqkv_fold_gemm_kernel(const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_x, const CacheView view,
                        const __grid_constant__ FoldParams prm)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // 128-byte swizzle atoms need 1024-byte alignment
    uint8_t* aligned = smem_raw + (base - raw);
    const uint32_t bar0 = base + STAGES * STAGE_BYTES;
    // barrier slots (same offsets in both CTAs): full[0..S) -- used in the leader only --, empty[S..2S), then
    // s_full, s_empty, d_full, d_empty (the two *_empty used in the leader only)
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto acc_full_bar = [&](int eo) { return bar0 + 8u * (2 * STAGES + 2 * eo); };
    auto acc_empty_bar = [&](int eo) { return bar0 + 8u * (2 * STAGES + 2 * eo + 1); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(aligned + STAGES * STAGE_BYTES + 8 * (2 * STAGES + 4));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster_rank();  // 0 = leader of the pair
    const int32_t cluster = blockIdx.x / 2, n_clusters = gridDim.x / 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);   // the leader's producer arrives; both producers' bytes are counted
            mbar_init(empty_bar(s), 1);  // one multicast commit
        }
        for (int eo = 0; eo < 2; ++eo) {
            mbar_init(acc_full_bar(eo), 1);               // one multicast commit
            mbar_init(acc_empty_bar(eo), 2 * EPI_WARPS);  // the epilogue warps of both CTAs
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {  // tensor memory of the pair: all 512 columns in each CTA
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // the peer's barriers exist before anything signals them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    // One setmaxnreg per warpgroup, inside the branch that only this warpgroup takes: where branches meet, ptxas
    // assumes the fewest registers.
    if (warp < 4) {
        set_registers<CONTROL_REGS, false>();
        if (warp == 0) {
            // ---------------- TMA producer (both CTAs) ----------------
            if (lane == 0) {
                uint32_t it = 0;  // global slice counter: stage = it % STAGES, phase = it / STAGES
                bool alive = true;
                for (int32_t tile = cluster; tile < prm.total_tiles && alive; tile += n_clusters) {
                    const int32_t pair = tile / prm.m_pairs, m0 = (tile % prm.m_pairs * 2 + (int32_t)rank) * BM;
                    for (int eo = 0; eo < 2 && alive; ++eo) {
                        const int32_t plane = (pair * 2 + (int32_t)rank) * 2 + eo;  // rank 0: K channels, rank 1: V
                        for (int32_t ks = 0; ks < prm.k_steps; ++ks, ++it) {
                            const int st = it % STAGES;
                            if (it >= STAGES &&
                                !mbar_wait(empty_bar(st), ((it / STAGES) - 1) & 1, abort_flag, prm.status, ERR_EMPTY_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            const uint32_t stage = base + st * STAGE_BYTES;
                            const uint32_t leader_full = cluster_addr(full_bar(st), 0);
                            if (rank == 0) mbar_expect_tx(full_bar(st), 2 * STAGE_BYTES);
                            const int32_t k0 = ks * BK;
                            tma_load_2d(stage, &map_p, leader_full, k0, eo * prm.basis_rows_pad + m0);
                            tma_load_3d(stage + A_BYTES, &map_x, leader_full, 0, k0, plane);
                            tma_load_3d(stage + A_BYTES + B_CHUNK_BYTES, &map_x, leader_full, 64, k0, plane);
                        }
                    }
                }
                if (*abort_flag) {  // let the copies in flight land before this CTA's shared memory goes away
                    const unsigned long long t0 = global_timer_ns();
                    while (global_timer_ns() - t0 < LANDING_NS) __nanosleep(1000);
                }
            }
        } else if (warp == 1) {
            // ---------------- MMA issuer (leader CTA only) ----------------
            if (lane == 0 && rank == 0) {
                uint32_t it = 0, phase = 0;  // phase: over all tiles; half of tensor memory = phase % 2
                bool alive = true;
                for (int32_t tile = cluster; tile < prm.total_tiles && alive; tile += n_clusters) {
                    for (int eo = 0; eo < 2 && alive; ++eo, ++phase) {
                        const uint32_t acc = phase & 1, use = phase >> 1;  // use: how often that half was filled before
                        if (use > 0) {  // both CTAs' epilogues must have read what this half held last
                            if (!mbar_wait(acc_empty_bar(acc), (use - 1) & 1, abort_flag, prm.status, ERR_ACC_EMPTY_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        }
                        for (int32_t ks = 0; ks < prm.k_steps; ++ks, ++it) {
                            const int st = it % STAGES;
                            if (!mbar_wait(full_bar(st), (it / STAGES) & 1, abort_flag, prm.status, ERR_FULL_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a0 = base + st * STAGE_BYTES, b0 = a0 + A_BYTES;
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk) {
                                // A: 128 rows per CTA, 8-row groups 1 KB apart; 16 k-elements = 32 bytes inside the swizzled row
                                const uint64_t ad = smem_desc(a0 + kk * 32, 16, 1024);
                                // B: per CTA 2 chunks of 64 channels 8 KB apart (leading offset), 8-row groups 1 KB apart
                                const uint64_t bd = smem_desc(b0 + kk * 2048, B_CHUNK_BYTES, 1024);
                                umma_bf16(tmem_base + acc * 256, ad, bd, (ks | kk) != 0);
                            }
                            umma_commit_both(empty_bar(st));  // frees the stage in both CTAs when these MMAs have read it
                        }
                        if (alive) umma_commit_both(acc_full_bar(acc));
                    }
                }
            }
        }
    } else {
        set_registers<EPILOGUE_REGS, true>();
        // ---------------- epilogue (both CTAs, each on its own 128 rows) ----------------
        const int ew = warp - 4, quarter = warp % 4, tensor = ew / 4;  // tensor: 0 = K columns, 1 = V columns
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + tensor * 128;
        uint32_t phase = 0;  // as the MMA issuer counts
        // wait for the accumulator that is complete next
        auto next_full = [&]() -> bool {
            const bool ok = mbar_wait(acc_full_bar(phase & 1), (phase >> 1) & 1, abort_flag, prm.status, ERR_ACC_FULL_WAIT, prm.wait_limit_ns);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            return ok;
        };
        // hand it back; both CTAs' warps tell the leader
        auto release = [&]() {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(acc_empty_bar(phase & 1), 0));
            ++phase;
        };
        for (int32_t tile = cluster; tile < prm.total_tiles; tile += n_clusters) {
            uint32_t s[128];
            // S = Pe U: park this thread's row (128 columns) in registers, hand that half back
            if (!next_full()) break;
            tmem_ld32<0>(lane_addr + (phase & 1) * 256 + 0, s);
            tmem_ld32<32>(lane_addr + (phase & 1) * 256 + 32, s);
            tmem_ld32<64>(lane_addr + (phase & 1) * 256 + 64, s);
            tmem_ld32<96>(lane_addr + (phase & 1) * 256 + 96, s);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            release();
            const int32_t n_keep = prm.n_keep;
            const int32_t m = (tile % prm.m_pairs * 2 + (int32_t)rank) * BM + quarter * 32 + lane;
            __nv_bfloat16* mat = static_cast<__nv_bfloat16*>(tensor_base(view, tensor)) +
                                 matrix_offset(view, prm.pair0 + tile / prm.m_pairs) + (int64_t)prm.sink * view.stride_token;
            // D = Po V: combine and store rows m and L-1-m
            if (!next_full()) break;
            const uint32_t addr = lane_addr + (phase & 1) * 256;
            const bool row_ok = m < prm.rows_half, mirror_ok = row_ok && n_keep - 1 - m != m;
            const float sgn = (float)prm.mirror_sign;
            __nv_bfloat16* out_p = mat + (int64_t)m * view.stride_token;
            __nv_bfloat16* out_m = mat + (int64_t)(n_keep - 1 - m) * view.stride_token;
            // The next 16 columns leave tensor memory while these are combined and stored (64 matrices 1497 -> 749 44.1 -> 42.1 us).
            uint32_t d2[2][16];
            tmem_ld16(addr, d2[0]);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (c < 7) tmem_ld16(addr + (c + 1) * 16, d2[(c + 1) & 1]);
                if (c == 7) release();
                const uint32_t(&d)[16] = d2[c & 1];
                uint32_t p[8], q[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float s0 = __uint_as_float(s[c * 16 + 2 * j]), s1 = __uint_as_float(s[c * 16 + 2 * j + 1]);
                    const float d0 = __uint_as_float(d[2 * j]), d1 = __uint_as_float(d[2 * j + 1]);
                    p[j] = pack_bf16(s0 + d0, s1 + d1);
                    q[j] = pack_bf16(sgn * (s0 - d0), sgn * (s1 - d1));
                }
                if (row_ok) store_row16(out_p + c * 16, p, prm.wide_rows);
                if (mirror_ok) store_row16(out_m + c * 16, q, prm.wide_rows);
            }
        }
    }

    // Neither CTA may leave (its barriers and tensor memory are used by the other) before both are done.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
    }
}

template <int MODE>
__global__ void __launch_bounds__(NUM_THREADS, 1)
freqkv_gemm_kernel(const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_x,
                   const __grid_constant__ CUtensorMap map_v, const CacheView view, const GemmParams prm)
{
    constexpr int PHASES = MODE == MODE_DIRECT ? 1 : 2;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // 128-byte swizzle atoms need 1024-byte alignment
    uint8_t* aligned = smem_raw + (base - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(aligned + STAGES * STAGE_BYTES);
    const uint32_t bar0 = base + STAGES * STAGE_BYTES;
    // barrier slots (same offsets in both CTAs): full[0..S) -- used in the leader only --,
    // empty[S..2S), then s_full, s_empty, d_full, d_empty (the two *_empty used in the leader only)
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto acc_full_bar = [&](int eo) { return bar0 + 8u * (2 * STAGES + 2 * eo); };
    auto acc_empty_bar = [&](int eo) { return bar0 + 8u * (2 * STAGES + 2 * eo + 1); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster_rank();  // 0 = leader of the pair
    const int32_t cluster = blockIdx.x / 2, n_clusters = gridDim.x / 2;
    // tiles of 256 folded rows x 256 columns
    const int32_t total_tiles = prm.pair_count * prm.m_pairs;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);   // the leader's producer arrives; both producers' bytes are counted
            mbar_init(empty_bar(s), 1);  // one multicast commit
        }
        for (int eo = 0; eo < 2; ++eo) {
            mbar_init(acc_full_bar(eo), 1);               // one multicast commit
            mbar_init(acc_empty_bar(eo), 2 * EPI_WARPS);  // the epilogue warps of both CTAs
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {  // tensor memory of the pair: all 512 columns in each CTA (S in 0..255, D in 256..511)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // the peer's barriers exist before anything signals them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    if (warp < 2) {
        if (warp == 0) {
            // ---------------- TMA producer (both CTAs) ----------------
            if (lane == 0) {
                uint32_t it = 0;  // global slice counter: stage = it % STAGES, phase = it / STAGES
                bool alive = true;
                for (int32_t tile = cluster; tile < total_tiles && alive; tile += n_clusters) {
                    const int32_t pair_local = tile / prm.m_pairs;
                    const int32_t m0 = (tile % prm.m_pairs * 2 + (int32_t)rank) * BM;
                    const int32_t pair = prm.pair0 + pair_local;  // direct mode: coordinates inside the cache tensor
                    const int32_t head = pair % view.kv_heads, layer = (pair / view.kv_heads) % view.layers,
                                  seq = pair / (view.kv_heads * view.layers);
                    for (int eo = 0; eo < PHASES && alive; ++eo) {
                        // rank 0: K channels, rank 1: V
                        const int32_t plane = (pair_local * 2 + (int32_t)rank) * 2 + eo;
                        for (int32_t ks = 0; ks < prm.k_steps; ++ks, ++it) {
                            const int s = it % STAGES;
                            if (it >= STAGES &&
                                !mbar_wait(empty_bar(s), ((it / STAGES) - 1) & 1, abort_flag, prm.status, ERR_EMPTY_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            const uint32_t stage = base + s * STAGE_BYTES;
                            const uint32_t leader_full = cluster_addr(full_bar(s), 0);
                            if (rank == 0) mbar_expect_tx(full_bar(s), 2 * STAGE_BYTES);
                            const int32_t k0 = ks * BK;
                            tma_load_2d(stage, &map_p, leader_full, k0, eo * prm.basis_rows_pad + m0);
                            if constexpr (MODE == MODE_DIRECT) {
                                const CUtensorMap* cache = rank ? &map_v : &map_x;
                                tma_load_5d(stage + A_BYTES, cache, leader_full, 0, k0, head, layer, seq);
                                tma_load_5d(stage + A_BYTES + B_CHUNK_BYTES, cache, leader_full, 64, k0, head, layer, seq);
                            } else {
                                tma_load_3d(stage + A_BYTES, &map_x, leader_full, 0, k0, plane);
                                tma_load_3d(stage + A_BYTES + B_CHUNK_BYTES, &map_x, leader_full, 64, k0, plane);
                            }
                        }
                    }
                }
                if (*abort_flag) {  // let the copies in flight land before this CTA's shared memory goes away
                    const unsigned long long t0 = global_timer_ns();
                    while (global_timer_ns() - t0 < LANDING_NS) __nanosleep(1000);
                }
            }
        } else if (warp == 1) {
            // ---------------- MMA issuer (leader CTA only) ----------------
            if (lane == 0 && rank == 0) {
                uint32_t it = 0, tile_no = 0;
                bool alive = true;
                for (int32_t tile = cluster; tile < total_tiles && alive; tile += n_clusters, ++tile_no) {
                    for (int eo = 0; eo < PHASES && alive; ++eo) {
                        const int acc = eo;                 // half of tensor memory
                        const uint32_t use = tile_no;       // how often that half was filled before
                        const int32_t k_steps = prm.k_steps;
                        if (use > 0) {  // both CTAs' epilogues must have read what this half held last
                            if (!mbar_wait(acc_empty_bar(acc), (use - 1) & 1, abort_flag, prm.status, ERR_ACC_EMPTY_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        }
                        for (int32_t ks = 0; ks < k_steps; ++ks, ++it) {
                            const int s = it % STAGES;
                            if (!mbar_wait(full_bar(s), (it / STAGES) & 1, abort_flag, prm.status, ERR_FULL_WAIT, prm.wait_limit_ns)) {
                                alive = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a0 = base + s * STAGE_BYTES, b0 = a0 + A_BYTES;
    #pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk) {
                                // A: 128 rows per CTA, 8-row groups 1 KB apart; 16 k-elements = 32 bytes inside the swizzled row
                                const uint64_t ad = smem_desc(a0 + kk * 32, 16, 1024);
                                // B: per CTA 2 chunks of 64 channels 8 KB apart (leading offset), 8-row groups 1 KB apart
                                const uint64_t bd = smem_desc(b0 + kk * 2048, B_CHUNK_BYTES, 1024);
                                umma_bf16(tmem_base + acc * 256, ad, bd, (ks | kk) != 0);
                            }
                            umma_commit_both(empty_bar(s));  // frees the stage in both CTAs when these MMAs have read it
                        }
                        if (alive) umma_commit_both(acc_full_bar(acc));
                    }
                }
            }
        }
    } else {
        // ---------------- epilogue (both CTAs, each on its own 128 rows) ----------------
        const int ew = warp - 2, quarter = warp % 4, tensor = ew / 4;  // tensor: 0 = K columns, 1 = V columns
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + tensor * 128;
        const uint32_t leader_s_empty = cluster_addr(acc_empty_bar(0), 0), leader_d_empty = cluster_addr(acc_empty_bar(1), 0);
        uint32_t tile_no = 0;
        if constexpr (MODE == MODE_DIRECT) {
            for (int32_t tile = cluster; tile < total_tiles; tile += n_clusters, ++tile_no) {
                if (!mbar_wait(acc_full_bar(0), tile_no & 1, abort_flag, prm.status, ERR_ACC_FULL_WAIT, prm.wait_limit_ns)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int32_t m = (int32_t)rank * BM + quarter * 32 + lane;
                __nv_bfloat16* mat = static_cast<__nv_bfloat16*>(tensor_base(view, tensor)) +
                                     matrix_offset(view, prm.pair0 + tile) + (int64_t)prm.sink * view.stride_token;
                uint4* out = reinterpret_cast<uint4*>(mat + (int64_t)m * view.stride_token);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    uint32_t y[16];
                    tmem_ld16(lane_addr + c * 16, y);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (m < prm.n_keep) {
                        uint32_t p[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) p[j] = pack_bf16(__uint_as_float(y[2 * j]), __uint_as_float(y[2 * j + 1]));
                        out[2 * c] = make_uint4(p[0], p[1], p[2], p[3]);
                        out[2 * c + 1] = make_uint4(p[4], p[5], p[6], p[7]);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(leader_s_empty);
            }
        } else {
            for (int32_t tile = cluster; tile < total_tiles; tile += n_clusters, ++tile_no) {
                const int32_t pair = prm.pair0 + tile / prm.m_pairs;
                const int32_t head = pair % view.kv_heads, layer = (pair / view.kv_heads) % view.layers;
                const int32_t m = ((tile % prm.m_pairs) * 2 + (int32_t)rank) * BM + quarter * 32 + lane;
                bool alive = true;
                for (int eo = 0; eo < 2; ++eo) {
                    if (!mbar_wait(acc_full_bar(eo), tile_no & 1, abort_flag, prm.status, ERR_ACC_FULL_WAIT, prm.wait_limit_ns)) {
                        alive = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    float sum = 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t r[32];
                        tmem_ld32<0>(lane_addr + eo * 256 + c * 32, r);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 32; ++j) sum = fmaf(__uint_as_float(r[j]), __uint_as_float(r[j]), sum);
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(eo ? leader_d_empty : leader_s_empty);
                    const int32_t t = 2 * m + eo;  // S holds the even components, D the odd ones
                    if (float* out = tensor ? prm.spectrum[1] : prm.spectrum[0]; t < prm.n_in && out)
                        atomicAdd(out + ((int64_t)layer * view.kv_heads + head) * prm.n_in + t,
                                  sum * prm.spectrum_scale);
                }
                if (!alive) break;
            }
        }
    }

    // Neither CTA may leave (its barriers and tensor memory are used by the other) before both are done.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
    }
}

// One CTA, one thread: a wait of the kernels above on an mbarrier nothing ever arrives on, so
// that the give-up path (status bit, abort flag, return) can be exercised without stalling a
// real launch.  No TMA, no tensor memory, no cluster.
__global__ void bounded_wait_probe_kernel(int32_t* status, unsigned long long limit_ns)
{
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_wait(smem_u32(&bar), 0, &abort_flag, status, ERR_FULL_WAIT, limit_ns);
    }
}

// ---- host side ----

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    }
    return fn;
}

// Pe stacked over Po: a 2-D tensor of 2 * fold_rows_pad rows x fold_ld columns.
bool encode_basis_map(CUtensorMap* map, const Basis& basis)
{
    const cuuint64_t dims[2] = {(cuuint64_t)basis.fold_ld, (cuuint64_t)2 * basis.fold_rows_pad};
    const cuuint64_t strides[1] = {(cuuint64_t)basis.fold_ld * 2};
    const cuuint32_t box[2] = {BK, BM};
    const cuuint32_t elem[2] = {1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, basis.fold, dims, strides, box, elem,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The scratch planes as a 3-D tensor (channel, folded row, plane); rows past n_half read as zero.
bool encode_scratch_map(CUtensorMap* map, void* scratch, int32_t n_half, int32_t planes)
{
    const cuuint64_t dims[3] = {128, (cuuint64_t)n_half, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {256, (cuuint64_t)n_half * 256};
    const cuuint32_t box[3] = {64, BK, 1};
    const cuuint32_t elem[3] = {1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, scratch, dims, strides, box, elem,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 64-row slices of one block of the four (gemm_blocks); the last runs on where L/2 is even.
int32_t quad_steps(int32_t n_in) { return (n_in / 4 + BK - 1) / BK; }
int32_t quad_last_steps(int32_t n_in, int32_t n_keep) { return n_keep / 2 % 2 ? quad_steps(n_in) : (n_in / 2 + BK - 1) / BK; }

constexpr size_t kFoldBufferBytes = size_t(2304) << 20;  // scratch for the folded inputs: a 7B-shaped cache of 4096 tokens fits in one pass

}  // namespace

bool gemm_supported(int32_t dtype, int32_t head_dim, int32_t n_in, int32_t n_keep)
{
    return dtype == FREQKV_BF16 && head_dim == 128 && n_in >= 1 && n_keep >= 1 && n_keep <= n_in;
}

// A device buffer of at least `bytes`; earlier launches may still use the one it replaces.
static cudaError_t grow(void** buffer, size_t* have, size_t bytes)
{
    if (bytes <= *have) return cudaSuccess;
    if (*buffer) {
        const cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return e;
        cudaFree(*buffer);
        *buffer = nullptr;
        *have = 0;
    }
    const cudaError_t e = cudaMalloc(buffer, bytes);
    if (e == cudaSuccess)
        *have = bytes;
    else
        *buffer = nullptr;
    return e;
}

// A launch of CTA pairs.
struct PairLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    PairLaunch(int ctas, int threads, int smem, cudaStream_t stream)
    {
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = (size_t)smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

// Everything a launch needs that is not a stream operation: kernel attributes, the count of
// resident CTA pairs, the scratch buffer for `pairs` (batch, layer, kv_head) triples of this basis
// (pairs = 0: none, the direct mode reads the cache itself).
// launch_gemm calls it itself; a caller that must not allocate later (stream capture) calls it first.
cudaError_t gemm_prepare(GemmState* state, int32_t pairs, const Basis& basis, int sm_count)
{
    state->last_error = nullptr;
    if (!encode_fn()) {
        state->last_error = "cuTensorMapEncodeTiled is not available from this driver";
        return cudaErrorNotSupported;
    }
    if (!state->attr_set) {
        const void* kernels[3] = {(const void*)freqkv_gemm_kernel<MODE_SPECTRUM>, (const void*)freqkv_gemm_kernel<MODE_DIRECT>,
                                  (const void*)freqkv_fold_gemm_kernel};
        for (int i = 0; i < 3; ++i) {
            const cudaError_t e = cudaFuncSetAttribute(kernels[i], cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
            if (e != cudaSuccess) {
                state->last_error = "cudaFuncSetAttribute(max dynamic shared memory)";
                return e;
            }
        }
        {  // the register shares are of what the block is launched with
            cudaFuncAttributes fa;
            const cudaError_t e = cudaFuncGetAttributes(&fa, kernels[2]);
            if (e != cudaSuccess || fa.numRegs < FOLD_LAUNCH_REGS) {
                state->last_error = "the kernel of the folded forms was not built with the registers it shares out";
                return e != cudaSuccess ? e : cudaErrorLaunchOutOfResources;
            }
        }
        // how many CTA pairs the device can hold at once (one CTA per SM; SMs pair up inside a GPC)
        PairLaunch launch(2 * (sm_count / 2), FOLD_THREADS, SMEM_BYTES, nullptr);
        int n = 0;
        const cudaError_t q = cudaOccupancyMaxActiveClusters(&n, freqkv_fold_gemm_kernel, &launch.cfg);
        if (q != cudaSuccess || n < 1) {
            state->last_error = "cudaOccupancyMaxActiveClusters: no CTA pair fits on this device";
            return q != cudaSuccess ? q : cudaErrorLaunchOutOfResources;
        }
        state->max_clusters = std::min(n, sm_count / 2);
        state->attr_set = true;
    }
    const int32_t n_half = (basis.n_in + 1) / 2;
    const size_t per_pair = (size_t)4 * n_half * 128 * 2;  // K and V, U and V planes
    const int64_t fit = std::max<int64_t>(1, (int64_t)(kFoldBufferBytes / per_pair));
    const int64_t pass = std::min<int64_t>(fit, pairs);
    const cudaError_t e = grow(&state->scratch, &state->scratch_bytes, (size_t)pass * per_pair);
    if (e != cudaSuccess) state->last_error = "cudaMalloc(fold scratch)";
    return e;
}

static FoldParams fold_params(const GemmState* state, const CacheView& view, const Basis& b, int32_t sink, int32_t* status_dev)
{
    FoldParams prm = {};
    prm.sink = sink;
    prm.mirror_sign = (b.first & 1) ? -1 : 1;
    prm.wide_rows = (((uintptr_t)view.base[0] | (uintptr_t)view.base[1]) & 31) == 0 &&
                    ((view.stride_token | view.stride_head | view.stride_layer | view.stride_batch) & 15) == 0;
    prm.n_keep = b.n_keep;
    prm.rows_half = (b.n_keep + 1) / 2;
    prm.basis_rows_pad = b.fold_rows_pad;
    prm.k_steps = ((b.n_in + 1) / 2 + BK - 1) / BK;
    prm.m_pairs = (prm.rows_half + 2 * BM - 1) / (2 * BM);
    prm.status = status_dev;
    prm.wait_limit_ns = state->wait_limit_ns;
    return prm;
}

static FoldJob fold_job(const Basis& b, int32_t pair0, int32_t pairs, int32_t sink, void* planes)
{
    FoldJob job;
    job.pair0 = pair0;
    job.pair_count = pairs;
    job.n_in = b.n_in;
    job.n_half = (b.n_in + 1) / 2;
    job.sink = sink;
    job.dst = static_cast<uint4*>(planes);
    return job;
}

// Blocks per matrix of a fold launch: each takes rounds of 1024 vectors.
static unsigned fold_blocks(int32_t n_half) { return (unsigned)std::min<int64_t>(((int64_t)n_half * 16 + 1023) / 1024, 64); }

// The product, after its fold launch.
static cudaError_t launch_product(GemmState* state, const CUtensorMap& map_p, const CUtensorMap& map_x, const CacheView& view,
                                  const FoldParams& prm, const LaunchHooks& hooks, cudaStream_t stream)
{
    PairLaunch launch(2 * std::min<int32_t>(prm.total_tiles, state->max_clusters), FOLD_THREADS, SMEM_BYTES, stream);
    if (hooks.before) hooks.before(hooks.user, stream);
    const cudaError_t e = cudaLaunchKernelEx(&launch.cfg, freqkv_fold_gemm_kernel, map_p, map_x, view, prm);
    if (hooks.after) hooks.after(hooks.user, stream);
    if (e != cudaSuccess) {
        state->last_error = "freqkv_fold_gemm_kernel launch";
        return e;
    }
    state->kernels_last_call += 2;
    return cudaSuccess;
}

cudaError_t launch_gemm(GemmState* state, const CacheView& view, const Basis& basis, int32_t sink, int32_t* status_dev,
                        int sm_count, const LaunchHooks& hooks, cudaStream_t stream)
{
    state->kernels_last_call = 0;
    const cudaError_t prepared = gemm_prepare(state, view.mats_per_tensor, basis, sm_count);
    if (prepared != cudaSuccess) return prepared;
    const int32_t pairs = view.mats_per_tensor;
    const size_t per_pair = (size_t)4 * ((basis.n_in + 1) / 2) * 128 * 2;
    // One pass when the folded inputs fit the scratch buffer, else several passes of `chunk` pairs.
    const int64_t chunk = std::min<int64_t>(std::max<int64_t>(1, (int64_t)(kFoldBufferBytes / per_pair)), pairs);
    CUtensorMap map_p;
    if (!encode_basis_map(&map_p, basis)) {
        state->last_error = "tensor map encoding rejected the basis";
        return cudaErrorInvalidValue;
    }
    const int32_t n_half = (basis.n_in + 1) / 2;
    FoldParams prm = fold_params(state, view, basis, sink, status_dev);
    for (int64_t p0 = 0; p0 < pairs; p0 += chunk) {
        const int32_t count = (int32_t)std::min<int64_t>(chunk, pairs - p0);
        CUtensorMap map_x;
        if (!encode_scratch_map(&map_x, state->scratch, n_half, count * 4)) {
            state->last_error = "tensor map encoding rejected the scratch planes";
            return cudaErrorInvalidValue;
        }
        prm.pair0 = (int32_t)p0;
        if ((int64_t)count * prm.m_pairs > 0x7fffffff) return cudaErrorInvalidValue;
        prm.total_tiles = count * prm.m_pairs;
        fold_kernel<<<dim3((unsigned)count * 2, fold_blocks(n_half)), 256, 0, stream>>>(
            view, fold_job(basis, (int32_t)p0, count, sink, state->scratch));
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            state->last_error = "fold_kernel launch";
            return e;
        }
        e = launch_product(state, map_p, map_x, view, prm, hooks, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The power spectrum: a fold pass and a pass of the spectrum kernel (two launches per scratch buffer full of planes).
cudaError_t launch_gemm_spectrum(GemmState* state, const CacheView& view, const Basis& basis, int32_t sink, int32_t* status_dev,
                                 int sm_count, const LaunchHooks& hooks, cudaStream_t stream, const SpectrumOut& spectrum)
{
    state->kernels_last_call = 0;
    const cudaError_t prepared = gemm_prepare(state, view.mats_per_tensor, basis, sm_count);
    if (prepared != cudaSuccess) return prepared;
    const int32_t n_half = (basis.n_in + 1) / 2, rows_half = (basis.n_keep + 1) / 2;
    const int32_t pairs = view.mats_per_tensor;
    const size_t per_pair = (size_t)4 * n_half * 128 * 2;
    const int64_t chunk = std::min<int64_t>(std::max<int64_t>(1, (int64_t)(kFoldBufferBytes / per_pair)), pairs);
    CUtensorMap map_p;
    if (!encode_basis_map(&map_p, basis)) {
        state->last_error = "tensor map encoding rejected the basis";
        return cudaErrorInvalidValue;
    }
    for (int64_t p0 = 0; p0 < pairs; p0 += chunk) {
        FoldJob job;
        job.pair0 = (int32_t)p0;
        job.pair_count = (int32_t)std::min<int64_t>(chunk, pairs - p0);
        job.n_in = basis.n_in;
        job.n_half = n_half;
        job.sink = sink;
        job.dst = static_cast<uint4*>(state->scratch);
        fold_kernel<<<dim3((unsigned)job.pair_count * 2, fold_blocks(n_half)), 256, 0, stream>>>(view, job);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            state->last_error = "fold_kernel launch";
            return e;
        }
        CUtensorMap map_x;
        if (!encode_scratch_map(&map_x, state->scratch, n_half, job.pair_count * 4)) {
            state->last_error = "tensor map encoding rejected the scratch planes";
            return cudaErrorInvalidValue;
        }
        GemmParams prm = {};
        prm.n_keep = basis.n_keep;
        prm.basis_rows_pad = basis.fold_rows_pad;
        prm.pair0 = job.pair0;
        prm.pair_count = job.pair_count;
        prm.m_pairs = (rows_half + 2 * BM - 1) / (2 * BM);
        prm.k_steps = (n_half + BK - 1) / BK;
        prm.sink = sink;
        prm.spectrum[0] = spectrum.k;
        prm.spectrum[1] = spectrum.v;
        prm.spectrum_scale = spectrum.scale;
        prm.n_in = basis.n_in;
        prm.status = status_dev;
        prm.wait_limit_ns = state->wait_limit_ns;
        PairLaunch launch(2 * std::min<int32_t>(job.pair_count * prm.m_pairs, state->max_clusters), NUM_THREADS, SMEM_BYTES, stream);
        if (hooks.before) hooks.before(hooks.user, stream);
        e = cudaLaunchKernelEx(&launch.cfg, freqkv_gemm_kernel<MODE_SPECTRUM>, map_p, map_x, map_x, view, prm);
        if (hooks.after) hooks.after(hooks.user, stream);
        if (e != cudaSuccess) {
            state->last_error = "freqkv_gemm_kernel launch";
            return e;
        }
        state->kernels_last_call += 2;
    }
    return cudaSuccess;
}

// The non-sink rows of one cache tensor as a 5-D tensor (channel, token, kv_head, layer, batch).
static bool encode_cache_map(CUtensorMap* map, const CacheView& view, int tensor, int32_t batch_count, int32_t n_in, int32_t sink)
{
    char* p = static_cast<char*>(tensor ? view.base[1] : view.base[0]) +
              ((int64_t)view.batch0 * view.stride_batch + (int64_t)sink * view.stride_token) * 2;
    const cuuint64_t dims[5] = {128, (cuuint64_t)n_in, (cuuint64_t)view.kv_heads, (cuuint64_t)view.layers,
                                (cuuint64_t)batch_count};
    // an axis of extent 1 is never stepped; give it a harmless stride
    const cuuint64_t row = (cuuint64_t)view.stride_token * 2;
    const cuuint64_t strides[4] = {row, view.kv_heads > 1 ? (cuuint64_t)view.stride_head * 2 : row,
                                   view.layers > 1 ? (cuuint64_t)view.stride_layer * 2 : row,
                                   batch_count > 1 ? (cuuint64_t)view.stride_batch * 2 : row};
    const cuuint32_t box[5] = {64, BK, 1, 1, 1};
    const cuuint32_t elem[5] = {1, 1, 1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, p, dims, strides, box, elem,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool gemm_is_direct(int32_t n_keep) { return n_keep <= 2 * BM; }

// Levels of the mirror symmetry alone: 0 = none (the direct mode), 2 where the lengths halve twice (n_in a
// multiple of 4, n_keep even, the lowest components kept) and a second level would mean fewer 64-row slices per
// matrix pair (tiles are 256 rows high: with few kept rows it can leave its last tile nearly empty), else 1.
int32_t gemm_fold_levels(int32_t n_in, int32_t n_keep, int32_t first)
{
    if (gemm_is_direct(n_keep)) return 0;
    if (first != 0 || n_in % 4 != 0 || n_keep % 2 != 0) return 1;
    const int32_t n_half = n_in / 2, rows_half = n_keep / 2, rows_quarter = (rows_half + 1) / 2;
    const int64_t slices1 = (int64_t)((rows_half + 2 * BM - 1) / (2 * BM)) * 2 * ((n_half + BK - 1) / BK);
    const int64_t slices2 =
        (int64_t)((rows_quarter + 2 * BM - 1) / (2 * BM)) * 2 * ((n_half / 2 + BK - 1) / BK + (n_half + BK - 1) / BK);
    return slices2 < slices1 ? 2 : 1;
}

bool gemm_quad(int32_t n_in, int32_t n_keep, int32_t first) { return gemm_fold_levels(n_in, n_keep, first) == 2; }

// In how many blocks the symmetries of the cosines would cut a compression of these lengths, and a call of this size run them: 1, 2
// (one level), or 4 (both levels, the odd part split by a rotation) where a count of 64-row slices, with 30 for the longer epilogue of a
// four-block tile, says they pay.  What this file runs is one level; plain compressions of more than 256 kept rows take nearfar.cu, whose
// work is not cut this way.
int32_t gemm_blocks(int32_t n_in, int32_t n_keep, int32_t first, int64_t triples)
{
    if (gemm_is_direct(n_keep)) return 1;
    if (!gemm_quad(n_in, n_keep, first)) return 2;
    constexpr int64_t CLUSTERS = 74;  // CTA pairs of a B200
    const int32_t rows_half = n_keep / 2, rows_quarter = (rows_half + 1) / 2;
    const int64_t tiles2 = (rows_half + 2 * BM - 1) / (2 * BM), tiles4 = (rows_quarter + 2 * BM - 1) / (2 * BM);
    const int64_t slices2 = 2 * ((n_in / 2 + BK - 1) / BK), slices4 = 3 * quad_steps(n_in) + quad_last_steps(n_in, n_keep);
    const int64_t waves2 = (triples * tiles2 + CLUSTERS - 1) / CLUSTERS, waves4 = (triples * tiles4 + CLUSTERS - 1) / CLUSTERS;
    return waves4 * (slices4 + 30) < waves2 * slices2 ? 4 : 2;
}

cudaError_t launch_gemm_direct(GemmState* state, const CacheView& view, const Basis& basis, int32_t sink,
                               int32_t* status_dev, int sm_count, const LaunchHooks& hooks, cudaStream_t stream)
{
    state->kernels_last_call = 0;
    const cudaError_t prepared = gemm_prepare(state, 0, basis, sm_count);
    if (prepared != cudaSuccess) return prepared;
    const int32_t pairs = view.mats_per_tensor;
    const int32_t batch_count = pairs / (view.layers * view.kv_heads);
    CUtensorMap map_p, map_k, map_v;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)basis.ld, (cuuint64_t)basis.dense_rows_pad};
        const cuuint64_t strides[1] = {(cuuint64_t)basis.ld * 2};
        const cuuint32_t box[2] = {BK, BM};
        const cuuint32_t elem[2] = {1, 1};
        if (encode_fn()(&map_p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, basis.dense, dims, strides, box, elem,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            state->last_error = "tensor map encoding rejected the basis";
            return cudaErrorInvalidValue;
        }
    }
    if (!encode_cache_map(&map_k, view, 0, batch_count, basis.n_in, sink) ||
        !encode_cache_map(&map_v, view, 1, batch_count, basis.n_in, sink)) {
        state->last_error = "tensor map encoding rejected this layout";
        return cudaErrorInvalidValue;
    }
    GemmParams prm = {};
    prm.n_keep = basis.n_keep;
    prm.basis_rows_pad = 0;
    prm.pair0 = 0;
    prm.pair_count = pairs;
    prm.m_pairs = 1;
    prm.k_steps = (basis.n_in + BK - 1) / BK;
    prm.sink = sink;
    prm.n_in = basis.n_in;
    prm.status = status_dev;
    prm.wait_limit_ns = state->wait_limit_ns;
    PairLaunch launch(2 * std::min<int32_t>(pairs, state->max_clusters), NUM_THREADS, SMEM_BYTES, stream);
    if (hooks.before) hooks.before(hooks.user, stream);
    const cudaError_t e = cudaLaunchKernelEx(&launch.cfg, freqkv_gemm_kernel<MODE_DIRECT>, map_p, map_k, map_v, view, prm);
    if (hooks.after) hooks.after(hooks.user, stream);
    if (e != cudaSuccess) {
        state->last_error = "freqkv_gemm_kernel launch";
        return e;
    }
    state->kernels_last_call = 1;
    return cudaSuccess;
}

cudaError_t launch_wait_probe(int32_t* status_dev, unsigned long long limit_ns, cudaStream_t stream)
{
    bounded_wait_probe_kernel<<<1, 32, 0, stream>>>(status_dev, limit_ns);
    return cudaGetLastError();
}

void gemm_release(GemmState* state)
{
    if (state->ragged_meta) cudaFree(state->ragged_meta);
    state->ragged_meta = nullptr;
    state->ragged_meta_bytes = 0;
    if (state->scratch) cudaFree(state->scratch);
    state->scratch = nullptr;
    state->scratch_bytes = 0;
}

}  // namespace freqkv
