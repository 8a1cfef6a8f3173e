// The compression Y = P X of bf16 caches, in place, in one pass over the cache.
//
// The basis as a Cauchy matrix.  With theta_m = pi (2m+1) / (2L), phi_n = pi (2n+1) / (2N) the entries of basis.cuh are
//     P[m][n] = (1/N) sum_{t<L} eps_t cos(t theta_m) cos(t phi_n)      (eps_0 = 1, eps_t = 2)
//             = (-1)^m sin(theta_m) * cos(L phi_n) / N * 1 / (cos(phi_n) - cos(theta_m)),
// the Christoffel-Darboux sum of the Chebyshev polynomials T_t at y_m = cos(theta_m), x_n = cos(phi_n): its second term
// drops out because T_L(y_m) = 0.  So apart from two diagonal factors P is 1 / (x_n - y_m), and for a tile of 128
// consecutive rows m and all columns n that are not close to it that is a function of few degrees of freedom.
//   near  columns [lo, lo + window) around the rows under a tile (the tile's own 128 N/L rows and a margin on either side):
//         the entries themselves, as one small dense product;
//   far   all other columns: interpolated over the tile by rational functions with `rank` nodes a_i and as many poles p_j,
//             1 / (x - y) ~ sum_i U_i(y) / (x - a_i),   U_i(y) = prod_{k != i} (y - a_k) / (a_i - a_k) * prod_j (a_i - p_j) / (y - p_j),
//         exact for x = p_j.  Nodes and poles are those of Zolotarev's rational function for the pair (tile, far columns)
//         -- sn at equidistant arguments, moved by the Moebius map that takes the two sets to [-1, 1] and |z| >= 1/k
//         (Beckermann, Townsend, "Bounds on the singular values of matrices with displacement structure", 2019) -- for
//         which the error falls by a constant factor per node.  So a tile needs `rank` numbers per channel of all its far
//         rows, E_i = sum_{n far} w_in x_n.
// The near products grow with N instead of N L, for every N and L: no length has to halve.  The far products are N for each 128
// far rows, `rank` of them a tile: one block up to 4096 kept rows, then N L / 4096 (16 blocks at 131072 -> 65536, with 0.5 GB of
// far basis and 180 MB of sums for a group in flight).
//
// The kernel.  One persistent CTA per SM takes jobs in the order of a ticket counter; a group of columns is 256 channels,
// the K and the V matrix of one (batch, layer, kv_head) of head_dim 128.  For every group come first its far jobs (a range of
// input slices times 128 far rows: partial sums, fp32, to a small ring in L2), a few groups ahead, then its tile jobs
// (near slices, then 16 more columns that add the far part).  Every job is a product of 128 rows x 256 columns; both read
// x as it lies in the cache, so nothing is folded or copied, and the second reading comes out of L2, since the groups
// between a far job and its tiles are few.  In each CTA:
//   warps 0,2,3  tickets; TMA: per slice 16 KB of basis (stored as the shared-memory image) and 64 rows x 256 channels
//   warp 1       tcgen05.mma 128 x 256 x 16, two accumulators of 256 columns of tensor memory in turn
//   warps 4-11   epilogue: partial far sums to the ring, or rows rounded to bf16 into the cache
//   warps 12-15  the far operand of the tiles: sums of the parts, as bf16 and its remainder in bf16 (16 rows of the product)
//   warps 16,17  far sums written and read: one release for all warps
// A tile overwrites rows that other tiles of its group read.  It waits until those have them in shared memory (flags):
// only tiles before it and the one after it can be among them, so every wait is for a job whose ticket is lower, or the
// very next one, which nothing keeps from loading (its accumulator is the other one, its far jobs have lower tickets).
//
// Its floor is HBM, (N + L) rows in and out; it runs at 0.46 to 0.59 of that: a job costs 7900 cycles and 770 for each of its slices
// (48 KB at the 64 bytes a clock that an SM takes from L2), and the first part hides behind nothing (4092 -> 2046 x 1024 groups 0.92 ms,
// 131 jobs an SM of 7.6 slices).
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "basis.cuh"
#include "nearfar.cuh"

namespace freqkv {
namespace {

constexpr int BM = 128, BK = 64, BN = 256;
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;        // 16 KB
constexpr int CHUNK_BYTES = BK * 128;       // 8 KB: 64 rows x 64 channels
constexpr int B_BYTES = 4 * CHUNK_BYTES;    // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int FAR_COLS = 16;                // columns of a near block that hold the far weights: of the values, of their remainders
constexpr int FAR_CHUNK = FAR_COLS * 128;   // 16 rows x 64 channels
constexpr int FAR_BYTES = 4 * FAR_CHUNK;
constexpr int JOBS = 4;                     // ring of jobs between the producer and the other roles
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 2 * FAR_BYTES + 1024 + 512;
constexpr int EPI_WARPS = 8, FAR_WARPS = 4, LOAD_WARPS = 3;
constexpr int EPI_WARP0 = 4, FAR_WARP0 = EPI_WARP0 + EPI_WARPS, WRITTEN_WARP = FAR_WARP0 + FAR_WARPS, READ_WARP = WRITTEN_WARP + 1;
constexpr int THREADS = 32 * (READ_WARP + 1);
constexpr int MAX_RANK = 8;
constexpr int TABLE = 4;                    // int32 per tile: first near column, first and last tile that reads its rows, -
constexpr int64_t AHEAD_BYTES = 40000000;
constexpr int64_t RING_BYTES = 256 << 20;   // the far sums of a call whose places are not all of one size (four places may take more)
constexpr unsigned long long LANDING_NS = 1000000ull;
constexpr uint32_t FAR_READ = 0x80000000u;  // in the counter of a group: every tile has read the far sums

// The matrices of one item of the call.
struct Seq {
    const uint8_t* blocks;      // near blocks, then far blocks
    const int32_t* table;
    int32_t group0, triple0, triples;
    int32_t n_keep, tiles, rank, slices, k_slices, part_slices, parts, far_tiles;
    int32_t read0;              // first of its tiles' flags
};

// Consecutive blocks of tickets that look alike: block i holds the far jobs of group i + ahead, then the tiles of group i.
struct Run {
    int32_t ticket0, block0, far_jobs, tiles, far_seq, tile_seq;
};

struct Params {
    Seq seq;                    // uniform calls
    Run run[3];
    const Seq* seqs;            // ragged batches
    const Run* runs;
    const CUtensorMap* maps;    // K and V of every item
    int32_t n_maps;
    int32_t n_runs, tickets, ahead, ring;
    int32_t sink, wide;
    float* far;                 // [ring][far_tiles x parts][tile][64][rank][4 columns]
    int64_t far_stride;         // floats per group
    uint32_t* flags;            // ticket | far sums written [groups] | far sums read [groups] | rows read [tiles]
    int32_t groups;
    int32_t* status;
    unsigned long long wait_limit_ns;
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
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// (The hint lets the hardware put the warp to sleep: twenty warps that spin leave the epilogue a fifth of the issue slots.)
constexpr uint32_t SUSPEND_NS = 20000;
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(SUSPEND_NS)
        : "memory");
    return ok != 0;
}
// Wait for something to become true, for at most `limit_ns`; gives up earlier when another role of the CTA has.  Where it
// gives up first it sets the status bit and the CTA's abort flag.
template <class F>
__device__ __forceinline__ bool bounded(F&& ready, volatile int* abort_flag, int32_t* status, unsigned long long limit_ns)
{
    if (ready()) return true;
    const unsigned long long t0 = global_timer_ns();
    for (;;) {
        for (int i = 0; i < 32; ++i)
            if (ready()) return true;
        if (*abort_flag) return false;
        if (global_timer_ns() - t0 > limit_ns) {
            atomicOr(status, NEARFAR_ERR_WAIT);
            *abort_flag = 1;
            __threadfence_block();
            return false;
        }
    }
}
__device__ __forceinline__ uint32_t load_acquire(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t load_relaxed(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// For waits on other CTAs: relaxed looks, one acquiring load at the end (an acquiring load empties the SM's L1).
template <class F>
__device__ __forceinline__ bool seen(const uint32_t* p, F&& good)
{
    if (!good(load_relaxed(p))) return false;
    return good(load_acquire(p));
}
__device__ __forceinline__ void store_relaxed(uint32_t* p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void store_release(uint32_t* p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t* p, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
// Counters in shared memory, one for each warp: the warp that publishes for all of them waits for every one.
__device__ __forceinline__ void count_up(uint32_t* p, uint32_t n) { asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(n) : "memory"); }
__device__ __forceinline__ uint32_t counted(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t c0, int32_t c1, int32_t c2,
                                            int32_t c3, int32_t c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}
// A tensor map that a copy has put into global memory, before the CTA's loads use it: what the SM holds of the map that lay
// there before (the call before had other lengths, another cache) is not read again.
__device__ __forceinline__ void map_acquire(const CUtensorMap* map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
                 "r"(bytes), "r"(bar)
                 : "memory");
}
// Shared-memory matrix descriptor of tcgen05.mma: start address, leading and stride byte offsets (16-byte units), version 1,
// 128-byte swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// kind::f16: D fp32, A and B bf16, A K-major, B MN-major, M = 128, N = 256.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (0u << 15) | (1u << 16) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(IDESC), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void store32(void* dst, const uint32_t* v, bool wide)
{
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                     "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    } else {
        static_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        static_cast<uint4*>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

// Where the four 64-channel chunks of a group lie: head_dim 128 K | V of one triple; 64 K K | V V of two; 256 K or V of one.
struct Chunk {
    int32_t tensor, triple, channel;
};
__device__ __forceinline__ Chunk chunk_of(int32_t head_dim, int32_t group, int32_t j)
{
    if (head_dim == 128) return {j >> 1, group, (j & 1) * 64};
    if (head_dim == 64) return {j >> 1, 2 * group + (j & 1), 0};
    return {group & 1, group >> 1, j * 64};
}

struct Job {
    int32_t kind, seq, group, idx;  // group: over the whole call; idx: tile, or far tile * parts + part
    int32_t row, first, last;       // tiles: their entry of the plan's table; far jobs: first input row
    int32_t steps;
    int32_t ready;                  // tiles: the far sums were written when the ticket was taken
};
constexpr int32_t JOB_FAR = 0, JOB_TILE = 1, JOB_STOP = 2;

template <bool RAGGED>
__global__ void __launch_bounds__(THREADS, 1)
freqkv_nearfar_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const CacheView view,
                      const __grid_constant__ Params prm)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t base = smem_u32(smem);
    const uint32_t far_base = base + STAGES * STAGE_BYTES;
    uint8_t* far_smem = smem + STAGES * STAGE_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(far_smem + 2 * FAR_BYTES);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8 * s; };
    auto empty_bar = [&](int s) { return bar0 + 8 * (STAGES + s); };
    auto acc_full = [&](int s) { return bar0 + 8 * (2 * STAGES + s); };
    auto acc_empty = [&](int s) { return bar0 + 8 * (2 * STAGES + 2 + s); };
    auto far_full = [&](int s) { return bar0 + 8 * (2 * STAGES + 4 + s); };
    auto far_empty = [&](int s) { return bar0 + 8 * (2 * STAGES + 6 + s); };
    auto job_full = [&](int s) { return bar0 + 8 * (2 * STAGES + 8 + s); };
    auto job_empty = [&](int s) { return bar0 + 8 * (2 * STAGES + 8 + JOBS + s); };
    constexpr int N_BARS = 2 * STAGES + 9 + 2 * JOBS;
    const uint32_t drained = bar0 + 8 * (N_BARS - 1);
    Job* jobs = reinterpret_cast<Job*>(bars + N_BARS);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(jobs + JOBS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint32_t* written = tmem_slot + 2;          // per epilogue warp: far jobs whose sums it has stored
    uint32_t* read = written + EPI_WARPS;       // per far warp: tiles whose sums it has read

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), LOAD_WARPS);
            mbar_init(empty_bar(s), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(acc_full(s), 1);
            mbar_init(acc_empty(s), EPI_WARPS);
            mbar_init(far_full(s), FAR_WARPS);
            mbar_init(far_empty(s), 1);
        }
        for (int s = 0; s < JOBS; ++s) {
            mbar_init(job_full(s), 1);
            mbar_init(job_empty(s), (LOAD_WARPS - 1) + 1 + EPI_WARPS + FAR_WARPS + 2);
        }
        mbar_init(drained, 1);
        *abort_flag = 0;
        for (int i = 0; i < EPI_WARPS + FAR_WARPS; ++i) written[i] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    // All maps by all threads side by side, ahead of the barrier that the loads come after: by the loading threads as they come to a
    // sequence the fences stand between its loads (a batch of eight 3056 against 3031 us).
    if (RAGGED)
        for (int32_t i = threadIdx.x; i < prm.n_maps; i += THREADS) map_acquire(prm.maps + i);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    uint32_t* const far_written = prm.flags + 16;
    uint32_t* const far_read = far_written + prm.groups;
    uint32_t* const rows_read = far_read + prm.groups;
    auto seq_of = [&](int32_t i) -> const Seq& { return RAGGED ? prm.seqs[i] : prm.seq; };
    auto wait_bar = [&](uint32_t bar, uint32_t parity) {
        return bounded([&] { return mbar_try_wait(bar, parity); }, abort_flag, prm.status, prm.wait_limit_ns);
    };
    auto wait_flag = [&](auto&& ready) { return bounded(ready, abort_flag, prm.status, prm.wait_limit_ns); };
    // by every lane of a warp, with one outcome for all of them
    auto warp_wait_bar = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, wait_bar(bar, parity)) != 0; };

    if (warp == 0 || warp == 2 || warp == 3) {
        // ---------------- loads: warp 0 takes the tickets and brings the basis, warps 2 and 3 half of the group's chunks each ----------------
        // (A thread issues a bulk or tensor copy every 250 to 300 cycles, whatever its size: five of them a slice from one thread
        // took twice as long as the slice's products.)
        if (lane == 0) {
            uint32_t it = 0;
            int32_t run_idx = 0;
            Run run = RAGGED ? prm.runs[0] : prm.run[0];
            int32_t ticket = warp == 0 ? (int32_t)atomicAdd(prm.flags, 1u) : 0;
            bool alive = true;
            for (uint32_t n = 0; alive; ++n) {
                const int slot = n % JOBS;
                Job job = {JOB_STOP, 0, 0, 0, 0, 0, 0, 0, 0};
                if (warp == 0) {
                    if (ticket < prm.tickets) {
                        while (run_idx + 1 < prm.n_runs) {
                            const Run next = RAGGED ? prm.runs[run_idx + 1] : prm.run[run_idx + 1 < 3 ? run_idx + 1 : 2];
                            if (ticket < next.ticket0) break;
                            run = next;
                            ++run_idx;
                        }
                        const int32_t per_block = run.far_jobs + run.tiles;
                        const int32_t block = (ticket - run.ticket0) / per_block, at = (ticket - run.ticket0) % per_block;
                        if (at < run.far_jobs) {
                            const Seq& s = seq_of(run.far_seq);
                            const int32_t s0 = at % s.parts * s.part_slices;
                            job = {JOB_FAR, run.far_seq, run.block0 + block + prm.ahead, at, s0 * BK, 0, 0, min(s.part_slices, s.k_slices - s0), 0};
                        } else {
                            const Seq& s = seq_of(run.tile_seq);
                            const int32_t tile = at - run.far_jobs;
                            const int32_t group = run.block0 + block;
                            const int4 t = __ldg(reinterpret_cast<const int4*>(s.table + tile * TABLE));
                            const int32_t ready = load_acquire(far_written + group) >= (uint32_t)(s.parts * s.far_tiles);
                            job = {JOB_TILE, run.tile_seq, group, tile, t.x, t.y, t.z, s.slices, ready};
                        }
                    }
                    if (n >= JOBS && !wait_bar(job_empty(slot), (n / JOBS - 1) & 1)) break;
                    jobs[slot] = job;
                    mbar_arrive(job_full(slot));
                } else {
                    if (!wait_bar(job_full(slot), (n / JOBS) & 1)) break;
                    job = jobs[slot];
                    mbar_arrive(job_empty(slot));
                }
                if (job.kind == JOB_STOP) break;

                const Seq& s = seq_of(job.seq);
                if (warp == 0) {
                    const size_t block0 = job.kind == JOB_FAR ? (size_t)s.tiles * s.slices + (size_t)(job.idx / s.parts) * s.k_slices + job.row / BK
                                                              : (size_t)job.idx * s.slices;
                    const uint8_t* a = s.blocks + block0 * A_BYTES;
                    int32_t next = 0;
                    for (int32_t ks = 0; ks < job.steps; ++ks, ++it) {
                        if (ks == max(0, job.steps - 4)) next = (int32_t)atomicAdd(prm.flags, 1u);
                        const int st = it % STAGES;
                        if (it >= STAGES && !wait_bar(empty_bar(st), (it / STAGES - 1) & 1)) {
                            alive = false;
                            break;
                        }
                        mbar_expect_tx(full_bar(st), A_BYTES);
                        bulk_load(base + st * STAGE_BYTES, a + (size_t)ks * A_BYTES, A_BYTES, full_bar(st));
                    }
                    ticket = next;
                    continue;
                }
                // chunks 2 (warp - 2) and the one after it: coordinates of their (kv_head, layer, batch)
                int32_t ch[2], h[2], l[2], b[2], valid = 0;
                const CUtensorMap* map[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const Chunk c = chunk_of(view.head_dim, job.group - s.group0, 2 * (warp - 2) + j);
                    if (c.triple < s.triples) valid |= 1 << j;
                    const int32_t t = s.triple0 + min(c.triple, s.triples - 1);
                    ch[j] = c.channel;
                    h[j] = t % view.kv_heads;
                    l[j] = t / view.kv_heads % view.layers;
                    b[j] = t / (view.kv_heads * view.layers);
                    map[j] = RAGGED ? prm.maps + 2 * job.seq + c.tensor : c.tensor ? &map_v : &map_k;
                }
                for (int32_t ks = 0; ks < job.steps; ++ks, ++it) {
                    const int st = it % STAGES;
                    if (it >= STAGES && !wait_bar(empty_bar(st), (it / STAGES - 1) & 1)) {
                        alive = false;
                        break;
                    }
                    const uint32_t dst = base + st * STAGE_BYTES + A_BYTES + 2 * (warp - 2) * CHUNK_BYTES;
                    mbar_expect_tx(full_bar(st), __popc(valid) * CHUNK_BYTES);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (valid >> j & 1)
                            tma_load_5d(dst + j * CHUNK_BYTES, map[j], full_bar(st), ch[j], job.row + ks * BK, h[j], l[j], b[j]);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t it = 0, tiles = 0;
            bool alive = true;
            for (uint32_t n = 0; alive; ++n) {
                const int slot = n % JOBS;
                if (!wait_bar(job_full(slot), (n / JOBS) & 1)) break;
                const Job job = jobs[slot];
                mbar_arrive(job_empty(slot));
                if (job.kind == JOB_STOP) break;
                const Seq& s = seq_of(job.seq);
                const bool tile = job.kind == JOB_TILE;
                const int32_t steps = job.steps;
                const uint32_t acc = n & 1, use = n >> 1;
                if (use > 0 && !wait_bar(acc_empty(acc), (use - 1) & 1)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d = tmem_base + acc * BN;
                for (int32_t ks = 0; ks < steps; ++ks, ++it) {
                    const int st = it % STAGES;
                    if (!wait_bar(full_bar(st), (it / STAGES) & 1)) {
                        alive = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const bool last = tile && ks == steps - 1;
                    const uint32_t a0 = base + st * STAGE_BYTES, b0 = a0 + A_BYTES;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        if (kk == 3 && last) break;
                        umma(d, smem_desc(a0 + kk * 32, 16, 1024), smem_desc(b0 + kk * 2048, CHUNK_BYTES, 1024), (ks | kk) != 0);
                    }
                    if (last) {
                        // Every row of the window is in shared memory (this thread has seen the barriers of its copies): they may be
                        // overwritten.  Nothing was written that the flag would have to publish, so it needs no release, which
                        // takes 4000 cycles here (it waits for the stores of the other warps).
                        store_relaxed(rows_read + s.read0 + (job.group - s.group0) * s.tiles + job.idx, 1u);
                        const uint32_t buf = tiles & 1;
                        if (!wait_bar(far_full(buf), (tiles >> 1) & 1)) {
                            alive = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        umma(d, smem_desc(a0 + 3 * 32, 16, 1024), smem_desc(far_base + buf * FAR_BYTES, FAR_CHUNK, 1024), 1u);
                        umma_commit(far_empty(buf));
                        ++tiles;
                    }
                    umma_commit(empty_bar(st));
                }
                if (alive) umma_commit(acc_full(acc));
            }
        }
    } else if (warp >= EPI_WARP0 && warp < EPI_WARP0 + EPI_WARPS) {
        const int quarter = warp % 4, half = (warp - EPI_WARP0) / 4;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + half * 128;
        const int32_t row = quarter * 32 + lane;
        uint32_t far_jobs = 0;
        for (uint32_t n = 0;; ++n) {
            const int slot = n % JOBS;
            if (!warp_wait_bar(job_full(slot), (n / JOBS) & 1)) break;
            const Job job = jobs[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(job_empty(slot));
            if (job.kind == JOB_STOP) break;
            const Seq& s = seq_of(job.seq);
            const int32_t group = job.group - s.group0;
            const uint32_t acc = n & 1, addr = lane_addr + acc * BN;
            auto release = [&] {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty(acc));
            };
            uint32_t r[32];
            if (job.kind == JOB_FAR) {
                // the ring's place is free once the tiles of the group before have read it
                if (job.group >= prm.ring) {
                    const uint32_t* p = far_read + job.group - prm.ring;
                    if (!__all_sync(0xffffffffu, wait_flag([&] { return seen(p, [](uint32_t v) { return (v & FAR_READ) != 0; }); }))) break;
                }
                if (!warp_wait_bar(acc_full(acc), (n >> 1) & 1)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // [tile][4 columns][value]: a warp stores whole lines, and what a tile reads lies together
                float4* out = reinterpret_cast<float4*>(prm.far + (int64_t)(job.group % prm.ring) * prm.far_stride + (int64_t)job.idx * BM * BN) +
                              (row / s.rank * (BN / 4) + half * 32) * s.rank + row % s.rank;
                const bool used = job.idx / s.parts * BM + row < s.rank * s.tiles;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    tmem_ld32(addr + c * 32, r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (c == 3) release();
                    if (used)
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            __stcg(out + (c * 8 + i) * s.rank, make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                                                           __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])));
                }
                __syncwarp();
                if (lane == 0) count_up(written + warp - EPI_WARP0, ++far_jobs);
                continue;
            }
            if (!warp_wait_bar(acc_full(acc), (n >> 1) & 1)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            {
                // the tiles that read the rows this one writes must have them
                const int32_t other = job.first + lane;
                bool ok = true;
                if (other <= job.last && other != job.idx) {
                    const uint32_t* p = rows_read + s.read0 + group * s.tiles + other;
                    ok = wait_flag([&] { return seen(p, [](uint32_t v) { return v != 0; }); });
                }
                if (!__all_sync(0xffffffffu, ok)) break;
                __syncwarp();  // what a lane has acquired holds for all of them (a vote alone orders no memory)
            }
            const int32_t m = job.idx * BM + row;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tmem_ld32(addr + c * 32, r);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (c == 3) release();
                uint32_t w[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_bf16(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                const Chunk ck = chunk_of(view.head_dim, group, half * 2 + (c >> 1));
                if (m < s.n_keep && ck.triple < s.triples) {
                    __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(tensor_base(view, ck.tensor)) +
                                         matrix_offset(view, s.triple0 + ck.triple) + (int64_t)(prm.sink + m) * view.stride_token +
                                         ck.channel + (c & 1) * 32;
                    store32(dst, w, prm.wide);
                    store32(dst + 16, w + 8, prm.wide);
                }
            }
        }
    } else if (warp >= FAR_WARP0 && warp < FAR_WARP0 + FAR_WARPS) {
        const int32_t tid = threadIdx.x - 32 * FAR_WARP0, i = tid % MAX_RANK;  // value i of columns 4 (tid / 8 + 16 j) and the three after
        uint32_t tiles = 0;
        for (uint32_t n = 0;; ++n) {
            const int slot = n % JOBS;
            if (!warp_wait_bar(job_full(slot), (n / JOBS) & 1)) break;
            const Job job = jobs[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(job_empty(slot));
            if (job.kind == JOB_STOP) break;
            if (job.kind != JOB_TILE) continue;
            const Seq& s = seq_of(job.seq);
            const uint32_t buf = tiles & 1;
            if (tiles >= 2 && !warp_wait_bar(far_empty(buf), ((tiles >> 1) - 1) & 1)) break;
            const uint32_t want = (uint32_t)(s.parts * s.far_tiles);
            bool ok = true;
            if (lane == 0 && !job.ready) ok = wait_flag([&] { return seen(far_written + job.group, [&](uint32_t v) { return v >= want; }); });
            if (!__all_sync(0xffffffffu, ok)) break;
            __syncwarp();  // lane 0 has acquired the sums, every lane reads them (a vote alone orders no memory)
            const int32_t row0 = job.idx * s.rank;
            const float4* in = reinterpret_cast<const float4*>(prm.far + (int64_t)(job.group % prm.ring) * prm.far_stride +
                                                               (int64_t)(row0 / BM) * s.parts * BM * BN) +
                               (row0 % BM) * (BN / 4) + tid / MAX_RANK * s.rank + i;
            float4 e[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) e[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < s.rank) {
#pragma unroll 4
                for (int32_t p = 0; p < s.parts; ++p, in += BM * BN / 4) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 x = __ldcg(in + j * 16 * s.rank);
                        e[j].x += x.x;
                        e[j].y += x.y;
                        e[j].z += x.z;
                        e[j].w += x.w;
                    }
                }
            }
            uint8_t* dst = far_smem + buf * FAR_BYTES + i * 128;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t col = 4 * (tid / MAX_RANK + 16 * j);
                const uint32_t at = col / 64 * FAR_CHUNK + ((col % 64 / 8 ^ (uint32_t)i) << 4) + col % 8 * 2;
                const uint2 hi = make_uint2(pack_bf16(e[j].x, e[j].y), pack_bf16(e[j].z, e[j].w));
                const uint2 lo = make_uint2(pack_bf16(e[j].x - __uint_as_float(hi.x << 16), e[j].y - __uint_as_float(hi.x & 0xffff0000u)),
                                            pack_bf16(e[j].z - __uint_as_float(hi.y << 16), e[j].w - __uint_as_float(hi.y & 0xffff0000u)));
                *reinterpret_cast<uint2*>(dst + at) = hi;
                *reinterpret_cast<uint2*>(dst + MAX_RANK * 128 + at) = lo;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(far_full(buf));
                count_up(read + warp - FAR_WARP0, tiles + 1);
            }
            ++tiles;
        }
    } else if (warp == WRITTEN_WARP || warp == READ_WARP) {
        // ---------------- far sums written, far sums read: told to the other CTAs for all warps of this one ----------------
        const bool writes = warp == WRITTEN_WARP;
        const uint32_t* counter = (writes ? written : read) + lane;
        uint32_t done = 0;
        for (uint32_t n = 0;; ++n) {
            const int slot = n % JOBS;
            if (!warp_wait_bar(job_full(slot), (n / JOBS) & 1)) break;
            const Job job = jobs[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(job_empty(slot));
            if (job.kind == JOB_STOP) break;
            if (job.kind != (writes ? JOB_FAR : JOB_TILE)) continue;
            ++done;
            bool ok = true;
            if (lane < (writes ? EPI_WARPS : FAR_WARPS)) ok = wait_flag([&] { return counted(counter) >= done; });
            if (!__all_sync(0xffffffffu, ok)) break;
            __syncwarp();
            if (lane == 0) {
                uint32_t* p = (writes ? far_written : far_read) + job.group;
                const uint32_t old = add_acq_rel(p, 1u);
                if (!writes && old + 1 == (uint32_t)seq_of(job.seq).tiles) store_release(p, FAR_READ);
            }
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*abort_flag) {
        // Some role gave up, whichever: copies that were issued may still be on their way to shared memory and products in the tensor
        // cores.  Both are waited for, with a limit, before either memory goes away.  (Every role is here, so none issues more.)
        if (threadIdx.x == 32) umma_commit(drained);
        if (threadIdx.x == 0 || threadIdx.x == 32) {
            const unsigned long long t0 = global_timer_ns();
            while (global_timer_ns() - t0 < LANDING_NS && !(threadIdx.x == 32 && mbar_try_wait(drained, 0))) __nanosleep(1000);
        }
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
}

// Tickets and flags of a call start at zero (a kernel of its own: what a call before left behind may still be in use until then).
__global__ void __launch_bounds__(256) nearfar_begin_kernel(uint4* flags, int32_t vectors)
{
    const int32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i < vectors) flags[i] = make_uint4(0, 0, 0, 0);
}

// ---- the plan ----

struct PlanJob {
    uint8_t* blocks;
    int32_t* table;
    double* nodes;  // per tile: rank nodes, rank poles
    int32_t n_in, n_keep, tiles, rank, slices, k_slices, near_columns, margin;
};

// Element (row i, column c) of a block as tcgen05 wants it in shared memory: K-major, 128-byte swizzle.
__device__ __forceinline__ void put(uint8_t* block, int32_t i, int32_t c, double x)
{
    *reinterpret_cast<__nv_bfloat16*>(block + i * 128 + ((((uint32_t)c >> 3) ^ (i & 7)) << 4) + (c & 7) * 2) = __double2bfloat16(x);
}

__global__ void __launch_bounds__(256) build_nearfar_kernel(const PlanJob job)
{
    const int64_t N = job.n_in, L = job.n_keep;
    const int32_t near_blocks = job.tiles * job.slices;
    const int32_t block = blockIdx.x;
    uint8_t* out = job.blocks + (size_t)block * A_BYTES;
    for (int32_t e = threadIdx.x; e < BM * BK; e += blockDim.x) {
        const int32_t i = e / BK, c = e % BK;
        double x = 0.0;
        if (block < near_blocks) {
            const int32_t tile = block / job.slices, col = block % job.slices * BK + c;
            const int64_t m = (int64_t)tile * BM + i;
            if (m < L && col < job.near_columns) {
                const int64_t n = job.table[tile * TABLE] + col;
                if (n < N) x = basis_entry(m, n, N, L, 0);
            } else if (m < L && (col - job.near_columns) % MAX_RANK < job.rank) {
                // weight of far value a in row m: (-1)^m sin(theta_m) U_a(cos theta_m) / sin(arccos(node a))
                const int32_t a = (col - job.near_columns) % MAX_RANK;
                const double* nodes = job.nodes + (size_t)tile * 2 * job.rank;
                const double* poles = nodes + job.rank;
                const double t = (double)(2 * m + 1) / (double)(2 * L), y = cospi(t);
                x = (m % 2 ? -1.0 : 1.0) * sinpi(t) / sqrt(fmax(1.0 - nodes[a] * nodes[a], 1e-300));
                for (int32_t k = 0; k < job.rank; ++k) {
                    if (k != a) x *= (y - nodes[k]) / (nodes[a] - nodes[k]);
                    x *= (nodes[a] - poles[k]) / (y - poles[k]);
                }
            }
        } else {
            const int32_t far = block - near_blocks, r = far / job.k_slices * BM + i, tile = r / job.rank;
            const int64_t n = (int64_t)(far % job.k_slices) * BK + c;
            if (tile < job.tiles && n < N) {
                const int32_t lo = job.table[tile * TABLE];
                if (n < lo || n >= lo + job.near_columns) {
                    const double a = job.nodes[(size_t)tile * 2 * job.rank + r % job.rank];
                    const int64_t phase = ((2 * n + 1) * L) % (4 * N);
                    x = sqrt(fmax(1.0 - a * a, 1e-300)) * cospi((double)phase / (double)(2 * N)) /
                        ((double)N * (cospi((double)(2 * n + 1) / (double)(2 * N)) - a));
                }
            }
        }
        put(out, i, c, x);
    }
}

// sn(u, k), 0 < k < 1, by descending Landen steps (Abramowitz and Stegun 16.4), and K(k) from the same means.
__device__ double elliptic_k(double k)
{
    double a = 1, b = sqrt((1 - k) * (1 + k));
    for (int i = 0; i < 15 && fabs(a - b) > 1e-15 * a; ++i) {
        const double t = 0.5 * (a + b);
        b = sqrt(a * b);
        a = t;
    }
    return 3.141592653589793 / (2 * a);
}
__device__ double elliptic_sn(double u, double k)
{
    double a[16], c[16];
    double b = sqrt((1 - k) * (1 + k));
    a[0] = 1;
    c[0] = k;
    int n = 0;
    while (n < 15 && fabs(c[n]) > 1e-16) {
        a[n + 1] = 0.5 * (a[n] + b);
        c[n + 1] = 0.5 * (a[n] - b);
        b = sqrt(a[n] * b);
        ++n;
    }
    double phi = ldexp(a[n] * u, n);
    for (int i = n; i > 0; --i) phi = 0.5 * (phi + asin(fmax(-1.0, fmin(1.0, c[i] * sin(phi) / a[i]))));
    return sin(phi);
}

// Nodes in the tile's interval [a, b] of cos(theta), poles in the far set outside (below, above): Zolotarev's, for
// [-1, 1] and |z| >= 1/k, moved by the Moebius map with the same cross ratio.
__device__ void tile_nodes(double a, double b, double below, double above, int32_t rank, double* nodes)
{
    if (b >= 1) above = -1;  // no far rows above: the far set is [-1, below]
    if (a <= -1) below = 1;  // none below: [above, 1]
    const double ratio = (a - below) * (above - b) / ((b - below) * (above - a));
    const double s = sqrt(ratio), k = (1 - s) / (1 + s);
    auto moved = [&](double z) {  // (x - a) (b - above) / ((x - above) (b - a)) = (z + 1) (1 - 1/k) / (2 (z - 1/k))
        const double c = (z + 1) * (1 - 1 / k) / (2 * (z - 1 / k));
        return (a * (b - above) - c * above * (b - a)) / ((b - above) - c * (b - a));
    };
    const double K = elliptic_k(k);
    for (int32_t i = 0; i < rank; ++i) {
        const double z = elliptic_sn((2.0 * i + 1 - rank) / rank * K, k);
        nodes[i] = moved(z);
        nodes[rank + i] = moved(1 / (k * z));
    }
}

// Per tile: first near column, the tiles that read the rows it writes, nodes and poles.
__global__ void __launch_bounds__(128) build_nearfar_tables_kernel(const PlanJob job)
{
    const int32_t i = blockIdx.x * 128 + threadIdx.x;
    if (i >= job.tiles) return;
    auto first_column = [&](int32_t j) { return max(0, (int32_t)((int64_t)j * BM * job.n_in / job.n_keep) - job.margin); };
    const int32_t m0 = i * BM, m1 = min(job.n_keep, m0 + BM), lo = first_column(i), hi = lo + job.near_columns;
    int32_t first = i, last = i;
    while (first > 0 && first_column(first - 1) + job.near_columns > m0) --first;
    while (first < i && first_column(first) >= m1) ++first;
    while (last + 1 < job.tiles && first_column(last + 1) < m1) ++last;
    int32_t* t = job.table + i * TABLE;
    t[0] = lo;
    t[1] = first;
    t[2] = last;
    t[3] = 0;
    auto x_of = [&](int64_t n) { return cospi((double)(2 * n + 1) / (double)(2 * (int64_t)job.n_in)); };
    auto y_of = [&](int64_t m) { return cospi((double)(2 * m + 1) / (double)(2 * (int64_t)job.n_keep)); };
    // Where the window reaches an end of the input there is no far set on that side, and the interval runs on to the end: also for
    // a tile before a short last one (with its own end kept, nodes for a far set that is not there: 3e-3 off at 8194 -> 4097, 2e-6 now).
    tile_nodes(hi < job.n_in ? y_of(m1 - 1) : -1.0, lo > 0 ? y_of(m0) : 1.0, hi < job.n_in ? x_of(hi) : -1.0,
               lo > 0 ? x_of(lo - 1) : 1.0, job.rank, job.nodes + (size_t)i * 2 * job.rank);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
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

// The non-sink rows of one cache tensor as a 5-D tensor (channel, token, kv_head, layer, batch); rows past n_in read as zero.
bool encode_rows(CUtensorMap* map, const CacheView& view, int tensor, int32_t batch_count, int32_t n_in, int32_t sink)
{
    char* p = static_cast<char*>(tensor ? view.base[1] : view.base[0]) +
              ((int64_t)view.batch0 * view.stride_batch + (int64_t)sink * view.stride_token) * 2;
    const cuuint64_t dims[5] = {(cuuint64_t)view.head_dim, (cuuint64_t)n_in, (cuuint64_t)view.kv_heads, (cuuint64_t)view.layers,
                                (cuuint64_t)batch_count};
    // an axis of extent 1 is never stepped; give it a harmless stride
    const cuuint64_t row = (cuuint64_t)view.stride_token * 2;
    const cuuint64_t strides[4] = {row, view.kv_heads > 1 ? (cuuint64_t)view.stride_head * 2 : row,
                                   view.layers > 1 ? (cuuint64_t)view.stride_layer * 2 : row,
                                   batch_count > 1 ? (cuuint64_t)view.stride_batch * 2 : row};
    const cuuint32_t box[5] = {64, BK, 1, 1, 1};
    const cuuint32_t elem[5] = {1, 1, 1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, p, dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int32_t groups_of(int32_t head_dim, int32_t triples)
{
    return head_dim == 64 ? (triples + 1) / 2 : head_dim == 256 ? 2 * triples : triples;
}

// How the tickets of a call are laid out, and what it needs of the scratch buffer.
struct Schedule {
    std::vector<Seq> seqs;
    std::vector<Run> runs;
    int32_t ahead = 0, ring = 0, groups = 0;
    int64_t tickets = 0, flags = 0;  // flags: in 32-bit words
    int64_t far_stride = 0;
    size_t far_offset = 0, bytes = 0;
};

// Groups of so many rows that the far jobs run ahead of the tiles (of calls with as many).
int64_t lead(int64_t rows) { return std::max<int64_t>(2, AHEAD_BYTES / (rows * BN * 2)); }

Schedule schedule(const CacheView& view, const std::vector<NearFarItem>& items)
{
    Schedule s;
    int64_t reads = 0, jobs = 0, groups = 0;
    for (const NearFarItem& item : items) {
        const NearFarShape sh = nearfar_shape(item.n_in, item.n_keep);
        Seq q = {};
        q.blocks = static_cast<const uint8_t*>(item.plan);
        q.table = reinterpret_cast<const int32_t*>(q.blocks + sh.near_bytes + sh.far_bytes);
        q.group0 = (int32_t)groups;
        q.triple0 = item.batch0 * view.layers * view.kv_heads;
        q.triples = item.batch_count * view.layers * view.kv_heads;
        q.n_keep = item.n_keep;
        q.tiles = sh.tiles;
        q.rank = sh.rank;
        q.slices = sh.slices;
        q.k_slices = sh.k_slices;
        q.part_slices = sh.part_slices;
        q.parts = sh.parts;
        q.far_tiles = sh.far_tiles;
        q.read0 = (int32_t)reads;
        const int64_t g = groups_of(view.head_dim, q.triples);
        groups += g;
        reads += g * sh.tiles;
        jobs += g * (sh.tiles + (int64_t)sh.parts * sh.far_tiles);
        s.far_stride = std::max<int64_t>(s.far_stride, (int64_t)sh.parts * sh.far_tiles * BM * BN);
        s.seqs.push_back(q);
    }
    s.groups = (int32_t)groups;
    s.tickets = jobs;
    // Far jobs run ahead of the tiles by what stays in L2 until those read it again (40 MB; with 1.5 jobs an SM, whatever their size, 7B
    // shape 1.10 against 0.93 ms, 8B shape 4.7 and 4.3 ms; 7B with 20 MB 1.57 ms, 30 1.05, 60 0.97, 90 1.00).
    int64_t rows = 0;
    for (const NearFarItem& item : items) rows += (int64_t)groups_of(view.head_dim, item.batch_count * view.layers * view.kv_heads) * item.n_in;
    // The ring's places are as large as the longest sequence needs, their number follows the mean: a long sequence among many short ones
    // would ask for many large places (131072 -> 65536 beside 31 of 600 -> 300: 33 of 180 MB), so there the lead gives way.
    s.ahead = (int32_t)std::min<int64_t>({groups, lead(rows / groups), std::max<int64_t>(2, RING_BYTES / (2 * s.far_stride * 4))});
    s.ring = (int32_t)std::min<int64_t>(groups, 2 * (int64_t)s.ahead);
    s.flags = (16 + 2 * groups + reads + 3) / 4 * 4;
    s.far_offset = ((size_t)s.flags * 4 + 255) / 256 * 256;
    s.bytes = s.far_offset + (size_t)s.ring * s.far_stride * 4;
    // runs: block i (from -ahead) holds the far jobs of group i + ahead and the tiles of group i
    size_t fs = 0, ts = 0;
    int64_t ticket = 0;
    auto end_of = [&](size_t q) { return q + 1 < s.seqs.size() ? (int64_t)s.seqs[q + 1].group0 : groups; };
    for (int64_t i = -s.ahead; i < groups;) {
        const int64_t fg = i + s.ahead;
        while (fs < s.seqs.size() && fg >= end_of(fs)) ++fs;
        while (i >= 0 && i >= end_of(ts)) ++ts;
        Run r = {};
        r.ticket0 = (int32_t)ticket;
        r.block0 = (int32_t)i;
        int64_t next = groups;
        if (fg < groups) {
            r.far_jobs = s.seqs[fs].parts * s.seqs[fs].far_tiles;
            r.far_seq = (int32_t)fs;
            next = std::min(next, end_of(fs) - s.ahead);
        }
        if (i >= 0) {
            r.tiles = s.seqs[ts].tiles;
            r.tile_seq = (int32_t)ts;
            next = std::min(next, end_of(ts));
        } else {
            next = std::min<int64_t>(next, 0);
        }
        s.runs.push_back(r);
        ticket += (next - i) * (r.far_jobs + r.tiles);
        i = next;
    }
    return s;
}

cudaError_t grow(void** buffer, size_t* have, size_t bytes)
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

cudaError_t prepare(GemmState* state, const Schedule& s)
{
    static PerDeviceOnce once;
    state->last_error = nullptr;
    if (!encode_fn()) {
        state->last_error = "cuTensorMapEncodeTiled is not available from this driver";
        return cudaErrorNotSupported;
    }
    cudaError_t e = once.run([] {
        cudaError_t r = cudaFuncSetAttribute(freqkv_nearfar_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        if (r == cudaSuccess) r = cudaFuncSetAttribute(freqkv_nearfar_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        return r;
    });
    if (e != cudaSuccess) {
        state->last_error = "cudaFuncSetAttribute(max dynamic shared memory)";
        return e;
    }
    if (s.tickets > 0x7fffffff || s.flags > 0x7fffffff) return cudaErrorInvalidValue;
    e = grow(&state->scratch, &state->scratch_bytes, s.bytes);
    if (e != cudaSuccess) state->last_error = "cudaMalloc(far sums)";
    return e;
}

}  // namespace

NearFarShape nearfar_shape(int32_t n_in, int32_t n_keep)
{
    NearFarShape s = {};
    s.tiles = (n_keep + BM - 1) / BM;
    // 128 far rows for the whole matrix where that is enough: the fewer nodes a tile has, the wider its margin
    s.rank = s.tiles <= 16 ? 8 : s.tiles <= 21 ? 6 : 4;
    const double under = (double)BM * n_in / n_keep;
    const int32_t rows = (int32_t)std::ceil(under) + 1;
    const int32_t least = (int32_t)std::ceil(under * (s.rank == 8 ? 0.05 : s.rank == 6 ? 0.1 : 0.2));
    s.slices = (rows + 2 * least + FAR_COLS + BK - 1) / BK;
    s.margin = (s.slices * BK - FAR_COLS - rows) / 2;
    s.k_slices = (n_in + BK - 1) / BK;
    s.parts = (s.k_slices + 23) / 24;  // 16 or 32 slices a job: 7B shape 1.03 and 1.01 times as long, ragged batches 1.08 and 0.98
    s.part_slices = (s.k_slices + s.parts - 1) / s.parts;
    s.parts = (s.k_slices + s.part_slices - 1) / s.part_slices;
    s.far_tiles = (s.tiles * s.rank + BM - 1) / BM;
    s.near_bytes = (size_t)s.tiles * s.slices * A_BYTES;
    s.far_bytes = (size_t)s.far_tiles * s.k_slices * A_BYTES;
    s.bytes = s.near_bytes + s.far_bytes + (size_t)s.tiles * (TABLE * sizeof(int32_t) + 2 * s.rank * sizeof(double));
    return s;
}

cudaError_t launch_build_nearfar(void* out, int32_t n_in, int32_t n_keep, cudaStream_t stream)
{
    const NearFarShape s = nearfar_shape(n_in, n_keep);
    PlanJob job = {};
    job.blocks = static_cast<uint8_t*>(out);
    job.table = reinterpret_cast<int32_t*>(job.blocks + s.near_bytes + s.far_bytes);
    job.nodes = reinterpret_cast<double*>(job.table + (size_t)s.tiles * TABLE);
    job.n_in = n_in;
    job.n_keep = n_keep;
    job.tiles = s.tiles;
    job.rank = s.rank;
    job.slices = s.slices;
    job.k_slices = s.k_slices;
    job.near_columns = s.slices * BK - FAR_COLS;
    job.margin = s.margin;
    build_nearfar_tables_kernel<<<(unsigned)((s.tiles + 127) / 128), 128, 0, stream>>>(job);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    build_nearfar_kernel<<<(unsigned)(s.tiles * s.slices + s.far_tiles * s.k_slices), 256, 0, stream>>>(job);
    return cudaGetLastError();
}

cudaError_t nearfar_reserve(GemmState* state, int32_t n_in, int32_t n_keep)
{
    const NearFarShape sh = nearfar_shape(n_in, n_keep);
    const size_t flags = size_t(1) << 20;
    return grow(&state->scratch, &state->scratch_bytes, flags + (size_t)(2 * lead(n_in)) * sh.parts * sh.far_tiles * BM * BN * sizeof(float));
}

cudaError_t nearfar_prepare(GemmState* state, const CacheView& view, const std::vector<NearFarItem>& items)
{
    return prepare(state, schedule(view, items));
}

cudaError_t launch_nearfar(GemmState* state, const CacheView& view, const std::vector<NearFarItem>& items, int32_t sink,
                           int32_t* status_dev, int sm_count, const LaunchHooks& hooks, cudaStream_t stream)
{
    state->kernels_last_call = 0;
    const Schedule s = schedule(view, items);
    cudaError_t e = prepare(state, s);
    if (e != cudaSuccess) return e;
    const bool ragged = items.size() > 1;
    std::vector<CUtensorMap> maps(2 * items.size());
    const int32_t batches = view.mats_per_tensor / (view.layers * view.kv_heads);
    for (size_t i = 0; i < items.size(); ++i)
        for (int t = 0; t < 2; ++t)
            if (!encode_rows(&maps[2 * i + t], view, t, batches, items[i].n_in, sink)) {
                state->last_error = "tensor map encoding rejected this layout";
                return cudaErrorInvalidValue;
            }
    Params prm = {};
    prm.n_runs = (int32_t)s.runs.size();
    prm.tickets = (int32_t)s.tickets;
    prm.ahead = s.ahead;
    prm.ring = s.ring;
    prm.sink = sink;
    prm.wide = (((uintptr_t)view.base[0] | (uintptr_t)view.base[1]) & 31) == 0 &&
               ((view.stride_token | view.stride_head | view.stride_layer | view.stride_batch) & 15) == 0;
    prm.flags = static_cast<uint32_t*>(state->scratch);
    prm.far = reinterpret_cast<float*>(static_cast<char*>(state->scratch) + s.far_offset);
    prm.far_stride = s.far_stride;
    prm.groups = s.groups;
    prm.status = status_dev;
    prm.wait_limit_ns = state->wait_limit_ns;
    if (ragged) {
        const size_t maps_bytes = maps.size() * sizeof(CUtensorMap), seqs_bytes = s.seqs.size() * sizeof(Seq),
                     runs_bytes = s.runs.size() * sizeof(Run);
        std::vector<char> host(maps_bytes + seqs_bytes + runs_bytes);
        memcpy(host.data(), maps.data(), maps_bytes);
        memcpy(host.data() + maps_bytes, s.seqs.data(), seqs_bytes);
        memcpy(host.data() + maps_bytes + seqs_bytes, s.runs.data(), runs_bytes);
        e = grow(&state->ragged_meta, &state->ragged_meta_bytes, host.size());
        if (e != cudaSuccess) {
            state->last_error = "cudaMalloc(tables of a ragged batch)";
            return e;
        }
        char* meta = static_cast<char*>(state->ragged_meta);
        e = cudaMemcpyAsync(meta, host.data(), host.size(), cudaMemcpyHostToDevice, stream);  // pageable: read when this returns
        if (e != cudaSuccess) return e;
        prm.maps = reinterpret_cast<const CUtensorMap*>(meta);
        prm.n_maps = (int32_t)maps.size();
        prm.seqs = reinterpret_cast<const Seq*>(meta + maps_bytes);
        prm.runs = reinterpret_cast<const Run*>(meta + maps_bytes + seqs_bytes);
    } else {
        prm.seq = s.seqs[0];
        for (size_t i = 0; i < s.runs.size() && i < 3; ++i) prm.run[i] = s.runs[i];
    }
    const int32_t vectors = (int32_t)(s.flags / 4);
    nearfar_begin_kernel<<<(unsigned)((vectors + 255) / 256), 256, 0, stream>>>(reinterpret_cast<uint4*>(prm.flags), vectors);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        state->last_error = "nearfar_begin_kernel launch";
        return e;
    }
    if (hooks.before) hooks.before(hooks.user, stream);
    const unsigned grid = (unsigned)std::min<int64_t>(sm_count, s.tickets);
    if (ragged)
        freqkv_nearfar_kernel<true><<<grid, THREADS, SMEM_BYTES, stream>>>(maps[0], maps[1], view, prm);
    else
        freqkv_nearfar_kernel<false><<<grid, THREADS, SMEM_BYTES, stream>>>(maps[0], maps[1], view, prm);
    e = cudaGetLastError();
    if (hooks.after) hooks.after(hooks.user, stream);
    if (e != cudaSuccess) {
        state->last_error = "freqkv_nearfar_kernel launch";
        return e;
    }
    state->kernels_last_call = 2;
    return cudaSuccess;
}

}  // namespace freqkv
