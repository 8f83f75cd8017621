// Tensor-core products of the S-STE linear layer (Sec. 5.1) for sm_100a:
//   forward      Z^T = S(W) X^T              sparse A (values + metadata), K-major B
//   grad weight  grad_W = MVUE(grad_Z^T) X   sparse A, MN-major B
//   grad input   grad_X = grad_Z S(W)        dense A, MN-major B
//
// One persistent, warp-specialised kernel template run by CTA PAIRS (cluster of two,
// tcgen05 cta_group::2).  A pair owns an output tile of 256 rows and 128 to 256 columns: each CTA holds its own
// 128 rows of A and HALF of the B tile, so the B operand is streamed from shared memory
// at half the rate per SM -- with one CTA per tile the sparse instruction is bound by that
// stream and runs no faster than the dense one -- and L2 -> SM traffic per flop drops.
//   warp 0    TMA producer (both CTAs; all transaction bytes land on the leader's barrier)
//   warp 1    leader CTA: tcgen05.cp of the stage's metadata, tcgen05.mma[.sp] issue; both CTAs: tensor-memory allocation
//   warps 2-9 epilogue, each on its own 32 accumulator rows and half of the columns: TMEM -> registers -> bf16 ->
//             shared memory -> TMA store
//   compressed B only (grad_X from the forward's operand): warps 2-5 epilogue on all columns, warps 6-9 expand values +
//             metadata into the dense shared-memory stage
// Output tiles are handed out band by band (tile_coords) so that operands are read from HBM about
// once; tile width, split-K plan and band height come from cost models on the host (make_plan).
// Every wait is bounded: on expiry the CTA records SSTE_ERR_TIMEOUT and leaves.
#include <cuda.h>

#include <array>
#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace {

constexpr int BM = 128;            // rows of A per CTA (a pair covers 256)
constexpr int TMEM_COLS = 512;
// Shared memory starts with a control block: barriers of the kernel's first product at 0 and of its second at 512, the
// expander's selector table at 256, the tensor-memory address at 1008 and the abort flag at 1016.
constexpr int CTRL_BYTES = 1024, CTRL_SECOND = 512, CTRL_LUT = 256, CTRL_TMEM = 1008, CTRL_ABORT = 1016;
constexpr int MAX_SPLITS = 16;     // split-K factor limit where the units exchange their partials
constexpr int MAX_PARTS = 2;       // parts that a warp's share of a split tile is exchanged in
constexpr int PANEL_BYTES = 2048;  // epilogue panel: 32 rows x 32 columns of bf16
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;   // two seconds of wall time (%globaltimer)

enum class BMajor { K, MN };

// ------------------------------------------------------------------ PTX wrappers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Arrive on a barrier that may live in the peer CTA (shared::cluster address).  CLUSTER: what this thread wrote to shared memory is
// for the peer too.  Without it the arrival only says that something has been read (tensor memory, behind its own fence), and
// need not wait until the thread's writes are visible in the cluster (cluster scope everywhere: forward of 3072 x 768, 8192 tokens,
// bf16 26.8 us, so 24.1).
template <bool CLUSTER>
__device__ __forceinline__ void mbar_arrive_at(uint32_t cluster_addr)
{
    if (CLUSTER) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
    else asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// One try: the thread is suspended by the hardware until the phase completes or a time limit of
// about a millisecond passes, so a waiting thread does not poll shared memory (the sparse MMA streams
// its operands at 3/4 of the shared-memory bandwidth and is slowed down by pollers).
// CLUSTER: the thread goes on to what the peer CTA's threads wrote (the others go on to what copies and MMAs, or nobody, wrote).
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if (CLUSTER)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(1000000u)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(1000000u)
            : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait of ONE thread.  Returns false (after recording a timeout) instead of spinning forever.
// The limit is wall time (nanoseconds of %globaltimer), so it does not depend on the SM clock.
struct WaitCtx {
    unsigned int *status;              // the context's device status word
    volatile int *abort_flag;          // this CTA's "a wait has expired" flag (shared memory)
    unsigned long long limit_ns;       // WAIT_LIMIT_NS, or the short limit of the stall-injection test hook
};
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx &wc)
{
    if (mbar_try_wait<CLUSTER>(bar, parity)) return true;
    const unsigned long long start = global_ns();
    while (true) {
        if (mbar_try_wait<CLUSTER>(bar, parity)) return true;
        if (*wc.abort_flag) return false;
        if (global_ns() - start > wc.limit_ns) {
            atomicMax(wc.status, static_cast<unsigned int>(SSTE_ERR_TIMEOUT));      // also over a recorded degenerate beta
            *wc.abort_flag = 1;
            return false;
        }
    }
}
// Bounded wait of a whole warp: lane 0 waits, the others park at the warp barrier.
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const WaitCtx &wc)
{
    uint32_t ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait<CLUSTER>(bar, parity, wc) ? 1u : 0u;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    return ok != 0;
}

// 2-D tiled TMA load into this CTA's shared memory; the transaction bytes are signalled on
// `bar`, which may be the pair leader's barrier (cta_group::2 form).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Arrive on the barrier at this shared-memory offset in BOTH CTAs of the pair once every
// tcgen05 operation issued so far by this thread has completed.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"(static_cast<uint16_t>(3))
        : "memory");
}
template <bool F8>
__device__ __forceinline__ void tc_mma_dense(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    if (F8)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
template <bool F8>
__device__ __forceinline__ void tc_mma_sparse(uint32_t d, uint64_t a, uint64_t b, uint32_t e, uint32_t idesc,
                                              uint32_t accumulate)
{
    if (F8)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "tcgen05.mma.sp.cta_group::2.kind::f8f6f4 [%0], %1, %2, [%3], %4, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(e), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "tcgen05.mma.sp.cta_group::2.kind::f16 [%0], %1, %2, [%3], %4, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(e), "r"(idesc), "r"(accumulate) : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns -> 32 registers per thread
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t r[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
// 32 lanes x 16 consecutive 32-bit columns -> 16 registers per thread
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// 16 lanes x 32 consecutive 32-bit columns in the fragment layout of the 8 x 8 matrix stores: for the 8-column block b
// thread t holds r[4b], r[4b + 1] = row t / 4, columns 2 (t % 4), + 1 and r[4b + 2], r[4b + 3] = the same of row t / 4 + 8
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// 32 accumulator columns of a warp's 32 rows -> 32 registers.  TRANSPOSED = false: r[c] = column c of row `lane`;
// true: r[16 h + i] = fragment i (above) of rows 16 h .. 16 h + 15.
template <bool TRANSPOSED>
__device__ __forceinline__ void tmem_ld_32cols(uint32_t taddr, uint32_t *r)
{
    if (TRANSPOSED) {
        tmem_ld_16x256_x4(taddr, r);
        tmem_ld_16x256_x4(taddr + (16u << 16), r + 16);
    } else {
        tmem_ld_32x32(taddr, r);
    }
}
// half h (registers 16 h .. 16 h + 15) of what tmem_ld_32cols loads
template <bool TRANSPOSED>
__device__ __forceinline__ void tmem_ld_half(uint32_t taddr, int h, uint32_t *r)
{
    if (TRANSPOSED) tmem_ld_16x256_x4(taddr + (static_cast<uint32_t>(16 * h) << 16), r);
    else tmem_ld_32x16(taddr + 16 * h, r);
}
// four 8 x 8 matrices of 16-bit elements, stored transposed: thread t gives the address of row t % 8 of matrix t / 8
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void pair_barrier(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
// Barrier of two warps that also combines a flag: true if all 64 threads passed true.
__device__ __forceinline__ bool pair_barrier_and(int id, bool ok)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, 64, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(ok ? 1u : 0u), "r"(id)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ uint32_t ld_acquire_gpu(const unsigned int *a)
{
    uint32_t r;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(r) : "l"(a) : "memory");
    return r;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// One metadata atom (128 lanes x 16 bytes, contiguous in shared memory) -> four tensor-memory columns, in both CTAs of
// the pair from their own shared memory at the same offset.  Issued by the thread that issues the MMAs: it executes in
// order with the MMAs that follow.
__device__ __forceinline__ void tc_cp_meta_atom(uint32_t taddr, uint64_t sdesc)
{
    asm volatile("tcgen05.cp.cta_group::2.128x128b [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------------ descriptors

// Shared-memory matrix descriptor: start address, leading / stride byte offsets (all >> 4),
// descriptor version 1, swizzle mode in the top three bits (0 none, 2 = 128 B, 4 = 64 B).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t swizzle)
{
    return static_cast<uint64_t>((addr & 0x3ffffu) >> 4) | (static_cast<uint64_t>(lbo_bytes >> 4) << 16) |
           (static_cast<uint64_t>(sbo_bytes >> 4) << 32) | (1ull << 46) | (static_cast<uint64_t>(swizzle) << 61);
}

// Instruction descriptor: sparse selector [0,2), sparse flag [2], D = fp32 [4,6), A format [7,10),
// B format [10,13), A major [15], B major [16] (1 = MN-major), N>>3 [17,23), M>>4 [24,29).
// M is 256: the pair's two 128-row halves.
__host__ __device__ constexpr uint32_t instr_desc(bool sparse, uint32_t afmt, uint32_t bfmt, bool b_mn_major, int bn)
{
    return (sparse ? 4u : 0u) | (1u << 4) | (afmt << 7) | (bfmt << 10) | ((b_mn_major ? 1u : 0u) << 16) |
           (static_cast<uint32_t>(bn >> 3) << 17) | (static_cast<uint32_t>((2 * BM) >> 4) << 24);
}

// ------------------------------------------------------------------ kernel

// Order in which output tiles are handed to the CTA pairs (pair p takes tiles p, p + pairs, ...).  Tiles are
// numbered band by band: a band is `group_m` consecutive rows of tiles, and inside a band the row index runs
// fastest.  The 74 tiles in flight at any time therefore cover group_m tile rows x 74 / group_m tile columns,
// and the A rows of a band stay in L2 while the band sweeps over all of B.  group_m = m_tiles is plain
// column-major order (all of A resident, B streamed once).
// Without integer divisions (450 clk of dependent instructions for each tile of each role): a quotient by an approximate reciprocal,
// put right by its remainder, whatever the numbers (FP8 forward of 3072 x 768, 8192 tokens: 20.0 -> 18.8 us, bf16 24.1 -> 24.0).
__host__ __device__ __forceinline__ int divide(int a, int b, int &rem)
{
#ifdef __CUDA_ARCH__
    int q = static_cast<int>(__fdividef(static_cast<float>(a), static_cast<float>(b)));
#else
    int q = static_cast<int>(static_cast<float>(a) / static_cast<float>(b));
#endif
    rem = a - q * b;
    while (rem < 0) { --q; rem += b; }
    while (rem >= b) { ++q; rem -= b; }
    return q;
}
__host__ __device__ __forceinline__ void tile_coords(int tile, int m_tiles, int n_tiles, int group_m, int &mt, int &nt)
{
    int within = tile, first = 0, rows = group_m;
    if (group_m < m_tiles) {
        first = divide(tile, group_m * n_tiles, within) * group_m;
        rows = (m_tiles - first < group_m) ? m_tiles - first : group_m;
    }
    nt = divide(within, rows, mt);
    mt += first;
}

struct GemmParams {
    int M, N, K;            // logical problem: D[M, N] = A[M, K] * B
    void *D;                // output (used by the direct-store fp32 epilogue)
    // FP8 operands (Sec. 5.2): device scalars max|a|, max|b| of the tensors the operands were quantised from and the
    // largest finite value of each operand's format; the epilogue multiplies by 1/scale_a * 1/scale_b.  Null for bf16.
    const float *a_amax, *b_amax;
    float a_fp8_max, b_fp8_max;
    unsigned int *out_amax; // nullable: receives max|D| (bit pattern of a non-negative fp32) by atomic maximum
    unsigned int *status;
    uint32_t afmt, bfmt;    // operand format codes of the instruction descriptor
    const uint8_t *b_vals;  // compressed-B kernels: the 2:4 values of B [K, N/2]; its metadata image is `meta`
    unsigned long long wait_limit_ns;   // limit of every device-side wait
    int skip_last_stage;    // stall-injection test hook: the producer leaves the last K stage of the launch unloaded
    int group_m;            // tile rows per band of the tile order (see tile_coords)
    int splits;             // split-K factor of the tiles from `split_from` on (1 = none)
    int split_from;         // first split tile: tiles below it are computed whole
    float *partials;        // split-K: fp32 partial tiles [split tile][cta][split][row quarter][BN / 4][32 lanes][4]
    unsigned int *tickets;  // split-K, null where splitk_sum_kernel follows: claims (low half) and finished partials (high half) per [split tile][cta][epilogue
                            // warp][part]; zero between launches
    unsigned int *zero_after; // nullable: a word to be zeroed once the kernels in front are done
};


// Shared-memory / tensor-memory plan of one CTA for a tile of 256 x BN.  A stage holds 128 bytes of K per
// A row and, for the sparse kernels, two B sub-tiles of 128 bytes of K each (the compressed A row covers
// twice the K of one B row) and the metadata atoms of that K; the dense kernel pairs it with one B sub-tile.
// Tensor memory: the accumulators, then the stages' metadata (four columns per atom, one region per stage, so a region
// is free again exactly when its stage is).  There are two accumulators, so the epilogue of a tile overlaps the next tile's main loop.
// Two of a sparse tile of BN = 256 do not fit beside the metadata: they share 32 columns, the last panel of the first and the first
// of the second, which their warps read first; the next main loop waits for that panel only.  (With one accumulator it waited
// for all tensor-memory reads, some 3100 clk of each tile by time stamps: forward 3840 x 1280, 16384 tokens, bf16 77.1 -> 75.5 us;
// 2304 x 768, 8192 tokens 19.2 -> 18.6.)
template <bool SPARSE, int ELT, int BN, bool BCOMP = false>
struct Cfg {
    static constexpr int A_STAGE = 16384;                        // 128 rows x 128 bytes
    static constexpr int B_SUB = (BN / 2) * 128;                 // this CTA's half of one B sub-tile
    static constexpr int B_STAGE = SPARSE ? 2 * B_SUB : B_SUB;
    static constexpr int ATOMS = SPARSE ? 256 / ELT / 128 : 0;   // metadata atoms (128 logical K, 2 KB) per stage
    static constexpr int STAGE = A_STAGE + B_STAGE + 2048 * ATOMS;
    static constexpr int EPI_WARPS = BCOMP ? 4 : 8;              // compressed B: the other four expand
    static constexpr int ROOM = 232448 - 1024 - CTRL_BYTES;      // 227 KB of shared memory per CTA, alignment slack, control block
    static constexpr int FIT = (ROOM - EPI_WARPS * PANEL_BYTES) / STAGE;
    static constexpr int STAGES = FIT > 8 ? 8 : FIT;
    // staging: panels per epilogue warp, two where they fit
    static constexpr int PANELS = (ROOM - STAGES * STAGE >= 2 * EPI_WARPS * PANEL_BYTES) ? 2 : 1;
    static constexpr int STAGING_BYTES = EPI_WARPS * PANELS * PANEL_BYTES;
    static constexpr bool SHARED_PANEL = SPARSE && BN == 256;
    static constexpr int ACC_STEP = SHARED_PANEL ? BN - 32 : BN; // columns from one accumulator to the other
    static constexpr int META_COL0 = ACC_STEP + BN;              // metadata regions follow the accumulators
    static constexpr int META_COLS = 4 * ATOMS;                  // tensor-memory columns of one stage's metadata
    static constexpr int THREADS = 320;
    static constexpr int SMEM_BYTES = 1024 /* alignment slack */ + CTRL_BYTES + STAGES * STAGE + STAGING_BYTES;
    static_assert(META_COL0 + STAGES * META_COLS <= TMEM_COLS, "tensor memory budget");
    static_assert(STAGES >= 3, "pipeline depth");
    static_assert(STAGE % 1024 == 0 && BN % 32 == 0, "swizzle alignment, epilogue panels");
};

// The units a pair works on, in order, until one is out of range: `early` rounds over `early_pairs` pairs only (those that
// have nothing to do before), then rounds over all `pairs` from unit `base` on.
struct UnitSeq {
    int early, early_pairs, early_rank, base, pairs, rank;
    __device__ __forceinline__ int first() const { return early > 0 ? early_rank : base + rank; }
    // the unit after `unit`; j: its number in the pair's order
    __device__ __forceinline__ int next(int unit, int j) const
    {
        return j < early ? unit + early_pairs : (early > 0 && j == early) ? base + rank : unit + pairs;
    }
};

template <typename C, bool BCOMP>
__device__ __forceinline__ void init_barriers(uint32_t bars)
{
    constexpr int NS = C::STAGES;
    static_assert(8 * (2 * NS + 5) <= CTRL_LUT, "barrier block");
    // full: the producer's arrival with the TMA byte count (+ the eight expander warps of the pair)
    for (int s = 0; s < NS; ++s) { mbar_init(bars + 8u * s, BCOMP ? 9 : 1); mbar_init(bars + 8u * (NS + s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bars + 8u * (2 * NS + b), 1); mbar_init(bars + 8u * (2 * NS + 2 + b), 2 * C::EPI_WARPS); }
    mbar_init(bars + 8u * (2 * NS + 4), C::EPI_WARPS);      // half of the warps of both CTAs
}

// One product on a CTA pair: all warp roles, from the first unit of `seq` to the last.
// ELT: operand element size in bytes (2 = bf16 via kind::f16, 1 = fp8 via kind::f8f6f4).
// OUT_T: store D transposed (out[n, m]); OUT_F32: fp32 output (direct stores) instead of bf16 (TMA stores).
// BCOMP: the (dense-product) B operand is given in compressed 2:4 form and expanded in shared memory.
// FINAL: nothing follows in the kernel (else another product reuses the shared memory).
template <bool SPARSE, BMajor BMAJ, int ELT, int BN, bool OUT_T, bool OUT_F32, bool BCOMP, bool FINAL>
__device__ __forceinline__ void
product(const CUtensorMap &map_a, const CUtensorMap &map_b, const CUtensorMap &map_d, const CUtensorMap &map_m,
        const uint8_t *__restrict__ meta, const GemmParams &p, const UnitSeq &seq, uint8_t *ctrl_generic, uint32_t bars,
        uint32_t smem_base, uint32_t tmem_base, const WaitCtx &wc)
{
    using C = Cfg<SPARSE, ELT, BN, BCOMP>;
    constexpr int NS = C::STAGES;
    constexpr int NB = 2;
    constexpr bool SHARED_PANEL = C::SHARED_PANEL;
    constexpr bool F8 = (ELT == 1);
    constexpr int BK = (SPARSE ? 256 : 128) / ELT;    // logical K per stage
    constexpr int B_SUBS = SPARSE ? 2 : 1;
    constexpr int SUB_K = 128 / ELT;                  // logical K of one B sub-tile
    constexpr int B_CHUNK_N = 128 / ELT;              // MN-major: N elements per 128-byte row
    constexpr int B_CHUNKS_HALF = (BN / 2) / B_CHUNK_N;
    constexpr uint32_t STAGE_TX = 2u * (BCOMP ? C::A_STAGE : C::STAGE);   // both CTAs' bytes that arrive by TMA
    static_assert(BMAJ == BMajor::K || (BN / 2) % B_CHUNK_N == 0, "MN-major B needs whole 128-byte chunks per CTA");
    static_assert(!BCOMP || (!SPARSE && BMAJ == BMajor::MN), "compressed B: dense A, MN-major B");

    const uint32_t staging = smem_base + NS * C::STAGE;
    auto full_bar = [&](int s) { return bars + 8u * s; };              // used in the leader only
    auto empty_bar = [&](int s) { return bars + 8u * (NS + s); };      // one per CTA
    auto acc_full_bar = [&](int b) { return bars + 8u * (2 * NS + b); };           // one per CTA
    auto acc_empty_bar = [&](int b) { return bars + 8u * (2 * NS + 2 + b); };      // leader only, one arrival per epilogue warp of the pair
    const uint32_t shared_read_bar = bars + 8u * (2 * NS + 4);                     // leader only: the panel that two accumulators share has been read

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader = (rank == 0);
    const int m_tiles = (p.M + 2 * BM - 1) / (2 * BM);
    const int n_tiles = (p.N + BN - 1) / BN;
    const int num_tiles = m_tiles * n_tiles;
    const int k_blocks_total = (p.K + BK - 1) / BK;   // a ragged last stage reads zero-filled K
    // Work units: tiles [0, split_from) are whole; every later tile is cut into `splits` K ranges that differ by
    // at most one stage.  Whole tiles fill complete waves, the split ones spread the last, partial wave over all pairs.
    const int num_units = p.split_from + (num_tiles - p.split_from) * p.splits;
    struct Unit { int tile, split, kb0, kb1; };
    auto decode = [&](int unit) {
        Unit u;
        if (unit < p.split_from) { u.tile = unit; u.split = 0; u.kb0 = 0; u.kb1 = k_blocks_total; }
        else {
            const int v = unit - p.split_from;
            u.tile = p.split_from + v / p.splits;
            u.split = v % p.splits;
            u.kb0 = u.split * k_blocks_total / p.splits;
            u.kb1 = (u.split + 1) * k_blocks_total / p.splits;
        }
        return u;
    };

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        if (lane == 0) {
            const int k_atoms = p.K / 128;
            uint32_t s = 0, ph = 0;          // stage of the ring and the parity of its round
            bool ok = true;
            for (int j = 0, unit = seq.first(); unit < num_units && ok; ++j, unit = seq.next(unit, j)) {
                const Unit u = decode(unit);
                int mt, nt;
                tile_coords(u.tile, m_tiles, n_tiles, p.group_m, mt, nt);
                const int m0 = mt * 2 * BM + static_cast<int>(rank) * BM;      // this CTA's rows of A
                const int n0 = nt * BN + static_cast<int>(rank) * (BN / 2);    // this CTA's half of B
                // rows beyond M (zero-filled values) take the codes of the last row block: zero is not one of the six codes
                const int meta_row = min(m0 / BM, p.M / BM - 1) * k_atoms * 4;
                if (j == 0) sste_pdl_wait();
                for (int kb = u.kb0; kb < u.kb1; ++kb) {
                    // test hook: the stage is never loaded nor announced, so the MMA warp's wait for it runs out
                    if (p.skip_last_stage && seq.next(unit, j + 1) >= num_units && kb == u.kb1 - 1) break;
                    if (!mbar_wait<BCOMP>(empty_bar(s), ph ^ 1u, wc)) { ok = false; break; }
                    const uint32_t lead_full = map_to_cta(full_bar(s), 0);
                    if (leader) mbar_arrive_expect_tx(full_bar(s), STAGE_TX);
                    const uint32_t a_dst = smem_base + s * C::STAGE;
                    const uint32_t b_dst = a_dst + C::A_STAGE;
                    // A: 128 bytes per row = BK/2 compressed (sparse) or BK dense elements
                    tma_load_2d(a_dst, &map_a, lead_full, kb * (SPARSE ? BK / 2 : BK), m0);
                    // metadata: the atoms of this K, 2 KB each, as rows of 512 bytes.  (With an odd number of atoms the last
                    // 8-bit stage also fetches what follows; no MMA reads it.)
                    if (SPARSE) tma_load_2d(b_dst + C::B_STAGE, &map_m, lead_full, 0, meta_row + kb * C::ATOMS * 4);
                    if (BCOMP) {
                        // B is written into the stage by the expander warps
                    } else if (BMAJ == BMajor::K) {
#pragma unroll
                        for (int u = 0; u < B_SUBS; ++u)
                            tma_load_2d(b_dst + u * C::B_SUB, &map_b, lead_full, kb * BK + u * SUB_K, n0);
                    } else {
                        // MN-major: one box per 128-byte N chunk spans the whole stage's K rows
#pragma unroll
                        for (int c = 0; c < B_CHUNKS_HALF; ++c)
                            tma_load_2d(b_dst + c * (BK * 128), &map_b, lead_full, n0 + c * B_CHUNK_N, kb * BK);
                    }
                    if (++s == NS) { s = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader CTA only)
        if (leader && lane == 0) {
            const uint32_t idesc = instr_desc(SPARSE, p.afmt, p.bfmt, BMAJ == BMajor::MN, BN);
            const int half_kb = p.K % BK != 0 ? k_blocks_total - 1 : -1;
            uint32_t s = 0, ph = 0, local_tile = 0;
            bool ok = true;
            sste_pdl_wait();                 // (the bounded waits below do not count the previous kernel's time)
            for (int unit = seq.first(); unit < num_units && ok; ++local_tile, unit = seq.next(unit, local_tile)) {
                const Unit u = decode(unit);
                const uint32_t buf = local_tile % NB, use = local_tile / NB;
                if (!mbar_wait<BCOMP>(acc_empty_bar(buf), (use & 1u) ^ 1u, wc)) { ok = false; break; }
                if (SHARED_PANEL && local_tile > 0 && !mbar_wait<BCOMP>(shared_read_bar, (local_tile - 1) & 1u, wc)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + buf * C::ACC_STEP;
                uint32_t acc = 0;
                for (int kb = u.kb0; kb < u.kb1; ++kb) {
                    if (!mbar_wait<BCOMP>(full_bar(s), ph, wc)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a_src = smem_base + s * C::STAGE;
                    const uint32_t b_src = a_src + C::A_STAGE;
                    const uint32_t meta_cols = tmem_base + C::META_COL0 + s * C::META_COLS;
                    // Metadata rides in the stage and is copied to tensor memory in front of the stage's MMAs.  (It used
                    // to go through the registers of four extra warps, tcgen05.st and a handshake per four atoms: their
                    // round trip paced the loop.  4096 x 8192 x 4096, clk per stage, bf16 / FP8: 783 / 1186 before,
                    // 639 / 612 now, against 594 / 562 with no metadata refreshed at all.)
                    if (SPARSE) {
#pragma unroll
                        for (int i = 0; i < C::ATOMS; ++i)
                            tc_cp_meta_atom(meta_cols + 4 * i, smem_desc(b_src + C::B_STAGE + 2048 * i, 128, 128, 0));
                    }
                    // the second half of the last stage of an 8-bit sparse product with an odd number of atoms (zero-filled
                    // values) takes the first half's metadata columns
                    const uint32_t back = (SPARSE && F8 && kb == half_kb) ? 4u : 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t adesc = smem_desc(a_src + 32 * j, 16, 1024, 2);
                        uint64_t bdesc;
                        if (BMAJ == BMajor::K) {
                            bdesc = SPARSE ? smem_desc(b_src + (j >> 1) * C::B_SUB + 64 * (j & 1), 16, 1024, 2)
                                           : smem_desc(b_src + 32 * j, 16, 1024, 2);
                        } else {
                            constexpr int ROWS_PER_MMA = BK / 4;     // K rows of 128 bytes per instruction
                            bdesc = smem_desc(b_src + ROWS_PER_MMA * 128 * j, BK * 128, 1024, 2);
                        }
                        if (SPARSE) {
                            // bf16: one 32-bit metadata column per instruction, the column pair is addressed and
                            // the descriptor's sparse selector picks the column; fp8: two columns per instruction
                            const uint32_t e = meta_cols + (F8 ? 2 * j - (j >= 2 ? back : 0u) : (j & 2));
                            const uint32_t id2 = F8 ? 0u : static_cast<uint32_t>(j & 1);
                            tc_mma_sparse<F8>(d_tmem, adesc, bdesc, e, idesc | id2, acc);
                        } else {
                            tc_mma_dense<F8>(d_tmem, adesc, bdesc, idesc, acc);
                        }
                        acc = 1u;
                    }
                    tc_commit_pair(empty_bar(s));     // frees the stage in both CTAs once these MMAs have read it
                    if (++s == NS) { s = 0; ph ^= 1u; }
                }
                if (ok) tc_commit_pair(acc_full_bar(buf));
            }
        }
    } else if (warp < 2 + C::EPI_WARPS) {
        // ------------------------------------------------------------ epilogue (warps 2.., both CTAs)
        // A warp owns 32 rows and a range of columns (half of them with eight warps) of the accumulator from tensor memory
        // to the output, two panels of 32 columns at a time: pulled into registers (packed bf16), staged and stored.  The
        // accumulator is released when the last panels are in registers, before they are stored; the next main loop has the other one.
        // What leaves is whole 128-byte lines: a row-major output by boxes of 32 rows x 64 columns of one warp, a transposed
        // one by boxes of 64 rows x 32 columns of a pair of warps (a warp alone has 64 bytes of each output row).  Half
        // lines by TMA were 2-3 % slower (3840 x 1280, 16384 tokens, bf16 forward: 82 -> 80 us), by plain stores 25 %.
        const int quarter = warp & 3;                  // tensor-memory lanes [32*quarter, 32*quarter + 32)
        constexpr int PANELS_MAX = C::EPI_WARPS == 8 ? (BN / 32 + 1) / 2 : BN / 32;   // 32-column panels per warp
        const int pnl0 = ((warp - 2) >> 2) * PANELS_MAX;                              // first panel of this warp
        const int n_pnl = (C::EPI_WARPS == 8 && pnl0 > 0) ? BN / 32 - PANELS_MAX : PANELS_MAX;
        constexpr int BOXP = (!OUT_T && C::PANELS == 2) ? 2 : 1;     // panels per box
        constexpr int BOXES = OUT_T ? C::PANELS : 1;                 // boxes that the group's staging holds
        const int group_bar = 1 + ((warp - 2) >> 1);                 // OUT_T: barrier of warps 2k, 2k + 1
        const bool elect = lane == 0 && (!OUT_T || (warp & 1) == 0); // issues the group's stores
        auto group_sync = [&] { if (OUT_T) pair_barrier(group_bar); else __syncwarp(); };
        auto group_all = [&](bool ok) -> bool { return OUT_T ? pair_barrier_and(group_bar, ok) : __all_sync(0xffffffffu, ok); };
        sste_pdl_wait();
        const float scale = sste_out_scale(p.a_amax, p.a_fp8_max, p.b_amax, p.b_fp8_max);
        const bool want_amax = (p.out_amax != nullptr);
        const int kind = want_amax ? 2 : scale != 1.0f ? 1 : 0;      // what a stored value needs besides the rounding
        uint32_t amax2 = 0;                            // bf16 output: running max of the magnitude bits, two lanes of 16
        float amaxf = 0.0f;                            // fp32 output
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t my_staging = staging + (OUT_T ? (warp - 2) & ~1 : warp - 2) * (C::PANELS * PANEL_BYTES);
        uint32_t local_tile = 0, box_it = 0;
        // Two accumulator values -> one word of two bf16 (packed conversion).  KIND 0: unit scale and no amax wanted
        // (every bf16 product of the path); 1: scale; 2: scale and running maximum.
        auto pack2 = [&](float lo, float hi, auto kind_tag) -> uint32_t {
            constexpr int KIND = decltype(kind_tag)::value;
            if (KIND >= 1) {
                lo = __fmul_rn(lo, scale);
                hi = __fmul_rn(hi, scale);
            }
            const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
            const uint32_t w = *reinterpret_cast<const uint32_t *>(&v);
            if (KIND == 2) amax2 = __vmaxu2(amax2, w & 0x7fff7fffu);
            return w;
        };
        // half h (tmem_ld_half) of 32 columns -> its 8 of the 16 packed words that store_box takes per panel
        auto pack_impl = [&](const uint32_t *r, uint32_t *w, int h, auto kind_tag) {
            if (OUT_T) {
#pragma unroll
                for (int b = 0; b < 4; ++b)            // 8-column blocks
#pragma unroll
                    for (int k = 0; k < 2; ++k)        // 8-row blocks
                        w[4 * b + 2 * h + k] = pack2(__uint_as_float(r[4 * b + 2 * k]), __uint_as_float(r[4 * b + 2 * k + 1]), kind_tag);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    w[8 * h + i] = pack2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]), kind_tag);
            }
        };
        auto pack_half = [&](const uint32_t *r, uint32_t *w, int h) {
            if (kind == 0) pack_impl(r, w, h, std::integral_constant<int, 0>{});
            else if (kind == 1) pack_impl(r, w, h, std::integral_constant<int, 1>{});
            else pack_impl(r, w, h, std::integral_constant<int, 2>{});
        };
        auto pack_chunk = [&](const uint32_t *r, uint32_t *w) {
            pack_half(r, w, 0);
            pack_half(r + 16, w, 1);
        };
        for (int unit = seq.first(); unit < num_units; ++local_tile, unit = seq.next(unit, local_tile)) {
            const Unit u = decode(unit);
            int mt, nt;
            tile_coords(u.tile, m_tiles, n_tiles, p.group_m, mt, nt);
            const int m0 = mt * 2 * BM + static_cast<int>(rank) * BM;
            const int n0 = nt * BN;
            const uint32_t buf = local_tile % NB, use = local_tile / NB;
            const uint32_t acc_base = lane_base + buf * C::ACC_STEP;
            // this warp reads the panel that the accumulators share: the last of the first, the first of the second
            const bool reads_shared = SHARED_PANEL && (buf == 0) == (pnl0 > 0);
            auto release_shared = [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at<BCOMP>(map_to_cta(shared_read_bar, 0));
            };
            auto release_acc = [&] {       // this warp has read its rows: count towards the buffer's release
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at<BCOMP>(map_to_cta(acc_empty_bar(buf), 0));
            };
            // (a pair of warps leaves together when a wait expired: its barriers need both)
            if (!group_all(mbar_wait_warp<BCOMP>(acc_full_bar(buf), use & 1u, wc))) break;
            tc_fence_after();
            if (OUT_F32) {
                const int m = m0 + quarter * 32 + lane;
#pragma unroll 1
                for (int c0 = 32 * pnl0; c0 < 32 * (pnl0 + n_pnl); c0 += 32) {
                    uint32_t r[32];
                    tmem_ld_32x32(acc_base + c0, r);
                    tmem_ld_wait();
                    if (m < p.M && n0 + c0 < p.N) {
                        float v[32];
#pragma unroll
                        for (int c = 0; c < 32; ++c) v[c] = __fmul_rn(__uint_as_float(r[c]), scale);
                        if (want_amax) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) amaxf = fmaxf(amaxf, fabsf(v[c]));
                        }
                        if (OUT_T) {
                            float *out = static_cast<float *>(p.D);
#pragma unroll
                            for (int c = 0; c < 32; ++c) out[static_cast<size_t>(n0 + c0 + c) * p.M + m] = v[c];
                        } else {
                            float4 *out = reinterpret_cast<float4 *>(static_cast<float *>(p.D) +
                                                                     static_cast<size_t>(m) * p.N + n0 + c0);
#pragma unroll
                            for (int c = 0; c < 8; ++c) out[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                        }
                    }
                }
                if (reads_shared) release_shared();
                release_acc();
                continue;
            }
            // packed panels of this warp -> staging (swizzled as the TMA store expects, conflict-free): one box of BOXP panels
            auto stage_box = [&](uint32_t sb, const uint32_t *w) {
                if (OUT_T) {
                    // staging row = column n of the accumulator, 64 m of the pair; matrix k = rows m 8k .. 8k + 7 of the warp
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const uint32_t n = 8u * b + (lane & 7);
                        stmatrix_x4_trans(sb + n * 128 + (((4 * (quarter & 1) + (lane >> 3)) ^ (n & 7)) << 4), w[4 * b],
                                          w[4 * b + 1], w[4 * b + 2], w[4 * b + 3]);
                    }
                } else if (BOXP == 2) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        st_shared_v4(sb + lane * 128 + ((c ^ (lane & 7)) << 4), w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                } else {
                    // no room for whole lines (256-wide weight gradient): 64-byte rows, 64-byte swizzle
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        st_shared_v4(sb + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4), w[4 * c], w[4 * c + 1], w[4 * c + 2],
                                     w[4 * c + 3]);
                }
            };
            // -> output, by one thread of the group
            auto put_box = [&](uint32_t sb, int pnl) {
                if (OUT_T) tma_store_2d(&map_d, sb, m0 + 64 * (quarter >> 1), n0 + 32 * pnl);
                else tma_store_2d(&map_d, sb, n0 + 32 * pnl, m0 + 32 * quarter);
            };
            auto store_box = [&](int pnl, const uint32_t *w) {
                const uint32_t sb = my_staging + (BOXES == 2 ? (box_it & 1u) * (2 * PANEL_BYTES) : 0u);
                ++box_it;
                // the buffer is writable once the store issued from it last has read it (in the newest group but one: a box is a
                // group of its own here, and nothing that store_two left is unread any more)
                if (elect) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(BOXES - 1) : "memory");
                group_sync();
                stage_box(sb, w);
                fence_proxy_async();
                group_sync();
                if (elect) {
                    put_box(sb, pnl);
                    tma_store_commit();
                }
            };
            // both buffers at once: one wait, one fence and two barriers for two boxes (the second is there if `two`; FP8 forward of
            // 3072 x 768, 8192 tokens: 18.8 -> 17.9 us, bf16 24.0 -> 23.8)
            auto store_two = [&](int pnl, const uint32_t *w, bool two) {
                if (elect) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                group_sync();
                stage_box(my_staging, w);
                if (two) stage_box(my_staging + 2 * PANEL_BYTES, w + 16);
                fence_proxy_async();
                group_sync();
                if (elect) {
                    put_box(my_staging, pnl);
                    if (two) put_box(my_staging + 2 * PANEL_BYTES, pnl + 1);
                    tma_store_commit();
                }
            };
            if (unit >= p.split_from && p.splits > 1) {
                // Split-K.  The group's panels are exchanged in up to MAX_PARTS parts, which the units of a tile take in
                // rotated order.  For each part a unit draws a number: all but the last to come leave their fp32 partial in
                // the workspace (512 contiguous bytes per warp and store) and count it as finished; the last one keeps its
                // own in tensor memory, waits for the others' (they are past their main loop and wait for nobody: the
                // wait ends whatever else the GPU runs), adds all in split order (bit-reproducible) and stores the result.  With
                // the rotation each unit ends up last for about its share of the parts.  (When the unit that came last
                // read all partials, its own too, and added up the whole tile, an exchange took 10 us; now 5-6 us between two
                // units, 8-10 between four.  3072 x 768, 8192 tokens, bf16 grad_W: 26.2 -> 22.5 us.)
                constexpr size_t PART = static_cast<size_t>(BN / 4) * 32;          // float4 per 32 rows and split
                const size_t slot = static_cast<size_t>(u.tile - p.split_from) * 2 + rank;
                float4 *part0 = reinterpret_cast<float4 *>(p.partials) + (slot * p.splits * 4 + quarter) * PART + lane;
                unsigned int *tickets = p.tickets + (slot * C::EPI_WARPS + (OUT_T ? (warp - 2) & ~1 : warp - 2)) * MAX_PARTS;
                const int n_box = n_pnl / BOXP;
                const int parts = min(n_box, MAX_PARTS);
                constexpr int AHEAD = 2;               // (three spill registers of the ordinary epilogue)
                bool ok = true;
                // store_two's group reads both buffers: store_box, which leaves the newest group unread, begins behind it.  (A group
                // per box there, and this wait left out, cost ordinary tiles 0.3 us of a forward of 3072 x 768, 8192 tokens.)
                if (BOXES == 2 && elect) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                if (!p.tickets) {
                    // summed by splitk_sum_kernel: lane = row, whatever the output's orientation
                    float4 *mine = part0 + static_cast<size_t>(u.split) * 4 * PART;
#pragma unroll 1
                    for (int pnl = pnl0; pnl < pnl0 + n_pnl; ++pnl) {
                        uint32_t r[32];
                        tmem_ld_32x32(acc_base + 32 * pnl, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            __stcg(mine + (8 * pnl + i) * 32,
                                   make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                               __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])));
                    }
                    if (reads_shared) release_shared();
                    release_acc();
                    continue;
                }
                uint32_t drawn = 0;
                if (elect) drawn = atomicAdd(tickets + u.split % parts, 1u);
#pragma unroll 1
                for (int k = 0; k < parts && ok; ++k) {
                    const int part = (u.split + k) % parts;
                    const int box_lo = part * n_box / parts, box_hi = (part + 1) * n_box / parts;
                    const int lo = pnl0 + box_lo * BOXP, hi = pnl0 + box_hi * BOXP;
                    unsigned int *ticket = tickets + part;
                    if (group_all(!elect || (drawn & 0xffffu) != static_cast<unsigned int>(p.splits) - 1u)) {
                        float4 *mine = part0 + static_cast<size_t>(u.split) * 4 * PART;
#pragma unroll 1
                        for (int pnl = lo; pnl < hi; ++pnl) {
                            uint32_t r[32];
                            tmem_ld_32cols<OUT_T>(acc_base + 32 * pnl, r);
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                __stcg(mine + (8 * pnl + i) * 32,
                                       make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                                   __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])));
                        }
                        group_sync();
                        if (elect) {
                            if (k + 1 < parts) drawn = atomicAdd(tickets + (u.split + k + 1) % parts, 1u);   // on its way meanwhile
                            __threadfence();               // the group's partial (ordered by group_sync) before the count
                            atomicAdd(ticket, 0x10000u);
                        }
                        continue;
                    }
                    if (elect) {
                        const uint32_t all = (static_cast<uint32_t>(p.splits) << 16) - 0x10000u + static_cast<uint32_t>(p.splits);
                        if (ld_acquire_gpu(ticket) != all) {
                            const unsigned long long start = global_ns();
                            while (ok && ld_acquire_gpu(ticket) != all) {
                                if (*wc.abort_flag) ok = false;
                                else if (global_ns() - start > wc.limit_ns) {
                                    atomicMax(wc.status, static_cast<unsigned int>(SSTE_ERR_TIMEOUT));      // also over a recorded degenerate beta
                                    *wc.abort_flag = 1;
                                    ok = false;
                                }
                            }
                        }
                        if (ok) *ticket = 0u;              // zero again for the next launch
                        if (k + 1 < parts) drawn = atomicAdd(tickets + (u.split + k + 1) % parts, 1u);
                    }
                    ok = group_all(ok);
                    if (!ok) break;
                    if (p.splits == 2) {
                        // one other partial, and a sum of two has no order: the next panel is on its way while one is stored
                        const float4 *src = part0 + static_cast<size_t>(1 - u.split) * 4 * PART;
                        sste_fresh(src);
                        float4 q[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) q[i] = __ldcg(src + (8 * lo + i) * 32);
                        uint32_t w[16 * BOXP];
#pragma unroll 1
                        for (int pnl = lo; pnl < hi; pnl += BOXP) {
#pragma unroll
                            for (int b = 0; b < BOXP; ++b) {
                                uint32_t own[32];
                                tmem_ld_32cols<OUT_T>(acc_base + 32 * (pnl + b), own);
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    own[4 * i] = __float_as_uint(__fadd_rn(__uint_as_float(own[4 * i]), q[i].x));
                                    own[4 * i + 1] = __float_as_uint(__fadd_rn(__uint_as_float(own[4 * i + 1]), q[i].y));
                                    own[4 * i + 2] = __float_as_uint(__fadd_rn(__uint_as_float(own[4 * i + 2]), q[i].z));
                                    own[4 * i + 3] = __float_as_uint(__fadd_rn(__uint_as_float(own[4 * i + 3]), q[i].w));
                                }
                                if (pnl + b + 1 < hi) {
#pragma unroll
                                    for (int i = 0; i < 8; ++i) q[i] = __ldcg(src + (8 * (pnl + b + 1) + i) * 32);
                                }
                                pack_chunk(own, w + 16 * b);
                            }
                            store_box(pnl, w);
                        }
                        continue;
                    }
#pragma unroll 1
                    for (int pnl = lo; pnl < hi; pnl += BOXP) {
                        uint32_t w[16 * BOXP];
#pragma unroll
                        for (int b = 0; b < BOXP; ++b) {
                            const float4 *src = part0 + (pnl + b) * 8 * 32;
                            sste_fresh(src);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                uint32_t v[16];
#pragma unroll 1
                                for (int sp = 0; sp < p.splits; sp += AHEAD) {
                                    uint32_t q[AHEAD][16];     // half a panel of AHEAD splits in flight
#pragma unroll
                                    for (int d = 0; d < AHEAD; ++d) {
                                        if (sp + d >= p.splits) break;
                                        if (sp + d == u.split) {
                                            tmem_ld_half<OUT_T>(acc_base + 32 * (pnl + b), h, q[d]);
                                        } else {
#pragma unroll
                                            for (int i = 0; i < 4; ++i) {
                                                const float4 x = __ldcg(src + static_cast<size_t>(sp + d) * 4 * PART + (4 * h + i) * 32);
                                                q[d][4 * i] = __float_as_uint(x.x);
                                                q[d][4 * i + 1] = __float_as_uint(x.y);
                                                q[d][4 * i + 2] = __float_as_uint(x.z);
                                                q[d][4 * i + 3] = __float_as_uint(x.w);
                                            }
                                        }
                                    }
                                    tmem_ld_wait();
#pragma unroll
                                    for (int d = 0; d < AHEAD; ++d) {
                                        if (sp + d >= p.splits) break;
#pragma unroll
                                        for (int i = 0; i < 16; ++i)
                                            v[i] = (d == 0 && sp == 0) ? q[0][i]
                                                                       : __float_as_uint(__fadd_rn(__uint_as_float(v[i]), __uint_as_float(q[d][i])));
                                    }
                                }
                                pack_half(v, w + 16 * b, h);
                            }
                        }
                        store_box(pnl, w);
                    }
                }
                if (reads_shared) release_shared();
                release_acc();
                if (!ok) break;
            } else {
                // panels held packed in registers at a time
                constexpr int HOLD = PANELS_MAX % 2 == 0 ? 2 : PANELS_MAX;
                static_assert(PANELS_MAX % HOLD == 0 && HOLD % BOXP == 0, "whole rounds of panels");
#pragma unroll
                for (int h = 0; h < PANELS_MAX; h += HOLD) {
                    const int h0 = (SHARED_PANEL && buf == 0 && pnl0 > 0) ? PANELS_MAX - HOLD - h : h;      // the shared panel first
                    uint32_t pk[16 * HOLD];
                    const uint32_t cols = acc_base + 32 * (pnl0 + h0);
#pragma unroll
                    for (int i = 0; i < HOLD; i += 2) {
                        uint32_t r[64];
                        const bool first = h0 + i < n_pnl, second = i + 1 < HOLD && h0 + i + 1 < n_pnl;
                        if (first) tmem_ld_32cols<OUT_T>(cols + 32 * i, r);
                        if (second) tmem_ld_32cols<OUT_T>(cols + 32 * i + 32, r + 32);
                        tmem_ld_wait();
                        if (SHARED_PANEL && h == 0 && reads_shared) release_shared();
                        if (first) pack_chunk(r, pk + 16 * i);
                        if (second) pack_chunk(r + 32, pk + 16 * i + 16);
                    }
                    if (h + HOLD == PANELS_MAX) release_acc();
                    if constexpr (BOXES == 2 && HOLD == 2) {
                        if (h0 < n_pnl) store_two(pnl0 + h0, pk, h0 + 1 < n_pnl);
                    } else {
#pragma unroll
                        for (int i = 0; i < HOLD; i += BOXP)
                            if (h0 + i < n_pnl) store_box(pnl0 + h0 + i, pk + 16 * i);
                    }
                }
            }
        }
        if (want_amax) {
            // max|D| of this warp's share, as the bits of a non-negative fp32 (they order like unsigned integers)
            uint32_t best = OUT_F32 ? __float_as_uint(amaxf) : (max(amax2 & 0xffffu, amax2 >> 16) << 16);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
            if (lane == 0 && best != 0) atomicMax(p.out_amax, best);
        }
        if (elect && !OUT_F32) {
            if (FINAL) tma_store_wait_all();
            else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
    } else if (BCOMP) {
        // ------------------------------------------------------------ expander warps (6..9, both CTAs)
        // grad_X = grad_Z S(W) reads S(W) [O, I] as its MN-major B operand.  Here S(W) is given as the forward's
        // compressed operand (2:4 values + metadata image) and every stage's K rows are expanded into the shared-
        // memory image a TMA load of the dense matrix would have left: rows of 128 bytes of N, 16-byte chunks
        // XOR-swizzled with the row, +0 in the pruned positions.  A unit is 16 bytes of values (8 groups of fp8,
        // 4 of bf16) = 32 bytes of the dense row; the loads of the next stage are in flight while this one is
        // expanded.
        constexpr int SEGS = (BN / 2) * ELT / 32;          // units per K row of this CTA's half of the tile
        constexpr int UNITS = BK * SEGS / 128;             // units per thread and stage
        static_assert(!BCOMP || (BK * SEGS) % 128 == 0, "units per stage");
        const int t = static_cast<int>(threadIdx.x) - 192;
        // byte-permute selectors per metadata nibble p0 | p1 << 2: which source byte feeds each output byte
        // (4 = a zero byte).  bf16: low / high 16 bits select the two output words of a group from the pair word;
        // fp8: 16 bits select the output word of a group from its two value bytes (0, 1).
        uint32_t *lut = reinterpret_cast<uint32_t *>(ctrl_generic + CTRL_LUT);
        if (t < 16) {
            const uint32_t p0 = t & 3, p1 = t >> 2;
            uint32_t sel = 0;
            for (uint32_t h = 0; h < 4; ++h) {
                if (F8) sel |= (h == p0 ? 0u : h == p1 ? 1u : 4u) << (4 * h);
                else sel |= (h == p0 ? 0x10u : h == p1 ? 0x32u : 0x44u) << (8 * h);
            }
            lut[t] = sel;
        }
        asm volatile("bar.sync 2, 128;" ::: "memory");
        // A thread's units of a stage: the same 32-byte column segment `seg` of rows r0 + j * ROWS_STEP.
        constexpr int ROWS_STEP = 128 / SEGS;
        constexpr int EPU = 32 / ELT;                      // dense elements per unit
        const int seg = t % SEGS, r0 = t / SEGS;
        const size_t row_bytes = static_cast<size_t>(p.N / 2) * ELT;     // one row of compressed values
        const size_t atom_row_bytes = static_cast<size_t>(p.N / 128) * 2048;
        uint32_t moff[UNITS];                              // metadata byte of unit j inside its (half) atom
#pragma unroll
        for (int j = 0; j < UNITS; ++j) {
            const uint32_t m = static_cast<uint32_t>(r0 + j * ROWS_STEP), k = static_cast<uint32_t>(seg * EPU);
            moff[j] = F8 ? sste_meta_atom_byte8(m, k) : sste_meta_atom_byte16(m, k);
        }
        // loader cursor: (unit, stage) of the next loads
        int e_j = 0, e_unit = seq.first(), e_kb = 0, e_kend = 0;
        const uint8_t *e_vals = nullptr, *e_meta = nullptr;
        bool e_cols = false;
        auto e_setup = [&]() {
            if (e_unit >= num_units) return;
            const Unit u = decode(e_unit);
            int mt, nt;
            tile_coords(u.tile, m_tiles, n_tiles, p.group_m, mt, nt);
            const int n0 = nt * BN + static_cast<int>(rank) * (BN / 2);
            e_cols = n0 < p.N;
            e_vals = p.b_vals + (static_cast<size_t>(n0 / 2) + seg * (EPU / 2)) * ELT + r0 * row_bytes;
            e_meta = meta + static_cast<size_t>(n0 >> 7) * 2048;
            e_kb = u.kb0;
            e_kend = u.kb1;
        };
        auto e_issue = [&](uint4 (&v)[UNITS], uint32_t (&m)[UNITS]) -> bool {
            if (e_unit >= num_units) return false;
            const uint32_t krow0 = static_cast<uint32_t>(e_kb) * BK;             // first K row of the stage
            const uint8_t *vp = e_vals + krow0 * row_bytes;
            const uint8_t *mp = e_meta + (krow0 >> 7) * atom_row_bytes + ((BK == 64 && (krow0 & 64u)) ? 1024u : 0u);
#pragma unroll
            for (int j = 0; j < UNITS; ++j) {
                if (e_cols) {
                    v[j] = sste_ld(reinterpret_cast<const uint4 *>(vp + static_cast<size_t>(j) * ROWS_STEP * row_bytes));
                    if (F8) m[j] = sste_ld(reinterpret_cast<const uint32_t *>(mp + moff[j]));
                    else m[j] = sste_ld(reinterpret_cast<const uint16_t *>(mp + moff[j]));
                } else {
                    v[j] = make_uint4(0, 0, 0, 0);         // columns beyond N: zeros (any valid code will do)
                    m[j] = 0x44444444u;
                }
            }
            if (++e_kb >= e_kend) {
                ++e_j;
                e_unit = seq.next(e_unit, e_j);
                e_setup();
            }
            return true;
        };
        e_setup();
        sste_pdl_wait(e_vals, e_meta);
        // three stages of loads in flight in registers: a round trip to L2 is longer than two stages of MMAs
        uint4 v0[UNITS], v1[UNITS], v2[UNITS];
        uint32_t m0[UNITS], m1[UNITS], m2[UNITS];
        bool h0 = e_issue(v0, m0), h1 = e_issue(v1, m1), h2 = e_issue(v2, m2);
        uint32_t it = 0;
        uint8_t *const ring = ctrl_generic + CTRL_BYTES;
        while (h0) {
            const int s = it % NS;
            const uint32_t ph = (it / NS) & 1u;
            if (!mbar_wait_warp<BCOMP>(empty_bar(s), ph ^ 1u, wc)) break;
            uint8_t *b_dst = ring + s * C::STAGE + C::A_STAGE + (seg >> 2) * (BK * 128);
            const int j0 = (seg & 3) * 2;
#pragma unroll
            for (int j = 0; j < UNITS; ++j) {
                const int r = r0 + j * ROWS_STEP;
                const uint32_t w[4] = {v0[j].x, v0[j].y, v0[j].z, v0[j].w};
                uint32_t o[8];
                if (F8) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        const uint32_t pairw = (g & 1) ? (w[g >> 1] >> 16) : w[g >> 1];    // value bytes 0, 1
                        o[g] = __byte_perm(pairw, 0, lut[(m0[j] >> (4 * g)) & 0xfu]);
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const uint32_t sel = lut[(m0[j] >> (4 * g)) & 0xfu];
                        o[2 * g] = __byte_perm(w[g], 0, sel & 0xffffu);
                        o[2 * g + 1] = __byte_perm(w[g], 0, sel >> 16);
                    }
                }
                uint8_t *rowp = b_dst + r * 128;
                *reinterpret_cast<uint4 *>(rowp + ((j0 ^ (r & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
                *reinterpret_cast<uint4 *>(rowp + (((j0 + 1) ^ (r & 7)) << 4)) = make_uint4(o[4], o[5], o[6], o[7]);
            }
            fence_proxy_async();        // the tensor core reads the stage through the async proxy
            __syncwarp();
            if (lane == 0) mbar_arrive_at<BCOMP>(map_to_cta(full_bar(s), 0));
#pragma unroll
            for (int j = 0; j < UNITS; ++j) { v0[j] = v1[j]; m0[j] = m1[j]; v1[j] = v2[j]; m1[j] = m2[j]; }
            h0 = h1;
            h1 = h2;
            h2 = e_issue(v2, m2);
            ++it;
        }
    }
}

// Shared-memory control block, tensor memory and the pair's barriers around one or two products.
struct Frame {
    uint8_t *ctrl;               // generic address of the control block
    uint32_t ctrl_u32, data_u32; // shared addresses: control block, first stage
    uint32_t tmem_base;
    WaitCtx wc;
};
template <typename F>
__device__ __forceinline__ Frame frame_begin(uint8_t *smem_raw, const GemmParams &p, F init)
{
    Frame f;
    f.ctrl_u32 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    f.data_u32 = f.ctrl_u32 + CTRL_BYTES;
    f.ctrl = smem_raw + (f.ctrl_u32 - smem_u32(smem_raw));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(f.ctrl + CTRL_ABORT);
    f.wc = WaitCtx{p.status, abort_flag, p.wait_limit_ns};
    if (threadIdx.x == 0) {
        init(f);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((threadIdx.x >> 5) == 1) {
        tmem_alloc(f.ctrl_u32 + CTRL_TMEM, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();          // the peer's barriers are initialised before anything signals them
    tc_fence_after();
    // (everything up to here overlaps the previous kernel.  Each role waits for it in front of its own first access to global
    // memory or bounded wait, the producer with the first tile's coordinates worked out: 0.2 to 0.4 us of every product, a forward of
    // 3072 x 768 with 128 tokens 6.55 -> 6.35.)
    if (blockIdx.x == 0 && threadIdx.x == 32 && p.zero_after) {
        sste_pdl_wait();
        *p.zero_after = 0u;
    }
    f.tmem_base = *reinterpret_cast<volatile uint32_t *>(f.ctrl + CTRL_TMEM);
    return f;
}
// every role of both CTAs is done: tensor memory and shared memory may be used for something else
__device__ __forceinline__ void pair_sync()
{
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
}

template <bool SPARSE, BMajor BMAJ, int ELT, int BN, bool OUT_T, bool OUT_F32, bool BCOMP = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Cfg<SPARSE, ELT, BN, BCOMP>::THREADS, 1)
gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_d, const __grid_constant__ CUtensorMap map_m,
            const uint8_t *__restrict__ meta, const __grid_constant__ GemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    sste_pdl_trigger();
    const Frame f = frame_begin(smem_raw, p, [&](const Frame &fr) {
        init_barriers<Cfg<SPARSE, ELT, BN, BCOMP>, BCOMP>(fr.ctrl_u32);
        prefetch_tensormap(&map_a);
        if (!BCOMP) prefetch_tensormap(&map_b);
        if (SPARSE) prefetch_tensormap(&map_m);
        if (!OUT_F32) prefetch_tensormap(&map_d);
    });
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    product<SPARSE, BMAJ, ELT, BN, OUT_T, OUT_F32, BCOMP, true>(map_a, map_b, map_d, map_m, meta, p,
                                                               UnitSeq{0, 0, 0, 0, pairs, pair}, f.ctrl, f.ctrl_u32, f.data_u32,
                                                               f.tmem_base, f.wc);
    pair_sync();             // neither CTA frees tensor memory while the pair still uses it
    if ((threadIdx.x >> 5) == 1) tmem_dealloc(f.tmem_base, TMEM_COLS);
}

// Sum of the partial tiles of a product whose few tiles were cut into many K ranges (p.tickets null).  In the product itself
// one warp would read the partials of all other units, a few at a time: at 16 ranges that chain of L2 round trips took 10 us
// and more.  Here every thread of a small grid adds up one float4 of the ranges, eight loads in flight, in split order.
// 128 x 8192, 128 tokens, bf16 forward: 13.3 us with 5 ranges that exchange -> 7.4 with 16; 8192 x 128, 128 tokens, both
// gradients: 21.7 -> 10.0; 128 x 128, 8192 tokens: 17.7 -> 8.6.  With many tiles the exchange moves half of the bytes and
// needs no second launch: it stays.
// (Blocks from `blocks` on do the same for a second product.)
template <bool OUT_T>
__global__ void __launch_bounds__(128) splitk_sum_kernel(const __grid_constant__ GemmParams p1, int bn1, int blocks,
                                                         const __grid_constant__ GemmParams p2, int bn2)
{
    sste_pdl_trigger();
    const bool second = static_cast<int>(blockIdx.x) >= blocks;
    const GemmParams &p = second ? p2 : p1;
    const int bn = second ? bn2 : bn1;
    const int lane = threadIdx.x & 31, warp = (blockIdx.x - (second ? blocks : 0)) * 4 + (threadIdx.x >> 5);
    const int groups = bn / 4;                               // warps per 32 rows of a tile
    const int q = warp / groups, g = warp - q * groups;
    const int slot = q >> 2, quarter = q & 3;                // slot: [split tile][cta]
    // row-major output: eight rows x 16 columns per warp (whole sectors); transposed: 32 rows x 4 columns
    const int c4 = OUT_T ? g : (g >> 2) * 4 + (lane & 3), row = OUT_T ? lane : (g & 3) * 8 + (lane >> 2);
    int mt, nt;
    tile_coords(p.split_from + (slot >> 1), (p.M + 2 * BM - 1) / (2 * BM), (p.N + bn - 1) / bn, p.group_m, mt, nt);
    const int m = mt * 2 * BM + (slot & 1) * BM + quarter * 32 + row, n = nt * bn + 4 * c4;
    const bool inside = m < p.M && n < p.N;
    sste_pdl_wait();
    const float scale = sste_out_scale(p.a_amax, p.a_fp8_max, p.b_amax, p.b_fp8_max);
    uint32_t best = 0;
    if (inside) {
        const size_t step = static_cast<size_t>(4) * groups * 32;       // float4 between two splits
        const float4 *src = reinterpret_cast<const float4 *>(p.partials) +
                            (static_cast<size_t>(slot) * p.splits * 4 + quarter) * (groups * 32) + c4 * 32 + row;
        sste_fresh(src);
        float4 v = __ldcg(src);
        auto add = [&](const float4 &x) {
            v.x = __fadd_rn(v.x, x.x); v.y = __fadd_rn(v.y, x.y); v.z = __fadd_rn(v.z, x.z); v.w = __fadd_rn(v.w, x.w);
        };
        int sp = 1;
        for (; sp + 8 <= p.splits; sp += 8) {
            float4 x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = __ldcg(src + (sp + i) * step);
#pragma unroll
            for (int i = 0; i < 8; ++i) add(x[i]);
        }
        float4 x[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) if (sp + i < p.splits) x[i] = __ldcg(src + (sp + i) * step);
#pragma unroll
        for (int i = 0; i < 7; ++i) if (sp + i < p.splits) add(x[i]);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(__fmul_rn(v.x, scale), __fmul_rn(v.y, scale));
        const __nv_bfloat162 hi = __floats2bfloat162_rn(__fmul_rn(v.z, scale), __fmul_rn(v.w, scale));
        const uint32_t w0 = *reinterpret_cast<const uint32_t *>(&lo), w1 = *reinterpret_cast<const uint32_t *>(&hi);
        __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(p.D);
        if (OUT_T) {
            out[static_cast<size_t>(n) * p.M + m] = lo.x;
            out[static_cast<size_t>(n + 1) * p.M + m] = lo.y;
            out[static_cast<size_t>(n + 2) * p.M + m] = hi.x;
            out[static_cast<size_t>(n + 3) * p.M + m] = hi.y;
        } else {
            *reinterpret_cast<uint2 *>(out + static_cast<size_t>(m) * p.N + n) = make_uint2(w0, w1);
        }
        const uint32_t a = __vmaxu2(w0 & 0x7fff7fffu, w1 & 0x7fff7fffu);
        best = max(a & 0xffffu, a >> 16) << 16;
    }
    if (p.out_amax) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
        if (lane == 0 && best != 0) atomicMax(p.out_amax, best);
    }
}

// grad_W and grad_X of a layer in one launch.  They are independent, and each alone quantises badly into waves of CTA pairs
// (3072 x 768, 8192 tokens: 36 and 96 tiles on 74 pairs).  Every pair computes its share of grad_W, then of grad_X: the
// pairs that come out of grad_W a round earlier (`late_pairs` is the number of the others, the first ones) take `early`
// rounds of grad_X tiles among themselves before all share the rest.
struct GradsPlan { int late_pairs, early, early_first; };
template <int ELT, int BNW, int BNX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(320, 1)
grads_kernel(const __grid_constant__ CUtensorMap wa, const __grid_constant__ CUtensorMap wb, const __grid_constant__ CUtensorMap wd,
             const __grid_constant__ CUtensorMap wm, const __grid_constant__ CUtensorMap xa, const __grid_constant__ CUtensorMap xb,
             const __grid_constant__ CUtensorMap xd, const __grid_constant__ GemmParams pw, const __grid_constant__ GemmParams px,
             const GradsPlan g)
{
    extern __shared__ uint8_t smem_raw[];
    sste_pdl_trigger();
    const Frame f = frame_begin(smem_raw, pw, [&](const Frame &fr) {
        init_barriers<Cfg<true, ELT, BNW>, false>(fr.ctrl_u32);
        init_barriers<Cfg<false, ELT, BNX>, false>(fr.ctrl_u32 + CTRL_SECOND);
        prefetch_tensormap(&wa); prefetch_tensormap(&wb); prefetch_tensormap(&wd); prefetch_tensormap(&wm);
        prefetch_tensormap(&xa); prefetch_tensormap(&xb); prefetch_tensormap(&xd);
    });
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    product<true, BMajor::MN, ELT, BNW, false, false, false, false>(wa, wb, wd, wm, nullptr, pw, UnitSeq{0, 0, 0, 0, pairs, pair},
                                                                    f.ctrl, f.ctrl_u32, f.data_u32, f.tmem_base, f.wc);
    pair_sync();
    const int n_early = pairs - g.late_pairs;
    const bool late = pair < g.late_pairs;
    const UnitSeq seq{late ? 0 : g.early, n_early, pair - g.late_pairs, g.early * n_early, pairs,
                      g.early_first ? (late ? n_early + pair : pair - g.late_pairs) : pair};
    product<false, BMajor::MN, ELT, BNX, false, false, false, true>(xa, xb, xd, xa, nullptr, px, seq, f.ctrl,
                                                                    f.ctrl_u32 + CTRL_SECOND, f.data_u32, f.tmem_base, f.wc);
    pair_sync();
    if ((threadIdx.x >> 5) == 1) tmem_dealloc(f.tmem_base, TMEM_COLS);
}

// ------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 2-D row-major tensor [rows, cols] of `elt`-byte elements; box = box_cols x box_rows.
bool make_map(const sste_ctx *ctx, CUtensorMap *map, const void *base, int elt, uint64_t rows, uint64_t cols,
              uint32_t box_cols, uint32_t box_rows, CUtensorMapSwizzle swz)
{
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * static_cast<uint64_t>(elt)};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = (elt == 4)   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : (elt == 2) ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                : CU_TENSOR_MAP_DATA_TYPE_UINT8;
    EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(ctx->cu_tensor_map_encode);
    return fn(map, dt, 2, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int g_inject_stall = 0;   // test hook: see sste_debug_inject_stall
int g_force_group_m = 0;  // test hook: 0 = automatic band height of the tile order

// Band height of the tile order from the operand sizes (a_tile / b_tile: bytes of one tile row of A / one tile
// column of B over the whole reduction).  L2 is 126 MB; an operand that takes less than half of it stays
// resident whatever the order.
//   A small: plain column-major order (every pair of a wave shares a few columns of B, B is read once).
//   else:    bands of about sqrt(pairs * b_tile / a_tile) tile rows: a wave then loads the least bytes, the band's
//            A rows are read once while B, if it fits, stays in L2 across bands.
int pick_group_m(int m_tiles, int n_tiles, int pairs, double a_tile, double b_tile)
{
    if (g_force_group_m > 0) return g_force_group_m < m_tiles ? g_force_group_m : m_tiles;
    const double l2_budget = 56e6;
    if (a_tile * m_tiles <= l2_budget || m_tiles <= 1 || n_tiles <= 1) return m_tiles;
    double g = __builtin_sqrt(static_cast<double>(pairs) * b_tile / a_tile);
    int gm = static_cast<int>(g + 0.5);
    if (gm < 1) gm = 1;
    if (gm > m_tiles) gm = m_tiles;
    return gm;
}

int g_force_splits = 0;   // test hook: 0 = automatic split-K factor
int g_force_bn = 0;       // test hook: 0 = automatic tile width

enum Product { FORWARD = 0, GRAD_WEIGHT = 1, GRAD_INPUT = 2 };

// Tile widths a product supports (0 ends the list).  The MN-major B of the two gradient products needs whole 128-byte
// chunks of N per CTA: 128 columns wide only with 2-byte operands.
struct Widths { int bn[4]; };
constexpr Widths widths_of(Product pr, int elt)
{
    return pr == FORWARD ? Widths{{256, 224, 192, 128}} : elt == 2 ? Widths{{256, 128, 0, 0}} : Widths{{256, 0, 0, 0}};
}

// Microseconds of one stage of the main loop and what a tile costs besides (the part of the epilogue that is not hidden, the
// output's share of the L2 traffic), all CTA pairs busy; fitted to timings of every width on B200 at K = 768 ... 16384.  (Fitted when a
// 256-wide sparse tile had one accumulator, and before the epilogue's and the coordinates' share fell: tiles cost less than this by
// now, most of all those; the choice between widths has not been fitted again.)  A narrower tile moves more operand bytes per flop, a wider one quantises worse into waves.
struct TileCost { double stage_us, tile_us; };
constexpr TileCost tile_cost(Product pr, int elt, int bn)
{
    if (pr == FORWARD && elt == 2)
        return bn == 256 ? TileCost{0.46, 1.6} : bn == 224 ? TileCost{0.44, 0.9} : bn == 192 ? TileCost{0.40, 0.8} : TileCost{0.31, 0.75};
    if (pr == FORWARD)
        return bn == 256 ? TileCost{0.53, 2.0} : bn == 224 ? TileCost{0.46, 1.65} : bn == 192 ? TileCost{0.41, 1.55} : TileCost{0.33, 1.3};
    if (pr == GRAD_WEIGHT) return bn == 256 ? TileCost{elt == 2 ? 0.405 : 0.47, 1.0} : TileCost{0.345, 0.9};
    return bn == 256 ? TileCost{0.34, elt == 2 ? 1.1 : 1.4} : TileCost{0.27, 1.0};
}

// Everything the host decides about one product launch.
struct LaunchPlan { int bn, splits, split_from, group_m; double us; bool sum_after; };

// Microseconds that a split costs on top of its units' main loops: the exchange between `s` units, `bytes` of partials.
double exchange_us(int s, int bn, double bytes)
{
    return (s == 2 ? 2.4 + 2.6 * bn / 256.0 : 2.5 + 0.65 * s + (2.6 + 0.4 * s) * bn / 256.0) + bytes / 15e6;
}

// The same where splitk_sum_kernel follows the product: its launch, the fp32 stores that the units end with, their bytes.
// (Measured against whole tiles and exchanges at 1 ... 32 tiles, 2 ... 44 ranges.)
double sum_us(int s, int bn, double bytes) { return 0.4 + 2.4 * bn / 256.0 + 0.04 * s + bytes / 2.9e6; }
// split factors tried there
constexpr int SUM_SPLITS[] = {2, 3, 4, 6, 8, 11, 16, 22, 32, 44, 64};

// L2-aware band height of a product with tiles `bn` wide.
int plan_group_m(Product pr, int elt, bool bcomp, int bn, int pairs, int M, int N, int K)
{
    const bool sparse = (pr != GRAD_INPUT);
    return pick_group_m((M + 2 * BM - 1) / (2 * BM), (N + bn - 1) / bn, pairs,
                        static_cast<double>(K) * (sparse ? 0.5 * elt + 0.125 : 1.0 * elt) * 2 * BM,
                        static_cast<double>(K) * ((bcomp ? 0.5 : 1.0) * elt) * bn);
}

// The plans of the last shapes of a thread: a search takes 0.4 us of host time for most products and 1.2 for most pairs of
// gradients, but some 30 us for 16384 tokens through 11008 x 4096 and more with more tokens (it tries every number of early
// rounds).  Sets of four: with one place per shape two products of a GPT-2-large block pushed each other out every step.
std::atomic<unsigned long long> g_plan_searches{0};
template <typename Plan>
struct PlanMemo {
    typedef std::array<long long, 6> Key;
    static constexpr int SETS = 32, WAYS = 4;
    struct Entry { Key key{}; Plan plan{}; bool set = false; };
    struct Set { Entry entry[WAYS]; int oldest = 0; } sets[SETS];
    template <typename F>
    const Plan &get(const Key &key, F make)
    {
        unsigned long long h = 0;
        for (long long k : key) h = (h ^ static_cast<unsigned long long>(k)) * 0x9e3779b97f4a7c15ull;
        Set &set = sets[h >> 59];
        for (const Entry &e : set.entry)
            if (e.set && e.key == key) return e.plan;
        g_plan_searches.fetch_add(1, std::memory_order_relaxed);
        Entry &e = set.entry[set.oldest];
        set.oldest = (set.oldest + 1) % WAYS;
        e = Entry{key, make(), true};
        return e.plan;
    }
};

// Tile width and split-K factor by the model's time.  Tiles that fill complete waves of CTA pairs are computed whole; the
// tiles of the last, partial wave (all of them when there are fewer tiles than pairs, as for the weight gradient of a
// GPT-2-sized layer: 36 tiles, 74 pairs) may be cut into `splits` K ranges of at least eight stages, so that the wave
// takes 1/splits of a tile time and the exchange of the partials on top: 2.4 + 2.6 bn/256 us between two units,
// 4.4 + 3.8 bn/256 between three and so on (measured at 9 ... 36 tiles), and their bytes.  Few tiles (all ranges run at once)
// of a long reduction take many short ranges and a sum afterwards instead.  Among widths within 3 % the first wins.
// (estimate: for the time of grad_X in joint_wins, whose line was drawn with these constants as they are.)
LaunchPlan find_plan(Product pr, int elt, int only_bn, bool out_f32, bool bcomp, int sm_count, size_t partial_bytes, int M,
                     int N, int K, bool estimate)
{
    const bool sparse = (pr != GRAD_INPUT);
    const int bk = (sparse ? 256 : 128) / elt, k_blocks = (K + bk - 1) / bk, pairs = sm_count / 2;
    const int m_tiles = (M + 2 * BM - 1) / (2 * BM);
    const Widths widths = widths_of(pr, elt);
    int forced = only_bn;
    for (int bn : widths.bn)
        if (!forced && bn && bn == g_force_bn) forced = bn;
    LaunchPlan best{0, 1, 0, m_tiles, 0.0, false};
    for (int bn : widths.bn) {
        if (!bn || (forced && bn != forced)) continue;
        const int tiles = m_tiles * ((N + bn - 1) / bn);
        const int whole = tiles / pairs * pairs, tail = tiles - whole;
        TileCost c = tile_cost(pr, elt, bn);
        // grad_X by itself, measured at 110 shapes with every width and split: a 128-wide stage costs more than beside grad_W
        // (few tiles, each paced by its own loads), and an exchange between more than two units 2 us more.  With both the
        // plan is within 0.6 % of the best on the mean and 10 % at worst, without 1.0 and 19 % (4864 x 1152, 640 tokens, bf16:
        // 21.3 -> 17.8 us; 4096 x 1664, 3200: 40.6 -> 38.1).
        const bool dense = pr == GRAD_INPUT && !estimate;
        if (dense && bn == 128) c.stage_us = 0.30;
        const double whole_us = (whole / pairs) * (k_blocks * c.stage_us + c.tile_us);
        for (int s = 1; s <= MAX_SPLITS; ++s) {
            double us = whole_us;
            if (s > 1) {
                // behind whole waves equal ranges only (an uneven split gains less than the exchange costs there)
                if (out_f32 || tail == 0 || k_blocks / s < 8 || (whole > 0 && k_blocks % s != 0)) continue;
                if (s > 4 && (whole > 0 || tail * s > pairs)) continue;      // many ranges: for a few tiles of a long reduction
                if (tail * 2 * 8 * MAX_PARTS > SSTE_SPLITK_TICKETS) continue;
                const size_t bytes = static_cast<size_t>(tail) * s * 2 * BM * bn * sizeof(float);
                if (bytes > partial_bytes) continue;
                us += exchange_us(s, bn, static_cast<double>(bytes)) + (dense && s > 2 ? 2.0 : 0.0);
            }
            if (tail) us += ((tail * s + pairs - 1) / pairs) * ((k_blocks + s - 1) / s * c.stage_us + c.tile_us);
            const bool wanted = (g_force_splits == s && best.bn == bn);      // the hook applies where the shape allows it
            if (!best.bn || us < best.us * (best.bn == bn ? 1.0 : 0.97) || wanted) {
                if (g_force_splits && best.bn == bn && best.splits == g_force_splits) continue;
                best = LaunchPlan{bn, s, s > 1 ? whole : tiles, m_tiles, us, false};
            }
            if (g_force_splits == 1) break;
        }
        for (int s : SUM_SPLITS) {
            const size_t bytes = static_cast<size_t>(tail) * s * 2 * BM * bn * sizeof(float);
            if (g_force_splits || g_inject_stall || out_f32 || whole > 0 || tail * s > pairs || k_blocks / s < 2 || bytes > partial_bytes) break;
            const double us = (k_blocks + s - 1) / s * c.stage_us + c.tile_us + sum_us(s, bn, static_cast<double>(bytes));
            if (us < best.us * (best.bn == bn ? 1.0 : 0.97)) best = LaunchPlan{bn, s, 0, m_tiles, us, true};
        }
    }
    best.group_m = plan_group_m(pr, elt, bcomp, best.bn, pairs, M, N, K);
    return best;
}

LaunchPlan make_plan(Product pr, int elt, int only_bn, bool out_f32, bool bcomp, int sm_count, size_t partial_bytes, int M,
                     int N, int K, bool estimate = false)
{
    if (g_force_splits || g_force_bn || g_force_group_m || g_inject_stall)
        return find_plan(pr, elt, only_bn, out_f32, bcomp, sm_count, partial_bytes, M, N, K, estimate);
    static thread_local PlanMemo<LaunchPlan> memo;
    const long long kind = ((((pr * 4 + elt) * 2 + out_f32) * 2 + bcomp) * 2 + estimate) * 1024 + only_bn;
    return memo.get({kind, sm_count, static_cast<long long>(partial_bytes), M, N, K},
                    [&] { return find_plan(pr, elt, only_bn, out_f32, bcomp, sm_count, partial_bytes, M, N, K, estimate); });
}

// One launch for both gradient products (grads_kernel): the plans of the two and how the pairs share grad_X.
struct JointPlan { LaunchPlan w, x; int pairs; GradsPlan g; double us; };

// grad_W units go round the pairs; the last, partial round leaves `late` pairs busy for one unit more.  For every width,
// split and number of early rounds the model gives the time at which the last pair ends; a pair that changes over from one
// product to the other drains and refills its pipeline (SWITCH_US, about what a kernel boundary costs).
constexpr double SWITCH_US = 2.5, SUM_WAIT_US = 1.5;
JointPlan find_joint_plan(int elt, int sm_count, size_t partial_bytes, int O, int I, int T)
{
    const int max_pairs = sm_count / 2;
    const int wk = (T + 256 / elt - 1) / (256 / elt), xk = (O + 128 / elt - 1) / (128 / elt);      // stages
    const Widths ww = widths_of(GRAD_WEIGHT, elt), xw = widths_of(GRAD_INPUT, elt);
    JointPlan best{};
    double best_rank = 0.0;
    for (int bnw : ww.bn) {
        if (!bnw) continue;
        const TileCost cw = tile_cost(GRAD_WEIGHT, elt, bnw);
        const int w_tiles = ((O + 2 * BM - 1) / (2 * BM)) * ((I + bnw - 1) / bnw);
        for (int bnx : xw.bn) {
            if (!bnx || (bnw == 256 && elt == 2 && bnx == 128)) continue;  // (no kernel for it)
            const TileCost cx = tile_cost(GRAD_INPUT, elt, bnx);
            const int x_tiles = ((T + 2 * BM - 1) / (2 * BM)) * ((I + bnx - 1) / bnx);
            // grad_W whole, split with an exchange (s = 2 .. MAX_SPLITS) or with a sum afterwards (the rest); grad_X whole or with
            // a sum.  Sums are for few tiles whose ranges all run at once; they wait for the last tile of the other product
            // too, which an exchange does not (128 x 2048, 8192 tokens, FP8: 19.1 us with an exchange, 21.4 with a sum): against
            // other plans of one launch they count SUM_WAIT_US more.
            constexpr int SUMS = sizeof(SUM_SPLITS) / sizeof(SUM_SPLITS[0]);
            for (int o = 1; o <= MAX_SPLITS + SUMS; ++o)
            for (int ox = -1; ox < SUMS; ++ox) {
                const bool w_sum = o > MAX_SPLITS;
                const int s = w_sum ? SUM_SPLITS[o - MAX_SPLITS - 1] : o, sx = ox < 0 ? 1 : SUM_SPLITS[ox];
                if (ox >= 0 && (w_tiles * s + x_tiles * sx > max_pairs || xk / sx < 2)) break;
                const double x_us = (xk + sx - 1) / sx * cx.stage_us + cx.tile_us;
                const int x_units = x_tiles * sx;
                const int all = w_tiles * s + x_units, P = all < max_pairs ? all : max_pairs;
                const int whole = w_tiles / P * P, tail = w_tiles - whole;
                const size_t w_bytes = s > 1 ? static_cast<size_t>(tail) * s * 2 * BM * bnw * sizeof(float) : 0;
                const size_t x_bytes = sx > 1 ? static_cast<size_t>(x_tiles) * sx * 2 * BM * bnx * sizeof(float) : 0;
                if (w_bytes + x_bytes > partial_bytes) continue;
                double extra = 0.0, after = 0.0;
                if (w_sum) {
                    if (whole > 0 || w_tiles * s > max_pairs || wk / s < 2) continue;
                } else if (s > 1) {
                    if (tail == 0 || wk / s < 8 || (whole > 0 && wk % s != 0) || tail * s > P) continue;
                    if (tail * 2 * 8 * MAX_PARTS > SSTE_SPLITK_TICKETS) continue;
                    extra = exchange_us(s, bnw, static_cast<double>(w_bytes));
                }
                if (w_sum || sx > 1)
                    after = sum_us(w_sum && s > sx ? s : sx, sx > 1 && (!w_sum || bnx > bnw) ? bnx : bnw,
                                   static_cast<double>((w_sum ? w_bytes : 0) + x_bytes));
                const int late = tail * s;                                  // pairs with one unit more
                const double w_us = wk * cw.stage_us + cw.tile_us;
                const double t_early = (whole / P) * w_us + (whole ? SWITCH_US : 0.0);
                const double t_late = late ? (whole / P) * w_us + (wk + s - 1) / s * cw.stage_us + cw.tile_us + extra + SWITCH_US : 0.0;
                const int n_early = P - late;
                for (int early = 0; early == 0 || (late && n_early && t_early + (early - 1) * x_us < t_late); ++early) {
                    const int rest = x_units - early * n_early;
                    const int rounds = rest > 0 ? (rest + P - 1) / P : 0, last = rest > 0 ? rest - (rounds - 1) * P : 0;
                    for (int ef = 0; ef < 2; ++ef) {
                        // rounds of the early / late pairs: the group that comes second lacks the last one if `last` is short
                        const int r_early = rounds - ((rounds && !ef && last <= late) ? 1 : 0);
                        const int r_late = rounds - ((rounds && ef && last <= n_early) ? 1 : 0);
                        // (a pair that gets no grad_X tile does not change over)
                        double us = n_early ? t_early + (early + r_early ? (early + r_early) * x_us : whole ? -SWITCH_US : 0.0) : 0.0;
                        const double late_us = t_late + (r_late ? r_late * x_us : -SWITCH_US);
                        if (late && late_us > us) us = late_us;
                        us += 0.05 * x_us + after;                          // among equals the shorter tile
                        const double rank = us + (after > 0.0 ? SUM_WAIT_US : 0.0);
                        if (best.pairs && rank >= best_rank - 1e-9) continue;
                        best_rank = rank;
                        best.w = LaunchPlan{bnw, s, s > 1 ? whole : w_tiles, 0, 0.0, w_sum};
                        best.x = LaunchPlan{bnx, sx, sx > 1 ? 0 : x_tiles, 0, 0.0, sx > 1};
                        best.pairs = P;
                        best.g = GradsPlan{late, early, ef};
                        best.us = us;
                    }
                    if (rest <= 0) break;
                }
            }
        }
    }
    best.w.group_m = plan_group_m(GRAD_WEIGHT, elt, false, best.w.bn, best.pairs, O, I, T);
    best.x.group_m = plan_group_m(GRAD_INPUT, elt, false, best.x.bn, best.pairs, T, I, O);
    return best;
}

JointPlan make_joint_plan(int elt, int sm_count, size_t partial_bytes, int O, int I, int T)
{
    if (g_force_splits || g_force_bn || g_force_group_m) return find_joint_plan(elt, sm_count, partial_bytes, O, I, T);
    static thread_local PlanMemo<JointPlan> memo;
    return memo.get({elt, sm_count, static_cast<long long>(partial_bytes), O, I, T},
                    [&] { return find_joint_plan(elt, sm_count, partial_bytes, O, I, T); });
}

// Tensor maps of a launch: A, B, output, metadata (those that it does not use repeat A's).
struct Maps { CUtensorMap a, b, d, m; };
template <bool SPARSE, BMajor BMAJ, int ELT, int BN, bool OUT_T, bool OUT_F32, bool BCOMP>
bool make_maps(const sste_ctx *ctx, const void *A, const void *B, const void *meta, const GemmParams &p, Maps &maps)
{
    using C = Cfg<SPARSE, ELT, BN, BCOMP>;
    constexpr int BK = (SPARSE ? 256 : 128) / ELT;
    // A: compressed values [M, K/2] or [M, K], 128 bytes per row per stage
    bool ok = make_map(ctx, &maps.a, A, ELT, p.M, SPARSE ? p.K / 2 : p.K, SPARSE ? BK / 2 : BK, BM, CU_TENSOR_MAP_SWIZZLE_128B);
    maps.b = maps.d = maps.m = maps.a;
    if (BCOMP) {             // B is expanded from its compressed form by the kernel
    } else if (BMAJ == BMajor::K) {   // B stored [N, K]: sub-tiles of BN/2 rows by 128 bytes of K
        ok = ok && make_map(ctx, &maps.b, B, ELT, p.N, p.K, 128 / ELT, BN / 2, CU_TENSOR_MAP_SWIZZLE_128B);
    } else {                 // B stored [K, N]: chunks of 128 bytes of N by BK rows of K
        ok = ok && make_map(ctx, &maps.b, B, ELT, p.K, p.N, 128 / ELT, BK, CU_TENSOR_MAP_SWIZZLE_128B);
    }
    if (OUT_F32) {           // the fp32 epilogue stores directly
    } else if (OUT_T) {      // out[N, M] bf16: boxes of 64 m x 32 n
        ok = ok && make_map(ctx, &maps.d, p.D, 2, p.N, p.M, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B);
    } else if (C::PANELS == 2) {   // out[M, N] bf16: boxes of 64 n x 32 m
        ok = ok && make_map(ctx, &maps.d, p.D, 2, p.M, p.N, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B);
    } else {                 // out[M, N] bf16: boxes of 32 n x 32 m
        ok = ok && make_map(ctx, &maps.d, p.D, 2, p.M, p.N, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
    }
    if (SPARSE)              // metadata image as rows of 512 bytes, four per atom
        ok = ok && make_map(ctx, &maps.m, meta, 4, static_cast<uint64_t>(p.M / 128) * (p.K / 128) * 4, 128, 128, 4 * C::ATOMS,
                            CU_TENSOR_MAP_SWIZZLE_NONE);
    return ok;
}

// the fields of a launch that its plan decides
void apply_plan(const sste_ctx *ctx, const LaunchPlan &plan, GemmParams &p)
{
    p.wait_limit_ns = WAIT_LIMIT_NS;
    p.skip_last_stage = 0;
    p.group_m = plan.group_m;
    p.splits = plan.splits;
    p.split_from = plan.split_from;
    p.partials = ctx->splitk_partials;
    p.tickets = plan.sum_after ? nullptr : ctx->splitk_tickets;
    p.zero_after = ctx->zero_after;
}

template <int BN>
int split_tiles(const GemmParams &p)
{
    return (p.M + 2 * BM - 1) / (2 * BM) * ((p.N + BN - 1) / BN) - p.split_from;
}

// The sum of a product's partials (the first `tiles` split tiles) and of a second one's.
template <bool OUT_T>
sste_status launch_sum(const GemmParams &p, int bn, int tiles, const GemmParams &p2, int bn2, int tiles2, cudaStream_t stream)
{
    // a thread per four elements: 2 CTAs x 4 row quarters x bn / 4 warps per tile, four warps a block
    const int blocks = tiles * bn / 2, blocks2 = tiles2 * bn2 / 2;
    if (sste_launch(splitk_sum_kernel<OUT_T>, dim3(blocks + blocks2), dim3(128), 0, stream, p, bn, blocks, p2, bn2) != cudaSuccess)
        return SSTE_ERR_CUDA;
    sste_count_launches(1);
    return SSTE_OK;
}

template <int ELT, int BNW, int BNX>
sste_status launch_grads(const sste_ctx *ctx, const void *gvals, const void *gmeta, const void *X, const void *dY, const void *w,
                         GemmParams pw, GemmParams px, const JointPlan &plan, cudaStream_t stream)
{
    Maps mw, mx;
    if (!make_maps<true, BMajor::MN, ELT, BNW, false, false, false>(ctx, gvals, X, gmeta, pw, mw) ||
        !make_maps<false, BMajor::MN, ELT, BNX, false, false, false>(ctx, dY, w, nullptr, px, mx))
        return SSTE_ERR_CUDA;
    auto kern = grads_kernel<ELT, BNW, BNX>;
    constexpr int SMEM = Cfg<true, ELT, BNW>::SMEM_BYTES > Cfg<false, ELT, BNX>::SMEM_BYTES ? Cfg<true, ELT, BNW>::SMEM_BYTES
                                                                                           : Cfg<false, ELT, BNX>::SMEM_BYTES;
    static DeviceOnce attr_done;
    if (!attr_done.run(ctx->device, [&] {
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) == cudaSuccess;
        }))
        return SSTE_ERR_CUDA;
    apply_plan(ctx, plan.w, pw);
    apply_plan(ctx, plan.x, px);
    if (plan.x.sum_after && plan.w.splits > 1)      // behind grad_W's partials
        px.partials += split_tiles<BNW>(pw) * static_cast<size_t>(plan.w.splits) * 2 * BM * BNW;
    if (sste_launch(kern, dim3(2 * plan.pairs), dim3(320), SMEM, stream, mw.a, mw.b, mw.d, mw.m, mx.a, mx.b, mx.d, pw, px,
                    plan.g) != cudaSuccess)
        return SSTE_ERR_CUDA;
    sste_count_launches(1);
    if (plan.w.sum_after) return launch_sum<false>(pw, BNW, split_tiles<BNW>(pw), px, BNX, plan.x.sum_after ? split_tiles<BNX>(px) : 0, stream);
    if (plan.x.sum_after) return launch_sum<false>(px, BNX, split_tiles<BNX>(px), px, BNX, 0, stream);
    return SSTE_OK;
}

template <bool SPARSE, BMajor BMAJ, int ELT, int BN, bool OUT_T, bool OUT_F32, bool BCOMP = false>
sste_status launch(const sste_ctx *ctx, const void *A, const void *B, const void *meta, const GemmParams &p,
                   const LaunchPlan &plan, cudaStream_t stream)
{
    using C = Cfg<SPARSE, ELT, BN, BCOMP>;
    Maps maps;
    if (!make_maps<SPARSE, BMAJ, ELT, BN, OUT_T, OUT_F32, BCOMP>(ctx, A, B, meta, p, maps)) return SSTE_ERR_CUDA;
    auto kern = gemm_kernel<SPARSE, BMAJ, ELT, BN, OUT_T, OUT_F32, BCOMP>;
    // The opt-in to more than 48 KB of dynamic shared memory is a per-DEVICE attribute of the kernel:
    // set once per (instantiation, device), under a lock (contexts may be used from several host threads).
    static DeviceOnce attr_done;
    if (!attr_done.run(ctx->device, [&] {
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES) == cudaSuccess;
        }))
        return SSTE_ERR_CUDA;
    const int m_tiles = (p.M + 2 * BM - 1) / (2 * BM), n_tiles = (p.N + BN - 1) / BN;
    GemmParams pp = p;
    apply_plan(ctx, plan, pp);
    if (g_inject_stall) {
        // Test hook (sste_debug_inject_stall): only a dense product of ONE output tile takes the fault, so that
        // exactly one CTA pair runs into the expired wait; every other launch refuses while the hook is armed.
        if (SPARSE || BCOMP || OUT_F32 || m_tiles * n_tiles != 1) return SSTE_ERR_INVALID_ARG;
        pp.wait_limit_ns = 1000000ull;      // one millisecond
        pp.skip_last_stage = 1;
    }
    if (BCOMP) pp.b_vals = static_cast<const uint8_t *>(B);
    if (pp.out_amax && cudaMemsetAsync(pp.out_amax, 0, sizeof(unsigned int), stream) != cudaSuccess) return SSTE_ERR_CUDA;
    const int tiles = m_tiles * n_tiles;
    const int n_split_tiles = tiles - pp.split_from;
    int pairs = pp.split_from + n_split_tiles * pp.splits;
    if (pairs > ctx->sm_count / 2) pairs = ctx->sm_count / 2;
    if (sste_launch(kern, dim3(2 * pairs), dim3(C::THREADS), C::SMEM_BYTES, stream, maps.a, maps.b, maps.d, maps.m,
                    static_cast<const uint8_t *>(meta), pp) != cudaSuccess)
        return SSTE_ERR_CUDA;
    if (cudaGetLastError() != cudaSuccess) return SSTE_ERR_CUDA;
    sste_count_launches(1);
    if (plan.sum_after) return launch_sum<OUT_T>(pp, BN, n_split_tiles, pp, BN, 0, stream);
    return SSTE_OK;
}

bool fmt_code(sste_dtype dt, int *elt, uint32_t *code)
{
    switch (dt) {
    case SSTE_BF16: *elt = 2; *code = 1; return true;   // kind::f16: 1 = bf16
    case SSTE_E4M3: *elt = 1; *code = 0; return true;   // kind::f8f6f4: 0 = e4m3
    case SSTE_E5M2: *elt = 1; *code = 1; return true;   //               1 = e5m2
    default: return false;
    }
}

// Dispatch on tile width and output dtype.  fp32 output (a test / debug path) always uses 256-wide tiles.
template <Product PR, int ELT>
sste_status launch_out(const sste_ctx *ctx, const void *A, const void *B, const void *meta, const GemmParams &p,
                       sste_dtype odt, cudaStream_t s)
{
    constexpr bool SPARSE = (PR != GRAD_INPUT), OUT_T = (PR == FORWARD);
    constexpr BMajor BMAJ = (PR == FORWARD) ? BMajor::K : BMajor::MN;
    if (odt != SSTE_F32 && odt != SSTE_BF16) return SSTE_ERR_DTYPE;
    const LaunchPlan plan = make_plan(PR, ELT, odt == SSTE_F32 || g_inject_stall ? 256 : 0, odt == SSTE_F32, false, ctx->sm_count,
                                      ctx->splitk_partials ? ctx->splitk_partial_bytes : 0, p.M, p.N, p.K);
    if (odt == SSTE_F32) return launch<SPARSE, BMAJ, ELT, 256, OUT_T, true>(ctx, A, B, meta, p, plan, s);
    if constexpr (PR == FORWARD) {
        if (plan.bn == 224) return launch<SPARSE, BMAJ, ELT, 224, OUT_T, false>(ctx, A, B, meta, p, plan, s);
        if (plan.bn == 192) return launch<SPARSE, BMAJ, ELT, 192, OUT_T, false>(ctx, A, B, meta, p, plan, s);
    }
    if constexpr (PR == FORWARD || ELT == 2) {
        if (plan.bn == 128) return launch<SPARSE, BMAJ, ELT, 128, OUT_T, false>(ctx, A, B, meta, p, plan, s);
    }
    return launch<SPARSE, BMAJ, ELT, 256, OUT_T, false>(ctx, A, B, meta, p, plan, s);
}

// Room for a dense copy of a compressed weight in the last bytes of the workspace, null if the partials in front of it
// would get too little; *partial_bytes: what is left to them.
void *dense_copy_in_workspace(const sste_ctx *ctx, int O, int I, int elt, size_t *partial_bytes)
{
    const size_t dense_bytes = (static_cast<size_t>(O) * I * elt + 255) / 256 * 256;
    if (!ctx->splitk_partials || dense_bytes + SSTE_DENSE_COPY_RESERVE > ctx->splitk_partial_bytes) return nullptr;
    const size_t at = (ctx->splitk_partial_bytes - dense_bytes) / 256 * 256;
    *partial_bytes = at;
    return reinterpret_cast<char *>(ctx->splitk_partials) + at;
}

bool test_hook_set() { return g_inject_stall || g_force_bn || g_force_splits || g_force_group_m; }

// The plan of both gradient products in one launch; whether that beats two in a row, or (beside) two side by side on two streams.
// Two win where the second launch and its own last wave, 5 us, cost less than what tiles lose beside the other product's, some 3 %
// (bf16: 6016 x 1152, 5504 tokens 100 us apart, 104 together; 3840 x 1280, 16384 tokens 183 and 168); the line was drawn over 146
// shapes timed both ways.  A caller that offers a second stream keeps it unless one launch is clearly ahead (512 x 7040, 1792 tokens
// 28.7 us side by side, 21.6 together).  That line is not the fastest one: of the 61 shapes that stay side by side most take 8 % less in
// one launch.
bool joint_wins(const sste_ctx *ctx, int elt, size_t partial_bytes, int O, int I, int T, bool beside, JointPlan *plan)
{
    *plan = make_joint_plan(elt, ctx->sm_count, partial_bytes, O, I, T);
    const double apart = make_plan(GRAD_WEIGHT, elt, 0, false, false, ctx->sm_count, partial_bytes, O, I, T).us +
                         make_plan(GRAD_INPUT, elt, 0, false, false, ctx->sm_count, partial_bytes, T, I, O, true).us;
    return beside ? 1.04 * plan->us <= apart + 3.0 : 1.03 * plan->us <= apart + 5.0;
}

// FP8 operands come with the amax of the tensors they were quantised from (both or neither); bf16 with none.
bool amax_args_ok(int elt, const float *a_amax, const float *b_amax)
{
    return elt == 1 ? (a_amax && b_amax) : (!a_amax && !b_amax);
}

}  // namespace

extern "C" sste_status sste_debug_force_splits(int splits)
{
    if (splits < 0 || splits > 4) return SSTE_ERR_INVALID_ARG;
    g_force_splits = splits;
    return SSTE_OK;
}
extern "C" sste_status sste_debug_plan(int product, sste_dtype opdt, int O, int I, int T, int sm_count,
                                       size_t workspace_bytes, int *tile_width, int *splits, int *split_from,
                                       int *group_m)
{
    int elt;
    uint32_t code;
    if (!fmt_code(opdt, &elt, &code) || product < 0 || product > 2 || sm_count < 2) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(T) || !sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    // the (M, N, K) of the launch, as in the three entry points below
    const int M = product == 2 ? T : O, N = product == 0 ? T : I, K = product == 0 ? I : product == 1 ? T : O;
    const size_t partial_bytes =
        workspace_bytes > SSTE_WS_SPLITK_PARTIALS_OFF + (size_t(1) << 20) ? workspace_bytes - SSTE_WS_SPLITK_PARTIALS_OFF : 0;
    const LaunchPlan plan = make_plan(static_cast<Product>(product), elt, 0, false, false, sm_count, partial_bytes, M, N, K);
    if (tile_width) *tile_width = plan.bn;
    if (splits) *splits = plan.splits;
    if (split_from) *split_from = plan.split_from;
    if (group_m) *group_m = plan.group_m;
    return SSTE_OK;
}
extern "C" sste_status sste_debug_joint_plan(sste_dtype opdt, int O, int I, int T, int sm_count, size_t workspace_bytes, int *out)
{
    int elt;
    uint32_t code;
    if (!fmt_code(opdt, &elt, &code) || sm_count < 2 || !out) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(T) || !sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    const size_t partial_bytes =
        workspace_bytes > SSTE_WS_SPLITK_PARTIALS_OFF + (size_t(1) << 20) ? workspace_bytes - SSTE_WS_SPLITK_PARTIALS_OFF : 0;
    const JointPlan plan = make_joint_plan(elt, sm_count, partial_bytes, O, I, T);
    const int v[12] = {plan.w.bn, plan.w.splits, plan.w.split_from, plan.w.group_m, plan.x.bn,
                       plan.x.group_m, plan.pairs, plan.g.late_pairs, plan.g.early, plan.g.early_first,
                       plan.x.splits, plan.w.sum_after};
    for (int i = 0; i < 12; ++i) out[i] = v[i];
    return SSTE_OK;
}
extern "C" unsigned long long sste_debug_plan_searches(void) { return g_plan_searches.load(std::memory_order_relaxed); }
// Host-only self-check of the once-per-device guard the launches use for per-device kernel attributes: `fn` must
// run once per device ordinal, again after a failure, and never for a device that already succeeded.
extern "C" sste_status sste_debug_selftest_device_once(void)
{
    DeviceOnce once;
    int calls[4] = {0, 0, 0, 0};
    bool fail_next = true;
    auto fn = [&](int dev) {
        return once.run(dev, [&] {
            ++calls[dev];
            if (dev == 2 && fail_next) { fail_next = false; return false; }   // first attempt on device 2 fails
            return true;
        });
    };
    const bool r0 = fn(0), r0b = fn(0), r1 = fn(1), r2 = fn(2), r2b = fn(2), r2c = fn(2), r3 = fn(3), r1b = fn(1);
    const bool ok = r0 && r0b && r1 && !r2 && r2b && r2c && r3 && r1b && calls[0] == 1 && calls[1] == 1 &&
                    calls[2] == 2 && calls[3] == 1;
    return ok ? SSTE_OK : SSTE_ERR_INVALID_ARG;
}
extern "C" sste_status sste_debug_tile_coords(int tile, int m_tiles, int n_tiles, int group_m, int *mt, int *nt)
{
    if (tile < 0 || m_tiles <= 0 || n_tiles <= 0 || group_m <= 0 || tile >= m_tiles * n_tiles || !mt || !nt)
        return SSTE_ERR_INVALID_ARG;
    tile_coords(tile, m_tiles, n_tiles, group_m < m_tiles ? group_m : m_tiles, *mt, *nt);
    return SSTE_OK;
}
extern "C" sste_status sste_debug_force_tile_order(int group_m)
{
    if (group_m < 0) return SSTE_ERR_INVALID_ARG;
    g_force_group_m = group_m;
    return SSTE_OK;
}
extern "C" sste_status sste_debug_inject_stall(int on)
{
    g_inject_stall = on ? 1 : 0;
    return SSTE_OK;
}
extern "C" sste_status sste_debug_force_tile_width(int bn)
{
    if (bn != 0 && bn != 128 && bn != 192 && bn != 224 && bn != 256) return SSTE_ERR_INVALID_ARG;
    g_force_bn = bn;
    return SSTE_OK;
}

extern "C" sste_status sste_linear_fwd(sste_ctx *ctx, const void *X, int T, const void *vals, const void *meta, int O,
                                       int I, sste_dtype opdt, const float *x_amax_dev, const float *w_amax_dev,
                                       void *Y, sste_dtype ydt, float *y_amax_out_dev, void *stream)
{
    if (!ctx || !X || !vals || !meta || !Y) return SSTE_ERR_INVALID_ARG;
    int elt;
    uint32_t code;
    if (!fmt_code(opdt, &elt, &code) || opdt == SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (ydt != SSTE_BF16 && ydt != SSTE_F32) return SSTE_ERR_DTYPE;
    if (!amax_args_ok(elt, w_amax_dev, x_amax_dev)) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(T) || !sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(X, 128) || !sste_aligned(vals, 128) || !sste_aligned(meta, 128) || !sste_aligned(Y, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    // Z^T[O, T] = S(W)[O, I] X^T: M = O, N = T, K = I; the output is stored transposed as Y[T, O]
    GemmParams p{O, T, I, Y, w_amax_dev, x_amax_dev, sste_fp8_max(opdt), sste_fp8_max(opdt),
                 reinterpret_cast<unsigned int *>(y_amax_out_dev), ctx->status_dev, code, code, nullptr};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (elt == 2) return launch_out<FORWARD, 2>(ctx, vals, X, meta, p, ydt, s);
    return launch_out<FORWARD, 1>(ctx, vals, X, meta, p, ydt, s);
}

extern "C" sste_status sste_linear_bwd_weight(sste_ctx *ctx, const void *gvals, const void *gmeta, int O, int T,
                                              sste_dtype gdt, const void *X, int I, sste_dtype xdt,
                                              const float *g_amax_dev, const float *x_amax_dev, void *dW,
                                              sste_dtype dwdt, void *stream)
{
    if (!ctx || !gvals || !gmeta || !X || !dW) return SSTE_ERR_INVALID_ARG;
    int ea, eb;
    uint32_t ca, cb;
    if (!fmt_code(gdt, &ea, &ca) || !fmt_code(xdt, &eb, &cb) || ea != eb) return SSTE_ERR_DTYPE;
    if (gdt == SSTE_E4M3 || xdt == SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (dwdt != SSTE_BF16 && dwdt != SSTE_F32) return SSTE_ERR_DTYPE;
    if (!amax_args_ok(ea, g_amax_dev, x_amax_dev)) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(T) || !sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(X, 128) || !sste_aligned(gvals, 128) || !sste_aligned(gmeta, 128) || !sste_aligned(dW, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    // grad_W[O, I] = G[O, T] X[T, I]: M = O, N = I, K = T; X is [K, N] row-major = MN-major B
    GemmParams p{O, I, T, dW, g_amax_dev, x_amax_dev, sste_fp8_max(gdt), sste_fp8_max(xdt), nullptr,
                 ctx->status_dev, ca, cb, nullptr};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (ea == 2) return launch_out<GRAD_WEIGHT, 2>(ctx, gvals, X, gmeta, p, dwdt, s);
    return launch_out<GRAD_WEIGHT, 1>(ctx, gvals, X, gmeta, p, dwdt, s);
}

extern "C" sste_status sste_linear_bwd_input(sste_ctx *ctx, const void *dY, int T, int O, sste_dtype gdt,
                                             const void *Wt_dense, const void *vals, const void *meta, int I,
                                             sste_dtype wdt, const float *g_amax_dev, const float *w_amax_dev,
                                             void *dX, sste_dtype xdt, float *dx_amax_out_dev, void *stream)
{
    if (!ctx || !dY || !dX) return SSTE_ERR_INVALID_ARG;
    if (!Wt_dense && !(vals && meta)) return SSTE_ERR_INVALID_ARG;
    int ea, eb;
    uint32_t ca, cb;
    if (!fmt_code(gdt, &ea, &ca) || !fmt_code(wdt, &eb, &cb) || ea != eb) return SSTE_ERR_DTYPE;
    if (gdt == SSTE_E4M3 || wdt == SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (xdt != SSTE_BF16 && xdt != SSTE_F32) return SSTE_ERR_DTYPE;
    if (!amax_args_ok(ea, g_amax_dev, w_amax_dev)) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(T) || !sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(dY, 128) || !sste_aligned(Wt_dense, 128) || !sste_aligned(vals, 128) || !sste_aligned(meta, 128) ||
        !sste_aligned(dX, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    // grad_X[T, I] = grad_Z[T, O] S(W)[O, I]: M = T, N = I, K = O; S(W) is [K, N] row-major = MN-major B
    GemmParams p{T, I, O, dX, g_amax_dev, w_amax_dev, sste_fp8_max(gdt), sste_fp8_max(wdt),
                 reinterpret_cast<unsigned int *>(dx_amax_out_dev), ctx->status_dev, ca, cb, nullptr};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!Wt_dense) {
        if (g_inject_stall) return SSTE_ERR_INVALID_ARG;      // the hook is for the dense operand only
        // S(W) from the forward's compressed operand.  Where the workspace has room for the dense copy (in its last bytes;
        // split-K partials stay in front of it), it is expanded there first and the dense product runs on it: the same
        // bits, and one pass over the weight costs little (1280 x 5120, 16384 tokens, bf16: 511 -> 152 us for both).
        size_t partial_bytes = 0;
        if (void *copy = dense_copy_in_workspace(ctx, O, I, ea, &partial_bytes)) {
            const sste_status st = sste_decompress(ctx, vals, meta, O, I, wdt, copy, stream);
            if (st != SSTE_OK) return st;
            sste_ctx rest = *ctx;
            rest.splitk_partial_bytes = partial_bytes;
            if (ea == 2) return launch_out<GRAD_INPUT, 2>(&rest, dY, copy, nullptr, p, xdt, s);
            return launch_out<GRAD_INPUT, 1>(&rest, dY, copy, nullptr, p, xdt, s);
        }
        // else expanded tile by tile in shared memory (256-wide tiles)
        const bool f32 = (xdt == SSTE_F32);
        const LaunchPlan plan = make_plan(GRAD_INPUT, ea, 256, f32, true, ctx->sm_count,
                                          ctx->splitk_partials ? ctx->splitk_partial_bytes : 0, p.M, p.N, p.K);
        if (ea == 2)
            return f32 ? launch<false, BMajor::MN, 2, 256, false, true, true>(ctx, dY, vals, meta, p, plan, s)
                       : launch<false, BMajor::MN, 2, 256, false, false, true>(ctx, dY, vals, meta, p, plan, s);
        return f32 ? launch<false, BMajor::MN, 1, 256, false, true, true>(ctx, dY, vals, meta, p, plan, s)
                   : launch<false, BMajor::MN, 1, 256, false, false, true>(ctx, dY, vals, meta, p, plan, s);
    }
    if (ea == 2) return launch_out<GRAD_INPUT, 2>(ctx, dY, Wt_dense, nullptr, p, xdt, s);
    return launch_out<GRAD_INPUT, 1>(ctx, dY, Wt_dense, nullptr, p, xdt, s);
}

bool sste_bwd_in_one_launch(const sste_ctx *ctx, int elt, int O, int I, int T, bool dense_copy, sste_dtype odt, bool beside)
{
    size_t partial_bytes = ctx->splitk_partials ? ctx->splitk_partial_bytes : 0;
    if (odt != SSTE_BF16 || test_hook_set()) return false;
    if (!dense_copy && !dense_copy_in_workspace(ctx, O, I, elt, &partial_bytes)) return false;
    JointPlan plan;
    return joint_wins(ctx, elt, partial_bytes, O, I, T, beside, &plan);
}

sste_status sste_bwd_products(sste_ctx *ctx, const void *gvals, const void *gmeta, const void *X, const void *dY, int O, int I,
                              int T, sste_dtype gdt, sste_dtype wdt, const void *w_dense, const void *vals, const void *meta,
                              const float *g_amax, const float *x_amax, const float *w_amax, void *dW, void *dX,
                              sste_dtype odt, void *stream)
{
    const int elt = wdt == SSTE_BF16 ? 2 : 1;
    const bool dims_ok = sste_mult128(T) && sste_mult128(O) && sste_mult128(I);
    const bool aligned = sste_aligned(X, 128) && sste_aligned(gvals, 128) && sste_aligned(gmeta, 128) && sste_aligned(dW, 128) &&
                         sste_aligned(dY, 128) && sste_aligned(w_dense, 128) && sste_aligned(vals, 128) &&
                         sste_aligned(meta, 128) && sste_aligned(dX, 128);
    const bool given = ctx && gvals && gmeta && X && dY && dW && dX && (w_dense || (vals && meta)) &&
                       amax_args_ok(elt, g_amax, x_amax) && amax_args_ok(elt, g_amax, w_amax);
    // One launch for bf16 outputs where joint_wins says so; test hooks, fp32 outputs and whatever the single calls refuse go there.
    if (given && dims_ok && aligned && odt == SSTE_BF16 && !test_hook_set()) {
        sste_device_guard guard(ctx->device);
        if (!guard.ok) return SSTE_ERR_CUDA;
        size_t partial_bytes = ctx->splitk_partials ? ctx->splitk_partial_bytes : 0;
        const void *w = w_dense;
        if (!w) {
            if (void *copy = dense_copy_in_workspace(ctx, O, I, elt, &partial_bytes)) {
                const sste_status st = sste_decompress(ctx, vals, meta, O, I, wdt, copy, stream);
                if (st != SSTE_OK) return st;
                w = copy;
            }
        }
        if (w) {
            uint32_t cg, cw;
            int unused;
            fmt_code(gdt, &unused, &cg);
            fmt_code(wdt, &unused, &cw);
            const GemmParams pw{O, I, T, dW, g_amax, x_amax, sste_fp8_max(gdt), sste_fp8_max(wdt), nullptr, ctx->status_dev, cg, cw, nullptr};
            const GemmParams px{T, I, O, dX, g_amax, w_amax, sste_fp8_max(gdt), sste_fp8_max(wdt), nullptr, ctx->status_dev, cg, cw, nullptr};
            cudaStream_t s = static_cast<cudaStream_t>(stream);
            JointPlan plan;
            if (joint_wins(ctx, elt, partial_bytes, O, I, T, false, &plan)) {
                if (elt == 1) return launch_grads<1, 256, 256>(ctx, gvals, gmeta, X, dY, w, pw, px, plan, s);
                if (plan.w.bn == 256) return launch_grads<2, 256, 256>(ctx, gvals, gmeta, X, dY, w, pw, px, plan, s);
                if (plan.x.bn == 256) return launch_grads<2, 128, 256>(ctx, gvals, gmeta, X, dY, w, pw, px, plan, s);
                return launch_grads<2, 128, 128>(ctx, gvals, gmeta, X, dY, w, pw, px, plan, s);
            }
            if (!w_dense) {      // grad_W's partials stay clear of the copy
                sste_ctx rest = *ctx;
                rest.splitk_partial_bytes = partial_bytes;
                sste_status st = elt == 2 ? launch_out<GRAD_WEIGHT, 2>(&rest, gvals, X, gmeta, pw, odt, s)
                                          : launch_out<GRAD_WEIGHT, 1>(&rest, gvals, X, gmeta, pw, odt, s);
                if (st == SSTE_OK)
                    st = elt == 2 ? launch_out<GRAD_INPUT, 2>(&rest, dY, w, nullptr, px, odt, s)
                                  : launch_out<GRAD_INPUT, 1>(&rest, dY, w, nullptr, px, odt, s);
                return st;
            }
        }
    }
    const sste_status st = sste_linear_bwd_weight(ctx, gvals, gmeta, O, T, gdt, X, I, wdt, g_amax, x_amax, dW, odt, stream);
    if (st != SSTE_OK) return st;
    return sste_linear_bwd_input(ctx, dY, T, O, gdt, w_dense, w_dense ? nullptr : vals, w_dense ? nullptr : meta, I, wdt, g_amax,
                                 w_amax, dX, odt, nullptr, stream);
}
