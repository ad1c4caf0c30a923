// GEMM with HiF8 operands decoded in-kernel, for sm_100a (tcgen05 + TMEM + TMA).
//
//   C[m,n] = 2^-(sa+sw) * sum_k value(Aq[m,k]) * value(Wq[k,n])       (Algorithm 1, "MatMul & Restore")
//
// Four kernels behind one entry point, chosen by the sizes and by what fits in the caller's workspace (see choose()):
//   warp     few activation rows and a small weight: every warp alone on a slice of K (hif8_gemm_warp.cuh)
//   narrow   up to 64 activation rows: bound by reading the weight bytes once
//   weights  weights decoded into tensor memory by the tensor-core kernel; the activations come expanded to BF16 from the
//            workspace, or, with no room there or too few of them, as bytes that are decoded in the kernel too
//   pair     both operands expanded to BF16 in the workspace (large products)
//
// Every HiF8 value has at most 4 significant bits and an exponent in [-22, 15], so it is exact in BF16 and every
// product of two of them is exact in the FP32 accumulator of the tensor core.
//
// The operand layout follows the shared-memory matrix descriptor of tcgen05: K-major operands are rows of 64 BF16
// (128 bytes), eight rows form a 1024-byte swizzle atom, 16-byte chunk j of row r is stored at chunk j ^ (r % 8).
// MN-major operands have atoms of 8 k-rows x 64 columns.
//
// Every wait on an mbarrier is bounded; a wait that runs out records a status word and makes all roles leave their
// loops.  Whoever issued copies or MMAs waits for them (again with a limit) before the block leaves and its shared memory may
// become another's; then TMEM is freed.  Copies whose barrier counts other parties too are made waitable by those parties.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "hif8.h"
#include "hif8_host_cache.h"
#include "hif8_internal.cuh"

namespace hif8 {
extern std::atomic<uint64_t> g_launches;

namespace {

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int kEpiWarps = 4, kDecodeWarps = 16;
// The decode warps work in groups, group g on the k-blocks kb = g (mod kDecodeGroups): several k-blocks are in the
// decode stage at once, which covers the latency of each one's lookups, proxy fence and barrier hand-over.  Group g
// owns byte stage g and operand stage g, so every barrier is waited on by one party in program order (a waiter is never
// more than one phase ahead of the barrier, which a parity wait could not tell apart).
constexpr int kDecodeGroups = 4, kGroupWarps = kDecodeWarps / kDecodeGroups, kGroupThreads = kGroupWarps * 32;
constexpr int kThreads = (kEpiWarps + 2 + kDecodeWarps) * 32;  // 704
constexpr int kTmaWarp = 4, kMmaWarp = 5, kFirstDecodeWarp = 6;
constexpr uint32_t kABfBytes = BM * BK * 2, kBBfBytes = (BN / 2) * BK * 2;  // BF16 tiles of one CTA of a pair: 16 KiB + 16 KiB
// tensor memory beside the accumulator: decoded operand stages
constexpr uint32_t kTmemColsAcc = 256, kTmemCols = 512;
constexpr uint32_t kSlotBytes = 16384, kLutBytesWide = 65536, kLutBytesNarrow = 256 * 32 * 4;  // decode tables with rows of 256 and 128 bytes
constexpr uint32_t kSmemBytesMax = 227 * 1024;  // the whole opt-in maximum; kernels that take it check that their layout fits
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s per wait

// ---------------------------------------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// A warp that issues copies or MMAs runs its loop as a whole, waits included, and one elected lane (the same one every time) issues:
// the compiler then keeps descriptors and addresses in uniform registers, which these instructions want.  In a branch of one lane
// four MMAs and their commit took that thread 555 cycles, so 246 (back to back, waits that do not wait; in the narrow kernel it took 1000, and its decode warps
// spent 43 of 101 thousand cycles waiting for MMAs), and a tile copy took 200.  us, a branch of lane 0 / elected: 16 x 28672 x 8192 59.5 / 48.5, 96 x 4096 x 4096 19.3 / 16.7,
// 256 x 1536 x 768 7.9 / 7.0, 201 x 7168 x 4096 19.9 / 18.8, 2048 x 7168 x 4096 101.4 / 96.0, without a workspace 127.8 / 125.5; 48 products in the mean 8 %.
// Whatever ends a loop is agreed on by the warp, since a lane of its own would be waited for at the next election.
__device__ __forceinline__ bool elect_one()
{
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ bool warp_all(bool x) { return __all_sync(0xFFFFFFFFu, x); }
__device__ __forceinline__ bool warp_any(bool x) { return __any_sync(0xFFFFFFFFu, x); }
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0); }
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Returns false when the barrier did not complete in time or another role already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int where,
                                          unsigned long long limit_ns = kWaitLimitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 1;; it++) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                atomicCAS(status, 0, where);
                return false;
            }
        }
    }
}

// Lets the use-th use of a ring of `stages` barriers complete, `bar` its own, within the limit of a wait.
__device__ __forceinline__ void wait_landed(uint32_t bar, int use, int stages)
{
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, (uint32_t)(use / stages) & 1u) && global_ns() - t0 < kWaitLimitNs) {}
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}

// the same with an L2 eviction policy for the lines the copy brings in
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 32 consecutive columns of this thread's tensor-memory lane (lane field of taddr = first lane of the warp's quarter)
__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
// 16 lanes x 32 columns (lane field of taddr = the first of the sixteen): thread t holds, for column octet j, columns
// 8 j + 2 (t % 4) and + 1 of lane t / 4 in r[4 j], r[4 j + 1] and of lane t / 4 + 8 in r[4 j + 2], r[4 j + 3]
__device__ __forceinline__ void tmem_st_16x256b_x4(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---- CTA pairs (cluster of two CTAs, cta_group::2)
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of `addr` (a shared::cta address of this CTA) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Arrival on a barrier of a CTA of the cluster with the default semantics (release at CTA scope).  For the decode warps of
// the fused kernel: what they hand over is read by the tensor core -- tensor memory, ordered by tcgen05.wait::st and
// tcgen05.fence::before_thread_sync, and shared memory, made visible to the async proxy by fence.proxy.async -- not by
// threads of the other CTA.  A release at cluster scope here cost about 2200 cycles per arrival (a per-k-block timeline of
// the groups showed it): it waits for every memory operation the SM has in flight.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// the same, its 16 bytes counted by a barrier of the CTA that gets them
__device__ __forceinline__ void st_async_v4(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t cluster_bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(cluster_addr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(cluster_bar) : "memory");
}

__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t cluster_addr)
{
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
    return v;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// Arrival that publishes nothing: "this CTA is through with what others may now overwrite".  One with release waits for every store
// the SM has in flight, results included (256 x 1536 x 768 split in two: the two such barriers of a call take 1500 and 410 cycles, with
// release 1700 and 1260).  At the end of a kernel it needs that no signal to another CTA is under way that nobody has waited for.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// TMA tile load of a CTA pair: data into this CTA's shared memory, completion on a barrier that may live in the peer.
// The tile comes from matrix c2 of a stack of matrices (three-dimensional tensor map, box one matrix deep).
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar_cluster)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// one-CTA forms (the narrow kernel)
__device__ __forceinline__ void tc_commit_cta(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// one-CTA form with the A operand (128 rows) in tensor memory
__device__ __forceinline__ void tc_mma_bf16_cta_a_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, uint32_t lead = 0)  // arrives on `bar` in both CTAs of the pair lead, lead + 1
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((unsigned short)(3u << lead)) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// the same with the A operand in tensor memory (K-major, row i of each CTA's 128 rows in lane i, two BF16 per column)
__device__ __forceinline__ void tc_mma_bf16_pair_a_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                        uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}


// shared-memory matrix descriptor: start address, leading / stride byte offsets (16-byte units), version 1,
// 128-byte swizzle
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of this architecture
    d |= (uint64_t)2 << 61;  // layout type: 128-byte swizzle
    return d;
}

// BF16 bits of one HiF8 byte (Eq. 1, Eq. 2, specials); used to fill the shared lookup table
__host__ __device__ constexpr uint32_t hif8_to_bf16_bits(uint32_t c)
{
    uint32_t sign = (c & 0x80u) << 8, m = c & 0x7Fu;
    if (m == 0) return sign ? 0x7FC0u : 0u;
    if (m == 0x6F) return sign | 0x7F80u;
    if (m < 8) return sign | ((m + 104u) << 7);
    int E = 0; uint32_t M = 0, w = 0;
    if (m < 0x10)      { E = 0; M = m & 7; w = 3; }
    else if (m < 0x20) { E = 1; M = m & 7; w = 3; if (m & 0x08) E = -E; }
    else if (m < 0x40) { E = 2 | ((m >> 3) & 1); M = m & 7; w = 3; if (m & 0x10) E = -E; }
    else if (m < 0x60) { E = 4 | ((m >> 2) & 3); M = m & 3; w = 2; if (m & 0x10) E = -E; }
    else               { E = 8 | ((m >> 1) & 7); M = m & 1; w = 1; if (m & 0x10) E = -E; }
    return sign | ((uint32_t)(E + 127) << 7) | (M << (7 - w));
}

struct Bf16OfCode { uint16_t v[256]; };
constexpr Bf16OfCode make_bf16_of_code()
{
    Bf16OfCode t{};
    for (uint32_t c = 0; c < 256; c++) t.v[c] = (uint16_t)hif8_to_bf16_bits(c);
    return t;
}
__device__ const Bf16OfCode g_bf16_of_code = make_bf16_of_code();

// Fills the decode table: entry (code c, lane l) at word c * ROW_WORDS + l holds the BF16 bits of code c (one copy per
// lane, so that a warp's lookups never meet in a bank).  A warp writes four rows per step, eight lanes with 16 bytes each to
// a row; STEPS steps, their values loaded together (three for the 22 warps or more of most blocks).  (What runs once at the head
// of a kernel costs its instruction fetches above all, so the values come from a table in global memory and not from the
// field definitions: 1050 -> 600 cycles; eight warps with 32 codes each, handed round by shuffles, took 1300.)
template <int ROW_WORDS, int STEPS = 3>
__device__ __forceinline__ void fill_decode_table(uint32_t* table, int warp, int lane, int n_warps)
{
    uint32_t v[STEPS];
#pragma unroll
    for (int k = 0; k < STEPS; k++) {
        const int i = warp + k * n_warps;
        v[k] = i < 64 ? __ldg(g_bf16_of_code.v + 4 * i + (lane >> 3)) : 0u;
    }
#pragma unroll
    for (int k = 0; k < STEPS; k++) {
        const int i = warp + k * n_warps;
        if (i < 64) *reinterpret_cast<uint4*>(table + (4 * i + (lane >> 3)) * ROW_WORDS + (lane & 7) * 4) = make_uint4(v[k], v[k], v[k], v[k]);
    }
}
static_assert(3 * (kThreads / 32) >= 64, "three steps fill the table");

// Shared-memory accesses by 32-bit shared-window address: the operand ring lives at a run-time offset inside the dynamic
// allocation, and spelling the state space out keeps every one of these an LDS / STS (never a generic access).
// (not volatile: the table is constant once it is built and every address derives from a byte read after the barrier
// wait, so the compiler is free to issue a whole batch of lookups before the first of them is consumed)
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint2 lds_v2(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
// Two 16 x 16 byte matrices, transposed: lane l gives the address of row l % 16 of matrix l / 16 (16 bytes); thread t gets
// bytes 4 (t % 4) .. + 3 of the first matrix's column t / 4 in v.x and of its column t / 4 + 8 in v.y, the second one's in
// v.z and v.w.
__device__ __forceinline__ uint4 ldmatrix_trans_bytes_x2(uint32_t addr)
{
    uint4 v;
    asm volatile("ldmatrix.sync.aligned.m16n16.x2.trans.shared.b8 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// eight HiF8 bytes -> eight BF16 (one 16-byte operand chunk) through the lane-replicated table: lane L only ever touches
// shared-memory bank L, so the lookups of a warp instruction never conflict.  `lut_lane` is the shared address of this
// lane's column.  ROW_SHIFT = 7: rows of 128 bytes, entry of byte c at lut_lane + 128 c (extract, scale, add).
// ROW_SHIFT = 8: rows of 256 bytes in a table that starts on a 64 KiB boundary of the shared window, so that bits 8-15 of
// lut_lane are zero and ONE byte permute drops the code into them: address = lut_lane with byte 1 replaced by c.
template <int ROW_SHIFT>
__device__ __forceinline__ uint4 decode8(uint2 v, uint32_t lut_lane)
{
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const uint32_t w = i < 2 ? v.x : v.y;
        if (ROW_SHIFT == 8) {
            const uint32_t a0 = __byte_perm(w, lut_lane, (i & 1) ? 0x7624 : 0x7604), a1 = __byte_perm(w, lut_lane, (i & 1) ? 0x7634 : 0x7614);
            o[i] = __byte_perm(lds_u32(a0), lds_u32(a1), 0x5410);
        } else {
            const uint32_t c0 = (w >> (16 * (i & 1))) & 0xFFu, c1 = (w >> (16 * (i & 1) + 8)) & 0xFFu;
            o[i] = __byte_perm(lds_u32(lut_lane + c0 * 128), lds_u32(lut_lane + c1 * 128), 0x5410);
        }
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// Groups of `group` tile-rows sweep N together: their W tiles stay in L2 (8 in the weights kernel, whose kGroupPieces is the same number; the pair kernel says its own).
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int& tile_m, int& tile_n, int group = 8)
{
    const int per_group = group * tiles_n;
    const int g = t / per_group, first_m = g * group;
    const int rows_in_group = min(group, tiles_m - first_m);
    tile_m = first_m + (t % per_group) % rows_in_group;
    tile_n = (t % per_group) / rows_in_group;
}


// One 32-column chunk of one accumulator row, descaled by f1 * f2 (two exact powers of two), added to BF16 results that are
// there already and rounded to nearest even; rows / columns outside the matrix are skipped.
__device__ __forceinline__ void add_chunk_bf16(const GemmParams& p, int row, int col, const uint32_t (&r)[32], float f1, float f2)
{
    if (row >= p.M || col >= p.N) return;
    const bool full = col + 32 <= p.N;
    unsigned short* out = reinterpret_cast<unsigned short*>(p.C) + (long long)row * p.ldc + col;
    uint32_t h[32];  // previous contents of C, widened exactly
    if (full) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
            const uint4 c = __ldcs(reinterpret_cast<const uint4*>(out + i));
            h[i] = c.x << 16; h[i + 1] = c.x & 0xFFFF0000u; h[i + 2] = c.y << 16; h[i + 3] = c.y & 0xFFFF0000u;
            h[i + 4] = c.z << 16; h[i + 5] = c.z & 0xFFFF0000u; h[i + 6] = c.w << 16; h[i + 7] = c.w & 0xFFFF0000u;
        }
    } else {
        // (every index a compile-time constant: a loop that stops at the ragged edge would index the chunk by a
        // variable and put it, for all paths, into local memory -- which has next to no L1 behind it in these kernels)
#pragma unroll
        for (int i = 0; i < 32; i++) h[i] = (col + i < p.N) ? (uint32_t)out[i] << 16 : 0u;
    }
    uint32_t pk[16];  // two BF16 per word, rounded to nearest even by the conversion instruction (a NaN stays a NaN)
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const float v0 = __uint_as_float(r[i]) * f1 * f2 + __uint_as_float(h[i]), v1 = __uint_as_float(r[i + 1]) * f1 * f2 + __uint_as_float(h[i + 1]);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[i >> 1]) : "f"(v1), "f"(v0));  // first source -> upper half
    }
    if (full) {
#pragma unroll
        for (int i = 0; i < 16; i += 4)
            __stcs(reinterpret_cast<uint4*>(out + 2 * i), make_uint4(pk[i], pk[i + 1], pk[i + 2], pk[i + 3]));
    } else {
#pragma unroll
        for (int i = 0; i < 32; i++)
            if (col + i < p.N) out[i] = (unsigned short)(pk[i >> 1] >> (16 * (i & 1)));
    }
}

// A chunk, descaled and rounded to BF16, into a staging tile in shared memory from which a tile store writes C:
// boxes of 64 columns x 128 rows in the 128-byte-swizzled layout of the tensor map (16-byte piece j of row r sits at
// piece j ^ (r % 8) of its 128-byte line; lines of eight rows form 1024-byte atoms).  `piece0` = first 16-byte piece of
// the chunk within its row of the box (0 or 4).  A thread's four stores hit four different pieces; the eight rows of an
// atom hit eight different ones: no bank conflicts.
__device__ __forceinline__ void stage_chunk_bf16(uint32_t box, int row, int piece0, const uint32_t (&r)[32], float f1, float f2)
{
    const uint32_t line = box + (uint32_t)(row >> 3) * 1024u + (uint32_t)(row & 7) * 128u;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        uint32_t pk[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float v0 = __uint_as_float(r[8 * i + 2 * j]) * f1 * f2, v1 = __uint_as_float(r[8 * i + 2 * j + 1]) * f1 * f2;
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(v1), "f"(v0));
        }
        sts_v4(line + ((uint32_t)((piece0 + i) ^ (row & 7)) << 4), make_uint4(pk[0], pk[1], pk[2], pk[3]));
    }
}
// tile store shared -> global (clipped at the edges of the matrix); the caller commits and waits for the group
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1) : "memory");
}

// Per-channel weight scales: multiply column col + i of the chunk by 2^-(sa + sw[col + i]).  Lane L fetches the
// exponent of column col + L once; every lane then walks the 32 columns of its own row.
__device__ __forceinline__ void apply_channel_scale(const GemmParams& p, int col, int lane, int sa, uint32_t (&r)[32])
{
    const int mine = (col + lane < p.N) ? -(sa + __ldg(p.d_sw_channel + col + lane)) : 0;
#pragma unroll
    for (int i = 0; i < 32; i++) {
        const int s = __shfl_sync(0xFFFFFFFFu, mine, i);
        const int s1 = s / 2, s2 = s - s1;
        r[i] = __float_as_uint(__uint_as_float(r[i]) * __uint_as_float((uint32_t)(s1 + 127) << 23) *
                               __uint_as_float((uint32_t)(s2 + 127) << 23));
    }
}

#include "hif8_gemm_warp.cuh"

// ---------------------------------------------------------------------------------------------------------
// Narrow products (M <= 64 rows of activations: the decode phase of inference).  The product is bound by reading the
// weight bytes once, so the roles are swapped: a CTA streams a slab of 128 weight columns as the 128-row MMA operand and
// the few activation rows are the narrow operand (MMA N = M rounded up to 16).  One CTA per SM, no pairs:
//   warp 4        copies: per pair block (two k-blocks) one tile of weight bytes and one of activation bytes
//                 (activations expanded to BF16 beforehand, when the workspace has room: their tiles instead, one per
//                 k-block, straight into the operand stages; the groups then decode weights only)
//   warps 6-21    four decode groups, group g on the k-blocks it = g (mod 4): a thread owns one weight column of the slab,
//                 decodes its 64 bytes of the k-block and stores them as its lane of a weight stage in tensor memory (the A
//                 operand of tcgen05.mma may live there); the group also decodes the activation tile into shared memory
//   warps 5, 22-24  MMA issuers (below)
//   warps 0-3     epilogue
// The accumulator holds C transposed (row = weight column n, column = activation row m); the epilogue writes C[m][n] with
// consecutive lanes on consecutive n.
// ---------------------------------------------------------------------------------------------------------
constexpr int kNarrowMaxM = 64;
constexpr uint32_t kNwW8 = BM * BK;  // weight bytes of a k-block: 8 KiB
// A copy brings two k-blocks (a "pair block": 128 bytes of k) of weights and of activations: a tile copy costs the same whatever its size.
constexpr int BK2 = 2 * BK;
// Byte stages (one pair block of weights each, and of activations when they are bytes).  The weight stream needs about
// 64 KiB per SM in flight for the rate of HBM, so six stages of 16 KiB where they fit: with four, and with the
// activation tiles issued by the thread that issues the weight copies (which then waited for MMAs before it asked for the next weights), a kernel without any lookups still took 54 of 63 us at 16 x 28672 x 8192; now 59 us with them (64 rows:
// 72 -> 67 us).  The number is even: each decode group then meets the same stages in every round.
constexpr int kNwMaxByteStages = 6, kNwMinByteStages = 4;
// Operand stages (32 tensor-memory columns of weights + mp rows of activations in shared memory each): two per group, so
// that a group starts its next k-block without waiting for the MMAs of its previous one
constexpr int kNwTmemStages = 2 * kDecodeGroups;
constexpr uint32_t kNwBars = 2 * kNwMaxByteStages + 2 * kNwTmemStages + 4;
// Where the narrow kernel keeps what (mp activation rows).  WIDE:
// the decode table has rows of 256 bytes and starts on a 64 KiB boundary of the shared window, so that one byte permute makes
// a lookup's address (see decode8); operand stages and then byte stages as they fit in front of it, the rest behind it.
// Otherwise: operand stages, byte stages and the 32 KiB table in a row, for more than 48 rows of activations given as bytes, beside which
// the larger table does not fit.  (With rows of 128 bytes a lookup's address takes three instructions: 16 x 28672 x 8192 with
// activations as bytes 75.9 us a call, with the larger table 68.2, and with their decode as a loop in front of the weights 61.7.)
constexpr int kNwWideBytesM = 48;
template <bool WIDE, bool ACT_BF16>
struct NarrowSmem {
    uint32_t base, lut, bars, end;  // shared-window addresses; base is 1024-byte aligned
    uint32_t behind_act, behind_u8, front_u8, act_bytes, u8_bytes;
    int act_front, u8_front, stages8;
    __device__ NarrowSmem(uint32_t raw, uint32_t limit, int mp)
    {
        base = (raw + 1023u) & ~1023u;
        act_bytes = ((uint32_t)mp * BK * 2u + 1023u) & ~1023u;
        u8_bytes = 2 * kNwW8 + (ACT_BF16 ? 0u : ((uint32_t)mp * BK2 + 1023u) & ~1023u);
        stages8 = kNwMaxByteStages;
        place();
        if (end > limit) { stages8 = kNwMinByteStages; place(); }
    }
    __device__ void place()
    {
        if (!WIDE) {
            act_front = kNwTmemStages; u8_front = stages8; behind_act = behind_u8 = 0;
            front_u8 = base + kNwTmemStages * act_bytes;
            lut = front_u8 + (uint32_t)stages8 * u8_bytes;
            bars = lut + kLutBytesNarrow;
        } else {
            lut = (base + kLutBytesWide - 1) & ~(kLutBytesWide - 1);
            const uint32_t front = lut - base;
            act_front = kNwTmemStages;
            while ((uint32_t)act_front * act_bytes > front) act_front--;
            front_u8 = base + (uint32_t)act_front * act_bytes;
            u8_front = (int)min((lut - front_u8) / u8_bytes, (uint32_t)stages8);
            behind_act = lut + kLutBytesWide;
            behind_u8 = behind_act + (uint32_t)(kNwTmemStages - act_front) * act_bytes;
            bars = behind_u8 + (uint32_t)(stages8 - u8_front) * u8_bytes;
        }
        end = bars + kNwBars * 8 + 8;
    }
    __device__ uint32_t bf(int s) const { return s < act_front ? base + (uint32_t)s * act_bytes : behind_act + (uint32_t)(s - act_front) * act_bytes; }
    __device__ uint32_t u8(int s) const { return s < u8_front ? front_u8 + (uint32_t)s * u8_bytes : behind_u8 + (uint32_t)(s - u8_front) * u8_bytes; }
    __device__ uint32_t tmem_slot() const { return bars + kNwBars * 8; }
    __device__ uint32_t abort_flag() const { return tmem_slot() + 4; }
};
// Tensor memory: the accumulators (two per issuer: the epilogue of one segment overlaps the next segment's MMAs), then
// one weight stage (128 rows x 64 BF16 = 32 columns) per operand stage.
// MMA issuers: four warps share the k-blocks, issuer q taking the k-blocks it = q (mod issuers) into accumulators of its own, which the
// epilogue adds (one lane that waited, issued and committed was busy 1000 cycles per k-block; see elect_one).  Up to 32
// activation rows every issuer has two accumulators, above that one: issuers x buffers x rows stays within 256 columns.
constexpr int kNwMaxIssuers = 4;
constexpr int kNwMaxSplit = 8;
// the first issuer is the MMA warp of the other kernels; the warp behind the others copies expanded activations
constexpr int kNwActWarp = kThreads / 32 + kNwMaxIssuers - 1, kThreadsN = (kNwActWarp + 1) * 32;  // 832
constexpr uint32_t kTmemAccN = 2 * 2 * kNarrowMaxM, kTmemColsN = 512;
static_assert(kTmemAccN + kNwTmemStages * (BK / 2) <= kTmemColsN, "weight stages fit beside the accumulators");
static_assert(2 * kNwMaxIssuers * 32 <= kTmemAccN, "four issuers x two buffers x 32 rows");

// Work split of the narrow kernel.  The unit is a pair block (two k-blocks; the second one of a slab's last pair may lie
// beyond K, where the copies fill zeros).  The (slab, pair block) units are numbered slab-major, and CTA c of G takes a
// contiguous range of q or q + 1 of them (the first `rem` CTAs one more): every SM streams the same number of weight bytes
// whatever the number of slabs.  A range cuts slabs into segments.  A segment that covers its whole slab is finished by
// its CTA; otherwise the CTA stores its FP32 partial sums as slice (slab, its position among the slab's contributors),
// and the last contributor to arrive (one ticket per slab and epilogue warp) adds the slices in position order - so the
// result does not depend on arrival order - and writes C.
// Few slabs go another way: a cluster of CTAs per slab, each an equal part of its pair blocks; the partial sums are exchanged
// through distributed shared memory and added in rank order.  Nothing of that is in the workspace, and after the last MMA it
// takes 4000 cycles where slices, tickets and a reduction by one warp take 8000 (16 rows) to 22000 (64 rows).  us a call: 64 x
// 4096 x 4096 21.2 -> 12.8, 16 rows 12.9 -> 11.4; with room for the status word only, where a slab had one CTA: 26.8 -> 12.4.
// (Everything in 32 bits, q and rem from the host: N K < 2^45 bytes, so slabs * pair blocks < 2^31.  What a call costs
// beyond its weight bytes is latency: with 64-bit products and divisions in the kernel, exponents loaded after the sums
// were complete, one accumulator read per wait and the first copies issued behind the table set-up, 16 x 512 x 512 took
// 10.2 us a call, 14.1 us with room for the status word only; now 7.5 and 10.3 us.  16 x 28672 x 8192: 67.7 -> 65.5 us.)
struct NarrowPlan {
    int q, rem;          // units per CTA; the first rem CTAs take one more
    float* part;         // [slab][pmax][mp][128] partial sums, or nullptr when every range is made of whole slabs
    unsigned* tickets;   // [slab][4], zero at launch
    int pmax;            // slices per slab
    int clear_status;    // nonzero: no launch in front of this one clears the status word
    int split;           // above 1: a cluster of `split` CTAs per slab, each a part of its pair blocks (see below)

    __device__ int first(int c) const { return c * q + (c < rem ? c : rem); }  // first unit of CTA c
    __device__ int owner(int x) const                                          // the CTA that takes unit x
    {
        const int cut = rem * (q + 1);
        return x < cut ? x / (q + 1) : rem + (x - cut) / q;
    }
};

// In front of the kernels that read expanded activations: the activations [M,K] (contiguous bytes) to BF16, and the status
// word (and the narrow kernel's tickets) cleared, in one launch.  It may itself start while the launch before it drains; its
// dependents may start once that one is complete (they read weights and exponents at once, and wait for this grid's
// completion before they read what it writes).
__global__ void __launch_bounds__(256) expand_activations_kernel(const uint4* __restrict__ a, uint4* __restrict__ a_bf, unsigned long long n_vec,
                                                                 uint32_t* __restrict__ clear, unsigned clear_words)
{
    __shared__ uint32_t lut[256];
    lut[threadIdx.x] = hif8_to_bf16_bits(threadIdx.x);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0)
        for (unsigned i = threadIdx.x; i < clear_words; i += 256) clear[i] = 0u;
    for (unsigned long long u = (unsigned long long)blockIdx.x * 256 + threadIdx.x; u < n_vec; u += (unsigned long long)gridDim.x * 256) {
        const uint4 v = a[u];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t o[8];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            o[2 * i] = lut[w[i] & 0xFFu] | (lut[(w[i] >> 8) & 0xFFu] << 16);
            o[2 * i + 1] = lut[(w[i] >> 16) & 0xFFu] | (lut[w[i] >> 24] << 16);
        }
        a_bf[2 * u] = make_uint4(o[0], o[1], o[2], o[3]);
        a_bf[2 * u + 1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// The same for many activations, with a table that has a copy per lane (the conflicts of one table for all lanes take longer than the
// transfer): 2048 x 4096 x 7168 with the activations expanded 97.1 -> 94.8 us, 2048 x 7168 x 4096 98.9 -> 97.4.  Below four million it
// has too few blocks, each with a table to fill (1024 x 4096 x 2048 21.3 / 21.4).
constexpr int kExpandThreads = 512, kExpandUnroll = 4;
constexpr unsigned long long kExpandStreamFrom = 1ull << 22;
__global__ void __launch_bounds__(kExpandThreads) expand_activations_stream_kernel(const uint2* __restrict__ a, uint4* __restrict__ a_bf, unsigned long long n_vec,
                                                                                   uint32_t* __restrict__ clear, unsigned clear_words)
{
    __shared__ __align__(16) uint32_t table[kLaneTableWords];
    fill_lane_table(table, hif8_to_bf16_bits(threadIdx.x & 255u));
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0)
        for (unsigned i = threadIdx.x; i < clear_words; i += kExpandThreads) clear[i] = 0u;
    const uint32_t lane4 = (threadIdx.x & 31u) * 4u;
    const unsigned long long u0 = (unsigned long long)blockIdx.x * (kExpandThreads * kExpandUnroll) + threadIdx.x;
    uint2 v[kExpandUnroll];
#pragma unroll
    for (int i = 0; i < kExpandUnroll; i++) v[i] = u0 + i * kExpandThreads < n_vec ? a[u0 + i * kExpandThreads] : make_uint2(0u, 0u);
#pragma unroll
    for (int i = 0; i < kExpandUnroll; i++) {
        const uint2 lo = lane_lookup4(table, v[i].x, lane4), hi = lane_lookup4(table, v[i].y, lane4);
        if (u0 + i * kExpandThreads < n_vec) a_bf[u0 + i * kExpandThreads] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
}

template <bool W_IS_NK, bool ACT_BF16, bool CLUSTER, bool WIDE>
__global__ void __launch_bounds__(kThreadsN, 1)
hif8_gemm_narrow_kernel(const __grid_constant__ CUtensorMap map_act, const __grid_constant__ CUtensorMap map_w, const GemmParams p, int mp,
                        const NarrowPlan plan)
{
    extern __shared__ unsigned char smem_raw[];
    constexpr int kLutShiftN = WIDE ? 8 : 7;
    uint32_t dyn_bytes;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
    // (a wait that gives up does so two seconds into the kernel, long after this; a separate launch cost 2 us)
    if (!ACT_BF16 && plan.clear_status && blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int*>(p.status) = 0;
    const NarrowSmem<WIDE, ACT_BF16> lay(smem_u32(smem_raw), smem_u32(smem_raw) + dyn_bytes, mp);
    unsigned char* sm = smem_raw - smem_u32(smem_raw);  // generic pointer of shared-window address 0
    {
        if (lay.end > smem_u32(smem_raw) + dyn_bytes) {  // the layout does not fit (the same answer in every thread)
            if (ACT_BF16) asm volatile("griddepcontrol.wait;" ::: "memory");  // (the launch in front clears the status word)
            if (threadIdx.x == 0) atomicCAS(p.status, 0, 7);
            return;
        }
    }
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    constexpr int S = kNwTmemStages;  // operand ring: the it-th k-block uses stage it % S
    static_assert(S % kDecodeGroups == 0, "an operand stage is always written by the same group");
    const int S8 = lay.stages8;         // byte ring: the i-th pair block of this CTA lands in stage i % S8
    constexpr int kS8 = kNwMaxByteStages;
    constexpr uint32_t kU8Act = 2 * kNwW8;  // byte stage: 128 weight columns x 128 k, then (activations as bytes) act rows x 128 k
    const uint32_t bars = lay.bars;
    auto bar_u8_full = [&](int s) { return bars + 8u * s; };
    auto bar_u8_empty = [&](int s) { return bars + 8u * (kS8 + s); };
    auto bar_bf_full = [&](int s) { return bars + 8u * (2 * kS8 + s); };
    auto bar_bf_empty = [&](int s) { return bars + 8u * (2 * kS8 + S + s); };
    auto bar_acc_full = [&](int b) { return bars + 8u * (2 * kS8 + 2 * S + b); };
    auto bar_acc_empty = [&](int b) { return bars + 8u * (2 * kS8 + 2 * S + 2 + b); };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + lay.abort_flag());
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + lay.tmem_slot());
    uint32_t* lut_all = reinterpret_cast<uint32_t*>(sm + lay.lut);
    const uint32_t lut = lay.lut + 4u * lane;
    const int num_pb = (p.K + BK2 - 1) / BK2, num_kb = 2 * num_pb;  // per slab
    // this CTA's (slab, pair block) range: where it starts, and its length
    const int split = CLUSTER ? plan.split : 1, part = CLUSTER ? (int)cluster_ctarank() : 0;
    int slab0, pb0, n_pairs;
    if (CLUSTER) {
        slab0 = (int)blockIdx.x / split;
        pb0 = num_pb * part / split;
        n_pairs = num_pb * (part + 1) / split - pb0;
    } else {
        const int pair0 = plan.first((int)blockIdx.x);
        slab0 = pair0 / num_pb; pb0 = pair0 - slab0 * num_pb;
        n_pairs = plan.first((int)blockIdx.x + 1) - pair0;
    }
    const int n_it = 2 * n_pairs;
    const uint32_t act_bytes = (uint32_t)mp * BK2;
    // Up to 32 activation rows every issuer has two accumulators (the epilogue of one segment overlaps the next segment's
    // MMAs).  Above that issuers x buffers x rows must stay within 256 columns, and four issuers with one accumulator each
    // are faster than two with two (91 against 94 us at 64 x 28672 x 8192 when that was the whole call).
    constexpr int issuers = kNwMaxIssuers;
    const int bufs = mp <= 32 ? 2 : 1;
    auto acc_col = [&](int q, int buf) { return (uint32_t)((q * bufs + buf) * mp); };  // accumulator of issuer q, buffer buf

    // (the whole copying warp) copies of the range's next unit: its weight bytes (and, as bytes, its activations) into stage s
    int cp_slab = slab0, cp_pb = pb0;
    auto copy_bytes = [&](int s) {
        const uint32_t dst_w = lay.u8(s), dst_a = dst_w + kU8Act;
        const uint64_t w_policy = l2_policy_evict_first();
        if (elect_one()) {
            mbar_arrive_expect_tx(bar_u8_full(s), 2 * kNwW8 + (ACT_BF16 ? 0u : act_bytes));
            // (the weight is read once: its lines are the first to leave L2 again, so that the expanded activations, which
            // every CTA reads, and the slices of the slabs that two CTAs share stay there)
            if (W_IS_NK) tma_load_2d_hint(dst_w, &map_w, cp_pb * BK2, cp_slab * BM, bar_u8_full(s), w_policy);
            else tma_load_2d_hint(dst_w, &map_w, cp_slab * BM, cp_pb * BK2, bar_u8_full(s), w_policy);
            if (!ACT_BF16) tma_load_2d(dst_a, &map_act, cp_pb * BK2, 0, bar_u8_full(s));
        }
        if (++cp_pb == num_pb) { cp_pb = 0; cp_slab++; }
    };
    const int n_early = min(2, n_pairs);
    if (warp == kTmaWarp) {
        if (elect_one()) {
            for (int s = 0; s < S8; s++) { mbar_init(bar_u8_full(s), 1); mbar_init(bar_u8_empty(s), 2 * kGroupWarps); }  // both halves' groups
            // operands ready: the group's warps, plus (ACT_BF16) the announcement of the activation tile's bytes
            for (int s = 0; s < S; s++) { mbar_init(bar_bf_full(s), kGroupWarps + (ACT_BF16 ? 1 : 0)); mbar_init(bar_bf_empty(s), 1); }
            for (int b = 0; b < 2; b++) { mbar_init(bar_acc_full(b), issuers); mbar_init(bar_acc_empty(b), kEpiWarps); }
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        // The first byte copies start here, under the table set-up (two of them: the block waits for this warp): nothing in front of this kernel writes the
        // operands (the launch before it writes the expanded activations and the cleared words only, and that launch itself
        // waits for everything before it).
        for (int i = 0; i < n_early; i++) copy_bytes(i);
    }
    fill_decode_table<(1 << (kLutShiftN - 2))>(lut_all, warp, lane, kThreadsN / 32);  // rows of 1 << kLutShiftN bytes
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(lay.tmem_slot()), "r"(kTmemColsN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // The launch in front of this kernel expands the activations and clears the status word and the tickets; this kernel was
    // started while that one ran, so that the set-up above overlaps it.  From here on its results are complete.
    // (Not the weight producer: it reads none of them.)
    if (ACT_BF16 && warp != kTmaWarp) asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == kTmaWarp) {
        int issued = n_early, s = n_early;
        uint32_t ph = 1;  // parity of the round before the one that fills stage s next
        for (int it = n_early; it < n_pairs; it++) {
            if (it >= S8 && !warp_all(mbar_wait(bar_u8_empty(s), ph, abort_flag, p.status, 31))) break;
            if (warp_any(*abort_flag)) break;
            copy_bytes(s);
            issued = it + 1;
            if (++s == S8) { s = 0; ph ^= 1u; }
        }
        if (*abort_flag)
            for (int it = max(0, issued - S8); it < issued; it++) wait_landed(bar_u8_full(it % S8), it, S8);
    } else if (warp == kNwActWarp) {
        // Activations expanded to BF16 beforehand (map_act is then the map of that copy): the tile of every k-block goes
        // straight into its operand stage, in the 128-byte-swizzled layout the MMA reads, once the MMAs of the stage's
        // previous use have read it.
        if (ACT_BF16) {
            int issued = 0, kb = 2 * pb0;
            for (int it = 0; it < n_it; it++) {
                const int sb = it % S, rb = it / S;
                if (rb > 0 && !warp_all(mbar_wait(bar_bf_empty(sb), (rb - 1) & 1, abort_flag, p.status, 37))) break;
                if (warp_any(*abort_flag)) break;
                const uint32_t dst = lay.bf(sb);
                if (elect_one()) {
                    mbar_arrive_expect_tx(bar_bf_full(sb), (uint32_t)mp * BK * 2u);
                    tma_load_2d(dst, &map_act, kb * BK, 0, bar_bf_full(sb));
                }
                issued = it + 1;
                if (++kb == num_kb) kb = 0;
            }
            if (*abort_flag)
                for (int it = max(0, issued - S); it < issued; it++) wait_landed(bar_bf_full(it % S), it, S);
        }
    } else if (warp == kMmaWarp || warp >= kFirstDecodeWarp + kDecodeWarps) {
        const int q = warp == kMmaWarp ? 0 : warp - (kFirstDecodeWarp + kDecodeWarps) + 1;  // issuer number
        if (q < issuers) {
            // FP32 accumulator, BF16 operands; A = weight slab (K-major for [N,K] weights, MN-major for [K,N]), B = activations
            // (K-major), N = mp, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(mp >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            // descriptor of stage 0; a stage or a 16-k step further on adds to the address field only
            const uint64_t da0 = make_smem_desc(lay.bf(0), 16, 1024);
            bool ok = true, first = true;
            int kb = 2 * pb0, seg = 0, it = 0;
            for (; it < n_it && ok; it++) {
                const int buf = bufs == 2 ? seg & 1 : 0, use = bufs == 2 ? seg >> 1 : seg;  // use: how often the buffer was filled before
                if ((it & (issuers - 1)) == q) {
                    const int s = it % S, round = it / S;
                    // a segment's first MMA overwrites the accumulator: the epilogue must have read its previous contents
                    if (first && use >= 1) ok = warp_all(mbar_wait(bar_acc_empty(buf), (use - 1) & 1, abort_flag, p.status, 36));
                    if (ok) ok = warp_all(mbar_wait(bar_bf_full(s), round & 1, abort_flag, p.status, 32));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + acc_col(q, buf), a_tmem = tmem_base + kTmemAccN + (uint32_t)(s * (BK / 2));
                    const uint64_t db = da0 + (uint64_t)((lay.bf(s) - lay.bf(0)) >> 4);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; kk++)  // weights from tensor memory: operand stage s, 16 k = 8 columns
                            tc_mma_bf16_cta_a_tmem(d_tmem, a_tmem + kk * 8, db + (uint64_t)(kk * 2), idesc, (!first || kk > 0) ? 1u : 0u);
                        tc_commit_cta(bar_bf_empty(s));
                    }
                    first = false;
                }
                if (++kb == num_kb || it == n_it - 1) {  // the segment ends with its slab or with this CTA's range
                    // An issuer without a k-block in the segment only arrives.  With one buffer that arrival must not fall
                    // into the barrier's previous phase (the other issuers' commits of the last segment may still be on
                    // their way): it waits until the epilogue has read the last segment, as a first MMA would have.
                    if (first && bufs == 1 && use >= 1) ok = warp_all(mbar_wait(bar_acc_empty(buf), (use - 1) & 1, abort_flag, p.status, 36));
                    if (!ok) break;
                    if (elect_one()) tc_commit_cta(bar_acc_full(buf));
                    kb = 0; seg++; first = true;
                }
            }
            if (!ok && it > q) {  // its last MMAs: of the last k-block before this one that it took
                const int last = it - 1 - ((it - 1 - q) & (issuers - 1));
                wait_landed(bar_bf_empty(last % S), last, S);
            }
        }
    } else if (warp >= kFirstDecodeWarp) {
        const int group = (warp - kFirstDecodeWarp) / kGroupWarps;
        const int dt = threadIdx.x - (kFirstDecodeWarp + group * kGroupWarps) * 32;
        const int act_chunks = mp * (BK / 8);  // 8-byte chunks of the activation tile
        bool ok = true;
        int s8 = group >> 1;  // byte stage of the group's next k-block, and the parity of its round
        uint32_t ph8 = 0;
        const int h = group & 1;  // which k-block of its pair block
        for (int it = group; it < n_it && ok; it += kDecodeGroups) {
            const int s = it % S, r = it / S;
            ok = mbar_wait(bar_u8_full(s8), ph8, abort_flag, p.status, 33);
            if (ok && r > 0) ok = mbar_wait(bar_bf_empty(s), (r - 1) & 1, abort_flag, p.status, 34);
            if (!ok) {
                // The barrier of an expanded activation tile counts this group too: its arrivals for the tiles that may have been
                // issued, one per stage, so that they can be waited for.
                if (ACT_BF16 && lane == 0)
                    for (int i = it; i < min(it + S, n_it); i += kDecodeGroups) mbar_arrive(bar_bf_full(i % S));
                break;
            }
            const uint32_t w8 = lay.u8(s8), a8 = w8 + kU8Act + (uint32_t)h * BK;
            const uint32_t abf = lay.bf(s);
            if (!ACT_BF16) {
                // (the tile's 8-byte chunks, up to four per thread; a loop, so that what a smaller tile does not have is not fetched either)
#pragma unroll 1
                for (int q = dt; q < act_chunks; q += kGroupThreads) {
                    const int row = q >> 3, jc = q & 7;
                    sts_v4(abf + (row >> 3) * 1024 + (row & 7) * 128 + ((jc ^ (row & 7)) << 4), decode8<kLutShiftN>(lds_v2(a8 + row * BK2 + jc * 8), lut));
                }
            }
            uint4 vr[BK / 16];
            // this warp's 32 weight columns (operand rows, tensor-memory lanes): quarter * 32 ..
            const int quarter = warp & 3;
            if (W_IS_NK) {
                // [N,K] weights, a thread per column: the byte tile (rows of 128 k) arrives with the 128-byte TMA swizzle (chunk
                // j of row r at chunk j ^ (r & 7)): conflict-free row reads
                const int wr = quarter * 32 + lane;
                const uint32_t w_row = w8 + (uint32_t)wr * BK2, sw = (uint32_t)wr & 7u;
#pragma unroll
                for (int jj = 0; jj < BK / 16; jj++) vr[jj] = lds_v4(w_row + (((uint32_t)(4 * h + jj) ^ sw) << 4));
            } else {
                // [K,N] weights: the rows of the tile are k, 128 columns each, with the same swizzle.  16 x 16 byte matrices
                // are read transposed, so that a thread holds four consecutive k of a column: vr[2 i + c] = k 32 i .. 32 i + 31
                // of the quarter's columns 16 c .. 16 c + 15.  (Read a byte per load, a k-block took 256 more shared-memory
                // wavefronts, as many as its lookups.)
                const int k = h * BK + lane;
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int c = 0; c < 2; c++)
                        vr[2 * i + c] = ldmatrix_trans_bytes_x2(w8 + (uint32_t)(k + 32 * i) * BM + ((uint32_t)((2 * quarter + c) ^ (lane & 7)) << 4));
            }
            __syncwarp();  // the byte stage has been read: the producer may refill it during the decode
            if (lane == 0) mbar_arrive(bar_u8_empty(s8));
            uint32_t o[BK / 2];  // two BF16 per tensor-memory column
            const uint32_t st_base = tmem_base + ((uint32_t)(quarter * 32) << 16) + kTmemAccN + (uint32_t)(s * (BK / 2));
            if (W_IS_NK) {
#pragma unroll
                for (int jj = 0; jj < BK / 16; jj++) {
                    const uint4 lo = decode8<kLutShiftN>(make_uint2(vr[jj].x, vr[jj].y), lut), hi = decode8<kLutShiftN>(make_uint2(vr[jj].z, vr[jj].w), lut);
                    o[8 * jj + 0] = lo.x; o[8 * jj + 1] = lo.y; o[8 * jj + 2] = lo.z; o[8 * jj + 3] = lo.w;
                    o[8 * jj + 4] = hi.x; o[8 * jj + 5] = hi.y; o[8 * jj + 6] = hi.z; o[8 * jj + 7] = hi.w;
                }
                tmem_st_32x32b_x32(st_base, o);
            } else {
#pragma unroll
                for (int c = 0; c < 2; c++) {
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const uint4 v = vr[2 * i + c];
                        const uint4 lo = decode8<kLutShiftN>(make_uint2(v.x, v.y), lut), hi = decode8<kLutShiftN>(make_uint2(v.z, v.w), lut);
                        uint32_t* d = o + 16 * c + 8 * i;
                        d[0] = lo.x; d[1] = lo.y; d[2] = lo.z; d[3] = lo.w; d[4] = hi.x; d[5] = hi.y; d[6] = hi.z; d[7] = hi.w;
                    }
                    tmem_st_16x256b_x4(st_base + ((uint32_t)(16 * c) << 16), o + 16 * c);
                }
            }
            tmem_st_wait();  // the weight column is in tensor memory
            if (!ACT_BF16) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_bf_full(s));
            s8 += 2;
            if (s8 >= S8) { s8 -= S8; ph8 ^= 1u; }
        }
    } else if (!CLUSTER) {
        // epilogue warps 0-3: TMEM lane = weight column n, TMEM column = activation row m.  Whatever does not need the sums
        // (exponents, the slab's contributors) is worked out before the wait for them: after it, it cost every segment
        // several thousand cycles of load latency and divisions.
        const int sa = p.d_sa ? *p.d_sa : 0, sw_all = (p.d_sw && !p.d_sw_channel) ? *p.d_sw : 0;
        const uint32_t tlane = tmem_base + ((uint32_t)(warp * 32) << 16);
        int slab = slab0, pb_a = pb0, done = 0;  // the segment: units [done, done + len) of the range, from pair block pb_a of the slab
        for (int seg = 0; done < n_pairs; seg++) {
            const int buf = bufs == 2 ? seg & 1 : 0, use = bufs == 2 ? seg >> 1 : seg;
            const int len = min(num_pb - pb_a, n_pairs - done);
            const bool whole = len == num_pb;
            const int n = slab * BM + warp * 32 + lane;
            const int sc = -(sa + (p.d_sw_channel ? (n < p.N ? __ldg(p.d_sw_channel + n) : 0) : sw_all)), s1 = sc / 2, s2 = sc - s1;
            const float f1 = __uint_as_float((uint32_t)(s1 + 127) << 23), f2 = __uint_as_float((uint32_t)(s2 + 127) << 23);
            // contributors of the slab: the CTAs from the owner of its first pair block to that of its last one
            const int c_first = whole ? 0 : plan.owner(slab * num_pb), c_last = whole ? 0 : plan.owner((slab + 1) * num_pb - 1);
            const int pos = (int)blockIdx.x - c_first, count = c_last - c_first + 1;
            float* slab_part = whole ? nullptr : plan.part + (size_t)slab * plan.pmax * mp * BM + warp * 32 + lane;
            float* mine = whole ? nullptr : slab_part + (size_t)pos * mp * BM;
            const int it_a = 2 * done, it_n = 2 * len;  // the segment's k-blocks, counted within this CTA's range
            // C[m0 .. m0 + 15][n] from complete sums
            auto finish16 = [&](int m0, const float (&acc)[16]) {
                if (n >= p.N) return;
                if (p.c_is_f32) {
                    float* out = reinterpret_cast<float*>(p.C) + (long long)m0 * p.ldc + n;
#pragma unroll
                    for (int h = 0; h < 16; h += 8) {
                        float old[8];
#pragma unroll
                        for (int u = 0; u < 8; u++) old[u] = (p.accumulate && m0 + h + u < p.M) ? out[(h + u) * p.ldc] : 0.f;
#pragma unroll
                        for (int u = 0; u < 8; u++)
                            if (m0 + h + u < p.M) out[(h + u) * p.ldc] = p.accumulate ? acc[h + u] * f1 * f2 + old[u] : acc[h + u] * f1 * f2;
                    }
                } else {
                    unsigned short* out = reinterpret_cast<unsigned short*>(p.C) + (long long)m0 * p.ldc + n;
#pragma unroll
                    for (int h = 0; h < 16; h += 8) {
                        uint32_t old[8];
#pragma unroll
                        for (int u = 0; u < 8; u++) old[u] = (p.accumulate && m0 + h + u < p.M) ? (uint32_t)out[(h + u) * p.ldc] << 16 : 0u;
#pragma unroll
                        for (int u = 0; u < 8; u++) {
                            float v = acc[h + u] * f1 * f2;
                            if (p.accumulate) v += __uint_as_float(old[u]);
                            unsigned short b;
                            asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(b) : "f"(v));  // round to nearest even; a NaN stays a NaN
                            if (m0 + h + u < p.M) out[(h + u) * p.ldc] = b;
                        }
                    }
                }
            };
            if (!mbar_wait(bar_acc_full(buf), use & 1, abort_flag, p.status, 35)) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < mp; c += 16) {
                float r[16];  // this lane's row of the segment's sum, columns c .. c + 15: the issuers' accumulators added in order
#pragma unroll
                for (int i = 0; i < 16; i++) r[i] = 0.f;
#pragma unroll 1
                for (int q = 0; q < issuers; q += 2) {
                    // issuer q took the k-blocks it = q (mod issuers): none of them in a short segment leaves its accumulator stale
                    const bool live0 = it_n >= issuers || ((q - it_a) & (issuers - 1)) < it_n;
                    const bool live1 = it_n >= issuers || ((q + 1 - it_a) & (issuers - 1)) < it_n;
                    uint32_t t0[16], t1[16];
                    tmem_ld_32x32b_x16(tlane + acc_col(q, buf) + c, t0);
                    tmem_ld_32x32b_x16(tlane + acc_col(q + 1, buf) + c, t1);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        if (live0) r[i] += __uint_as_float(t0[i]);
                        if (live1) r[i] += __uint_as_float(t1[i]);
                    }
                }
                if (whole) finish16(c, r);
                else {
#pragma unroll
                    for (int i = 0; i < 16; i++) __stcg(mine + (c + i) * BM, r[i]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty(buf));  // the accumulator has been read: it may be overwritten
            if (!whole) {
                // the warp's slice is complete; lane 0's release covers what the other lanes stored before the barrier
                unsigned prior = 0;
                if (lane == 0)
                    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(prior) : "l"(plan.tickets + slab * kEpiWarps + warp) : "memory");
                prior = __shfl_sync(0xFFFFFFFFu, prior, 0);
                if (prior == (unsigned)(count - 1)) {  // every slice of this quarter slab is complete
                    __threadfence();
                    // sixteen rows at a time: their loads are independent, so the L2 latency is paid once per two slices
#pragma unroll 1
                    for (int m0 = 0; m0 < mp; m0 += 16) {
                        const float* sl = slab_part + (size_t)m0 * BM;  // m0 + 15 < mp: mp is a multiple of 16
                        float acc[16], v[16];
#pragma unroll
                        for (int u = 0; u < 16; u++) acc[u] = __ldcg(sl + u * BM);
                        sl += (size_t)mp * BM;  // (a slab that is not whole has two contributors at least)
#pragma unroll
                        for (int u = 0; u < 16; u++) v[u] = __ldcg(sl + u * BM);
#pragma unroll
                        for (int u = 0; u < 16; u++) acc[u] = (0.f + acc[u]) + v[u];
#pragma unroll 1
                        for (int i = 2; i < count; i++) {
                            sl += (size_t)mp * BM;
#pragma unroll
                            for (int u = 0; u < 16; u++) v[u] = __ldcg(sl + u * BM);
#pragma unroll
                            for (int u = 0; u < 16; u++) acc[u] += v[u];
                        }
                        finish16(m0, acc);
                    }
                }
            }
            done += len; pb_a = 0; slab++;
        }
    }
    if (CLUSTER) {
        // Exchange and epilogue of a slab shared by a cluster: pieces of eight activation rows, dealt to the CTAs in runs of `per`.
        // Every CTA sends its sums of a piece to the owner (itself included), which adds them in rank order.
        __syncwarp();
        const int quarter = warp & 3, shares = quarter < 2 ? 7 : 6, pieces = mp / 8, per = (pieces + split - 1) / split;
        static_assert(kThreadsN / 32 == 26, "seven warps on the lanes of quarters 0 and 1, six on the others");
        const int sa = p.d_sa ? *p.d_sa : 0, sw_all = (p.d_sw && !p.d_sw_channel) ? *p.d_sw : 0;
        const bool ok = mbar_wait(bar_acc_full(0), 0, abort_flag, p.status, 38);
        tc_fence_after();
        __syncwarp();
        cluster_arrive_relaxed();
        cluster_wait();  // all CTAs are done with their stages
        if (ok) {
#pragma unroll 1
            for (int j = warp >> 2; j < pieces; j += shares) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; i++) v[i] = 0.f;
#pragma unroll 1
                for (int q = 0; q < issuers; q++) {
                    if (q >= n_it) break;  // (an issuer without a k-block left its accumulator as it was)
                    uint32_t r[8];
                    tmem_ld_32x32b_x8(tmem_base + ((uint32_t)(quarter * 32) << 16) + acc_col(q, 0) + j * 8, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; i++) v[i] += __uint_as_float(r[i]);
                }
                const int owner = j / per;
                const uint32_t to = map_to_cta(lay.base + (uint32_t)(((part * per + j - owner * per) * 2 * BM + quarter * 32 + lane) * 16), (uint32_t)owner);
                st_cluster_v4(to, __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
                st_cluster_v4(to + BM * 16, __float_as_uint(v[4]), __float_as_uint(v[5]), __float_as_uint(v[6]), __float_as_uint(v[7]));
            }
        }
        __syncwarp();
        cluster_sync_all();
        // four activation rows of a quarter's columns per warp and step
        const int items = max(0, min(pieces - part * per, per)) * 8;
#pragma unroll 1
        for (int u = warp; ok && u < items; u += kThreadsN / 32) {
            const int nl = (u & 3) * 32 + lane, n = slab0 * BM + nl, m = (part * per + (u >> 3)) * 8 + ((u >> 2) & 1) * 4;
            const int sc = -(sa + (p.d_sw_channel ? (n < p.N ? __ldg(p.d_sw_channel + n) : 0) : sw_all)), s1 = sc / 2, s2 = sc - s1;
            const float f1 = __uint_as_float((uint32_t)(s1 + 127) << 23), f2 = __uint_as_float((uint32_t)(s2 + 127) << 23);
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            for (int q = 0; q < split; q++) {
                const uint4 w = lds_v4(lay.base + (uint32_t)((((q * per + (u >> 3)) * 2 + ((u >> 2) & 1)) * BM + nl) * 16));
                v[0] += __uint_as_float(w.x); v[1] += __uint_as_float(w.y); v[2] += __uint_as_float(w.z); v[3] += __uint_as_float(w.w);
            }
            if (n < p.N) {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    if (m + i >= p.M) continue;
                    float x = v[i] * f1 * f2;
                    const long long at = (long long)(m + i) * p.ldc + n;
                    if (p.c_is_f32) {
                        float* out = reinterpret_cast<float*>(p.C) + at;
                        *out = p.accumulate ? x + *out : x;
                    } else {
                        unsigned short* out = reinterpret_cast<unsigned short*>(p.C) + at;
                        if (p.accumulate) x += __uint_as_float((uint32_t)*out << 16);
                        unsigned short b;
                        asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(b) : "f"(x));  // round to nearest even; a NaN stays a NaN
                        *out = b;
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemColsN) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------------------
// Weights decoded into tensor memory: C^T = W^T A^T.
// A pair of CTAs computes 256 weight columns x bn activation rows: each CTA decodes 128 weight columns straight into its
// tensor memory (the 128-row A operand of the MMA; nothing decoded there touches shared memory) and provides bn / 2 activation
// rows (the B operand): expanded to BF16 beforehand in the caller's workspace and brought by TMA (a k-block is 128 k then), or,
// when there is no room for them, as bytes [M,K] or [K,M] that the decode groups decode into shared memory as well (64 k).
// Warp roles per CTA:
//   warps 0-3   epilogue: accumulator column = activation row m, lane = weight column n
//   warp  4     copies of weight bytes, four stages of 16 KiB       warp 22  copies of the activation tiles, four stages
//   warp  5     MMA issuer (even CTA)                               warps 6-21  four decode groups, group g on it = g (mod 4),
//                                                                              and the epilogue
// Two forms, one kernel:
//   split = 1   persistent: pair p of P takes tiles p, p + P, ..  A decode group that is through with a tile decodes one k-block
//               of the next (which fills the four stages) and then joins the epilogue: with warps 0-3 alone the accumulator was
//               occupied for 13400 cycles (against 64000 for the k-blocks at K = 7168), now 5000.
//   split > 1   a cluster of `split` pairs per tile, each pair a part of K; the pairs exchange their partial sums through
//               distributed shared memory, every pair finishes a part of the activation rows, adding in pair order.  For
//               products with too few tiles for the device and for the last, incomplete round of the persistent form.
// What bounds it: per k-block and SM 256 x 2 lookup wavefronts (one per 32 bytes), the byte tile in and out and the
// activation tile in and out, about 1100 cycles of shared memory against 1024 of the tensor pipe at bn = 256.
// ---------------------------------------------------------------------------------------------------------
constexpr int kWdStages = 4, kWdActWarp = kThreads / 32, kThreadsWd = kThreads + 32;  // 736
constexpr int kWdMaxSplit = 4;
static_assert(kWdStages == kDecodeGroups, "group g owns stage g, so every barrier is waited on in program order");
enum Activations { kActExpanded, kActRows, kActColumns };  // BF16 [M,K], bytes [M,K], bytes [K,M]

// Shared memory.  Expanded activations: four operand stages of 32 KiB, four stages of weight bytes of 16 KiB, the 32 KiB table.
// Activations as bytes: eight slots of 16 KiB (four operand stages; four byte stages, weights then activations) around the 64 KiB
// table, which starts on a 64 KiB boundary of the shared window (see decode8).  The partial sums that a pair receives in the
// split form go to `base` and up, over stages and table: nothing there is needed any more.
template <int ACT>
struct WdSmem {
    static constexpr int KB = ACT == kActExpanded ? 2 * BK : BK;  // k per k-block
    static constexpr uint32_t kActStage = (BN / 2) * KB * 2, kW8 = BM * KB;
    static constexpr uint32_t n_bars = 4 * kWdStages + 3;
    uint32_t base, lut, bars, end;
    int front;
    __device__ explicit WdSmem(uint32_t raw)
    {
        base = (raw + 1023u) & ~1023u;
        if (ACT == kActExpanded) {
            lut = base + kWdStages * (kActStage + kW8); bars = lut + kLutBytesNarrow; front = 0;
        } else {
            lut = (base + kLutBytesWide - 1) & ~(kLutBytesWide - 1);
            front = min((int)((lut - base) / kSlotBytes), 2 * kWdStages);
            bars = lut + kLutBytesWide + (uint32_t)(2 * kWdStages - front) * kSlotBytes;
        }
        end = bars + n_bars * 8 + 16;
    }
    __device__ uint32_t slot(int i) const { return i < front ? base + (uint32_t)i * kSlotBytes : lut + kLutBytesWide + (uint32_t)(i - front) * kSlotBytes; }
    __device__ uint32_t act(int s) const { return ACT == kActExpanded ? base + (uint32_t)s * kActStage : slot(s); }
    __device__ uint32_t u8(int s) const { return ACT == kActExpanded ? base + kWdStages * kActStage + (uint32_t)s * kW8 : slot(kWdStages + s); }
    __device__ uint32_t tmem_slot() const { return bars + n_bars * 8; }
    __device__ uint32_t abort_flag() const { return tmem_slot() + 4; }
    __device__ uint32_t gave_up() const { return tmem_slot() + 12; }  // a CTA of the cluster gave up
    __device__ uint32_t issued() const { return tmem_slot() + 8; }  // 1 + the activation tiles that this CTA issued in all (0: not through yet)
};
static_assert(WdSmem<kActRows>::kActStage == kSlotBytes && 2 * WdSmem<kActRows>::kW8 == kSlotBytes, "one stage per slot");
static_assert((kWdMaxSplit - 1) * (BN / kWdMaxSplit) * BM * 4 <= 2 * kWdStages * kSlotBytes && (2 - 1) * (BN / 2) * BM * 4 <= 2 * kWdStages * kSlotBytes,
              "the partial sums received stay below the barriers");

struct TilePlan {
    int first, count;  // tiles [first, first + count) of the product
    int chunks, bn;    // activation rows in `chunks` pieces of bn (a multiple of 32)
    // Tiles in groups of eight pieces that sweep the `slabs` of 256 weight columns together (tile_coords).  Slab by slab, with 32
    // pieces one round of 74 tiles read all of the activations: 8192 x 28672 x 8192 with expanded activations (134 MB, more than
    // L2 holds) 2905 us, in groups 2614 to 2636.
    int slabs;
    int split;
    int clear_status;  // nonzero: no launch in front of this one clears the status word
    // nonzero: the launch in front of this one is the same product's other tiles.  It lets this one start once everything before itself
    // is complete, so nothing is waited for at the start, and its end at this one's end, for whoever comes after.
    int follows;
    // kParts: `first` and `count` are in parts of tiles, `parts` to a tile, whose activation rows are `tile_rows`; bn is a part's
    int parts, tile_rows;
};

// Eight results that are there already, `pitch` bytes apart.  All loads go out before the first is used: left to the compiler, an
// instantiation that is short of registers waited for each of them (3872 x 3200 x 1680, [K,N] weights, operands as bytes, added
// to FP32: 87.5 us a call, so 77.8; BF16 86 and 75.7).  BATCH: where that matters, in the instantiations for more than eight pieces of
// activation rows; with it in the one for up to eight, 2048 x 7168 x 4096 that adds to nothing took 134.7 us instead of 134.0.
__device__ __forceinline__ void load_column_f32(const unsigned char* at, unsigned long long pitch, float (&v)[8])
{
    asm volatile("{\n\t.reg .u64 a;\n\t"
                 "ld.global.cs.f32 %0, [%8];\n\tadd.u64 a, %8, %9;\n\tld.global.cs.f32 %1, [a];\n\tadd.u64 a, a, %9;\n\tld.global.cs.f32 %2, [a];\n\t"
                 "add.u64 a, a, %9;\n\tld.global.cs.f32 %3, [a];\n\tadd.u64 a, a, %9;\n\tld.global.cs.f32 %4, [a];\n\tadd.u64 a, a, %9;\n\t"
                 "ld.global.cs.f32 %5, [a];\n\tadd.u64 a, a, %9;\n\tld.global.cs.f32 %6, [a];\n\tadd.u64 a, a, %9;\n\tld.global.cs.f32 %7, [a];\n\t}"
                 : "=&f"(v[0]), "=&f"(v[1]), "=&f"(v[2]), "=&f"(v[3]), "=&f"(v[4]), "=&f"(v[5]), "=&f"(v[6]), "=&f"(v[7]) : "l"(at), "l"(pitch) : "memory");
}
__device__ __forceinline__ void load_column_bf16(const unsigned char* at, unsigned long long pitch, unsigned short (&v)[8])
{
    asm volatile("{\n\t.reg .u64 a;\n\t"
                 "ld.global.b16 %0, [%8];\n\tadd.u64 a, %8, %9;\n\tld.global.b16 %1, [a];\n\tadd.u64 a, a, %9;\n\tld.global.b16 %2, [a];\n\t"
                 "add.u64 a, a, %9;\n\tld.global.b16 %3, [a];\n\tadd.u64 a, a, %9;\n\tld.global.b16 %4, [a];\n\tadd.u64 a, a, %9;\n\t"
                 "ld.global.b16 %5, [a];\n\tadd.u64 a, a, %9;\n\tld.global.b16 %6, [a];\n\tadd.u64 a, a, %9;\n\tld.global.b16 %7, [a];\n\t}"
                 : "=&h"(v[0]), "=&h"(v[1]), "=&h"(v[2]), "=&h"(v[3]), "=&h"(v[4]), "=&h"(v[5]), "=&h"(v[6]), "=&h"(v[7]) : "l"(at), "l"(pitch) : "memory");
}

// Eight finished sums of this thread's weight column, activation rows m .. m + 7 of which `rows` exist, to C: `out` is the
// place of the first, `pitch` the bytes from row to row.  For one row a warp writes 32 consecutive columns.  Issue slots bound
// this: with two scale factors, 64-bit row addresses and a test per row the epilogue of a 256 x 256 tile took 5300 cycles, 19
// instructions a store.  So the pitch has 32 bits, one multiply-add per row, unless rows lie 4 GiB apart or more (a few rows of
// a large buffer): that is an instantiation of its own, since 64-bit products for all cost 1 % (4096 x 28672 x 8192 with
// expanded activations: 1320 -> 1352 us).
template <bool BATCH, typename Pitch>
__device__ __forceinline__ void store_columns(unsigned char* out, Pitch pitch, int is_f32, int accumulate, int rows, float (&v)[8])
{
    auto at = [&](int i) { return out + (unsigned long long)pitch * (uint32_t)i; };
    if (accumulate) {
        if (BATCH && is_f32 && rows >= 8) {
            float old[8];
            load_column_f32(out, (unsigned long long)pitch, old);
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] += old[i];
        } else if (is_f32) {
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] += i < rows ? __ldcs(reinterpret_cast<const float*>(at(i))) : 0.f;
        } else if (BATCH && rows >= 8) {
            unsigned short old[8];
            load_column_bf16(out, (unsigned long long)pitch, old);
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] += __uint_as_float((uint32_t)old[i] << 16);
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] += i < rows ? __uint_as_float((uint32_t)*reinterpret_cast<const unsigned short*>(at(i)) << 16) : 0.f;
        }
    }
    if (is_f32) {
        if (rows >= 8) {
#pragma unroll
            for (int i = 0; i < 8; i++) __stcs(reinterpret_cast<float*>(at(i)), v[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (i < rows) __stcs(reinterpret_cast<float*>(at(i)), v[i]);
        }
    } else {
        unsigned short b[8];
#pragma unroll
        for (int i = 0; i < 8; i++) asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(b[i]) : "f"(v[i]));  // round to nearest even; a NaN stays a NaN
        if (rows >= 8) {
#pragma unroll
            for (int i = 0; i < 8; i++) *reinterpret_cast<unsigned short*>(at(i)) = b[i];
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (i < rows) *reinterpret_cast<unsigned short*>(at(i)) = b[i];
        }
    }
}

// Instantiations by tile order and row pitch.  (With the choice of the order made in the kernel, the divisions of the other one in
// the way of the first copies, 128 x 512 x 512 took 10.0 us instead of 9.8.)
// kParts is the last, incomplete round of a large product in tiles of fewer activation rows: divided along K alone, two tiles of
// 2048 x 7168 x 4096 kept 8 pairs of 74 busy (103.7 us, with it 101.5; with activations as bytes 138.4 and 135.8; that launch waits
// for nothing of the one in front of it, see TilePlan::follows, which is 1 us of it).
enum WeightsForm { kOneGroup, kGroups, kFarRows, kParts };  // up to eight pieces (or sixteen, see launch_weights_gemm); more; the rows of C 4 GiB apart or more (any number of pieces); parts of tiles
constexpr int kGroupPieces = 8;

template <bool W_IS_NK, int ACT, int FORM>
__global__ void __launch_bounds__(kThreadsWd, 1)
hif8_gemm_weights_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_act, const GemmParams p, const TilePlan tp)
{
    extern __shared__ unsigned char smem_raw[];
    using Smem = WdSmem<ACT>;
    constexpr int KB = Smem::KB, kLutShift = ACT == kActExpanded ? 7 : 8;
    const Smem lay(smem_u32(smem_raw));
    const uint32_t base = lay.base;
    unsigned char* sm = smem_raw - smem_u32(smem_raw);  // generic pointer of shared-window address 0
    if (ACT != kActExpanded) {
        uint32_t dyn_bytes;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
        if (lay.end > smem_u32(smem_raw) + dyn_bytes) {  // the layout does not fit (the same answer in every thread of the grid)
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int*>(p.status) = 7;
            return;
        }
    }
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), half = rank & 1u, lead = rank & ~1u;  // half 0: leader of its pair (issues the MMAs)
    const bool leader = half == 0;
    const uint32_t bars = lay.bars;
    auto bar_u8_full = [&](int s) { return bars + 8u * s; };                       // per CTA
    auto bar_u8_empty = [&](int s) { return bars + 8u * (kWdStages + s); };        // per CTA
    auto bar_bf_full = [&](int s) { return bars + 8u * (2 * kWdStages + s); };     // leader: both CTAs' decode warps and activation tiles
    auto bar_bf_empty = [&](int s) { return bars + 8u * (3 * kWdStages + s); };    // per CTA, leader's commits
    const uint32_t bar_acc_full = bars + 8u * (4 * kWdStages);                     // per CTA, leader's commit
    const uint32_t bar_acc_empty = bars + 8u * (4 * kWdStages + 1);                // leader: both CTAs' epilogue warps
    const uint32_t bar_sums = bars + 8u * (4 * kWdStages + 2);                     // per CTA: the sums of the other pairs have arrived
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + lay.abort_flag());
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + lay.tmem_slot());
    const uint32_t lut = lay.lut + 4u * lane;

    const int num_kb = (p.K + KB - 1) / KB, split = tp.split, part = split > 1 ? (int)(rank >> 1) : 0;
    const int kb0 = split > 1 ? num_kb * part / split : 0, kb1 = split > 1 ? num_kb * (part + 1) / split : num_kb;
    const int t0 = tp.first + (int)(split > 1 ? blockIdx.x / (2 * split) : blockIdx.x >> 1);
    const int t_end = tp.first + tp.count, t_step = split > 1 ? tp.count : (int)(gridDim.x >> 1);

    // ---- set-up.  A call of a small product is mostly latency: the first weight copies go out under the table set-up, and only
    // what touches the other CTAs waits for the cluster (its barrier takes 1400 to 1900 cycles from the start of the kernel,
    // in which a first k-block is copied and decoded).
    auto place = [&](int t, int& slab, int& m0) {  // tile t: its weight slab and its first activation row
        int piece;
        if (FORM == kOneGroup) {
            slab = t / tp.chunks;
            piece = t - slab * tp.chunks;
        } else tile_coords(FORM == kParts ? t / tp.parts : t, tp.chunks, tp.slabs, piece, slab);
        m0 = FORM == kParts ? piece * tp.tile_rows + t % tp.parts * tp.bn : piece * tp.bn;
    };
    auto copy_bytes = [&](int it, int t, int kb) {  // (the whole copying warp) tile t's bytes of k-block kb into stage it % kWdStages, which is free
        int slab, m0;
        place(t, slab, m0);
        const int s = it % kWdStages, n0 = slab * 2 * BM + (int)half * BM;
        const uint32_t dst = lay.u8(s), bar = bar_u8_full(s);
        m0 += (int)half * (tp.bn / 2);
        if (elect_one()) {
            mbar_arrive_expect_tx(bar, Smem::kW8 + (ACT == kActExpanded ? 0u : (uint32_t)(tp.bn / 2) * KB));
            if (W_IS_NK) tma_load_2d(dst, &map_w, kb * KB, n0, bar);
            else tma_load_2d(dst, &map_w, n0, kb * KB, bar);
            if (ACT == kActRows) tma_load_2d(dst + Smem::kW8, &map_act, kb * KB, m0, bar);
            else if (ACT == kActColumns) tma_load_2d(dst + Smem::kW8, &map_act, m0, kb * KB, bar);
        }
    };
    if (warp == kTmaWarp) {
        if (elect_one()) {
            for (int s = 0; s < kWdStages; s++) {
                mbar_init(bar_u8_full(s), 1); mbar_init(bar_u8_empty(s), kGroupWarps);
                // operands ready: both CTAs' groups, plus (expanded activations) the leader's announcement of the tile bytes
                mbar_init(bar_bf_full(s), 2 * kGroupWarps + (ACT == kActExpanded ? 1 : 0)); mbar_init(bar_bf_empty(s), 1);
            }
            mbar_init(bar_acc_full, 1); mbar_init(bar_acc_empty, 2 * (kEpiWarps + kDecodeWarps)); mbar_init(bar_sums, 1);
            // (The others touch these two words when a wait has given up, seconds later, and the block's barrier stands in front of the
            // cluster's: no fence at cluster scope, which would make every call 0.8 us longer, 201 x 7168 x 4096 19.9 -> 20.6.)
            *reinterpret_cast<volatile int*>(sm + lay.gave_up()) = 0;
            *reinterpret_cast<volatile uint32_t*>(sm + lay.issued()) = 0u;
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        if (ACT == kActExpanded) copy_bytes(0, t0, kb0);
    }
    fill_decode_table<(1 << (kLutShift - 2))>(reinterpret_cast<uint32_t*>(sm + lay.lut), warp, lane, kThreadsWd / 32);
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(lay.tmem_slot()), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_relaxed();  // (the barriers' initialisation has been released) barriers and tensor memory of this CTA are there; every warp waits for the other CTAs' once
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (ACT != kActExpanded) {
        // Nothing was launched in front of this kernel to order it behind what produces its operands.
        if (!tp.follows) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (tp.clear_status && blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int*>(p.status) = 0;  // (a wait gives up seconds later)
    }

    if (warp == kTmaWarp) {
        // ------------------------------------------------------------------ bytes (each CTA feeds itself).  Beside expanded
        // activations nothing is read here that the launch in front of this one writes, and what came before that is complete.
        const int n_early = min(kWdStages, kb1 - kb0);  // of the first tile, without waiting for anybody
        for (int i = ACT == kActExpanded ? 1 : 0; i < n_early; i++) copy_bytes(i, t0, kb0 + i);
        __syncwarp();
        cluster_wait();
        int it = 0;
        bool ok = true;
        for (int t = t0; t < t_end && ok; t += t_step) {
            for (int kb = kb0; kb < kb1; kb++, it++) {
                if (it < n_early) continue;
                if (it >= kWdStages) ok = warp_all(mbar_wait(bar_u8_empty(it % kWdStages), (it / kWdStages - 1) & 1, abort_flag, p.status, 41));
                if (!ok || warp_any(*abort_flag)) { ok = false; break; }
                copy_bytes(it, t, kb);
            }
        }
        if (*abort_flag)
            for (int i = max(0, it - kWdStages); i < it; i++) wait_landed(bar_u8_full(i % kWdStages), i, kWdStages);
    } else if (warp == kWdActWarp) {
        // ------------------------------------------------------------------ expanded activations: this CTA's bn / 2 rows, two boxes of
        // 64 k (the swizzle span); both CTAs' copies complete on the leader's "operands ready" barrier
        cluster_wait();
        {
            if (!tp.follows) asm volatile("griddepcontrol.wait;" ::: "memory");  // the launch in front expands them
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
            // A tile's barrier (in the pair's leader) counts the bytes of both CTAs' halves.  A thread that is through says how many tiles
            // it has issued, and one that gives up reads that of the other CTA and issues its halves of the tiles that the other
            // one issued: their stages were free for both, and hold nothing that anybody still wants.  (It is read from there, and not
            // sent here by every run: a store that nobody waits for could arrive after this CTA has left.)
            constexpr int kNoLimit = 0x7FFFFFFF;
            int it = 0, limit = kNoLimit;
            bool ok = ACT == kActExpanded;
            auto tell = [&]() { *reinterpret_cast<volatile uint32_t*>(sm + lay.issued()) = (uint32_t)it + 1u; };
            for (int t = t0; t < t_end && ok; t += t_step) {
                int slab, m0;
                if (FORM == kOneGroup) m0 = t % tp.chunks * tp.bn;
                else place(t, slab, m0);
                m0 += (int)half * (tp.bn / 2);
                for (int kb = kb0; kb < kb1; kb++, it++) {
                    const int s = it % kWdStages;
                    if (limit == kNoLimit && ((it >= kWdStages && !warp_all(mbar_wait(bar_bf_empty(s), (it / kWdStages - 1) & 1, abort_flag, p.status, 46))) || warp_any(*abort_flag))) {
                        tell();
                        const unsigned long long c0 = global_ns();
                        do limit = (int)ld_cluster_u32(map_to_cta(lay.issued(), rank ^ 1u)) - 1;  // (the other CTA's waits are bounded as well)
                        while (limit < 0 && global_ns() - c0 < 2 * kWaitLimitNs);
                        limit = __shfl_sync(0xFFFFFFFFu, limit, 0);
                    }
                    if (it >= limit) { ok = false; break; }
                    const uint32_t full = map_to_cta(bar_bf_full(s), lead);
                    if (elect_one()) {
                        if (leader) mbar_arrive_expect_tx(bar_bf_full(s), (uint32_t)tp.bn * KB * 2u);
                        tma_load_3d_pair(lay.act(s), &map_act, kb * KB, m0, 0, full);
                        tma_load_3d_pair(lay.act(s) + Smem::kActStage / 2, &map_act, kb * KB + BK, m0, 0, full);
                    }
                }
            }
            if (ACT == kActExpanded) {
                if (limit == kNoLimit) tell();
                if (leader && *abort_flag) {
                    for (int i = max(0, it - kWdStages); i < it; i++) wait_landed(bar_bf_full(i % kWdStages), i, kWdStages);
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer (leader CTA only)
        cluster_wait();
        if (leader) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((ACT == kActColumns ? 1u : 0u) << 16) | ((uint32_t)(tp.bn >> 3) << 17) |
                                   ((uint32_t)((2 * BM) >> 4) << 24);
            int it = 0, local = 0;
            bool ok = true;
            for (int t = t0; t < t_end && ok; t += t_step, local++) {
                if (local > 0) ok = mbar_wait(bar_acc_empty, (local - 1) & 1, abort_flag, p.status, 45);
                ok = warp_all(ok);
                for (int kb = kb0; kb < kb1 && ok; kb++, it++) {
                    const int s = it % kWdStages;
                    ok = warp_all(mbar_wait(bar_bf_full(s), (it / kWdStages) & 1, abort_flag, p.status, 42));
                    if (!ok) break;
                    tc_fence_after();
                    // [M,K]: 16 k = 32 bytes inside the 128-byte rows (the second 64 k of an expanded block are the stage's second
                    // half); [K,M]: 16 k = two 1024-byte atoms
                    const uint64_t db = ACT == kActColumns ? make_smem_desc(lay.act(s), 8192, 1024) : make_smem_desc(lay.act(s), 16, 1024);
                    const uint32_t a_tmem = tmem_base + kTmemColsAcc + (uint32_t)(s * (KB / 2));
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < KB / 16; kk++) {
                            const uint32_t off = ACT == kActColumns ? kk * 2048 : (kk >> 2) * (Smem::kActStage / 2) + (kk & 3) * 32;
                            tc_mma_bf16_pair_a_tmem(tmem_base, a_tmem + kk * 8, db + (uint64_t)(off >> 4), idesc, (kb > kb0 || kk > 0) ? 1u : 0u);
                        }
                        tc_commit_pair(bar_bf_empty(s), lead);
                    }
                }
                if (ok && elect_one()) tc_commit_pair(bar_acc_full, lead);
                __syncwarp();
            }
            if (!ok && it > 0) wait_landed(bar_bf_empty((it - 1) % kWdStages), it - 1, kWdStages);
        }
    } else if (warp < kFirstDecodeWarp) cluster_wait();  // warps 0-3

    const bool one_tile = tp.count <= t_step, decodes = warp >= kFirstDecodeWarp && warp < kFirstDecodeWarp + kDecodeWarps;
    if (one_tile || warp < kEpiWarps || decodes) {
        // ------------------------------------------------------------------ decode and epilogue.  An epilogue is done in pieces of
        // eight columns by five warps per quarter of the lanes; with one tile per pair all warps take part, six (five) to a
        // quarter.  In the split form the pairs exchange first: each finishes `per` of the pieces.
        __syncwarp();
        const int group = (warp - kFirstDecodeWarp) / kGroupWarps, quarter = warp & 3;
        const int shares = one_tile && quarter < 3 ? 6 : 5;
        const int share = one_tile ? warp >> 2 : (decodes ? (warp - quarter) / 4 - (quarter < 2 ? 1 : 0) : 0);
        static_assert(kThreadsWd / 32 == 23 && kFirstDecodeWarp == 6 && kDecodeWarps == 16,
                      "six warps on the lanes of quarters 0 to 2, five on those of quarter 3; five each without warps 4, 5 and 22");
        const int row = quarter * 32 + lane, sa = p.d_sa ? *p.d_sa : 0, sw_all = (p.d_sw && !p.d_sw_channel) ? *p.d_sw : 0;
        const int c_size = p.c_is_f32 ? 4 : 2;
        const long long pitch = p.ldc * c_size;
        const uint32_t tl = tmem_base + ((uint32_t)(quarter * 32) << 16), mine = base + (uint32_t)row * 16u, tlane = tl + kTmemColsAcc;
        const int n_kb = kb1 - kb0;
        constexpr int kGaveUp = 1 << 30;
        int it = decodes ? group : kGaveUp, tile_it = 0, local = 0;  // next k-block of the group; first k-block of the tile to finish next
        bool joined = !decodes;
        for (int t = t0; t < t_end;) {
            // the group's k-blocks of this tile, and one of the next
            const int n_it_known = t + t_step < t_end ? tile_it + 2 * n_kb : tile_it + n_kb;
            if (it < tile_it + n_kb || (it < n_it_known && it - kDecodeGroups < tile_it + n_kb)) {
                const int s = it % kWdStages, r = it / kWdStages;
                bool ok = mbar_wait(bar_u8_full(s), r & 1, abort_flag, p.status, 43);
                if (ok && r > 0) ok = mbar_wait(bar_bf_empty(s), (r - 1) & 1, abort_flag, p.status, 44);
                if (!ok) { it += kGaveUp; continue; }  // (no further k-block: gives up at the next wait)
                const uint32_t w8 = lay.u8(s), dst = tlane + (uint32_t)(s * (KB / 2));
                if (ACT != kActExpanded) {
                    // activations as bytes: the tile's 8-byte chunks, up to eight per thread (it lies in a row, [M,K] or [K,M]), two at a time and in
                    // front of the weights.  Unrolled to eight behind them, with what smaller tiles do not have skipped, they took as long as four
                    // times as many weights (256 x 1536 x 768 8.2 -> 7.9 us, 1024 x 7168 x 4096 [K,M] 82.8 -> 78.8, 4096 x 4096 x 4096 159.3 -> 155.8; four
                    // at a time 8.0, 79.6, 155.6).
                    const int dt = threadIdx.x - (kFirstDecodeWarp + group * kGroupWarps) * 32, n_chunks = tp.bn / 2 * (BK / 8);
                    const uint32_t abf = lay.act(s);
                    const int per_row = tp.bn >> 4;  // [K,M]: 8-byte chunks per k (8 or 16)
                    auto put = [&](int q, uint2 bytes) {
                        uint32_t at;
                        if (ACT == kActRows) at = abf + (q >> 6) * 1024 + ((q >> 3) & 7) * 128 + (((q ^ (q >> 3)) & 7) << 4);
                        else {
                            const int kr = per_row == 16 ? q >> 4 : q >> 3, jn = q & (per_row - 1);
                            at = abf + ((jn >> 3) * 8 + (kr >> 3)) * 1024 + (kr & 7) * 128 + (((jn ^ kr) & 7) << 4);
                        }
                        sts_v4(at, decode8<kLutShift>(bytes, lut));
                    };
#pragma unroll 1
                    for (int q = dt; q < n_chunks; q += 2 * kGroupThreads) {
                        const bool two = q + kGroupThreads < n_chunks;  // (the same for the whole group)
                        const uint2 v0 = lds_v2(w8 + Smem::kW8 + (uint32_t)q * 8u);
                        uint2 v1 = v0;
                        if (two) v1 = lds_v2(w8 + Smem::kW8 + (uint32_t)(q + kGroupThreads) * 8u);
                        put(q, v0);
                        if (two) put(q + kGroupThreads, v1);
                    }
                }
                // 64 bytes of weights per thread and pass, one piece of code for both passes of an expanded block (unrolled, the first
                // time through cost every group a thousand cycles of instruction fetches)
#pragma unroll 1
                for (int h = 0; h < KB / BK; h++) {
                    uint4 v[4];
                    if (W_IS_NK) {
                        // a thread per weight column; rows of KB k with the swizzle of that span: chunk j of row r at j ^ (r & 7), or
                        // with 64 bytes at j ^ ((r >> 1) & 3)
                        const uint32_t w_row = w8 + (uint32_t)row * KB, sw = KB == 2 * BK ? (uint32_t)row & 7u : (uint32_t)(row >> 1) & 3u;
#pragma unroll
                        for (int j = 0; j < 4; j++) v[j] = lds_v4(w_row + (((uint32_t)(4 * h + j) ^ sw) << 4));
                    } else {
                        // rows of 128 columns, one per k, read transposed (see the narrow kernel): 128 k of sixteen columns a pass, or
                        // 64 k of sixteen columns in v[0], v[1] and of the next sixteen in v[2], v[3]
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const int i = KB == 2 * BK ? j : j & 1, c = KB == 2 * BK ? h : j >> 1;
                            v[j] = ldmatrix_trans_bytes_x2(w8 + (uint32_t)(32 * i + lane) * BM + ((uint32_t)((2 * quarter + c) ^ (lane & 7)) << 4));
                        }
                    }
                    if (h == KB / BK - 1) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_u8_empty(s));
                    }
                    uint32_t o[32];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const uint4 lo = decode8<kLutShift>(make_uint2(v[j].x, v[j].y), lut), hi = decode8<kLutShift>(make_uint2(v[j].z, v[j].w), lut);
                        o[8 * j + 0] = lo.x; o[8 * j + 1] = lo.y; o[8 * j + 2] = lo.z; o[8 * j + 3] = lo.w;
                        o[8 * j + 4] = hi.x; o[8 * j + 5] = hi.y; o[8 * j + 6] = hi.z; o[8 * j + 7] = hi.w;
                    }
                    if (W_IS_NK) tmem_st_32x32b_x32(dst + (uint32_t)(h * (BK / 2)), o);
                    else if (KB == 2 * BK) {
                        tmem_st_16x256b_x4(dst + ((uint32_t)(16 * h) << 16), o);
                        tmem_st_16x256b_x4(dst + ((uint32_t)(16 * h) << 16) + BK / 2, o + 16);
                    } else {
                        tmem_st_16x256b_x4(dst, o);
                        tmem_st_16x256b_x4(dst + (16u << 16), o + 16);
                    }
                }
                if (ACT != kActExpanded) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (!joined) { cluster_wait(); joined = true; }  // before the first signal to another CTA
                if (lane == 0) mbar_arrive_remote(map_to_cta(bar_bf_full(s), lead));
                it += kDecodeGroups;
                continue;
            }
            if (!joined) { __syncwarp(); cluster_wait(); joined = true; }
            int slab, m0;
            place(t, slab, m0);
            const int n = slab * 2 * BM + (int)half * BM + row;
            // 2^sc as one factor, and a second one for the few scales that need it
            const int sc = -(sa + (p.d_sw_channel ? (n < p.N ? __ldg(p.d_sw_channel + n) : 0) : sw_all)), s1 = max(-126, min(126, sc));
            const float f1 = __uint_as_float((uint32_t)(s1 + 127) << 23), f2 = __uint_as_float((uint32_t)(sc - s1 + 127) << 23);
            const int past = FORM == kParts ? min(p.M, (m0 / tp.tile_rows + 1) * tp.tile_rows) : p.M;  // (the last part of a tile may be a shorter one)
            const int cols = max(0, min(tp.bn, past - m0)), pieces = (cols + 7) / 8, per = split == 1 ? pieces : (pieces + split - 1) / split;
            unsigned char* out = reinterpret_cast<unsigned char*>(p.C) + (long long)m0 * pitch + (long long)n * c_size;
            const bool ok = mbar_wait(bar_acc_full, local & 1, abort_flag, p.status, 47);
            if (!ok && split == 1) break;
            tc_fence_after();
            const int j0 = part * per, j1 = min(pieces, j0 + per);
            if (split > 1) {
                if (threadIdx.x == 0) mbar_arrive_expect_tx(bar_sums, (uint32_t)((split - 1) * max(0, j1 - j0)) * 8u * BM * 4u);
                __syncwarp();
                cluster_arrive_relaxed();
                cluster_wait();  // every pair's MMAs and copies are done: the stages of all CTAs are free
                if (ok) {
#pragma unroll 1
                    for (int j = share; j < pieces; j += shares) {
                        const int owner = j / per;
                        if (owner == part) continue;
                        uint32_t r[8];
                        tmem_ld_32x32b_x8(tl + j * 8, r);
                        tmem_ld_wait();
                        const int slot = part < owner ? part : part - 1;
                        const uint32_t to = map_to_cta(mine + (uint32_t)((slot * per + (j - owner * per)) * 8 * BM) * 4u, 2u * owner + half);
                        const uint32_t bar = map_to_cta(bar_sums, 2u * owner + half);
                        st_async_v4(to, r[0], r[1], r[2], r[3], bar);
                        st_async_v4(to + BM * 16, r[4], r[5], r[6], r[7], bar);
                    }
                }
                // (counted by a barrier here: a cluster barrier with release and acquire took 1800 cycles, this 800; in the narrow kernel, whose exchange is smaller, nothing is gained)
                if (!ok || !mbar_wait(bar_sums, 0, abort_flag, p.status, 48)) break;
            }
#pragma unroll 1
            for (int j = j0 + share; j < j1; j += shares) {
                uint32_t r[8];
                float v[8];
                tmem_ld_32x32b_x8(tl + j * 8, r);
                tmem_ld_wait();
                if (split > 1) {  // the pairs' sums in pair order
#pragma unroll
                    for (int i = 0; i < 8; i++) v[i] = 0.f;
#pragma unroll 1
                    for (int q = 0; q < split; q++) {
                        const uint32_t from = mine + (uint32_t)(((q < part ? q : q - 1) * per + (j - j0)) * 8 * BM) * 4u;
                        uint4 lo = make_uint4(r[0], r[1], r[2], r[3]), hi = make_uint4(r[4], r[5], r[6], r[7]);
                        if (q != part) { lo = lds_v4(from); hi = lds_v4(from + BM * 16); }
                        v[0] += __uint_as_float(lo.x); v[1] += __uint_as_float(lo.y); v[2] += __uint_as_float(lo.z); v[3] += __uint_as_float(lo.w);
                        v[4] += __uint_as_float(hi.x); v[5] += __uint_as_float(hi.y); v[6] += __uint_as_float(hi.z); v[7] += __uint_as_float(hi.w);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
                }
#pragma unroll
                for (int i = 0; i < 8; i++) v[i] *= f1;
                if (sc != s1) {
#pragma unroll
                    for (int i = 0; i < 8; i++) v[i] *= f2;
                }
                if (n < p.N) store_columns<FORM != kOneGroup>(out + j * 8 * pitch, (std::conditional_t<FORM == kFarRows, unsigned long long, uint32_t>)pitch, p.c_is_f32, p.accumulate, cols - j * 8, v);
            }
            tc_fence_before();
            __syncwarp();
            // (not after the last tile: nobody waits for that one, so it could reach the leader after the leader has left)
            if (t + t_step < t_end && lane == 0) mbar_arrive_remote(map_to_cta(bar_acc_empty, lead));
            t += t_step; tile_it += n_kb; local++;
        }
        if (!joined) { __syncwarp(); cluster_wait(); }
        // (gave up: the barrier of an expanded activation tile counts this group too; its arrival, so that the tile can be waited for)
        if (ACT == kActExpanded && decodes && it >= kGaveUp && lane == 0) mbar_arrive_remote(map_to_cta(bar_bf_full((it - kGaveUp) % kWdStages), lead));
    }

    // ---- teardown: all waits are bounded, so everybody arrives; nobody leaves while the peer may still read this
    // CTA's operands or signal its barriers; then the allocating warps free TMEM
    if (tp.follows) asm volatile("griddepcontrol.wait;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    // (unlikely, so that what follows a wait that gave up stands behind the rest of the code.  The question itself costs a small product
    // 0.1 us; asked by one warp a CTA alone it costs the same.)
    if (__builtin_expect(*abort_flag != 0, 0)) {
        if (threadIdx.x < 2u * split) st_cluster_u32(map_to_cta(lay.gave_up(), threadIdx.x), 1u);
        __syncwarp();
        cluster_arrive();
    } else cluster_arrive_relaxed();  // (in a run that succeeds every signal to another CTA has been waited for)
    cluster_wait();
    if (__builtin_expect(*reinterpret_cast<volatile int*>(sm + lay.gave_up()) != 0, 0)) {
        // A wait gave up in one of the CTAs (the same answer in all of them), so the others may have signalled to it and it to them
        // what nobody waited for: the partial sums are waited for here, the rest is released by a second barrier.
        if (split > 1 && threadIdx.x == 0) wait_landed(bar_sums, 0, 1);
        __syncwarp();
        cluster_sync_all();
    }
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------------------
// Decode-once path: operands already decoded to BF16 (by the conversion kernels of this library, into the caller's
// workspace).  Persistent kernel on CTA pairs (cta_group::2), 64-wide k-blocks.
//   warps 0-3  epilogue (TMEM -> global), overlapped with the next tile through two TMEM accumulators
//   warp  4    TMA producer of the A tiles: BF16 tiles land directly in the 128-byte-swizzled operand layout
//   warp  5    MMA issuer
//   warp  6    TMA producer of the W tiles
// A cluster of two CTAs on two SMs computes one 256 x 256 tile: each CTA stages its own 128 rows of A and its own 128
// columns of W (so the tensor core reads half as many operand bytes per SM and flop as with one CTA per tile, which is
// what bounds a one-CTA kernel), both accumulate their 128 rows in their own TMEM.  The even CTA of the pair (the
// leader) issues every tcgen05.mma; its commits arrive on the barriers of both CTAs.  TMA copies of both CTAs complete
// on the leader's "full" barrier (no multicast loads).
// The result leaves in pieces of 32 rows x 128 bytes, staged in shared memory by the warp that owns the rows and written by
// tile stores; FP32 results that are added to C have the old piece brought in by a tile copy two pieces ahead.  (With plain
// stores, 16 bytes a lane to 32 different rows, an FP32 tile took 26000 cycles to drain, longer than its k-blocks take at
// K = 2048: 4096 x 7168 x 2048 took
// 126 us a call, now 95; with BF16 results 102 and 89.)  BF16 results that are added to C and the squared error keep the plain loop.
// ---------------------------------------------------------------------------------------------------------
constexpr int kThreadsP = 7 * 32;
constexpr int kTmaWarpW = 6;
constexpr int kStages2 = 6;
constexpr uint32_t kStageBytes2 = kABfBytes + kBBfBytes;            // 32 KiB per CTA and stage
constexpr uint32_t kOutBytes = 32 * 128;                              // one piece of the result: 32 rows of 128 bytes
struct SmemLayout2 {
    static constexpr uint32_t out = kStages2 * kStageBytes2;          // 192 KiB; two pieces per epilogue warp
    static constexpr uint32_t bars = out + kEpiWarps * 2 * kOutBytes;
    static constexpr uint32_t n_bars = 2 * kStages2 + 4 + 2 * kEpiWarps;
    static constexpr uint32_t tmem_slot = bars + n_bars * 8;
    static constexpr uint32_t abort_flag = tmem_slot + 4;
    static constexpr uint32_t gave_up = abort_flag + 4;    // a CTA of the pair gave up
    static constexpr uint32_t issued = gave_up + 4;        // k-blocks issued by the pair's four copying threads
    static constexpr uint32_t total = issued + 4 * 4;
};
constexpr uint32_t kSmemBytes2 = SmemLayout2::total + 1024;
static_assert(kSmemBytes2 <= 227 * 1024, "shared memory of one CTA");

template <bool W_IS_NK>
__global__ void __launch_bounds__(kThreadsP, 1)
bf16_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_c,
                      const GemmParams p)
{
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - smem_u32(smem_raw));
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();          // 0: leader (issues the MMAs), 1: peer
    const bool leader = rank == 0;
    const uint32_t bars = base + SmemLayout2::bars;
    auto bar_full = [&](int s) { return bars + 8u * s; };                       // used in the leader only
    auto bar_empty = [&](int s) { return bars + 8u * (kStages2 + s); };         // per CTA, released by the leader's commits
    auto bar_acc_full = [&](int a) { return bars + 8u * (2 * kStages2 + a); };  // per CTA
    auto bar_acc_empty = [&](int a) { return bars + 8u * (2 * kStages2 + 2 + a); };  // leader: both epilogues arrive
    auto bar_old = [&](int i) { return bars + 8u * (2 * kStages2 + 4 + i); };        // per epilogue warp and staging piece
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + SmemLayout2::abort_flag);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + SmemLayout2::tmem_slot);
    const int num_kb = (p.K + BK - 1) / BK;
    // Up to K = 4096 the A tiles of sixteen tile-rows (32 MiB) stay in L2 beside the W tiles, and W is read half as often; beyond, those of eight (8192 x 28672
    // x 8192 in a sequence of calls 2600 us, with sixteen 2655, with four 2676; x 4096 1255 and with sixteen 1240; 3000 x 11008 x 4096 203.5 and 197.9).
    const int group = p.K <= 4096 ? 16 : 8;
    const int tiles_m2 = (p.M + 2 * BM - 1) / (2 * BM), tiles_n2 = p.tiles_n;
    // a batch of n x n products (A variant ia, W variant iw) is one list of tiles: product b = ia * n + iw owns tiles
    // [b * tiles_one, (b + 1) * tiles_one)
    const int tiles_one = tiles_m2 * tiles_n2, nb = p.batch_n > 0 ? p.batch_n : 1;
    const int tiles = tiles_one * nb * nb, pairs = gridDim.x >> 1, pair_id = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages2; s++) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int a = 0; a < 2; a++) { mbar_init(bar_acc_full(a), 1); mbar_init(bar_acc_empty(a), 2 * kEpiWarps); }
        for (int i = 0; i < 2 * kEpiWarps; i++) mbar_init(bar_old(i), 1);
        *abort_flag = 0;
        *reinterpret_cast<volatile int*>(sm + SmemLayout2::gave_up) = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + SmemLayout2::tmem_slot), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // barriers of both CTAs are initialised before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // (set-up above runs under the launch in front, which expands the weights)

    int progress = 0;  // of this thread's role: k-blocks issued or committed
    const bool loads_a = warp == kTmaWarp;
    auto copy_block = [&](int m0, int n0, int ia, int iw, int kb, int s) {  // this thread's operand of k-block kb into stage s, which is free
        const uint32_t dst_a = base + s * kStageBytes2, dst_b = dst_a + kABfBytes;
        const uint32_t full = map_to_cta(bar_full(s), 0);
        if (loads_a) {
            if (leader) mbar_arrive_expect_tx(bar_full(s), 2 * kStageBytes2);  // bytes of both CTAs, both operands
            tma_load_3d_pair(dst_a, &map_a, kb * BK, m0, ia, full);
        } else if (W_IS_NK) tma_load_3d_pair(dst_b, &map_w, kb * BK, n0, iw, full);
        else {
#pragma unroll
            for (int c = 0; c < BN / 2 / 64; c++)
                tma_load_3d_pair(dst_b + c * 8192, &map_w, n0 + c * 64, kb * BK, iw, full);
        }
    };
    if (warp == kTmaWarp || warp == kTmaWarpW) {
        {
            int s = 0;            // stage of the next k-block
            uint32_t ph = 0;      // parity of the round the ring is in
            bool ok = true, wrapped = false;
            for (int t = pair_id; t < tiles && ok; t += pairs) {
                int tile_m, tile_n;
                const int b = t / tiles_one, ia = b / nb, iw = b - ia * nb;
                tile_coords(t - b * tiles_one, tiles_m2, tiles_n2, tile_m, tile_n, group);
                const int m0 = tile_m * 2 * BM + (int)rank * BM, n0 = tile_n * BN + (int)rank * (BN / 2);
                for (int kb = 0; kb < num_kb; kb++) {
                    if (wrapped) ok = warp_all(mbar_wait(bar_empty(s), ph ^ 1u, abort_flag, p.status, 21));  // the previous round's use of the stage
                    if (!ok || warp_any(*abort_flag)) { ok = false; break; }
                    if (elect_one()) copy_block(m0, n0, ia, iw, kb, s);
                    progress++;
                    if (++s == kStages2) { s = 0; ph ^= 1u; wrapped = true; }
                }
            }
            if (lane == 0)
                for (uint32_t r = 0; r < 2; r++) st_cluster_u32(map_to_cta(base + SmemLayout2::issued + 4u * (2u * rank + (loads_a ? 0u : 1u)), r), (uint32_t)progress);
        }
    } else if (warp == kMmaWarp) {
        if (leader) {
            // M = 256 over the pair, N = 256
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((W_IS_NK ? 0u : 1u) << 16) |
                                   ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
            int local = 0, s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = pair_id; t < tiles && ok; t += pairs, local++) {
                const int acc = local & 1, use = local >> 1;
                if (use > 0) ok = warp_all(mbar_wait(bar_acc_empty(acc), (uint32_t)((use - 1) & 1), abort_flag, p.status, 22));
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * 256;
                for (int kb = 0; kb < num_kb; kb++) {
                    ok = warp_all(mbar_wait(bar_full(s), ph, abort_flag, p.status, 23));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_addr = base + s * kStageBytes2, b_addr = a_addr + kABfBytes;
                    const uint64_t da = make_smem_desc(a_addr, 16, 1024), db = W_IS_NK ? make_smem_desc(b_addr, 16, 1024) : make_smem_desc(b_addr, 8192, 1024);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; kk++)
                            tc_mma_bf16_pair(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * (W_IS_NK ? 2 : 128)), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                        tc_commit_pair(bar_empty(s));
                    }
                    progress++;
                    if (++s == kStages2) { s = 0; ph ^= 1u; }
                }
                if (ok && elect_one()) tc_commit_pair(bar_acc_full(acc));
                __syncwarp();
            }
        }
    } else if (warp < kEpiWarps) {
        int local = 0, b_held = -1;
        double err_acc = 0.0;  // squared-error variant: this thread's share of product b_held
        const bool ref_vec = !(reinterpret_cast<uintptr_t>(p.err_ref) & 15) && !(p.ld_ref & 3);
        auto flush_error = [&]() {  // all lanes of the warp
            for (int off = 16; off > 0; off >>= 1) err_acc += __shfl_xor_sync(0xFFFFFFFFu, err_acc, off);
            if (lane == 0 && err_acc != 0.0 && b_held >= 0) atomicAdd(p.err_sum + b_held, err_acc);
            err_acc = 0.0;
        };
        const int piece_cols = p.c_is_f32 ? 32 : 64;
        const uint32_t staging = base + SmemLayout2::out + (uint32_t)warp * 2 * kOutBytes;  // this warp's two pieces
        uint32_t n_old = 0, n_fetched = 0;  // old pieces waited for and (lane 0) asked for, over all tiles: parities of the two buffers
        for (int t = pair_id; t < tiles; t += pairs, local++) {
            const int acc = local & 1, use = local >> 1;
            int tile_m, tile_n;
            const int b = t / tiles_one, ia = b / nb, iw = b - ia * nb;
            tile_coords(t - b * tiles_one, tiles_m2, tiles_n2, tile_m, tile_n, group);
            const int row0 = tile_m * 2 * BM + (int)rank * BM + warp * 32, row = row0 + lane, n0 = tile_n * BN;
            const int pieces = p.c_by_tma && row0 < p.M ? (min(BN, p.N - n0) + piece_cols - 1) / piece_cols : 0;
            auto fetch_old = [&](int i) {  // lane 0; the staging piece is free
                const uint32_t bar = bar_old(2 * warp + (i & 1));
                mbar_arrive_expect_tx(bar, kOutBytes);
                tma_load_2d(staging + (uint32_t)(i & 1) * kOutBytes, &map_c, n0 + i * piece_cols, row0, bar);
                n_fetched ^= 1u << (i & 1);
            };
            if (p.c_by_tma && p.accumulate && lane == 0) {
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                for (int i = 0; i < min(2, pieces); i++) fetch_old(i);
            }
            if (!mbar_wait(bar_acc_full(acc), (uint32_t)(use & 1), abort_flag, p.status, 24)) break;
            tc_fence_after();
            if (p.err_sum && b != b_held) { flush_error(); b_held = b; }
            // exponents of this product (in a batch: entry ia / iw of the two device arrays)
            const int sa = p.d_sa ? p.d_sa[ia] : 0;
            const int sdesc = p.d_sw_channel ? 0 : -(sa + (p.d_sw ? p.d_sw[iw] : 0));
            const int s1 = sdesc / 2, s2 = sdesc - s1;
            const float f1 = __uint_as_float((uint32_t)(s1 + 127) << 23), f2 = __uint_as_float((uint32_t)(s2 + 127) << 23);
            const uint32_t tlane = tmem_base + ((uint32_t)(warp * 32) << 16) + acc * 256;
#pragma unroll 1
            for (int i = 0; i < pieces; i++) {
                const uint32_t buf = staging + (uint32_t)(i & 1) * kOutBytes, line = buf + (uint32_t)lane * 128u;
                if (!p.accumulate) {  // the store of two pieces ago has been read out
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                }
                if (p.c_is_f32) {
                    uint32_t r[32];
                    tmem_ld_32x32b_x32(tlane + i * 32, r);
                    tmem_ld_wait();
                    if (p.d_sw_channel) apply_channel_scale(p, n0 + i * 32, lane, sa, r);
                    if (p.accumulate) {
                        if (!mbar_wait(bar_old(2 * warp + (i & 1)), (n_old >> (i & 1)) & 1, abort_flag, p.status, 25)) break;
                        n_old ^= 1u << (i & 1);
                    }
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const uint32_t at = line + (uint32_t)((j ^ (lane & 7)) << 4);
                        float v[4];
#pragma unroll
                        for (int u = 0; u < 4; u++) v[u] = __uint_as_float(r[4 * j + u]) * f1 * f2;
                        if (p.accumulate) {
                            const uint4 o = lds_v4(at);
                            v[0] += __uint_as_float(o.x); v[1] += __uint_as_float(o.y); v[2] += __uint_as_float(o.z); v[3] += __uint_as_float(o.w);
                        }
                        sts_v4(at, make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3])));
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        uint32_t r[32];
                        tmem_ld_32x32b_x32(tlane + i * 64 + h * 32, r);
                        tmem_ld_wait();
                        if (p.d_sw_channel) apply_channel_scale(p, n0 + i * 64 + h * 32, lane, sa, r);
                        stage_chunk_bf16(buf, lane, 4 * h, r, f1, f2);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&map_c, buf, n0 + i * piece_cols, row0);
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    if (p.accumulate && i + 2 < pieces) {
                        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        fetch_old(i + 2);
                    }
                }
            }
#pragma unroll 1
            for (int c = 0; c < (p.c_by_tma ? 0 : BN); c += 32) {
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(warp * 32) << 16) + acc * 256 + c, r);
                tmem_ld_wait();
                const int col = n0 + c;
                if (p.d_sw_channel) apply_channel_scale(p, col, lane, sa, r);
                if (p.err_sum) {
                    if (row < p.M && col < p.N) {
                        // exact differences of the FP32 result and the FP32 reference, squared and summed in double
                        const float* ref = p.err_ref + (long long)row * p.ld_ref + col;
                        if (col + 32 <= p.N && ref_vec) {
#pragma unroll
                            for (int i = 0; i < 32; i += 4) {
                                const float4 o = __ldg(reinterpret_cast<const float4*>(ref + i));
                                const double d0 = (double)(__uint_as_float(r[i]) * f1 * f2) - (double)o.x;
                                const double d1 = (double)(__uint_as_float(r[i + 1]) * f1 * f2) - (double)o.y;
                                const double d2 = (double)(__uint_as_float(r[i + 2]) * f1 * f2) - (double)o.z;
                                const double d3 = (double)(__uint_as_float(r[i + 3]) * f1 * f2) - (double)o.w;
                                err_acc += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < 32; i++) {  // (constant indices: see add_chunk_bf16)
                                if (col + i < p.N) {
                                    const double d = (double)(__uint_as_float(r[i]) * f1 * f2) - (double)__ldg(ref + i);
                                    err_acc += d * d;
                                }
                            }
                        }
                    }
                } else add_chunk_bf16(p, row, col, r, f1, f2);
            }
            tc_fence_before();
            __syncwarp();
            // (default semantics: what the leader's MMAs must not overtake are this warp's tensor-memory loads, ordered by
            // tcgen05.wait::ld and the fence above -- not its stores to C, which a release at cluster scope would wait for)
            if (lane == 0) mbar_arrive_remote(map_to_cta(bar_acc_empty(acc), 0));  // tell the leader: accumulator drained
        }
        if (p.err_sum) flush_error();
        if (p.c_by_tma && lane == 0) {
            // old pieces still on their way (a wait gave up) land before this CTA's shared memory goes away
            for (uint32_t i = 0; i < 2; i++)
                if (((n_fetched ^ n_old) >> i) & 1u) wait_landed(bar_old(2 * warp + i), (int)(n_old >> i), 1);
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
    }

    // nobody leaves while the other CTA may still read this CTA's shared memory or signal its barriers
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0)
        for (uint32_t r = 0; r < 2; r++) st_cluster_u32(map_to_cta(base + SmemLayout2::gave_up, r), 1u);
    __syncwarp();
    cluster_sync_all();
    if (*reinterpret_cast<volatile int*>(sm + SmemLayout2::gave_up)) {
        // A wait gave up in one of the CTAs (the same answer in both).  A stage's barrier counts the copies of four threads: those
        // that are behind issue theirs of the k-blocks that another one issued (whose stages were free for all), and the leader
        // waits for them all, and for its last MMAs.
        if (lane == 0) {
            if (warp == kTmaWarp || warp == kTmaWarpW) {
                const volatile int* issued = reinterpret_cast<const volatile int*>(sm + SmemLayout2::issued);
                const int top = max(max(issued[0], issued[1]), max(issued[2], issued[3]));
#pragma unroll 1
                for (int i = progress; i < top; i++) {
                    int tile_m, tile_n;
                    const int t = pair_id + i / num_kb * pairs, b = t / tiles_one, ia = b / nb;
                    tile_coords(t - b * tiles_one, tiles_m2, tiles_n2, tile_m, tile_n, group);
                    copy_block(tile_m * 2 * BM + (int)rank * BM, tile_n * BN + (int)rank * (BN / 2), ia, b - ia * nb, i % num_kb, i % kStages2);
                }
                if (leader && loads_a)
                    for (int i = max(0, top - kStages2); i < top; i++) wait_landed(bar_full(i % kStages2), i, kStages2);
            } else if (warp == kMmaWarp && leader && progress > 0) wait_landed(bar_empty((progress - 1) % kStages2), progress - 1, kStages2);
        }
        __syncwarp();
        cluster_sync_all();
    }
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// Self-test of the bounded wait: one warp waits on a barrier that nothing will ever complete, with a short limit.
// The wait must give up, record its status word and let the kernel finish normally.
__global__ void wait_selftest_kernel(int* status, unsigned long long limit_ns)
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) (void)mbar_wait(smem_u32(&bar), 0, &abort_flag, status, 99, limit_ns);
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------
cudaError_t launch_expand_activations(const uint8_t* a, void* a_bf, unsigned long long n, void* clear, size_t clear_bytes, int sm_count, cudaStream_t st)
{
    // (K is a multiple of 16)
    const bool stream = n >= kExpandStreamFrom && n < (1ull << 44);
    const unsigned long long per_block = stream ? 8ull * kExpandThreads * kExpandUnroll : 16ull * 256, cap = (unsigned long long)sm_count * 32;
    const unsigned long long want = (n + per_block - 1) / per_block;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(stream || want < cap ? want : cap));
    cfg.blockDim = dim3(stream ? kExpandThreads : 256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (stream)
        return cudaLaunchKernelEx(&cfg, expand_activations_stream_kernel, reinterpret_cast<const uint2*>(a), reinterpret_cast<uint4*>(a_bf), n / 8,
                                  reinterpret_cast<uint32_t*>(clear), (unsigned)(clear_bytes / 4));
    return cudaLaunchKernelEx(&cfg, expand_activations_kernel, reinterpret_cast<const uint4*>(a), reinterpret_cast<uint4*>(a_bf), n / 16,
                              reinterpret_cast<uint32_t*>(clear), (unsigned)(clear_bytes / 4));
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    });
    return fn;
}

// Tensor maps are cached per (pointer, shape, leading dimension, box): encoding one costs a driver call of a few
// microseconds, which matters for the narrow products of ~100 us when the same operands come back call after call.
struct MapKey {
    const void* ptr;
    uint64_t inner, rows, count, ld;  // ld: row pitch in elements (2-D) or distance between stacked matrices (3-D)
    uint32_t box_inner, box_rows;
    uint32_t kind;                    // 0: bytes, 2-D; 1: BF16, 2-D, 128-byte swizzle; 2: BF16, 3-D stack, 128-byte swizzle;
                                      // 3: bytes, 2-D, 64-byte swizzle; 4: bytes, 2-D, 128-byte swizzle; 5: FP32, 2-D, 128-byte swizzle;
                                      // 6: as 4, lines of 128 bytes brought to L2
    uint32_t pad;
};
LruCache<MapKey, CUtensorMap, 64> g_map_cache;

bool encode_map(const MapKey& k, CUtensorMap* map)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const bool bf16 = k.kind == 1 || k.kind == 2;
    if (k.kind == 2) {
        cuuint64_t dims[3] = {k.inner, k.rows, k.count};
        cuuint64_t strides[2] = {k.inner * 2u, (k.count > 1 ? k.ld : k.inner * k.rows) * 2u};
        cuuint32_t box[3] = {k.box_inner, k.box_rows, 1};
        cuuint32_t estr[3] = {1, 1, 1};
        return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(k.ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    if (k.kind == 5) {
        cuuint64_t dims[2] = {k.inner, k.rows};
        cuuint64_t strides[1] = {k.ld * 4u};
        cuuint32_t box[2] = {k.box_inner, k.box_rows};
        cuuint32_t estr[2] = {1, 1};
        return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(k.ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    cuuint64_t dims[2] = {k.inner, k.rows};
    cuuint64_t strides[1] = {k.ld * (bf16 ? 2u : 1u)};
    cuuint32_t box[2] = {k.box_inner, k.box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(k.ptr), dims,
              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              (bf16 || k.kind == 4 || k.kind == 6) ? CU_TENSOR_MAP_SWIZZLE_128B : (k.kind == 3 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE),
              k.kind == 6 ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B : CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D tensor [rows][ld elements] with a box of box_inner x box_rows elements, zero fill out of bounds.
// bf16 = false: bytes, with no swizzle or the 64- or 128-byte one (box_inner at most that many bytes).  bf16 = true: 16-bit
// elements, 128-byte swizzle (box_inner must be 64).  lines_128: a copy brings lines of 128 bytes to L2 and not of 256.
bool make_map(CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t rows, uint64_t ld, uint32_t box_inner, uint32_t box_rows,
              bool bf16 = false, uint32_t bytes_swizzle = 0, bool lines_128 = false)
{
    MapKey k;
    std::memset(&k, 0, sizeof k);
    k.ptr = ptr; k.inner = inner; k.rows = rows; k.count = 1; k.ld = ld; k.box_inner = box_inner; k.box_rows = box_rows;
    k.kind = bf16 ? 1u : (bytes_swizzle == 64 ? 3u : (bytes_swizzle == 128 ? (lines_128 ? 6u : 4u) : 0u));
    return g_map_cache.lookup_or_make(k, map, encode_map);
}

// FP32 matrix (a result), 128-byte swizzle, boxes of 32 columns
bool make_map_f32(CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t rows, uint64_t ld, uint32_t box_rows)
{
    MapKey k;
    std::memset(&k, 0, sizeof k);
    k.ptr = ptr; k.inner = inner; k.rows = rows; k.count = 1; k.ld = ld; k.box_inner = 32; k.box_rows = box_rows; k.kind = 5u;
    return g_map_cache.lookup_or_make(k, map, encode_map);
}

// BF16 stack of `count` matrices [rows, inner], `stack_stride` elements apart (box: one matrix deep)
bool make_map3(CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t rows, uint64_t count, uint64_t stack_stride,
               uint32_t box_inner, uint32_t box_rows)
{
    MapKey k;
    std::memset(&k, 0, sizeof k);
    k.ptr = ptr; k.inner = inner; k.rows = rows; k.count = count; k.ld = count > 1 ? stack_stride : 0; k.box_inner = box_inner;
    k.box_rows = box_rows; k.kind = 2u;
    return g_map_cache.lookup_or_make(k, map, encode_map);
}

// Kernel attributes (opt-in to more than 48 KiB of dynamic shared memory) and the SM count are facts of one device:
// they are set up once per device ordinal, by the first GEMM call made with that device current.
struct GemmDeviceSetup {
    cudaError_t rc;
    int sm_count;
    int nw_clusters[kNwMaxSplit + 1];  // clusters of s CTAs of the narrow kernel, s = 1, 2, 4, 8
    int wp_clusters[kWarpMaxCluster + 1];  // clusters of s blocks of hif8_gemm_warp_kernel, s = 1 .. 8
    int wd_clusters[kWdMaxSplit + 1];  // clusters of s pairs of hif8_gemm_weights_kernel that fit on the device at once, s = 1, 2, 4
};
PerDevice<GemmDeviceSetup> g_gemm_setup;

template <bool ACT_BF16, bool WIDE>
void narrow_kernels(const void** k)
{
    k[0] = (const void*)hif8_gemm_narrow_kernel<false, ACT_BF16, false, WIDE>; k[1] = (const void*)hif8_gemm_narrow_kernel<true, ACT_BF16, false, WIDE>;
    k[2] = (const void*)hif8_gemm_narrow_kernel<false, ACT_BF16, true, WIDE>; k[3] = (const void*)hif8_gemm_narrow_kernel<true, ACT_BF16, true, WIDE>;
}
template <int FORM>
void weights_kernels(const void** k)
{
    k[0] = (const void*)hif8_gemm_weights_kernel<false, kActExpanded, FORM>; k[1] = (const void*)hif8_gemm_weights_kernel<true, kActExpanded, FORM>;
    k[2] = (const void*)hif8_gemm_weights_kernel<false, kActRows, FORM>; k[3] = (const void*)hif8_gemm_weights_kernel<true, kActRows, FORM>;
    k[4] = (const void*)hif8_gemm_weights_kernel<false, kActColumns, FORM>; k[5] = (const void*)hif8_gemm_weights_kernel<true, kActColumns, FORM>;
}

template <int MT>
void warp_kernels(const void** k)
{
    k[0] = (const void*)hif8_gemm_warp_kernel<false, false, MT>; k[1] = (const void*)hif8_gemm_warp_kernel<true, false, MT>;
}

bool gemm_kernels_ready(int dev, int* sm_count_out, const int** wd_clusters = nullptr, const int** nw_clusters = nullptr, const int** wp_clusters = nullptr)
{
    const GemmDeviceSetup* s = g_gemm_setup.get(dev, [](int d, GemmDeviceSetup* out) {
        out->rc = cudaSuccess;
        out->sm_count = 0;
        std::memset(out->wd_clusters, 0, sizeof out->wd_clusters);
        std::memset(out->nw_clusters, 0, sizeof out->nw_clusters);
        const void* pair[2] = {(const void*)bf16_gemm_pair_kernel<false>, (const void*)bf16_gemm_pair_kernel<true>};
        const void* wd[24];
        weights_kernels<kOneGroup>(wd); weights_kernels<kGroups>(wd + 6); weights_kernels<kFarRows>(wd + 12); weights_kernels<kParts>(wd + 18);
        for (int i = 0; i < 2 && out->rc == cudaSuccess; i++)
            out->rc = cudaFuncSetAttribute(pair[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes2);
        for (int i = 0; i < 24 && out->rc == cudaSuccess; i++)
            out->rc = cudaFuncSetAttribute(wd[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytesMax);
        for (int s = 1; s <= kWdMaxSplit && out->rc == cudaSuccess; s *= 2) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 2 * s; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(2 * s); cfg.blockDim = dim3(kThreadsWd); cfg.dynamicSmemBytes = kSmemBytesMax;
            cfg.attrs = attr; cfg.numAttrs = 1;
            out->rc = cudaOccupancyMaxActiveClusters(&out->wd_clusters[s], wd[1], &cfg);
        }
        const void* narrow[12];
        narrow_kernels<false, true>(narrow); narrow_kernels<true, true>(narrow + 4); narrow_kernels<false, false>(narrow + 8);
        for (int i = 0; i < 12 && out->rc == cudaSuccess; i++)
            out->rc = cudaFuncSetAttribute(narrow[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytesMax);
        for (int s = 1; s <= kNwMaxSplit && out->rc == cudaSuccess; s *= 2) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = s; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(s); cfg.blockDim = dim3(kThreadsN); cfg.dynamicSmemBytes = kSmemBytesMax;
            cfg.attrs = attr; cfg.numAttrs = 1;
            out->rc = cudaOccupancyMaxActiveClusters(&out->nw_clusters[s], narrow[7], &cfg);  // (all of them take the same)
        }
        std::memset(out->wp_clusters, 0, sizeof out->wp_clusters);
        const void* wp[8];
        warp_kernels<1>(wp); warp_kernels<2>(wp + 2); warp_kernels<4>(wp + 4);
        wp[6] = (const void*)hif8_gemm_warp_kernel<false, true, 4>; wp[7] = (const void*)hif8_gemm_warp_kernel<true, true, 4>;
        for (int i = 0; i < 8 && out->rc == cudaSuccess; i++)
            out->rc = cudaFuncSetAttribute(wp[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytesMax);
        for (int s = 1; s <= kWarpMaxCluster && out->rc == cudaSuccess; s++) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = s; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(s); cfg.blockDim = dim3(kWarpThreads); cfg.dynamicSmemBytes = kSmemBytesMax;
            cfg.attrs = attr; cfg.numAttrs = 1;
            out->rc = cudaOccupancyMaxActiveClusters(&out->wp_clusters[s], wp[7], &cfg);
        }
        if (out->rc == cudaSuccess) out->rc = cudaDeviceGetAttribute(&out->sm_count, cudaDevAttrMultiProcessorCount, d);
    });
    if (!s) return false;
    *sm_count_out = s->sm_count;
    if (wd_clusters) *wd_clusters = s->wd_clusters;
    if (nw_clusters) *nw_clusters = s->nw_clusters;
    if (wp_clusters) *wp_clusters = s->wp_clusters;
    return s->rc == cudaSuccess && s->sm_count > 0 && s->wd_clusters[1] > 0;
}

// The status word of the most recent GEMM-class call per stream, for hif8_last_device_status.
struct StatusKey {
    const void* stream;
};
struct StatusVal {
    const int* word;
    int dev;
};
LruCache<StatusKey, StatusVal, 64> g_last_status;

constexpr size_t kGemmWorkspaceBytes = 256;

}  // namespace

void note_status_word(cudaStream_t st, const int* word)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    StatusKey k;
    std::memset(&k, 0, sizeof k);
    k.stream = st;
    g_last_status.put(k, StatusVal{word, dev});
}

int launch_bf16_pair_gemm(const void* a_bf, const void* w_bf, int w_is_nk, GemmParams p, cudaStream_t st,
                          long long a_stack_stride, long long w_stack_stride)
{
    int dev = 0, sm_count = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || !gemm_kernels_ready(dev, &sm_count)) return HIF8_ERR_CUDA;
    const int M = p.M, N = p.N, K = p.K;
    const uint64_t nb = p.batch_n > 0 ? (uint64_t)p.batch_n : 1;
    p.tiles_m = (M + BM - 1) / BM;
    p.tiles_n = (N + BN - 1) / BN;
    const long long tiles2 = (long long)((M + 2 * BM - 1) / (2 * BM)) * p.tiles_n * (long long)(nb * nb);
    if (M <= 0 || N <= 0 || K <= 0 || tiles2 > 0x3FFFFFFF) return HIF8_ERR_SHAPE;
    if (nb > 1 && ((a_stack_stride & 7) || (w_stack_stride & 7))) return HIF8_ERR_ALIGN;  // 16-byte strides
    CUtensorMap ma, mw;
    // A boxes: this CTA's 128 rows of [M,K]
    if (!make_map3(&ma, a_bf, (uint64_t)K, (uint64_t)M, nb, (uint64_t)a_stack_stride, BK, BM)) return HIF8_ERR_CUDA;
    // W boxes are one CTA's half of the 256-column tile: 128 rows of [N,K], or two boxes of 64 columns of [K,N]
    const bool okw = w_is_nk ? make_map3(&mw, w_bf, (uint64_t)K, (uint64_t)N, nb, (uint64_t)w_stack_stride, BK, BN / 2)
                             : make_map3(&mw, w_bf, (uint64_t)N, (uint64_t)K, nb, (uint64_t)w_stack_stride, 64, BK);
    if (!okw) return HIF8_ERR_CUDA;
    // the result through tile stores, except the squared error and BF16 sums
    CUtensorMap mc = ma;  // (a valid map in any case; only used when c_by_tma is set)
    p.c_by_tma = (!p.err_sum && (p.c_is_f32 || !p.accumulate)) ? 1 : 0;
    if (p.c_by_tma) {
        const bool okc = p.c_is_f32 ? make_map_f32(&mc, p.C, (uint64_t)N, (uint64_t)M, (uint64_t)p.ldc, 32)
                                    : make_map(&mc, p.C, (uint64_t)N, (uint64_t)M, (uint64_t)p.ldc, 64, 32, true);
        if (!okc) return HIF8_ERR_CUDA;
    }
    const int pairs = (int)(tiles2 < sm_count / 2 ? tiles2 : sm_count / 2);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2u * (unsigned)pairs);
    cfg.blockDim = dim3(kThreadsP);
    cfg.dynamicSmemBytes = kSmemBytes2;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t lrc = w_is_nk ? cudaLaunchKernelEx(&cfg, bf16_gemm_pair_kernel<true>, ma, mw, mc, p)
                                    : cudaLaunchKernelEx(&cfg, bf16_gemm_pair_kernel<false>, ma, mw, mc, p);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return (lrc == cudaSuccess && cudaGetLastError() == cudaSuccess) ? HIF8_OK : HIF8_ERR_CUDA;
}

}  // namespace hif8

using namespace hif8;

// Time of the weights kernel in cycles, from measurements: a k-block (128 k with expanded activations; 64 k with bytes, where the
// activations' lookups count too) and a tile's drain; what the exchange of a split tile costs beyond that (a cluster barrier, the
// sums at 20 bytes a cycle and the wait for them, less what the shared epilogue saves).  A launch of its own for the last round:
// from 90 products with and without one.  (With 4200 cycles for it and nothing in proportion 17 of them lost 3 to 16 % by it; behind a
// transposing expansion 4200 it is.)  The exchange's terms were measured when a second cluster barrier, both with release, stood in
// the place of that wait, and are up to 1200 cycles too high now: some products that would gain from it are not split.
struct WeightsCost {
    int num_kb, bn, unit;  // unit: the activation rows of a tile are a multiple of this
    bool expanded, transposed;  // the activations are expanded by the launch in front, from [K,M]
    const int* clusters;  // clusters of s pairs that the device holds
    double tiles(long long n, int split) const
    {
        if (split > num_kb || clusters[split] <= 0) return 1e30;
        const double f = bn / 256.0, exchange = split == 1 ? 0.0 : (split == 2 ? 1300.0 + 2000.0 * f : 2100.0 + 5300.0 * f);
        const double kblock = expanded ? 1150.0 : 730.0 + 270.0 * f;
        return (double)((n + clusters[split] - 1) / clusters[split]) * ((num_kb + split - 1) / split * kblock + 5000.0 * f + exchange);
    }
    int best_split(long long n) const
    {
        int best = 1;
        for (int s = 2; s <= kWdMaxSplit; s *= 2)
            if (tiles(n, s) < tiles(n, best)) best = s;
        return best;
    }
    // The tiles of the last, incomplete round, in a launch of their own when that finishes earlier: in parts of fewer activation
    // rows, each split along K.
    struct Rest {
        long long tiles = 0;  // 0: no such launch
        int parts = 1, rows = 0, split = 1;
        double cycles = 0.0;
    };
    Rest rest(long long n) const
    {
        Rest r;
        const long long rem = n > clusters[1] ? n % clusters[1] : 0;
        if (!rem) return r;
        r.cycles = tiles(rem, 1);
        for (int want = 1; want <= 8; want *= 2) {
            WeightsCost c = *this;
            c.bn = (bn + want * unit - 1) / (want * unit) * unit;
            const int parts = (bn + c.bn - 1) / c.bn, split = c.best_split(rem * parts);
            const double t = transposed ? c.tiles(rem * parts, split) + 4200.0 : 1.08 * c.tiles(rem * parts, split) + 7000.0;
            if ((split > 1 || parts > 1) && rem * parts <= clusters[split] && t < r.cycles) r = Rest{rem, parts, c.bn, split, t};
        }
        return r;
    }
    double all(long long n) const
    {
        if (n <= clusters[1]) return tiles(n, best_split(n));
        const long long rem = n % clusters[1];
        return tiles(n - rem, 1) + rest(n).cycles;
    }
};

// How the weights kernel divides a product for one form of the activations.  Pieces of up to 256 activation rows, a multiple of 32
// (of 128 as bytes [K,M]: whole 64-column atoms per CTA): as few as possible, or, where that leaves the device idle, more and
// smaller ones, which need no exchange between pairs (256 x 768 x 1536 with bytes, one piece split in four 12.8 us, four pieces
// split in four 9.9; 128 x 512 x 512 9.1 in one piece, 6.9 in four).
struct WeightsTiling {
    int act = kActExpanded, chunks = 0, bn = 0;
    long long tiles = 0;
    WeightsCost cost{};
    double cycles = 1e30;  // of the kernel and of the launch that expands the activations, from call to results
    WeightsTiling() = default;
    WeightsTiling(int M, int N, int K, int act_, bool a_is_km, const int* clusters) : act(act_)
    {
        const int unit = act == kActColumns ? 128 : 32, kb = act == kActExpanded ? 2 * BK : BK, least = (M + BN - 1) / BN;
        const long long slabs = (N + 2 * BM - 1) / (2 * BM);
        // (Expanded: the launch that does it, its passing over to the kernel, and so much of a cycle per element; transposed, the first
        // three million cost more.)
        const double elements = (double)M * K, transposed = 0.0039 * elements < 8000.0 + 0.0013 * elements ? 0.0039 * elements : 8000.0 + 0.0013 * elements;
        const double before = act == kActExpanded ? 11000.0 + (a_is_km ? transposed : 0.0009 * elements) : 7500.0;
        int next;  // (the fewest pieces with fewer rows each: many numbers of pieces round up to the same rows)
        for (int pieces = least; pieces == least || slabs * pieces <= clusters[1]; pieces = next) {
            const int rows = ((M + pieces - 1) / pieces + unit - 1) / unit * unit, n = (M + rows - 1) / rows;
            next = rows > unit ? (M + rows - unit - 1) / (rows - unit) : 0x7FFFFFFF;
            const WeightsCost c{(K + kb - 1) / kb, rows, unit, act == kActExpanded, act == kActExpanded && a_is_km, clusters};
            const double t = before + c.all(slabs * n);
            if (t < cycles) { cycles = t; chunks = n; bn = rows; tiles = slabs * n; cost = c; }
        }
    }
};

template <int ACT, int FORM>
static cudaError_t launch_weights_form(const cudaLaunchConfig_t& cfg, int w_is_nk, const CUtensorMap& map_w, const CUtensorMap& map_act, const GemmParams& p,
                                       const TilePlan& tp)
{
    return w_is_nk ? cudaLaunchKernelEx(&cfg, hif8_gemm_weights_kernel<true, ACT, FORM>, map_w, map_act, p, tp)
                   : cudaLaunchKernelEx(&cfg, hif8_gemm_weights_kernel<false, ACT, FORM>, map_w, map_act, p, tp);
}

template <int ACT>
static cudaError_t launch_weights_kernel(const cudaLaunchConfig_t& cfg, int w_is_nk, const CUtensorMap& map_w, const CUtensorMap& map_act, const GemmParams& p,
                                         const TilePlan& tp, bool one_group)
{
    if ((p.ldc * (p.c_is_f32 ? 4 : 2)) >> 32) return launch_weights_form<ACT, kFarRows>(cfg, w_is_nk, map_w, map_act, p, tp);
    if (tp.parts > 1) return launch_weights_form<ACT, kParts>(cfg, w_is_nk, map_w, map_act, p, tp);
    return one_group ? launch_weights_form<ACT, kOneGroup>(cfg, w_is_nk, map_w, map_act, p, tp)
                     : launch_weights_form<ACT, kGroups>(cfg, w_is_nk, map_w, map_act, p, tp);
}

// C = A W with the weights decoded inside the kernel.  act = kActExpanded: `a` is BF16 [M,K], written by the launch in front of
// this one, which also clears the status word; otherwise the caller's bytes.
static int launch_weights_gemm(const uint8_t* Wq, int64_t ldw, int w_is_nk, const WeightsTiling& tl, const void* a, int64_t lda, const GemmParams& p,
                               const int* clusters, cudaStream_t st)
{
    const int M = p.M, N = p.N, K = p.K, act = tl.act, kb = act == kActExpanded ? 2 * BK : BK;
    if (tl.tiles > 0x3FFFFFFF) return HIF8_ERR_SHAPE;
    const int tiles = (int)tl.tiles, pairs = clusters[1];
    CUtensorMap map_w;
    const bool okw = w_is_nk ? make_map(&map_w, Wq, (uint64_t)K, (uint64_t)N, (uint64_t)ldw, (uint32_t)kb, BM, false, (uint32_t)kb)
                             : make_map(&map_w, Wq, (uint64_t)N, (uint64_t)K, (uint64_t)ldw, BM, (uint32_t)kb, false, 128);
    if (!okw) return HIF8_ERR_CUDA;
    WeightsCost::Rest rest = tl.cost.rest(tiles);
    if (rest.parts > 1 && (p.ldc * (p.c_is_f32 ? 4 : 2)) >> 32) rest = WeightsCost::Rest{};  // (rows of C 4 GiB apart have an instantiation for whole tiles)
    const int rem = (int)rest.tiles, clear = act != kActExpanded, slabs = tiles / tl.chunks;
    // Sixteen pieces of K up to 4096 stay in L2 as eight of more do, and the instantiation for one group has the cheaper tiles; the other has the
    // cheaper sums (us in groups / as one group, activations as bytes: 4000 x 11008 x 1024 119.9 / 118.4, 3072 x 1024 x 4096 36.0 / 34.4, 3000 x 1024 x 1024 13.3 / 13.0;
    // added to FP32 171.1 / 172.4, 38.2 / 37.0 and 15.2 / 15.4, to BF16 162.1 / 190.8, 37.8 / 37.3 and 15.0 / 15.8).
    // (Not where a launch for the last round follows: both number the tiles in the same order, parts of tiles are numbered in groups, and which tiles
    // are divided along K, so how their sums are rounded, is as it is in groups.)
    const bool one_group = tl.chunks <= (K <= 4096 && !p.accumulate && rem == 0 ? 2 * kGroupPieces : kGroupPieces);
    TilePlan launch[2];
    launch[0] = TilePlan{0, tiles - rem, tl.chunks, tl.bn, slabs, tiles <= pairs ? tl.cost.best_split(tiles) : 1, clear, 0, 1, tl.bn};
    launch[1] = TilePlan{(tiles - rem) * rest.parts, rem * rest.parts, tl.chunks, rest.rows, slabs, rest.split, 0, 1, rest.parts, tl.bn};
    for (int i = 0; i < (rem ? 2 : 1); i++) {
        const TilePlan& tp = launch[i];
        CUtensorMap map_act;
        const bool oka = act == kActExpanded ? make_map3(&map_act, a, (uint64_t)K, (uint64_t)M, 1, 0, BK, (uint32_t)tp.bn / 2)
                         : act == kActRows   ? make_map(&map_act, a, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, (uint32_t)tp.bn / 2)
                                             : make_map(&map_act, a, (uint64_t)M, (uint64_t)K, (uint64_t)lda, (uint32_t)tp.bn / 2, BK);
        if (!oka) return HIF8_ERR_CUDA;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(2u * (unsigned)(tp.split > 1 ? tp.count * tp.split : (tp.count < pairs ? tp.count : pairs)));
        cfg.blockDim = dim3(kThreadsWd);
        cfg.dynamicSmemBytes = kSmemBytesMax;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2u * (unsigned)tp.split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 2;
        const cudaError_t rc = act == kActExpanded ? launch_weights_kernel<kActExpanded>(cfg, w_is_nk, map_w, map_act, p, tp, one_group)
                               : act == kActRows   ? launch_weights_kernel<kActRows>(cfg, w_is_nk, map_w, map_act, p, tp, one_group)
                                                   : launch_weights_kernel<kActColumns>(cfg, w_is_nk, map_w, map_act, p, tp, one_group);
        if (rc != cudaSuccess) return HIF8_ERR_CUDA;
        g_launches.fetch_add(1, std::memory_order_relaxed);
    }
    return cudaGetLastError() == cudaSuccess ? HIF8_OK : HIF8_ERR_CUDA;
}

template <bool W_IS_NK, bool ACT_BF16, bool WIDE>
static cudaError_t launch_narrow_form(const cudaLaunchConfig_t& cfg, bool cluster, const CUtensorMap& map_act, const CUtensorMap& map_w, const GemmParams& p,
                                      int mp, const NarrowPlan& plan)
{
    return cluster ? cudaLaunchKernelEx(&cfg, hif8_gemm_narrow_kernel<W_IS_NK, ACT_BF16, true, WIDE>, map_act, map_w, p, mp, plan)
                   : cudaLaunchKernelEx(&cfg, hif8_gemm_narrow_kernel<W_IS_NK, ACT_BF16, false, WIDE>, map_act, map_w, p, mp, plan);
}
template <bool W_IS_NK>
static cudaError_t launch_narrow_kernel(const cudaLaunchConfig_t& cfg, bool cluster, bool act_bf16, const CUtensorMap& map_act, const CUtensorMap& map_w,
                                        const GemmParams& p, int mp, const NarrowPlan& plan)
{
    if (act_bf16) return launch_narrow_form<W_IS_NK, true, true>(cfg, cluster, map_act, map_w, p, mp, plan);
    return mp <= kNwWideBytesM ? launch_narrow_form<W_IS_NK, false, true>(cfg, cluster, map_act, map_w, p, mp, plan)
                               : launch_narrow_form<W_IS_NK, false, false>(cfg, cluster, map_act, map_w, p, mp, plan);
}

// How the warp kernel divides a product, and what that takes in cycles from call to results.  The terms are fitted to 670 measured
// calls (1 to 256 rows, N and K 512 to 8192, all divisions; within 15 % of most): the activations that a block decodes, the weights
// that go through its shared memory, deposits, and what a unit costs a warp one after the other.
struct WarpTiling {
    WarpPlan plan{};
    int mt = 0, row_blocks = 0;
    double cycles = 1e30;
    struct Limits {
        int cols, chunks;  // columns of a unit; 64-k blocks of a slice at most
        uint32_t deposit;
    };
    template <bool W_IS_NK, int MT>
    static Limits limits()
    {
        using S = WarpShape<W_IS_NK, MT>;
        return Limits{S::kCols, S::CH, S::kDeposit};
    }
    WarpTiling() = default;
    // the division that takes the fewest cycles, if it takes fewer than `below` (otherwise mt = 0)
    WarpTiling(int M, int N, int K, bool w_is_nk, bool a_is_km, const int* clusters, double below) : cycles(below)
    {
        if ((double)M * N * K > 4e9 || K > 4096 * kWarpMaxCluster || (!w_is_nk && (N & 3))) return;  // (far beyond what it is good for; a thread loads four columns of [K,N] in one piece)
        for (int m = a_is_km ? 4 : 1; m <= 4; m *= 2)
            if (m == 1 ? M <= 8 : (a_is_km || 4 * m < M)) divide(M, N, K, w_is_nk, m, clusters);
    }
    void divide(int M, int N, int K, bool w_is_nk, int m, const int* clusters)
    {
        const int blocks = (M + 8 * m - 1) / (8 * m);
        if (blocks > 65535) return;  // the second dimension of a grid
        const Limits l = w_is_nk ? (m == 1 ? limits<true, 1>() : (m == 2 ? limits<true, 2>() : limits<true, 4>()))
                                 : (m == 1 ? limits<false, 1>() : (m == 2 ? limits<false, 2>() : limits<false, 4>()));
        const int units = (N + l.cols - 1) / l.cols, kb = (K + 63) / 64;
        for (int c = 1; c <= kWarpMaxCluster; c++) {
            if (clusters[c] <= 0) continue;
            const int fit = clusters[c] / blocks, n = fit < 1 ? 1 : (fit < units ? fit : units), nu = (units + n - 1) / n;
            const int rounds = fit < 1 ? (blocks + clusters[c] - 1) / clusters[c] : 1;
            if ((uint32_t)(units / n + 1) * l.deposit > kWarpSumBytes) continue;
            const int least = (kb + c * l.chunks - 1) / (c * l.chunks);  // (with fewer slices a slice is longer than a warp can hold)
            // (what no division into this many blocks goes below: most are not looked at)
            if (rounds * (w_is_nk ? 4840.0 + 46.0 * nu * least * m : 5510.0 + 122.0 * nu * (kb / c) + 34.0 * nu * least * m) >= cycles) continue;
            for (int s = least; s <= kWarpWarps; s++) {
                const int chunks = (kb + c * s - 1) / (c * s), lanes = kWarpWarps / s;
                if (chunks > l.chunks || (kb + chunks - 1) / chunks <= (c - 1) * s) continue;  // (the latter: a block of the cluster without work)
                const int turns = (nu + lanes - 1) / lanes, active = s * (lanes < nu ? lanes : nu);
                const double t = rounds * (w_is_nk ? 3500.0 + 40.0 * active * chunks * m + 46.0 * nu * s * m + 450.0 * turns + 890.0 * turns * chunks + (c > 1 ? 4100.0 : 0.0)
                                                   : 3300.0 + 24.0 * active * chunks * m + 122.0 * nu * s * chunks + 34.0 * nu * s * m + 970.0 * turns +
                                                         1240.0 * turns * chunks + (c > 1 ? 4400.0 : 0.0));
                if (t < cycles) {
                    cycles = t; mt = m; row_blocks = blocks;
                    plan.chunks = chunks; plan.slices = s; plan.lanes = lanes; plan.cluster = c; plan.units = units;
                    plan.q = units / n; plan.rem = units % n;
                }
            }
        }
    }
    int clusters_used() const { return (plan.units - plan.rem) / plan.q; }  // (no more clusters than units: q > 0)
};

template <int MT>
static cudaError_t launch_warp_kernel(const cudaLaunchConfig_t& cfg, bool w_is_nk, const uint8_t* A, long long lda, const uint8_t* W, long long ldw,
                                      const GemmParams& p, const WarpPlan& plan)
{
    return w_is_nk ? cudaLaunchKernelEx(&cfg, hif8_gemm_warp_kernel<true, false, MT>, A, lda, W, ldw, p, plan)
                   : cudaLaunchKernelEx(&cfg, hif8_gemm_warp_kernel<false, false, MT>, A, lda, W, ldw, p, plan);
}

static int launch_warp_gemm(const uint8_t* A, int64_t lda, int a_is_km, const uint8_t* W, int64_t ldw, int w_is_nk, const GemmParams& p, const WarpTiling& tl,
                            cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(tl.clusters_used() * tl.plan.cluster), (unsigned)tl.row_blocks);
    cfg.blockDim = dim3(kWarpThreads);
    cfg.dynamicSmemBytes = kSmemBytesMax;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)tl.plan.cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = tl.plan.cluster > 1 ? 2 : 1;
    cudaError_t rc;
    if (a_is_km)
        rc = w_is_nk ? cudaLaunchKernelEx(&cfg, hif8_gemm_warp_kernel<true, true, 4>, A, (long long)lda, W, (long long)ldw, p, tl.plan)
                     : cudaLaunchKernelEx(&cfg, hif8_gemm_warp_kernel<false, true, 4>, A, (long long)lda, W, (long long)ldw, p, tl.plan);
    else if (tl.mt == 1) rc = launch_warp_kernel<1>(cfg, w_is_nk, A, lda, W, ldw, p, tl.plan);
    else if (tl.mt == 2) rc = launch_warp_kernel<2>(cfg, w_is_nk, A, lda, W, ldw, p, tl.plan);
    else rc = launch_warp_kernel<4>(cfg, w_is_nk, A, lda, W, ldw, p, tl.plan);
    if (rc != cudaSuccess) return HIF8_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? HIF8_OK : HIF8_ERR_CUDA;
}

static std::atomic<int> g_path_policy{HIF8_GEMM_PATH_AUTO};

extern "C" int hif8_gemm_path_policy(int policy)
{
    if (policy != HIF8_GEMM_PATH_AUTO && policy != HIF8_GEMM_PATH_EXPAND_BOTH && policy != HIF8_GEMM_PATH_NO_WARP &&
        policy != HIF8_GEMM_PATH_EXPAND_A && policy != HIF8_GEMM_PATH_WARP)
        return HIF8_ERR_FLAGS;
    return g_path_policy.exchange(policy, std::memory_order_relaxed);
}

// How the narrow kernel divides a product.  Cycles: a k-block was taken to cost 500 (mp = 16) to 590 (64); it is 390 to 423 now, 530 to 828 with activations as
// bytes, but with those figures in its place 250 products came out no faster in the mean and some 10 to 25 % slower.  A cluster's exchange 4000, and
// clusters of eight start later; ranges of slabs end in a reduction of 2500 + 290 mp.  A cluster per slab (or one CTA: split 1), or,
// when the workspace holds the partial sums of the slabs that a range boundary cuts, one CTA per SM with equal ranges: for many
// slabs that do not divide among the SMs, and few rows.
struct NarrowTiling {
    int split = 0;         // of the best clusters
    bool ranges = false;   // ranges are better
    long long grid = 0, pmax = 0;
    double cycles = 1e30;
    NarrowTiling(int M, int N, int K, int sm_count, const int* clusters, bool with_ranges)
    {
        const int mp = (M + 15) & ~15;
        const long long slabs = (N + BM - 1) / BM, num_pb = (K + BK2 - 1) / BK2, total = slabs * num_pb;  // pair blocks: two k-blocks
        const double c_pb = 2.0 * (470.0 + 1.9 * mp);
        for (int s = 1; s <= kNwMaxSplit && s <= num_pb; s *= 2) {
            if (clusters[s] <= 0) continue;
            const long long rounds = (slabs + clusters[s] - 1) / clusters[s];
            const double c = (double)rounds * ((double)((num_pb + s - 1) / s) * c_pb + 4500.0 + (s == 1 ? 0.0 : (s < 8 ? 4000.0 : 6000.0)));
            if (c < cycles) { cycles = c; split = s; }
        }
        // four or more pair blocks per CTA, but never fewer CTAs than slabs
        grid = total / 4 < sm_count ? total / 4 : sm_count;
        const long long floor_g = slabs < sm_count ? slabs : sm_count;
        if (grid < floor_g) grid = floor_g;
        const long long per = total / grid;
        pmax = (num_pb + per - 1) / per + 1;
        const double c = (double)(per + 1) * c_pb + 4500.0 + 2500.0 + 290.0 * mp;
        if (with_ranges && c < cycles) { cycles = c; ranges = true; }
    }
};

// Which kernel takes a product, and how it divides it: a function of the sizes, the layouts and what the workspace has room for, so
// it is kept for the 64 used last.  (The search over divisions takes 0.5 us on the host, 2 us at most: products of 1 to 8192 rows, N and K 16
// to 28672.  It runs outside the lock, so that threads with new sizes do not wait for one another.)
enum GemmForm { kFormWarp, kFormNarrow, kFormWeights, kFormPair };
struct GemmKey {
    int M, N, K, dev, w_is_nk, a_is_km, room, policy;
};
struct GemmChoice {
    GemmForm form;
    WarpTiling warp;
    WeightsTiling weights;
};
static LruCache<GemmKey, GemmChoice, 64> g_choices;

// false: the kernel that hif8_gemm_path_policy asks for has no division of this product
static bool choose(const GemmKey& k, int sm_count, const int* wd_clusters, const int* nw_clusters, const int* wp_clusters, GemmChoice* out)
{
    if (k.policy == HIF8_GEMM_PATH_WARP) {
        out->form = kFormWarp;
        out->warp = WarpTiling(k.M, k.N, k.K, k.w_is_nk, k.a_is_km, wp_clusters, 1e30);
        return out->warp.mt > 0;
    }
    const bool narrow = !k.a_is_km && k.M <= kNarrowMaxM;
    out->form = narrow ? kFormNarrow : kFormWeights;
    if (!narrow) {
        const WeightsTiling bytes(k.M, k.N, k.K, k.a_is_km ? kActColumns : kActRows, k.a_is_km, wd_clusters);
        const WeightsTiling expanded(k.M, k.N, k.K, kActExpanded, k.a_is_km, wd_clusters);
        // (3000: bytes [K,M] of 16 rows, of which every pair copies the same few lines)
        const double crowded = k.a_is_km && k.M < 32 ? 3000.0 * (bytes.tiles < wd_clusters[1] ? (double)bytes.tiles / wd_clusters[1] : 1.0) : 0.0;
        out->weights = k.room && (k.policy == HIF8_GEMM_PATH_EXPAND_A || expanded.cycles < bytes.cycles + crowded) ? expanded : bytes;
        // Expanding W as well only pays when the product is large enough to win back the pass over W (3 bytes per element moved, at
        // 3300 bytes a cycle, and a launch) by the cheaper k-blocks and tiles of the pair kernel: 545 cycles per
        // 64 k and nothing between tiles, against the weights kernel's cost above.  Measured (us, both expanded / weights decoded in
        // the kernel): 2048 x 7168 x 4096 105 / 98, 3072 rows 130 / 133, 4096 rows 172 / 176; 1536 x 8192 x 1024 28.5 / 33;
        // 2048 x 16384 x 8192 381 / 357, 4096 rows 702 / 732.
        const long long pair_rounds = ((long long)((k.M + 2 * BM - 1) / (2 * BM)) * ((k.N + BN - 1) / BN) + sm_count / 2 - 1) / (sm_count / 2);
        const double expand_w = 6000.0 + 3.0 * (double)k.K * k.N / 3300.0, pair_cycles = (double)pair_rounds * ((k.K + BK - 1) / BK * 545.0 + 500.0);
        if (k.room == 2 && k.policy != HIF8_GEMM_PATH_EXPAND_A &&
            (k.policy == HIF8_GEMM_PATH_EXPAND_BOTH ||
             expand_w + pair_cycles < 1.03 * expanded.cost.all(expanded.tiles))) {  // (equal at 1.03: the lookups also cost clock under the power limit)
            out->form = kFormPair;
            return true;
        }
    }
    if (k.policy != HIF8_GEMM_PATH_AUTO) return true;
    // (1.2: the search takes the division whose time is underestimated most; 6000: the launch in front of the narrow kernel, its start and end)
    const double other = narrow ? NarrowTiling(k.M, k.N, k.K, sm_count, nw_clusters, k.room > 0).cycles + 6000.0 : out->weights.cycles;
    out->warp = WarpTiling(k.M, k.N, k.K, k.w_is_nk, k.a_is_km, wp_clusters, other / 1.2);
    if (out->warp.mt > 0) out->form = kFormWarp;
    return true;
}

static int gemm_entry(const uint8_t* Aq, int64_t lda, int a_is_km, const uint8_t* Wq, int64_t ldw, int w_is_nk, void* C,
                      int64_t ldc, int c_dtype, int M, int N, int K, const int* d_scale_exp_a, const int* d_scale_exp_w,
                      const int* d_scale_exp_w_channel, int accumulate, void* workspace, size_t workspace_bytes,
                      hif8_stream_t stream)
{
    if (c_dtype != HIF8_BF16 && c_dtype != HIF8_F32) return HIF8_ERR_DTYPE;
    if (M < 0 || N < 0 || K < 0 || (K & 15)) return HIF8_ERR_SHAPE;
    if (lda < (a_is_km ? M : K) || ldc < N || ldw < (w_is_nk ? K : N)) return HIF8_ERR_SHAPE;
    if (M == 0 || N == 0) return HIF8_OK;
    if (!Aq || !Wq || !C) return HIF8_ERR_NULL;
    const size_t c_item = c_dtype == HIF8_F32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(Aq) & 15) || (reinterpret_cast<uintptr_t>(Wq) & 15) || (reinterpret_cast<uintptr_t>(C) & 15) ||
        (lda & 15) || (ldw & 15) || ((ldc * c_item) & 15))
        return HIF8_ERR_ALIGN;
    if (!workspace || workspace_bytes < kGemmWorkspaceBytes || (reinterpret_cast<uintptr_t>(workspace) & 15))
        return HIF8_ERR_WORKSPACE;
    if (K == 0) return HIF8_ERR_SHAPE;
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HIF8_ERR_CUDA;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (major != 10) return HIF8_ERR_CUDA;

    GemmParams p{};
    p.C = C; p.ldc = ldc; p.c_is_f32 = c_dtype == HIF8_F32; p.M = M; p.N = N; p.K = K;
    p.d_sa = d_scale_exp_a; p.d_sw = d_scale_exp_w; p.d_sw_channel = d_scale_exp_w_channel;
    p.accumulate = accumulate ? 1 : 0;
    p.status = reinterpret_cast<int*>(workspace);
    cudaStream_t st = (cudaStream_t)stream;
    note_status_word(st, reinterpret_cast<const int*>(workspace));

    int sm_count = 0;
    const int *wd_clusters = nullptr, *nw_clusters = nullptr, *wp_clusters = nullptr;
    if (!gemm_kernels_ready(dev, &sm_count, &wd_clusters, &nw_clusters, &wp_clusters)) return HIF8_ERR_CUDA;

    // Operands as BF16 in the workspace: none, the activations, both.
    const size_t bytes_a = (((size_t)M * K * 2) + 255) & ~(size_t)255, bytes_w = (((size_t)K * N * 2) + 255) & ~(size_t)255;
    const bool a_contiguous = lda == (a_is_km ? M : K), w_contiguous = ldw == (w_is_nk ? K : N), ws_aligned = !(reinterpret_cast<uintptr_t>(workspace) & 255);
    const bool room_a = a_contiguous && ws_aligned && workspace_bytes >= kGemmWorkspaceBytes + bytes_a;
    const bool room_w = room_a && w_contiguous && workspace_bytes >= kGemmWorkspaceBytes + bytes_a + bytes_w;
    GemmKey key;
    std::memset(&key, 0, sizeof key);
    key.M = M; key.N = N; key.K = K; key.dev = dev;
    key.w_is_nk = w_is_nk != 0; key.a_is_km = a_is_km != 0; key.room = room_w ? 2 : (room_a ? 1 : 0);
    key.policy = g_path_policy.load(std::memory_order_relaxed);
    GemmChoice choice;
    if (!g_choices.find(key, &choice)) {
        if (!choose(key, sm_count, wd_clusters, nw_clusters, wp_clusters, &choice)) return HIF8_ERR_SHAPE;
        g_choices.put(key, choice);
    }
    if (choice.form == kFormWarp) return launch_warp_gemm(Aq, lda, a_is_km, Wq, ldw, w_is_nk, p, choice.warp, st);
    // the status word is cleared on the stream before the kernels; the narrow path clears its tickets in the same operation
    size_t clear_bytes = 4;

    // Narrow products: the weight-streaming kernel, whatever the workspace
    if (choice.form == kFormNarrow) {
        const int mp = (M + 15) & ~15;
        CUtensorMap map_act, map_ws;
        if (!make_map(&map_act, Aq, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK2, (uint32_t)mp)) return HIF8_ERR_CUDA;
        // (Weight tiles: 128-byte rows with the 128-byte swizzle, of 128 k or of 128 columns.  Columns: the other half of a line of 256 bytes is
        // another slab's, which another CTA reads at another time, and is not brought along: 16 x 28672 x 8192 58.0 -> 48.8 us a call, 64 rows 68.2 -> 64.4.)
        const bool okn = w_is_nk ? make_map(&map_ws, Wq, (uint64_t)K, (uint64_t)N, (uint64_t)ldw, BK2, BM, false, 128)
                                 : make_map(&map_ws, Wq, (uint64_t)N, (uint64_t)K, (uint64_t)ldw, BM, BK2, false, 128, true);
        if (!okn) return HIF8_ERR_CUDA;
        const long long slabs = (N + BM - 1) / BM, num_pb = (K + BK2 - 1) / BK2;  // pair blocks: two k-blocks
        NarrowPlan plan{};
        const long long total = slabs * num_pb;
        if (total > 0x3FFFFFFF) return HIF8_ERR_SHAPE;
        const NarrowTiling nt(M, N, K, sm_count, nw_clusters, true);
        plan.split = nt.split;
        long long grid = slabs * plan.split;
        if (nt.ranges) {
            const size_t ticket_bytes = (((size_t)slabs * kEpiWarps * 4) + 255) & ~(size_t)255;
            const size_t part_bytes = (size_t)slabs * nt.pmax * mp * BM * 4;
            if (workspace_bytes >= kGemmWorkspaceBytes + ticket_bytes + part_bytes && ws_aligned) {
                unsigned char* wsb = reinterpret_cast<unsigned char*>(workspace) + kGemmWorkspaceBytes;
                plan.tickets = reinterpret_cast<unsigned*>(wsb);
                plan.part = reinterpret_cast<float*>(wsb + ticket_bytes);
                plan.pmax = (int)nt.pmax;
                plan.split = 0;
                grid = nt.grid;
                clear_bytes = kGemmWorkspaceBytes + ticket_bytes;  // the tickets follow the status block
            }
        }
        if (grid > 0x7FFFFFFFll) return HIF8_ERR_SHAPE;
        plan.q = (int)(total / grid); plan.rem = (int)(total % grid);
        // With room left for the activations as BF16 (2 M K bytes behind the partial sums) they are expanded once, here,
        // and their tiles are copied straight into the operand stages: otherwise every CTA decodes the activation tile of
        // every k-block again for each of its slabs, a seventh (16 rows) to a third (64 rows) of the kernel's table lookups.
        bool act_bf16 = false;
        {
            const size_t used = clear_bytes > 4 ? clear_bytes + (size_t)slabs * plan.pmax * mp * BM * 4 : kGemmWorkspaceBytes;
            const size_t off = (used + 255) & ~(size_t)255, bytes_act = (size_t)M * K * 2;
            if (lda == K && workspace_bytes >= off + bytes_act && !(reinterpret_cast<uintptr_t>(workspace) & 255)) {
                unsigned char* a_bf = reinterpret_cast<unsigned char*>(workspace) + off;
                if (!make_map(&map_act, a_bf, (uint64_t)K, (uint64_t)M, (uint64_t)K, BK, (uint32_t)mp, true)) return HIF8_ERR_CUDA;
                if (launch_expand_activations(Aq, a_bf, (unsigned long long)M * K, workspace, clear_bytes, sm_count, st) != cudaSuccess) return HIF8_ERR_CUDA;
                act_bf16 = true;
            }
        }
        plan.clear_status = !act_bf16 && !plan.tickets;
        if (!act_bf16 && plan.tickets && cudaMemsetAsync(workspace, 0, clear_bytes, st) != cudaSuccess) return HIF8_ERR_CUDA;
        cudaLaunchConfig_t cn{};
        cn.gridDim = dim3((unsigned)grid);
        cn.blockDim = dim3(kThreadsN);
        cn.dynamicSmemBytes = kSmemBytesMax;
        cn.stream = st;
        // with the preparing kernel right in front: programmatic stream serialization (that kernel lets its dependents start
        // at once; this one waits for its completion once its own set-up is done)
        cudaLaunchAttribute an[2];
        int n_an = 0;
        if (act_bf16) {
            an[n_an].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            an[n_an++].val.programmaticStreamSerializationAllowed = 1;
        }
        if (plan.split > 1) {
            an[n_an].id = cudaLaunchAttributeClusterDimension;
            an[n_an].val.clusterDim.x = (unsigned)plan.split; an[n_an].val.clusterDim.y = 1; an[n_an++].val.clusterDim.z = 1;
        }
        cn.attrs = an; cn.numAttrs = (unsigned)n_an;
        cudaError_t nrc;
        const bool cluster = plan.split > 1;
        nrc = w_is_nk ? launch_narrow_kernel<true>(cn, cluster, act_bf16, map_act, map_ws, p, mp, plan)
                      : launch_narrow_kernel<false>(cn, cluster, act_bf16, map_act, map_ws, p, mp, plan);
        if (nrc != cudaSuccess) return HIF8_ERR_CUDA;
        g_launches.fetch_add(1, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess ? HIF8_OK : HIF8_ERR_CUDA;
    }

    if (choice.form == kFormWeights && choice.weights.act != kActExpanded) return launch_weights_gemm(Wq, ldw, w_is_nk, choice.weights, Aq, lda, p, wd_clusters, st);
    // The activations are expanded once (an A given as [K,M] is written as [M,K] meanwhile); either launch clears the status word.
    // For the pair kernel the weights too: each HiF8 byte is then decoded exactly once.
    unsigned char* a_bf = reinterpret_cast<unsigned char*>(workspace) + kGemmWorkspaceBytes;
    int rc = HIF8_OK;
    if (a_is_km) rc = decode_transpose_bf16(Aq, a_bf, K, M, reinterpret_cast<uint32_t*>(workspace), st);
    else if (launch_expand_activations(Aq, a_bf, (unsigned long long)M * K, workspace, 4, sm_count, st) != cudaSuccess) rc = HIF8_ERR_CUDA;
    if (rc != HIF8_OK) return rc;
    if (choice.form == kFormWeights) return launch_weights_gemm(Wq, ldw, w_is_nk, choice.weights, a_bf, K, p, wd_clusters, st);
    unsigned char* w_bf = a_bf + bytes_a;
    // (a block of the pair kernel, which starts under this launch, has no room beside blocks that hold a 32 KiB table: below eight
    // million codes that costs more than such a table saves, 2758 x 2816 x 848 21.1 -> 22.3 us)
    rc = decode_codes(Wq, w_bf, HIF8_BF16, (size_t)K * N, 0, (size_t)1 << 23, st);
    return rc != HIF8_OK ? rc : launch_bf16_pair_gemm(a_bf, w_bf, w_is_nk, p, st);
}

extern "C" int hif8_gemm(const uint8_t* Aq, int64_t lda, const uint8_t* Wq, int64_t ldw, int w_is_nk, void* C, int64_t ldc,
                         int c_dtype, int M, int N, int K, const int* d_scale_exp_a, const int* d_scale_exp_w,
                         void* workspace, size_t workspace_bytes, hif8_stream_t stream)
{
    return gemm_entry(Aq, lda, 0, Wq, ldw, w_is_nk, C, ldc, c_dtype, M, N, K, d_scale_exp_a, d_scale_exp_w, nullptr, 0, workspace,
                      workspace_bytes, stream);
}

extern "C" int hif8_gemm_channel_scaled(const uint8_t* Aq, int64_t lda, const uint8_t* Wq, int64_t ldw, int w_is_nk, void* C,
                                        int64_t ldc, int c_dtype, int M, int N, int K, const int* d_scale_exp_a,
                                        const int* d_scale_exp_w_channel, void* workspace, size_t workspace_bytes,
                                        hif8_stream_t stream)
{
    if (!d_scale_exp_w_channel && M > 0 && N > 0) return HIF8_ERR_NULL;
    return gemm_entry(Aq, lda, 0, Wq, ldw, w_is_nk, C, ldc, c_dtype, M, N, K, d_scale_exp_a, nullptr, d_scale_exp_w_channel, 0,
                      workspace, workspace_bytes, stream);
}

extern "C" int hif8_gemm_ex(const uint8_t* Aq, int64_t lda, int a_is_km, const uint8_t* Wq, int64_t ldw, int w_is_nk, void* C,
                            int64_t ldc, int c_dtype, int M, int N, int K, const int* d_scale_exp_a, const int* d_scale_exp_w,
                            const int* d_scale_exp_w_channel, int accumulate, void* workspace, size_t workspace_bytes,
                            hif8_stream_t stream)
{
    return gemm_entry(Aq, lda, a_is_km ? 1 : 0, Wq, ldw, w_is_nk ? 1 : 0, C, ldc, c_dtype, M, N, K, d_scale_exp_a,
                      d_scale_exp_w_channel ? nullptr : d_scale_exp_w, d_scale_exp_w_channel, accumulate, workspace,
                      workspace_bytes, stream);
}

extern "C" int hif8_gemm_status(const void* workspace, hif8_stream_t stream)
{
    if (!workspace) return HIF8_ERR_NULL;
    int v = 0;
    if (cudaMemcpyAsync(&v, workspace, sizeof v, cudaMemcpyDeviceToHost, (cudaStream_t)stream) != cudaSuccess) return HIF8_ERR_CUDA;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return HIF8_ERR_CUDA;
    return v == 0 ? HIF8_OK : HIF8_ERR_DEVICE_TIMEOUT;
}

extern "C" int hif8_last_device_status(hif8_stream_t stream)
{
    StatusKey k;
    std::memset(&k, 0, sizeof k);
    k.stream = (cudaStream_t)stream;
    StatusVal v;
    if (!g_last_status.find(k, &v)) return HIF8_OK;  // no GEMM-class call was made on this stream
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != v.dev) return HIF8_ERR_CUDA;
    return hif8_gemm_status(v.word, stream);
}

extern "C" int hif8_selftest_host_caches(int* failed_check)
{
    int check = 0;
    auto fail = [&](int c) { if (failed_check) *failed_check = c; return HIF8_ERR_SHAPE; };
    {   // set-up record: one initialisation per device ordinal, each with its own value
        static PerDevice<int> rec;
        static int calls;
        calls = 0;
        auto init = [](int dev, int* out) { calls++; *out = 1000 + dev; };
        const int* a = rec.get(3, init);
        const int* b = rec.get(5, init);
        const int* c = rec.get(3, init);
        check = 1; if (!a || !b || a != c || *a != 1003 || *b != 1005) return fail(check);
        check = 2; if (calls > 2) return fail(check);   // at most one per ordinal (zero when run before in this process)
        check = 3; if (rec.get(-1, init) || rec.get(kMaxDevices, init)) return fail(check);
    }
    {   // keyed cache: hit after miss, a failed build is not kept, the least recently used entry is replaced
        struct K { uint64_t a; uint32_t b; uint32_t pad; };
        LruCache<K, int, 4> cache;
        int builds = 0;
        auto make = [&](const K& k, int* v) { builds++; *v = (int)(k.a * 10 + k.b); return k.b != 99; };
        auto key = [](uint64_t a, uint32_t b) { K k; std::memset(&k, 0, sizeof k); k.a = a; k.b = b; return k; };
        int v = 0;
        check = 4; if (!cache.lookup_or_make(key(1, 2), &v, make) || v != 12 || builds != 1) return fail(check);
        check = 5; if (!cache.lookup_or_make(key(1, 2), &v, make) || v != 12 || builds != 1) return fail(check);
        check = 6; if (cache.lookup_or_make(key(7, 99), &v, make) || builds != 2) return fail(check);
        check = 7; if (cache.lookup_or_make(key(7, 99), &v, make) || builds != 3) return fail(check);
        for (uint64_t a = 2; a <= 4; a++) cache.lookup_or_make(key(a, 0), &v, make);   // cache now holds (1,2), 2, 3, 4
        check = 8; if (!cache.lookup_or_make(key(1, 2), &v, make) || builds != 6) return fail(check);   // refreshes (1,2)
        cache.lookup_or_make(key(5, 0), &v, make);                                     // replaces key 2, the oldest
        check = 9; if (builds != 7 || !cache.lookup_or_make(key(1, 2), &v, make) || builds != 7) return fail(check);
        check = 10; if (!cache.lookup_or_make(key(2, 0), &v, make) || builds != 8) return fail(check);
        check = 11; if (cache.hits() != 3 || cache.misses() != 6) return fail(check);
        int w = 0;
        cache.put(key(1, 2), 77);
        check = 12; if (!cache.find(key(1, 2), &w) || w != 77 || cache.find(key(42, 0), &w)) return fail(check);
    }
    if (failed_check) *failed_check = 0;
    return HIF8_OK;
}

extern "C" int hif8_selftest_wait_timeout(void* workspace, unsigned limit_ms, hif8_stream_t stream)
{
    if (!workspace) return HIF8_ERR_NULL;
    if (limit_ms == 0 || limit_ms > 1000) return HIF8_ERR_SHAPE;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(workspace, 0, 4, st) != cudaSuccess) return HIF8_ERR_CUDA;
    note_status_word(st, reinterpret_cast<const int*>(workspace));
    wait_selftest_kernel<<<1, 32, 0, st>>>(reinterpret_cast<int*>(workspace), (unsigned long long)limit_ms * 1000000ull);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? HIF8_OK : HIF8_ERR_CUDA;
}
