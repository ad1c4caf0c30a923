// The GEMM kernel for few activation rows (included by hif8_gemm.cu, whose helpers it uses).
//
// Every warp works alone on a slice of K: it keeps the slice's activations as BF16 in registers (the B operand of mma.sync, up to
// 32 rows a block, decoded once), streams the weight bytes of one unit of columns after the other from global memory into
// registers, looks their values up and multiplies.  No operand is staged in shared memory, no barrier stands between a load and
// its use, and next to nothing has to be set up.  What is shared: the decode table, and the partial sums.  The warps of a block
// that work on the same columns deposit their sums of a unit in shared memory, and in the middle of their next unit each adds
// its share of the deposits, pairwise.  When K takes more slices than a block has warps, a cluster of blocks works on the
// same columns, and the blocks' sums are added in rank order through distributed shared memory at the end.
//
// What bounds it: for the small products it is chosen for, latency (loads, the activations' decoding, a unit's deposit and sum:
// about 5000 cycles with one unit a warp), which is why it exists: the tensor-memory kernels spend 12000 on barriers, tensor memory,
// descriptors, hand-overs between their roles and another launch that expands the activations.  us a call in a graph, [N,K] weights,
// the kernel that would take it otherwise / this: 4 x 512 x 512 6.7 / 2.7, 16 x 1024 x 1024 7.1 / 3.8, 16 x 2048 x 2048 8.4 / 5.2,
// 128 x 512 x 1024 6.8 / 5.4; [K,N]: 16 x 512 x 512 7.0 / 3.9; too large for it: 256 x 768 x 1536 8.6 / 9.3.  A stream of weights it does not sustain (16 x 28672 x 8192: 100 us against 60): all warps of a block
// wait for one another once per unit, and four warps a scheduler do not cover the lookups' latency with 64 registers of activations each.
//
// Column units.  [N,K] weights: 16 columns, the rows of one m16n8k16 operand.  A thread (g = lane / 4, t = lane % 4) loads 16
// consecutive k of the columns g and g + 8; which k of a block of 64 are multiplied together is the operands' own business as
// long as both agree, so step s of the block takes bytes 4 s .. 4 s + 3 of every thread's sixteen.  [K,N] weights: 2 UT columns per
// thread from four k rows, transposed four by four with byte permutes.
template <bool W_IS_NK, int MT>
struct WarpShape {
    static constexpr int UT = W_IS_NK ? 1 : 2;      // m16 tiles per unit
    static constexpr int kCols = 16 * UT;           // columns per unit
    static constexpr int CH = (W_IS_NK ? 4 : 2) / (MT == 4 ? 2 : 1);  // 64-k blocks per slice at most: the registers of the activations and weights
    static constexpr int kRows = 8 * MT;            // activation rows per block
    static constexpr int kSums = kCols * kRows;     // sums of a unit
    static constexpr uint32_t kDeposit = kSums * 4; // bytes a warp deposits per unit
};
constexpr int kWarpWarps = 16, kWarpThreads = kWarpWarps * 32, kWarpMaxCluster = 8;
constexpr uint32_t kWarpSumBytes = 62 * 1024;  // sums of a block at most: what lies in front of the 64 KiB boundary of the table

struct WarpPlan {
    int chunks;      // 64-k blocks per slice
    int slices;      // slices (warps that work on the same columns) per block
    int lanes;       // column lanes per block: warps / slices
    int cluster;     // blocks along K
    int units;       // column units
    int q, rem;      // units per cluster; the first rem clusters take one more
};

// Shared memory: the sums of the block's units, the 64 KiB table on a 64 KiB boundary (see decode8), deposits, barriers.  The sums
// go in front of the table (up to 63 KiB).
struct WarpSmem {
    uint32_t sums, lut, dep, bars, end;
    __device__ WarpSmem(uint32_t raw, uint32_t dep_bytes)
    {
        sums = (raw + 127u) & ~127u;
        lut = (raw + kLutBytesWide - 1) & ~(kLutBytesWide - 1);
        dep = lut + kLutBytesWide;
        bars = dep + dep_bytes;
        end = bars + 2 * kWarpWarps * 8 + 16;
    }
    __device__ uint32_t abort_flag() const { return bars + 2 * kWarpWarps * 8; }
};

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// weights are read once: not kept in L1, first to leave L2
__device__ __forceinline__ uint4 ld_weights_v4(const uint8_t* p, uint64_t policy)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_weights_u32(const uint8_t* p, uint64_t policy)
{
    uint32_t v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(policy) : "memory");
    return v;
}
// four codes -> two words of two BF16 (table with rows of 256 bytes)
__device__ __forceinline__ void decode4(uint32_t w, uint32_t lut_lane, uint32_t& lo, uint32_t& hi)
{
    const uint32_t c0 = lds_u32(__byte_perm(w, lut_lane, 0x7604)), c1 = lds_u32(__byte_perm(w, lut_lane, 0x7614));
    const uint32_t c2 = lds_u32(__byte_perm(w, lut_lane, 0x7624)), c3 = lds_u32(__byte_perm(w, lut_lane, 0x7634));
    lo = __byte_perm(c0, c1, 0x5410);
    hi = __byte_perm(c2, c3, 0x5410);
}
// byte j of r[i] -> byte i of out[j]
__device__ __forceinline__ void transpose4x4(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3, uint32_t (&out)[4])
{
    const uint32_t a = __byte_perm(r0, r1, 0x5140), b = __byte_perm(r0, r1, 0x7362), c = __byte_perm(r2, r3, 0x5140), d = __byte_perm(r2, r3, 0x7362);
    out[0] = __byte_perm(a, c, 0x5410); out[1] = __byte_perm(a, c, 0x7632);
    out[2] = __byte_perm(b, d, 0x5410); out[3] = __byte_perm(b, d, 0x7632);
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }
__device__ __forceinline__ float lds_volatile_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.volatile.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <bool W_IS_NK, bool A_IS_KM, int MT>
__global__ void __launch_bounds__(kWarpThreads, 1)
hif8_gemm_warp_kernel(const uint8_t* __restrict__ A, long long lda, const uint8_t* __restrict__ W, long long ldw, const GemmParams p, const WarpPlan plan)
{
    using S = WarpShape<W_IS_NK, MT>;
    constexpr int UT = S::UT, CH = S::CH;
    extern __shared__ unsigned char smem_raw[];
    const WarpSmem lay(smem_u32(smem_raw), (uint32_t)(plan.slices * plan.lanes) * S::kDeposit);
    unsigned char* sm = smem_raw - smem_u32(smem_raw);  // generic pointer of shared-window address 0
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int c = plan.cluster, rank = c > 1 ? (int)cluster_ctarank() : 0, cid = c > 1 ? (int)blockIdx.x / c : (int)blockIdx.x;
    const int m0 = (int)blockIdx.y * S::kRows;
    const int cl = warp / plan.slices, sl = warp - cl * plan.slices;  // column lane, slice
    const bool works = cl < plan.lanes;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + lay.abort_flag());
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // units of this cluster, and of this column lane among them: u0 + cl, + lanes, ..
    const int u0 = cid * plan.q + min(cid, plan.rem), nu = plan.q + (cid < plan.rem ? 1 : 0);
    {
        uint32_t dyn_bytes;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
        // the layout does not fit (the same answer in every thread of the grid)
        if (lay.sums + (uint32_t)(plan.q + 1) * S::kDeposit > lay.lut || lay.end > smem_u32(smem_raw) + dyn_bytes) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int*>(p.status) = 7;
            return;
        }
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < plan.lanes; i++) { mbar_init(lay.bars + 8u * i, plan.slices); mbar_init(lay.bars + 8u * (kWarpWarps + i), plan.slices); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fill_decode_table<64, 64 / kWarpWarps>(reinterpret_cast<uint32_t*>(sm + lay.lut), warp, lane, kWarpWarps);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int*>(p.status) = 0;  // (a wait gives up seconds later)

    const int n_it = works && nu > cl ? (nu - cl + plan.lanes - 1) / plan.lanes : 0;
    const int k0 = (rank * plan.slices + sl) * plan.chunks * 64, k_len = min(plan.chunks * 64, p.K - k0);  // (k_len may be below one: nothing to do)
    const uint32_t lut = lay.lut + 4u * lane;
    const uint64_t policy = l2_policy_evict_first();

    // ---- weights.  [N,K]: a slot per 64 k of the slice, refilled with the next unit's bytes as soon as its own have been used.  [K,N]:
    // the slots are the four steps of 64 k, refilled with the next 64 k's.
    constexpr int kSlots = W_IS_NK ? CH : 4 * CH, kSlotWords = W_IS_NK ? 8 * UT : 2 * UT;
    uint32_t v[kSlots][kSlotWords];
    int n_next = (u0 + cl) * S::kCols + (W_IS_NK ? g : 2 * UT * g);  // this thread's first column of the unit to load next
    const uint8_t* w_next = W_IS_NK ? W + (long long)n_next * ldw + k0 + 16 * t : W + (long long)(k0 + 16 * t) * ldw + n_next;
    const long long w_unit = W_IS_NK ? (long long)plan.lanes * S::kCols * ldw : plan.lanes * S::kCols;
    const long long row8 = 8 * ldw;
    int k_blocks = 0;  // bit j: this thread's k of block j exist
#pragma unroll
    for (int j = 0; j < CH; j++)
        if (j < plan.chunks && 64 * j + 16 * t < k_len) k_blocks |= 1 << j;
    auto load_slot = [&](const uint8_t* from, int n, int j, int s) {  // slot j of a unit, or step s of its 64-k block j
        const bool in_k = (k_blocks >> j) & 1;
        if (W_IS_NK) {
#pragma unroll
            for (int i = 0; i < 2 * UT; i++) {
                const uint4 a = in_k && n + 8 * i < p.N ? ld_weights_v4(from + i * row8 + 64 * j, policy) : make_uint4(0, 0, 0, 0);
                v[j][(4 * i) % kSlotWords] = a.x; v[j][(4 * i + 1) % kSlotWords] = a.y; v[j][(4 * i + 2) % kSlotWords] = a.z; v[j][(4 * i + 3) % kSlotWords] = a.w;
            }
        } else {
            const bool in = n < p.N && in_k;
            const uint8_t* src = from + (long long)(64 * j + 4 * s) * ldw;
#pragma unroll
            for (int i = 0; i < 4; i++) v[4 * j + s][i] = in ? ld_weights_u32(src + i * ldw, policy) : 0u;
        }
    };
    // ---- activations of the slice: b[64-k block][step][8 rows][register].  Row of column x of n8 tile i: [M,K] 8 i + x, [K,M] MT x + i.
    // Their loads go out in front of the weights', which would keep them waiting.
    uint32_t b[CH][4][MT][2];
#pragma unroll
    for (int j = 0; j < CH; j++)
#pragma unroll
        for (int s = 0; s < 4; s++)
#pragma unroll
            for (int i = 0; i < MT; i++) b[j][s][i][0] = 0u;  // the codes, until they are decoded
    if (n_it > 0) {
#pragma unroll
        for (int j = 0; j < CH; j++) {
            if (j >= plan.chunks) break;
            if (!A_IS_KM) {
#pragma unroll
                for (int i = 0; i < MT; i++) {
                    const int m = m0 + 8 * i + g;
                    const uint8_t* src = A + (long long)m * lda + k0 + 64 * j;
                    if (m >= p.M) continue;
                    if ((k_blocks >> j) & 1) {
                        const uint4 x = __ldg(reinterpret_cast<const uint4*>(src + 16 * t));
                        b[j][0][i][0] = x.x; b[j][1][i][0] = x.y; b[j][2][i][0] = x.z; b[j][3][i][0] = x.w;
                    }
                }
            } else {
                const int m = m0 + 4 * g;  // (MT = 4)
#pragma unroll
                for (int s = 0; s < 4; s++) {
                    const int k = 64 * j + 16 * t + 4 * s;
                    uint32_t r[4] = {0u, 0u, 0u, 0u};
                    if (k < k_len) {
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            const uint8_t* src = A + (long long)(k0 + k + i) * lda + m;
                            if (m + 4 <= p.M) r[i] = __ldg(reinterpret_cast<const uint32_t*>(src));
                            else
                                for (int e = 0; m + e < p.M; e++) r[i] |= (uint32_t)src[e] << (8 * e);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < MT; i++) b[j][s][i][0] = r[i & 3];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < CH; j++) {
            if (j < plan.chunks) {
#pragma unroll
                for (int s = 0; s < 4; s++) {
                    if (!W_IS_NK) load_slot(w_next, n_next, j, s);
                    if (W_IS_NK && s == 0) load_slot(w_next, n_next, j, 0);
                    uint32_t w[MT];
#pragma unroll
                    for (int i = 0; i < MT; i++) w[i] = b[j][s][i][0];
                    if constexpr (A_IS_KM) {
                        uint32_t o[4];
                        transpose4x4(w[0], w[1], w[2], w[3], o);
#pragma unroll
                        for (int i = 0; i < 4; i++) w[i] = o[i];
                    }
#pragma unroll
                    for (int i = 0; i < MT; i++) decode4(w[i], lut, b[j][s][i][0], b[j][s][i][1]);
                }
            }
        }
    }

    // ---- units
    const uint32_t bar_full = lay.bars + 8u * cl, bar_empty = lay.bars + 8u * (kWarpWarps + cl);
    const uint32_t dep_lane = lay.dep + (uint32_t)(cl * plan.slices) * S::kDeposit, dep_mine = dep_lane + (uint32_t)sl * S::kDeposit + 4u * lane;
    bool ok = true;
    // this warp's share of the deposits of the lane's it-th unit, added pairwise, to the sums: [row][column] of the unit
    auto reduce = [&](int it) {
        ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait(bar_full, it & 1, abort_flag, p.status, 51));
        if (!ok) return;
        const uint32_t sums = lay.sums + (uint32_t)(cl + it * plan.lanes) * S::kDeposit;
        for (int e = sl * 32; e < S::kSums; e += plan.slices * 32) {  // deposits are [register][lane]; register r = (tile, n8 tile, quarter)
            const int r = e >> 5, q = r & 3, i = (r >> 2) & (MT - 1), ut = (r >> 2) / MT;
            const uint32_t from = dep_lane + 4u * (uint32_t)(e + lane);
            float part[kWarpWarps];
#pragma unroll
            for (int s = 0; s < kWarpWarps; s++) part[s] = s < plan.slices ? lds_volatile_f32(from + (uint32_t)s * S::kDeposit) : 0.f;
#pragma unroll
            for (int h = 1; h < kWarpWarps; h *= 2)
#pragma unroll
                for (int s = 0; s < kWarpWarps; s += 2 * h) part[s] += part[s + h];
            const int col = W_IS_NK ? 16 * ut + g + 8 * (q >> 1) : 2 * UT * g + 2 * ut + (q >> 1), x = 2 * t + (q & 1), row = A_IS_KM ? MT * x + i : 8 * i + x;
            sts_f32(sums + 4u * (uint32_t)(row * S::kCols + col), part[0]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_empty);
    };
#pragma unroll 1
    for (int it = 0; it < n_it && ok; it++) {
        n_next += plan.lanes * S::kCols;
        w_next += w_unit;
        float acc[UT][MT][4];
#pragma unroll
        for (int u = 0; u < UT; u++)
#pragma unroll
            for (int i = 0; i < MT; i++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[u][i][q] = 0.f;
#pragma unroll
        for (int j = 0; j < CH; j++) {
            if (j < plan.chunks) {
                uint32_t x[kSlotWords];
                if (W_IS_NK) {
#pragma unroll
                    for (int i = 0; i < kSlotWords; i++) x[i] = v[j][i];
                    if (it + 1 < n_it) load_slot(w_next, n_next, j, 0);
                }
#pragma unroll
                for (int s = 0; s < 4; s++) {
                    uint32_t codes[UT][2];  // four k of column g's (or the thread's first) and of column g + 8's (second) of each tile
                    if (W_IS_NK) {
#pragma unroll
                        for (int u = 0; u < UT; u++) { codes[u][0] = x[(8 * u + s) % kSlotWords]; codes[u][1] = x[(8 * u + 4 + s) % kSlotWords]; }
                    } else {
#pragma unroll
                        for (int i = 0; i < kSlotWords; i++) x[i] = v[4 * j + s][i];
                        if (it + 1 < n_it) load_slot(w_next, n_next, j, s);
                        uint32_t o[4];
                        transpose4x4(x[0], x[1], x[2], x[3], o);
                        codes[0][0] = o[0]; codes[0][1] = o[1]; codes[UT - 1][0] = o[2]; codes[UT - 1][1] = o[3];
                    }
#pragma unroll
                    for (int u = 0; u < UT; u++) {
                        uint32_t a0, a1, a2, a3;
                        decode4(codes[u][0], lut, a0, a2);
                        decode4(codes[u][1], lut, a1, a3);
#pragma unroll
                        for (int i = 0; i < MT; i++) mma_16816(acc[u][i], a0, a1, a2, a3, b[j][s][i][0], b[j][s][i][1]);
                    }
                }
            }
            if (j == 0 && it > 0) reduce(it - 1);
        }
        if (it > 0) ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait(bar_empty, (it - 1) & 1, abort_flag, p.status, 52));
        if (!ok) break;
#pragma unroll
        for (int u = 0; u < UT; u++)
#pragma unroll
            for (int i = 0; i < MT; i++)
#pragma unroll
                for (int q = 0; q < 4; q++) sts_f32(dep_mine + 128u * (uint32_t)((u * MT + i) * 4 + q), acc[u][i][q]);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full);
    }
    if (n_it > 0 && ok) reduce(n_it - 1);

    // ---- results: four consecutive columns of a row per thread and step; in a cluster each block finishes the units u = rank (mod c)
    const int sa = p.d_sa ? *p.d_sa : 0, sw_all = (p.d_sw && !p.d_sw_channel) ? *p.d_sw : 0;
    __syncthreads();
    if (c > 1) cluster_sync_all();
    if (!*abort_flag) {
        const int mine = nu > rank ? (nu - rank + c - 1) / c : 0;
        constexpr int kQuads = S::kSums / 4, kRowQuads = S::kCols / 4;
        for (int e = threadIdx.x; e < mine * kQuads; e += kWarpThreads) {
            const int ul = rank + c * (e / kQuads), r = e % kQuads, row = m0 + r / kRowQuads, n = (u0 + ul) * S::kCols + 4 * (r % kRowQuads);
            if (row >= p.M || n >= p.N) continue;
            const uint32_t at = lay.sums + (uint32_t)ul * S::kDeposit + 16u * (uint32_t)r;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            for (int k = 0; k < c; k++) {
                const uint32_t from = c > 1 ? map_to_cta(at, (uint32_t)k) : at;
#pragma unroll
                for (int i = 0; i < 4; i++) x[i] += ld_cluster_f32(from + 4u * i);
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int sc = -(sa + (p.d_sw_channel ? (n + i < p.N ? __ldg(p.d_sw_channel + n + i) : 0) : sw_all)), s1 = sc / 2, s2 = sc - s1;
                x[i] = x[i] * __uint_as_float((uint32_t)(s1 + 127) << 23) * __uint_as_float((uint32_t)(s2 + 127) << 23);
            }
            const long long o = (long long)row * p.ldc + n;
            if (p.c_is_f32) {
                float* out = reinterpret_cast<float*>(p.C) + o;
                if (n + 4 <= p.N) {
                    if (p.accumulate) {
                        const float4 old = *reinterpret_cast<const float4*>(out);
                        x[0] += old.x; x[1] += old.y; x[2] += old.z; x[3] += old.w;
                    }
                    *reinterpret_cast<float4*>(out) = make_float4(x[0], x[1], x[2], x[3]);
                } else
                    for (int i = 0; n + i < p.N; i++) out[i] = p.accumulate ? x[i] + out[i] : x[i];
            } else {
                unsigned short* out = reinterpret_cast<unsigned short*>(p.C) + o;
                const bool full = n + 4 <= p.N;
                uint2 w = make_uint2(0, 0);
                if (p.accumulate) {
                    if (full) w = *reinterpret_cast<const uint2*>(out);
                    else
                        for (int i = 0; n + i < p.N; i++) (i < 2 ? w.x : w.y) |= (uint32_t)out[i] << (16 * (i & 1));
                    x[0] += __uint_as_float(w.x << 16); x[1] += __uint_as_float(w.x & 0xFFFF0000u);
                    x[2] += __uint_as_float(w.y << 16); x[3] += __uint_as_float(w.y & 0xFFFF0000u);
                }
                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w.x) : "f"(x[1]), "f"(x[0]));  // round to nearest even; a NaN stays a NaN
                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w.y) : "f"(x[3]), "f"(x[2]));
                if (full) *reinterpret_cast<uint2*>(out) = w;
                else
                    for (int i = 0; n + i < p.N; i++) out[i] = (unsigned short)((i < 2 ? w.x : w.y) >> (16 * (i & 1)));
            }
        }
    }
    if (c > 1) {  // nobody leaves while another block reads its sums
        cluster_arrive_relaxed();
        cluster_wait();
    }
}
