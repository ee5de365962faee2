// Int8 GEMM with the fused epilogue for problems whose tiles do not fill the device and whose K is long: a cluster of CTAs shares
// one tile, each CTA multiplying its own part of K.
//
// With one CTA per 128 x 32 tile such a problem is a serial chain of K / 128 steps in a few CTAs, bound by the bytes that one SM
// keeps in flight (20 KB per step, 0.2 us).  Here a CTA runs a half or a quarter of the steps, mostly all in flight at once.
// Then the partial Int32 sums are exchanged through distributed shared memory and added (exactly: Int32), the sums go back
// into tensor memory and the epilogue shared with the other kernels runs on them.  Two forms:
//   rows     four CTAs share a 128 x 32 tile, each finishes one lane quarter (32 rows): for the smallest problems, four times as
//            many CTAs as 128 x 32 tiles.  128 x 3072 -> 768: 7.9 -> 5.4 us, 128 x 4096 -> 1024: 9.4 -> 6.0.
//   columns  two CTAs share a 128 x 64 tile, each finishes 32 columns: as many CTAs as 128 x 32 tiles, half the X_q traffic.
//            509 x 4096 -> 1024: 9.8 -> 8.0 us, 384 x 3072 -> 768: 8.0 -> 6.9.
// The exchange costs 0.3 (rows) to 0.8 us (columns), so with K <= 1024 nothing is gained (128 x 768 -> 768 4.3 / 4.6 us).  Wider
// tiles or more splits were slower: one warp per CTA then finishes several blocks, or the exchange grows.
//
// Warps 0 and 2 fetch operands by TMA (even and odd steps), warp 1 issues the MMAs, warps 3..6 are the epilogue.  A CTA has one
// tile.  Waits are bounded as in q8_gemm_sm100.cu; the cluster barrier is reached on every path.

#include <cuda.h>

#include "q8_gemm_common.cuh"

namespace q8 {

namespace {

using namespace ptx;
using namespace gemm_detail;

constexpr int kThreads = 224;

template <bool ROWS>
struct SplitCfg {
    static constexpr int KS = ROWS ? 4 : 2;        // CTAs per cluster = parts of K
    static constexpr int BN = ROWS ? 32 : 64;      // tile width
    static constexpr int kFinishers = ROWS ? 1 : 4;  // epilogue warps that finish a 32 x 32 block
    static constexpr int kABytes = BLOCK_M * BLOCK_K, kBBytes = BN * BLOCK_K;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStagingBytes = kFinishers * kStagingBytesPerWarp;
    static constexpr int kSlotRows = 32 * kFinishers;
    static constexpr int kSlotBytes = kSlotRows * 32 * 4;  // one CTA's partial sums of another's block(s)
    static constexpr int kExchangeBytes = (KS - 1) * kSlotBytes;
    static constexpr int kBiasBytes = kFinishers * 32 * 4;
    static constexpr int kStages = ROWS ? 8 : 7;
    static constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kStagingBytes + kExchangeBytes + kBiasBytes + (2 * kStages + 1) * 8 + 16;
    static_assert(kSmemBytes <= 232448, "shared memory budget");
    static constexpr uint32_t kInstrDesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                           ((uint32_t)(BLOCK_M >> 4) << 24);
};

__device__ __forceinline__ void tmem_st_32x32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// Place of the 16-byte piece g of a row in an exchange slot: a warp's store is one run of 512 bytes (rows of 128 bytes, 32
// segments per store, took 0.5 us longer).
template <int SLOT_ROWS>
__device__ __forceinline__ uint32_t exchange_at(int row, int g) { return (uint32_t)((g * SLOT_ROWS + row) * 16); }

template <bool ROWS, bool ABSMAX, int OUT>
__global__ void __launch_bounds__(kThreads, 1)
gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                   const __grid_constant__ CUtensorMap tmap_y, GemmArgs a, int tma_store)
{
    using C = SplitCfg<ROWS>;
    constexpr int KS = C::KS, BN = C::BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *smem_a = smem, *smem_b = smem + C::kStages * C::kABytes;
    uint8_t *smem_stage = smem + C::kStages * C::kStageBytes;
    uint8_t *smem_exchange = smem_stage + C::kStagingBytes;
    int32_t *smem_bq = reinterpret_cast<int32_t *>(smem_exchange + C::kExchangeBytes);
    uint64_t *full_bar = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(smem_bq) + C::kBiasBytes);
    uint64_t *empty_bar = full_bar + C::kStages;
    uint64_t *done_bar = full_bar + 2 * C::kStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done_bar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int64_t tile = blockIdx.x / KS, tiles_n = (a.N + BN - 1) / BN;
    const int64_t m0 = tile / tiles_n * BLOCK_M, n0 = tile % tiles_n * BN;
    const int num_kb = (int)((a.K + BLOCK_K - 1) / BLOCK_K);
    const int kb0 = (int)((int64_t)num_kb * rank / KS), kb1 = (int)((int64_t)num_kb * (rank + 1) / KS);  // (the host: num_kb >= KS)

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(smem_u32(full_bar + s), 1);
            mbar_init(smem_u32(empty_bar + s), 1);
        }
        mbar_init(smem_u32(done_bar), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), (uint32_t)BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    cluster_arrive();  // this CTA has started.  Every role waits for the others' arrivals off the critical path (and when aborting)
    if (warp == 3 && lane == 0 && m0 == 0)  // the weights on their way into L2 while the kernel before this one still runs
        for (int kb = kb0; kb < kb1; ++kb) tma_prefetch_2d(&tmap_w, kb * BLOCK_K, (int32_t)n0);
    grid_dependency_release_next(true);  // small by construction: one tile per cluster
    grid_dependency_wait();

    bool ok = true;
    if (warp == 0 || warp == 2) {
        const uint32_t elected = elect_one();
        for (int kb = kb0 + (warp >> 1); kb < kb1; kb += 2) {
            const int i = kb - kb0, s = i % C::kStages;
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(empty_bar + s), (uint32_t)((i / C::kStages) & 1) ^ 1u, abort_flag, a.status));
            if (!ok) break;
            const uint32_t fb = smem_u32(full_bar + s);
            mbar_expect_tx_elected(elected, fb, (uint32_t)C::kStageBytes);
            tma_load_2d_elected(elected, smem_u32(smem_a + s * C::kABytes), &tmap_x, kb * BLOCK_K, (int32_t)m0, fb);
            tma_load_2d_elected(elected, smem_u32(smem_b + s * C::kBBytes), &tmap_w, kb * BLOCK_K, (int32_t)n0, fb);
        }
        if (!ok) {  // aborting: let the copies already issued land before the shared memory is given up
            const uint64_t t0 = global_timer_ns();
            while (global_timer_ns() - t0 < 1000000ull) {}
        }
        __syncwarp();
        cluster_wait();
    } else if (warp == 1) {
        const uint32_t elected = elect_one();
        for (int kb = kb0; kb < kb1; ++kb) {
            const int i = kb - kb0, s = i % C::kStages;
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(full_bar + s), (uint32_t)((i / C::kStages) & 1), abort_flag, a.status));
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = smem_desc_sw128(smem_u32(smem_a + s * C::kABytes)), db = smem_desc_sw128(smem_u32(smem_b + s * C::kBBytes));
#pragma unroll
            for (int k = 0; k < BLOCK_K / 32; ++k)  // +32 bytes along K inside the swizzle span == +2 in the (addr >> 4) field
                umma_i8_elected(elected, tmem_base, da + 2 * k, db + 2 * k, C::kInstrDesc, (uint32_t)((i | k) != 0));
            umma_commit_elected(elected, smem_u32(empty_bar + s));
        }
        if (ok) umma_commit_elected(elected, smem_u32(done_bar));
        else {  // aborting: let the MMAs issued so far finish before the tensor memory is freed
            const uint64_t t0 = global_timer_ns();
            while (global_timer_ns() - t0 < 1000000ull) {}
        }
        __syncwarp();
        cluster_wait();
    } else {
        cluster_wait();  // (before any CTA stores into another's shared memory)
        // Partial sums of the blocks that another CTA finishes go to that CTA's exchange slot: with ROWS the block of lane quarter
        // q is CTA q's, else the block of columns 32 r .. of every quarter is CTA r's.
        const int quarter = warp & 3;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(done_bar), 0, abort_flag, a.status));
        tc_fence_after();
        const uint32_t peer = ROWS ? (uint32_t)quarter : rank ^ 1u;
        if (ok && peer != rank) {
            const uint32_t slot = (rank + KS - peer) % KS - 1;  // 0 .. KS - 2: this CTA as seen from the peer
            const uint32_t at = map_to_cta(smem_u32(smem_exchange) + slot * C::kSlotBytes, peer);
            const int row = (ROWS ? 0 : quarter * 32) + lane;
            uint32_t v[32];
            tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (ROWS ? 0u : 32u * peer), v);
            tmem_ld_wait();
#pragma unroll
            for (int g = 0; g < 8; ++g)
                asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};"
                             ::"r"(at + exchange_at<C::kSlotRows>(row, g)), "r"(v[4 * g]), "r"(v[4 * g + 1]), "r"(v[4 * g + 2]),
                             "r"(v[4 * g + 3])
                             : "memory");
        }
    }
    __syncwarp();
    cluster_sync_all();  // every partial sum is in place (release / acquire); reached by all threads, also when aborting
    if (warp >= 3 && (!ROWS || (uint32_t)(warp & 3) == rank) && ok && *abort_flag == 0) {
        const int quarter = warp & 3, mine = ROWS ? 0 : quarter, row = mine * 32 + lane;
        const uint32_t col = ROWS ? 0u : 32u * rank;
        const uint32_t t_own = tmem_base + ((uint32_t)(quarter * 32) << 16) + col, slots = smem_u32(smem_exchange);
        const int64_t n = n0 + col;  // (w_seg is a multiple of 32: a block never straddles two weight scales)
        const float S_out = __fmul_rn(__ldg(a.S_x), __ldg(a.S_w + (a.w_seg > 0 && n < a.N ? n / a.w_seg : 0)));
        const float invv[1] = {__fdiv_rn(1.0f, S_out)};
        const int32_t bqv[1] = {quantize_bias(a.bias != nullptr && n + lane < a.N ? __ldg(a.bias + n + lane) : 0.0f, S_out)};
        uint32_t part[32];
        tmem_ld_32x32(t_own, part);
        tmem_ld_wait();
#pragma unroll
        for (int p = 0; p < KS - 1; ++p)
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                uint32_t v[4];
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                             : "r"(slots + (uint32_t)(p * C::kSlotBytes) + exchange_at<C::kSlotRows>(row, g))
                             : "memory");
#pragma unroll
                for (int j = 0; j < 4; ++j) part[4 * g + j] += v[j];
            }
        tmem_st_32x32(t_own, part);
        tmem_st_wait();
        float am = 0.0f;
        epilogue_warp<32, ABSMAX, false, false, false, OUT>(a, &tmap_y, tma_store == 1, &tmap_y, false, t_own, m0 + quarter * 32, n, bqv, invv,
                                                     smem_stage + mine * kStagingBytesPerWarp, smem_bq + mine * 32, lane, 1, [] {}, am);
        if (ABSMAX) warp_fold_absmax(am, a.y_absmax);
        if (lane == 0) tma_store_wait_all();
    }

    // ---------------- teardown (reached by every thread, also when aborting)
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)BN);
    }
}

template <bool ROWS, bool ABSMAX, int OUT>
cudaError_t launch_out(const GemmArgs &a, cudaStream_t s)
{
    using C = SplitCfg<ROWS>;
    constexpr int KS = C::KS, BN = C::BN;
    auto kernel = gemm_splitk_kernel<ROWS, ABSMAX, OUT>;
    static bool attr_set[64] = {};  // the opt-in shared-memory size is a per-device, per-function attribute
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    CUtensorMap tx, tw, ty;
    if (!make_tmap(&tx, a.Xq, a.M, a.K, BLOCK_M) || !make_tmap(&tw, a.Wq, a.N, a.K, BN)) return cudaErrorInvalidValue;
    const int tma_store = a.Y != nullptr && (a.N & 3) == 0 && (reinterpret_cast<uintptr_t>(a.Y) & 15u) == 0;
    ty = tx;  // never dereferenced unless tma_store
    if (tma_store && !make_tmap_out(&ty, a.Y, a.M, a.N)) return cudaErrorInvalidValue;
    const int64_t tiles = ((a.M + BLOCK_M - 1) / BLOCK_M) * ((a.N + BN - 1) / BN);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * KS));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = KS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kernel, tx, tw, ty, a, tma_store);
    LaunchInfo &li = last_launch_info();
    li.gemm_kernel = 1;
    li.block_n = BN;
    li.ctas = KS;
    li.epilogue_warps = 4;
    li.grid = (int)(tiles * KS);
    li.tail_split = 1;
    li.store_mode = tma_store;
    li.launches += 1;
    return e;
}

template <bool ROWS>
cudaError_t launch_split(const GemmArgs &a, cudaStream_t s)
{
    const bool int8_only = a.Yq != nullptr && a.Y == nullptr && a.dbg_acc == nullptr, plain = a.Yq == nullptr && a.dbg_acc == nullptr;
    const bool gelu = a.act == Q8_ACT_GELU;
    if (a.y_absmax != nullptr && plain) return gelu ? launch_out<ROWS, true, kOutPlain | kOutGelu>(a, s) : launch_out<ROWS, true, kOutPlain>(a, s);
    if (a.y_absmax != nullptr) return launch_out<ROWS, true, kOutFull>(a, s);
    if (int8_only) return gelu ? launch_out<ROWS, false, kOutInt8 | kOutGelu>(a, s) : launch_out<ROWS, false, kOutInt8>(a, s);
    if (plain) return gelu ? launch_out<ROWS, false, kOutPlain | kOutGelu>(a, s) : launch_out<ROWS, false, kOutPlain>(a, s);
    return launch_out<ROWS, false, kOutFull>(a, s);
}

}  // namespace

cudaError_t launch_gemm_splitk(const GemmArgs &a, bool rows, cudaStream_t s)
{
    return rows ? launch_split<true>(a, s) : launch_split<false>(a, s);
}

}  // namespace q8
