// Projections of a prefill pass (Sec. 2.2: the target model's pass over the prompt): Y[r][n] = bf16(sum_k W[n][k] X[r][k]) for up to
// kPrefillRows rows, with the bits that a row gets from the verification projection (verify_gemm.cu).
//
// What fixes those bits is that the K ranges of a projection are summed apart, each by MMAs in order from a zero accumulator, and
// the ranges' fp32 sums are then added in order.  Here one pair of CTAs goes through all ranges of its tile: the tensor memory holds
// two accumulators in turn, and while one range is multiplied, eight warps add the range before to sums in their registers.  No
// fp32 part leaves the SM (the split-K kernel writes and its consumers read 4 bytes a range, feature and row, most of the time of
// norms, SwiGLU and RoPE in a prefill).
//
// cta_group::2: the pair multiplies 256 features x BN rows per MMA, each CTA holding 128 features of the weights and half of the rows,
// so that an SM takes 64 bytes a cycle from L2 at full tensor rate; a CTA of its own with 128 x 256 would need 96.  CTA 0 issues the
// MMAs; both copy (TMA, 128-byte swizzle) and signal CTA 0's barriers.  Persistent pairs, one CTA an SM; the row tiles of a feature
// tile run side by side, so that the weights come from memory once.
// Bound: the tensor pipe and the steps around it.  28672 x 4096 with 1000 rows 168 us (1.40 PFLOP/s, 85 % of measured with 6.05 rounds
// of the pairs taken as 7), four calls of the split-K kernel with their additions 501; four layers' prompt of 1000 tokens 4.28 -> 2.69 ms.
// A stage's barriers and commit cost some 0.2 us, hence two K blocks a stage where those are small (128 rows: 4096 x 14336 140 -> 99 us;
// at 256 rows six stages of one block are as fast), and the issuing thread is found by elect.sync instead of its lane's
// number (140 -> 116 us of that).  Ten warps are three on one quarter of the SM, which leaves a thread 168 registers; at 256 rows the 128 sums do
// not quite fit beside the rest (11 words spilled).
#include "tc.cuh"
#include "kernels.cuh"

namespace cass {

constexpr int kWgBM = 128, kWgBK = 64;          // features and K values of a CTA's tile
constexpr int kWgThreads = 320;                 // warp 0: TMA; warp 1: MMA issue (CTA 0) and tensor memory; warps 2-9: sums and stores
constexpr int kWgEpiWarps = 8;
constexpr int wg_step(int bn) { return bn <= 192 ? 2 : 1; }               // K blocks a stage
constexpr int kWgABytes = kWgBM * kWgBK * 2;
constexpr int wg_b_bytes(int bn) { return bn / 2 * kWgBK * 2; }
constexpr int wg_stages(int bn) { return bn <= 192 ? 4 : 6; }
constexpr int wg_smem(int bn) { return wg_stages(bn) * wg_step(bn) * (kWgABytes + wg_b_bytes(bn)) + 256 + 1024; }     // + barriers + alignment slack
constexpr int kWgAccCols = 256, kWgTmemCols = 512;                                                  // two accumulators
constexpr int kPairs = kSms / 2;

__device__ __forceinline__ uint32_t wg_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t wg_leader_addr(const void* p) {          // the same place in CTA 0 of the pair
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
    return r;
}
__device__ __forceinline__ void wg_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void wg_tma_load(void* dst, const CUtensorMap* map, int x, int y, uint32_t leader_bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
                     smem_u32(dst)),
                 "l"(map), "r"(leader_bar), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void wg_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void wg_commit(uint64_t* bar) {                   // arrives at this place of both CTAs when the MMAs so far are done
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "h"((uint16_t)3)
                 : "memory");
}
// Bounded wait for arrivals of either CTA.
__device__ __forceinline__ bool wg_wait_cluster(uint64_t* bar, uint32_t parity) {
    for (uint32_t i = 0; i < (1u << 22); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// grid: pairs of CTAs; tile t = (t / r_tiles)-th 256 features x (t % r_tiles)-th BN rows.
// A role whose bounded wait runs out flags the status and goes to the end; the others' waits run out in turn, and both CTAs meet before
// either leaves.
template <int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kWgThreads, 1)
    k_wide_gemm(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, uint16_t* __restrict__ out, int rows, int n,
                int kb_total, int kb_per_split, int r_tiles, int n_tiles, int32_t* __restrict__ d_status, int w_static) {
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);     // swizzled tiles: 1024-byte aligned
    constexpr int S = wg_stages(BN), kStep = wg_step(BN), kBBytes = wg_b_bytes(BN);
    constexpr uint32_t kIdesc = tc_idesc_mn(2 * kWgBM, BN, false), kBlockTx = 2 * (kWgABytes + kBBytes);      // a K block in both CTAs
    uint8_t *sA = base, *sB = base + S * kStep * kWgABytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(sB + S * kStep * kBBytes);          // of CTA 0: a stage has arrived in both CTAs
    uint64_t* empty = full + S;                                              // of each: the stage has been multiplied with
    uint64_t* acc_full = empty + S;                                          // of each: a range's sums are complete
    uint64_t* acc_empty = acc_full + 2;                                      // of CTA 0: they have been read in both CTAs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)wg_rank(), pair = blockIdx.x / 2, n_pairs = gridDim.x / 2;
    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * kWgEpiWarps); }
        fence_mbar_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kWgTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    wg_cluster_sync();                                                       // the pair's barriers are set up
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int my_tiles = pair < n_tiles ? (n_tiles - pair + n_pairs - 1) / n_pairs : 0;
    auto tile_at = [&](int i, int& m0, int& r0) {
        const int t = pair + i * n_pairs;
        m0 = t / r_tiles * 2 * kWgBM + rank * kWgBM;
        r0 = t % r_tiles * BN;
    };
    // The producer's stages in order: up to kStep blocks of a K range.  The first ring's weights, which nobody writes, are asked for
    // ahead of the wait (`pre`), the rows behind it.
    auto produce = [&](bool pre) {
        int it = 0;
        for (int i = 0; i < my_tiles; ++i) {
            int m0, r0;
            tile_at(i, m0, r0);
            for (int k0 = 0; k0 < kb_total; k0 += kb_per_split) {
                const int k1 = min(kb_total, k0 + kb_per_split);
                for (int kb = k0; kb < k1; kb += kStep, ++it) {
                    if (pre && it >= S) return;
                    const int s = it % S, nb = min(kStep, k1 - kb);
                    const uint32_t bar = wg_leader_addr(&full[s]);
                    if (!mbar_wait_bounded(&empty[s], ((uint32_t)(it / S) & 1u) ^ 1u)) { atomicExch(d_status, CASS_ERR_TIMEOUT); return; }
                    if (pre || it >= S || w_static != kWeightsStatic) {
                        if (rank == 0) mbar_expect_tx(&full[s], nb * kBlockTx);
                        for (int j = 0; j < nb; ++j) wg_tma_load(sA + (s * kStep + j) * kWgABytes, &map_w, (kb + j) * kWgBK, m0, bar);
                    }
                    if (!pre)
                        for (int j = 0; j < nb; ++j) wg_tma_load(sB + (s * kStep + j) * kBBytes, &map_x, (kb + j) * kWgBK, r0 + rank * (BN / 2), bar);
                }
            }
        }
    };
    if (warp == 0 && w_static == kWeightsStatic && tc_elect()) produce(true);
    __syncwarp();
    pdl_wait();
    pdl_early<5>();

    if (warp == 0) {
        if (tc_elect()) produce(false);                                      // this CTA's half of every stage
    } else if (warp == 1) {
        if (rank == 0 && tc_elect()) {                                       // the MMAs of both CTAs
            int it = 0, rng = 0;
            bool ok = true;
            for (int i = 0; i < my_tiles && ok; ++i)
                for (int k0 = 0; k0 < kb_total && ok; k0 += kb_per_split, ++rng) {
                    const int b = rng & 1, k1 = min(kb_total, k0 + kb_per_split);
                    if (!wg_wait_cluster(&acc_empty[b], ((uint32_t)(rng >> 1) & 1u) ^ 1u)) { ok = false; break; }
                    tc_fence_after();
                    for (int kb = k0; kb < k1; kb += kStep, ++it) {
                        const int s = it % S;
                        if (!mbar_wait_bounded(&full[s], (uint32_t)(it / S) & 1u)) { ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int j = 0; j < kStep; ++j) {
                            if (kb + j >= k1) break;
                            const uint64_t ad = tc_smem_desc(sA + (s * kStep + j) * kWgABytes), bd = tc_smem_desc(sB + (s * kStep + j) * kBBytes);
#pragma unroll
                            for (int kk = 0; kk < kWgBK / 16; ++kk)
                                wg_mma(tmem + (uint32_t)(b * kWgAccCols), ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), kIdesc,
                                       (uint32_t)(kb != k0 || j != 0 || kk != 0));
                        }
                        wg_commit(&empty[s]);
                    }
                    wg_commit(&acc_full[b]);
                }
            if (!ok) {
                atomicExch(d_status, CASS_ERR_TIMEOUT);
                for (int j = it; j < it + S; ++j)                            // what is in flight in either CTA lands before they end (bounded)
                    mbar_wait_bounded(&full[j % S], (uint32_t)(j / S) & 1u);
            }
        }
    } else {
        // ---- sums of the ranges: warp w reads the 32 accumulator lanes of quarter w % 4, half of the columns ----
        constexpr int NC = BN / 2;
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t col0 = ((uint32_t)(q * 32) << 16) + (uint32_t)(half * NC);
        int rng = 0;
        bool ok = true;
        for (int i = 0; i < my_tiles && ok; ++i) {
            float acc[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = 0.f;
            for (int k0 = 0; k0 < kb_total; k0 += kb_per_split, ++rng) {
                const int b = rng & 1;
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[b], (uint32_t)(rng >> 1) & 1u));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < NC; c0 += 16) {                        // 16 at a time: the sums take 128 registers
                    uint32_t v[16];
                    tmem_ld16(tmem + col0 + (uint32_t)(b * kWgAccCols + c0), v);
#pragma unroll
                    for (int c = 0; c < 16; ++c) acc[c0 + c] += __uint_as_float(v[c]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(wg_leader_addr(&acc_empty[b])) : "memory");
            }
            if (!ok) break;
            int m0, r0;
            tile_at(i, m0, r0);
            const int feat = m0 + q * 32 + lane, row0 = r0 + half * NC;
            if (feat < n) {
                uint16_t* o = out + (size_t)row0 * n + feat;
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (row0 + c < rows) o[(size_t)c * n] = float_to_bf16_bits(acc[c]);
            }
        }
        if (!ok && lane == 0) atomicExch(d_status, CASS_ERR_TIMEOUT);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    wg_cluster_sync();                                                       // nobody leaves while its barriers or tensor memory are in use
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kWgTmemCols) : "memory");
    }
}

template <int BN>
static int launch_wide(const CUtensorMap& mw, const CUtensorMap& mx, uint16_t* out, int rows, int n, int kbt, int kbs, int32_t* d_status,
                       int w_static, cudaStream_t s) {
    CASS_ALLOW_SMEM(k_wide_gemm<BN>);
    const int r_tiles = ceil_div(rows, BN), tiles = ceil_div(n, 2 * kWgBM) * r_tiles;
    CASS_PDL_LAUNCH(k_wide_gemm<BN>, dim3(2 * (tiles < kPairs ? tiles : kPairs)), dim3(kWgThreads), (size_t)wg_smem(BN), s, mw, mx, out, rows, n, kbt, kbs,
                    r_tiles, tiles, d_status, w_static);
    return CASS_OK;
}

// Rows of a tile: the one whose rounds of all pairs take least, a K block of a round being 0.22, 0.27 and 0.37 us at 128, 192 and 256
// rows (4096 x 14336, 1000 rows).  1000 rows: 28672 x 4096 186, 178 and 168 us, 6144 x 4096 49, 43 and 56.
struct WidePlan { int bn, rounds, block_us100; };
static WidePlan wide_gemm_plan(int rows, int n) {
    const int us100[3] = {37, 27, 22};
    WidePlan best{0, 0, 0};
    for (int i = 0; i < 3; ++i) {
        const int bn = 256 - 64 * i, rounds = ceil_div(ceil_div(n, 2 * kWgBM) * ceil_div(rows, bn), kPairs);
        if (i == 0 || rounds * us100[i] < best.rounds * best.block_us100) best = WidePlan{bn, rounds, us100[i]};
    }
    return best;
}

// Where the split-K kernel takes the rows too (up to kSplitRows): it spreads the K ranges over the chip but writes each one's sums, which
// the next kernel reads; here they follow one another, each at least as long as its sums' addition to the registers (1.2 us for 128 rows).
// Both sides in hundredths of a us, fitted to kernel times (split-K with what its parts cost the next kernel) of six models' projections, 256 to
// 5120 wide, at 33 to 256 rows: the faster one is chosen but for 10 of 216, by 0.2 % of the time over all.  Split-K / this one: 256 x 688
// 5 / 9 us for 64 rows, 11 / 10 for 160; 2048 x 2048 6 / 17 for 64, 12 / 17 for 256; 6144 x 4096 17 / 22 for 128, 26 / 22 for 256; 28672 x
// 4096 52 / 48 for 64, 92 / 62 for 256; 4096 x 14336 36 / 53 for 256.
bool wide_gemm_pays(int rows, int n, int k) {
    if (rows > kSplitRows) return true;
    if (rows <= 32) return false;
    int kbt, kbs, ns;
    verify_gemm_split(n, k, &kbt, &kbs, &ns);
    const WidePlan plan = wide_gemm_plan(rows, n);
    const int range = kbs * plan.block_us100, add = 120 * plan.bn / 128;
    const int c = rows <= 64 ? 0 : rows <= 128 ? 1 : 2;                      // columns of the split-K kernel's tile: 64, 128, 256
    constexpr int kCall[3] = {200, 350, 500}, kBlock[3] = {74, 74, 98}, kRound[3] = {0, 0, 400}, kParts[3] = {16, 12, 8};
    const int rounds = ceil_div(ceil_div(n, kWgBM) * ns, 2 * kSms);
    return 700 + plan.rounds * ns * (range > add ? range : add) <
           kCall[c] + rounds * (kbs * kBlock[c] + kRound[c]) + (long long)ns * rows * n * kParts[c] / 100000;
}

int launch_wide_gemm(const uint16_t* W, const uint16_t* X, int x_rows, int rows, int n, int k, uint16_t* out, int32_t* d_status, cudaStream_t s,
                     int w_static) {
    if (rows < 1 || rows > x_rows || (k % 8) || n < 1 || !out || !d_status) return CASS_ERR_INVALID_ARG;
    if (((uintptr_t)W & 15) || ((uintptr_t)X & 15)) return CASS_ERR_INVALID_ARG;
    const int bn = wide_gemm_plan(rows, n).bn;
    CUtensorMap mw, mx;
    int rc = tc_matrix_map(&mw, W, n, k, kWgBM);
    if (rc) return rc;
    rc = tc_matrix_map(&mx, X, x_rows, k, bn / 2);
    if (rc) return rc;
    int kbt, kbs, ns;
    verify_gemm_split(n, k, &kbt, &kbs, &ns);
    if (bn == 256) return launch_wide<256>(mw, mx, out, rows, n, kbt, kbs, d_status, w_static, s);
    if (bn == 192) return launch_wide<192>(mw, mx, out, rows, n, kbt, kbs, d_status, w_static, s);
    return launch_wide<128>(mw, mx, out, rows, n, kbt, kbs, d_status, w_static, s);
}

}  // namespace cass
