// Verification attention on the tensor cores (Sec. 2.2: the gamma+1 rows are verified in one pass; bf16 KV cache).
// One CTA = one (128-token chunk, KV head, sequence).  Both products of the chunk run as tcgen05 MMAs with the
// accumulators in tensor memory:
//   scores^T [128 tokens x NP pairs] = K tile [128 x d] . Q^T          (pairs = (row, query head of the group), padded
//   out^T    [d x NP pairs]          = V tile^T [d x 128 tokens] . P^T   to NP = 32 or 64; P = chunk-local softmax
//                                                                        numerators, bf16)
// K and V tiles arrive by TMA (128-byte swizzle); Q and P are written to shared memory by threads in the same
// swizzled layout.  The V tile is used as it lies in memory (rows = tokens), i.e. as an M-contiguous A operand.
// Chunk results (o, running maximum m, sum l) go to the split-K scratch and k_attn_merge combines the chunks, as for
// the SIMT kernel.  A (row, head) pair is one accumulator column, so its result does not depend on the other rows.
// Needs head_dim = 128 and rows x group <= 64; other shapes use k_verify_attn.  More rows than that (a prefill over more chunks
// than prefill_attn.cu takes) are cut into groups, one CTA each; where the fp32-pipe kernel would have taken them 16 at a time,
// P is kept as two bf16 terms and the second product runs twice, so that the accuracy is that kernel's.
#include "tc.cuh"
#include "kernels.cuh"

namespace cass {

constexpr int kVtTok = 128;            // tokens per CTA: M of the score product, K of the output product
constexpr int kVtMaxPairs = 64;        // largest N of both products (template NP = 32 or 64)
constexpr int kVtD = 128;              // head_dim
constexpr int kVtThreads = 192;        // warp 0: TMA; warp 1: MMA issue and tensor-memory allocation; warps 2-5: softmax, epilogue
constexpr int kVtTileBytes = kVtTok * 64 * 2;          // one TMA box: 128 tokens x 64 dims
constexpr int vt_q_bytes(int np) { return np * 64 * 2; }               // one K-block of the Q or P operand: NP rows x 64 elements
// K tiles (32 KB) | V tiles (32 KB) | Q (2 blocks) | [P (2 blocks) when np = 64] | barriers.  The scores (np x 128
// floats) reuse the K tiles' memory, and with np = 32 so does P: both are written only after the first product has
// finished reading K.  The low term of P takes Q's place.
constexpr int vt_smem(int np) { return 4 * kVtTileBytes + (np == 32 ? 2 : 4) * vt_q_bytes(np) + 256 + 1024; }
static_assert(32 * kVtTok * 4 + 2 * vt_q_bytes(32) <= 2 * kVtTileBytes && 64 * kVtTok * 4 <= 2 * kVtTileBytes, "scores (and P) fit the K tiles");
constexpr int vt_tmem_cols(int np) { return 2 * np; }                  // scores^T in columns 0..NP-1, out^T in columns NP..2NP-1

// Byte offset of element (row, col) in a K-major operand block of rows x 64 bf16 with 128-byte swizzle.
__device__ __forceinline__ uint32_t swz_off(int row, int col) {
    return (uint32_t)(row * 128 + ((((col >> 3) ^ (row & 7)) & 7) << 4) + ((col & 7) << 1));
}

__device__ __forceinline__ void named_sync_128() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

template <int NP>
__global__ void __launch_bounds__(kVtThreads) k_verify_attn_tc(const __grid_constant__ CUtensorMap map_k,
                                                                const __grid_constant__ CUtensorMap map_v,
                                                                const uint16_t* __restrict__ qkv, AttnRows ar, int n_groups, int fine,
                                                                int n_q, int n_kv, const DevState* __restrict__ st, AttnScratch sc,
                                                                int32_t* __restrict__ d_status) {
    extern __shared__ uint8_t smem_dyn[];
    pdl_wait();
    const int chunk = blockIdx.x, head = blockIdx.y, seq = blockIdx.z / n_groups;
    const int first = ar.lo + (int)(blockIdx.z % n_groups) * ar.group;        // the group's rows: row r of it sits at position len + r
    const int rows = min(ar.group, ar.hi - first);
    const bool two_terms = first < fine;
    const int len = st->len[seq] + first;
    const int t0 = chunk * kVtTok;
    if (t0 >= len + rows) return;                              // no row of this call sees the chunk
    constexpr int kVtPairs = NP, kVtQBytes = vt_q_bytes(NP), kVtTmemCols = vt_tmem_cols(NP);
    uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    uint8_t* sK = base;                                        // 2 boxes [128 tok][64 d]
    uint8_t* sV = sK + 2 * kVtTileBytes;                       // 2 boxes [128 tok][64 d]
    uint8_t* sQ = sV + 2 * kVtTileBytes;                       // 2 blocks [NP pairs][64 d]
    float* sS = reinterpret_cast<float*>(sK);                  // [NP pairs][128 tok] scores: over the K tiles, once consumed
    uint8_t* sP = NP == 32 ? sK + NP * kVtTok * 4 : sQ + 2 * kVtQBytes;      // 2 blocks [NP pairs][64 tok], 1024-aligned
    uint64_t* bar_k = reinterpret_cast<uint64_t*>(sQ + (NP == 32 ? 2 : 4) * kVtQBytes);
    uint64_t* bar_v = bar_k + 1;
    uint64_t* bar_s = bar_k + 2;       // scores complete in tensor memory
    uint64_t* bar_p = bar_k + 3;       // P written to shared memory (128 arrivals)
    uint64_t* bar_o = bar_k + 4;       // output complete in tensor memory
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_k + 5);
    // per pair: the last position it sees (-1: no such pair), and its place in the scratch; divisions by the group size and
    // 64-bit products for every pair and thread took most of the instructions
    __shared__ __align__(16) int s_lim[NP];
    __shared__ __align__(16) uint32_t s_at[NP];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int G = n_q / n_kv, P = rows * G;
    const int qkv_dim = (n_q + 2 * n_kv) * kVtD;
    if (tid == 0) {
        mbar_init(bar_k, 1); mbar_init(bar_v, 1); mbar_init(bar_s, 1); mbar_init(bar_p, 128); mbar_init(bar_o, 1);
        fence_mbar_init();
        // the chunk's K and V tiles start travelling now, while the other warps stage Q and tensor memory is allocated
        mbar_expect_tx(bar_k, 2 * kVtTileBytes);
        tma_load_3d(sK, &map_k, head * kVtD, t0, seq, bar_k);
        tma_load_3d(sK + kVtTileBytes, &map_k, head * kVtD + 64, t0, seq, bar_k);
        mbar_expect_tx(bar_v, 2 * kVtTileBytes);
        tma_load_3d(sV, &map_v, head * kVtD, t0, seq, bar_v);
        tma_load_3d(sV + kVtTileBytes, &map_v, head * kVtD + 64, t0, seq, bar_v);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kVtTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == 1)
        for (int p = lane; p < NP; p += 32) {
            s_lim[p] = p < P ? len + p / G : -1;
            s_at[p] = (uint32_t)((((size_t)seq * (ar.hi - ar.lo) + first - ar.lo + p / G) * n_q + head * G + p % G) * ar.chunks + chunk);
        }
    if (warp >= 2) {
        // Q of this sequence's rows and this group's heads -> sQ (pair p = row * G + head-in-group), zero beyond P
        const int et = tid - 64;
        const uint16_t* q0 = qkv + ((size_t)seq * ar.rps + first) * qkv_dim + (size_t)head * G * kVtD;
        for (int i = et; i < kVtPairs * (kVtD / 8); i += 128) {
            const int p = i / (kVtD / 8), c8 = i % (kVtD / 8);           // 8 dims = 16 bytes per item
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (p < P) v = *reinterpret_cast<const uint4*>(q0 + (size_t)(p / G) * qkv_dim + (size_t)(p % G) * kVtD + c8 * 8);
            const int blk = c8 >> 3;                                     // which 64-dim block
            *reinterpret_cast<uint4*>(sQ + blk * kVtQBytes + swz_off(p, (c8 & 7) * 8)) = v;
        }
        fence_proxy_async();                                             // generic-proxy writes -> visible to the MMA
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_early<4>();                                    // not before the tensor memory is held: a successor takes its own ahead of its wait
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    if (warp == 1) {
        if (tc_elect()) {
            // ---- scores^T = K . Q^T: A = K tile (K-major over d), B = Q (K-major over d) ----
            if (mbar_wait_bounded(bar_k, 0)) {
                tc_fence_after();
                constexpr uint32_t idesc1 = tc_idesc_mn(kVtTok, kVtPairs, false);
#pragma unroll
                for (int kb = 0; kb < 2; ++kb) {
                    const uint64_t ad = tc_smem_desc(sK + kb * kVtTileBytes), bd = tc_smem_desc(sQ + kb * kVtQBytes);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma(tmem, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc1, (uint32_t)((kb | kk) != 0));
                }
            } else {
                atomicExch(d_status, CASS_ERR_TIMEOUT); ok = false;
            }
            if (!ok) {                                     // what is in flight lands before the CTA ends (bounded)
                mbar_wait_bounded(bar_k, 0);
                mbar_wait_bounded(bar_v, 0);
            }
            tc_commit(bar_s);
            // ---- out^T = V^T . P^T: A = V tile as stored (rows = tokens: M-contiguous), B = P (K-major over tokens) ----
            if (ok && mbar_wait_bounded(bar_v, 0) && mbar_wait_bounded(bar_p, 0)) {
                tc_fence_after();
                constexpr uint32_t idesc2 = tc_idesc_mn(kVtD, kVtPairs, true);
#pragma unroll
                for (int kk = 0; kk < kVtTok / 16; ++kk) {                   // 16 tokens per MMA
                    // A: 16 token rows of 128 bytes = 2048 bytes further per step; the second 64-dim block is the other box
                    const uint64_t ad = tc_smem_desc(sV + kk * 2048, kVtTileBytes);
                    // B: block kk / 4 of P (64 tokens each), 32 bytes per 16 tokens inside the swizzled row
                    const uint64_t bd = tc_smem_desc(sP + (kk >> 2) * kVtQBytes) + (uint64_t)((kk & 3) * 2);
                    tc_mma(tmem + (uint32_t)NP, ad, bd, idesc2, (uint32_t)(kk != 0));
                    if (two_terms)
                        tc_mma(tmem + (uint32_t)NP, ad, tc_smem_desc(sQ + (kk >> 2) * kVtQBytes) + (uint64_t)((kk & 3) * 2), idesc2, 1u);
                }
            } else if (ok) {
                atomicExch(d_status, CASS_ERR_TIMEOUT);
                mbar_wait_bounded(bar_v, 0);
            }
            tc_commit(bar_o);
        }
    } else if (warp >= 2) {
        const int q = warp & 3;                       // the tensor-memory lane quarter this warp may read
        const int et = q * 32 + lane;                 // this thread's token (scores) and dim (output)
        const float scale = rsqrtf((float)kVtD);
        uint32_t v[32];
        const bool have = mbar_wait_bounded(bar_s, 0);
        if (have) { __syncwarp(); tc_fence_after(); }
        else atomicExch(d_status, CASS_ERR_TIMEOUT);
        // scores^T -> sS[pair][token], scaled, causal: row r of the call sits at position len + r
#pragma unroll
        for (int c0 = 0; c0 < NP; c0 += 32) {
            if (have) tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int p = c0 + i;
                const bool vis = have && (t0 + et) <= s_lim[p];
                sS[p * kVtTok + et] = vis ? __uint_as_float(v[i]) * scale : -INFINITY;
            }
        }
        named_sync_128();
        // chunk softmax of every pair (warp q: pairs q, q + 4, ...), numerators rounded to bf16 into the P operand
#pragma unroll 2
        for (int p = q; p < kVtPairs; p += 4) {
            float a[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) a[k] = sS[p * kVtTok + lane + 32 * k];
            const float m = warp_max(fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3])));
            float l = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float e = (m == -INFINITY) ? 0.f : expf(a[k] - m);
                const uint16_t eb = float_to_bf16_bits(e);
                const int t = lane + 32 * k;
                float used = bf16_bits_to_float(eb);
                if (two_terms) {                              // Q has been consumed: the remainder goes there
                    const uint16_t lo = float_to_bf16_bits(e - used);
                    used += bf16_bits_to_float(lo);
                    *reinterpret_cast<uint16_t*>(sQ + (t >> 6) * kVtQBytes + swz_off(p, t & 63)) = lo;
                }
                l += used;                                    // the sum of what the MMA multiplies
                *reinterpret_cast<uint16_t*>(sP + (t >> 6) * kVtQBytes + swz_off(p, t & 63)) = eb;
            }
            l = warp_sum(l);
            if (lane == 0 && t0 <= s_lim[p]) {
                sc.m[s_at[p]] = m;
                sc.l[s_at[p]] = l;
            }
        }
        fence_proxy_async();
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar_p)) : "memory");
        if (mbar_wait_bounded(bar_o, 0)) {
            __syncwarp();
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < NP; c0 += 32) {
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(NP + c0), v);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int p = c0 + i;
                    if (t0 <= s_lim[p]) sc.o[(size_t)s_at[p] * kVtD + et] = __uint_as_float(v[i]);
                }
            }
        } else {
            atomicExch(d_status, CASS_ERR_TIMEOUT);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kVtTmemCols) : "memory");
    }
}

bool verify_attn_tc_usable(const KvGeom& g, int rps, int n_q) {
    return g.d == kVtD && rps * (n_q / g.n_kv) <= kVtMaxPairs && (g.seq_stride % 16) == 0;
}

int launch_verify_attn_tc(const KvGeom& g, const uint16_t* k_cache, const uint16_t* v_cache, const uint16_t* qkv, int n_seq,
                          const AttnRows& ar, int fine, int n_q, int np_cols, const DevState* st, const AttnScratch& sc, uint16_t* out,
                          int32_t* d_status, cudaStream_t s) {
    if (!verify_attn_tc_usable(g, ar.group, n_q) || (np_cols != 32 && np_cols != 64) || ar.group * (n_q / g.n_kv) > np_cols)
        return CASS_ERR_UNSUPPORTED;
    CUtensorMap mk, mv;
    int rc = tc_cache_map(&mk, g, k_cache, n_seq);
    if (!rc) rc = tc_cache_map(&mv, g, v_cache, n_seq);
    if (rc) return rc;
    const int n_groups = ceil_div(ar.hi - ar.lo, ar.group);
    dim3 grid(ar.chunks, g.n_kv, n_seq * n_groups);
    if (np_cols == 32) {
        CASS_ALLOW_SMEM(k_verify_attn_tc<32>);
        CASS_PDL_LAUNCH(k_verify_attn_tc<32>, grid, dim3(kVtThreads), (size_t)vt_smem(32), s, mk, mv, qkv, ar, n_groups, fine, n_q,
                        g.n_kv, st, sc, d_status);
    } else {
        CASS_ALLOW_SMEM(k_verify_attn_tc<64>);
        CASS_PDL_LAUNCH(k_verify_attn_tc<64>, grid, dim3(kVtThreads), (size_t)vt_smem(64), s, mk, mv, qkv, ar, n_groups, fine, n_q,
                        g.n_kv, st, sc, d_status);
    }
    return launch_attn_merge(sc, kVtTok, n_seq, ar, n_q, g.d, st, 0, 0, out, s);
}

}  // namespace cass
