// Log-sum-exp merge of the attention kernels' partial results, and the dispatch of the draft attention (Sec. 4.1 draft
// inference over the compressed KV cache of Sec. 4.2; the kernel itself is in draft_attn_tc.cu).
#include "kernels.cuh"

namespace cass {

// Merge the chunk partials of every (row, query head): out = sum_c e^{m_c - M} o_c / sum_c e^{m_c - M} l_c.
// Row i of a sequence sees positions < len + (draft: inflight + 1 | verify: i + 1);
// chunks hold `chunk_tokens` positions.
// The reductions run in a fixed order that depends on the number of visible chunks only.
constexpr int kMergeThreads = 256;
constexpr int kMergeWarps = kMergeThreads / 32;

__global__ void __launch_bounds__(kMergeThreads) k_attn_merge(AttnScratch sc, int chunk_tokens, AttnRows ar, int n_q, int d,
                                                              const DevState* __restrict__ st, int draft_mode, int draft_units,
                                                              uint16_t* __restrict__ out) {
    extern __shared__ __align__(16) float w_s[];    // [n_chunks_alloc] weights e^{m_c - M}, then [kMergeWarps][d] partial outputs
    __shared__ float s_red[kMergeWarps];
    pdl_wait();
    pdl_early<3>();
    const int hq = blockIdx.x, r = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = ar.hi - ar.lo, seq = r / sub, n_chunks_alloc = ar.chunks;
    const int row = ar.lo + r % sub;                                        // of the sequence's rps rows
    const int vis = st->len[seq] + (draft_mode ? st->inflight[seq] + 1 : row + 1);
    if (draft_units < 0) chunk_tokens = tc_run_tokens(vis, -draft_units);     // the draft attention's runs follow the visible length
    const int n_ch = ceil_div(vis, chunk_tokens);
    const size_t pair = (size_t)r * n_q + hq;
    const float* mp = sc.m + pair * n_chunks_alloc;
    const float* lp = sc.l + pair * n_chunks_alloc;
    float* part_s = w_s + ((n_chunks_alloc + 3) & ~3);
    // What the first round of every loop below needs is requested here, before any of it is used: the statistics of
    // chunk tid and the partial outputs of this warp's first two chunks share one round trip to L2.
    const float* op = sc.o + pair * n_chunks_alloc * d;
    const bool has0 = tid < n_ch;
    const float m_first = has0 ? __ldcg(mp + tid) : -INFINITY, l_first = has0 ? __ldcg(lp + tid) : 0.f;
    const int dim0 = lane * 4;
    float4 o_first[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int c = warp + k * kMergeWarps;
        o_first[k] = (c < n_ch && dim0 < d) ? __ldcg(reinterpret_cast<const float4*>(op + (size_t)c * d + dim0)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float M = m_first;
    for (int c = tid + kMergeThreads; c < n_ch; c += kMergeThreads) M = fmaxf(M, mp[c]);
    M = warp_max(M);
    if (lane == 0) s_red[warp] = M;
    __syncthreads();
    M = s_red[0];
#pragma unroll
    for (int w = 1; w < kMergeWarps; ++w) M = fmaxf(M, s_red[w]);
    __syncthreads();
    float L = 0.f;
    if (has0) {
        const float w = expf(m_first - M);
        w_s[tid] = w;
        L += w * l_first;
    }
    for (int c = tid + kMergeThreads; c < n_ch; c += kMergeThreads) {
        const float w = expf(mp[c] - M);
        w_s[c] = w;
        L += w * lp[c];
    }
    L = warp_sum(L);
    if (lane == 0) s_red[warp] = L;
    __syncthreads();
    L = s_red[0];
#pragma unroll
    for (int w = 1; w < kMergeWarps; ++w) L += s_red[w];
    // warp w adds the chunks w, w + 8, ... (four dims per lane, 16-byte loads); the warps' sums are then added in warp
    // order: the order of every addition depends on the number of visible chunks only
    for (int dim = dim0; dim < d; dim += 128) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        int c = warp;
        if (dim == dim0) {
#pragma unroll
            for (int k = 0; k < 2; ++k, c += kMergeWarps) {
                if (c < n_ch) {
                    const float w = w_s[c];
                    const float4 o = o_first[k];
                    acc.x = fmaf(w, o.x, acc.x); acc.y = fmaf(w, o.y, acc.y); acc.z = fmaf(w, o.z, acc.z); acc.w = fmaf(w, o.w, acc.w);
                }
            }
        }
#pragma unroll 4
        for (; c < n_ch; c += kMergeWarps) {
            const float w = w_s[c];
            const float4 o = *reinterpret_cast<const float4*>(op + (size_t)c * d + dim);
            acc.x = fmaf(w, o.x, acc.x); acc.y = fmaf(w, o.y, acc.y); acc.z = fmaf(w, o.z, acc.z); acc.w = fmaf(w, o.w, acc.w);
        }
        *reinterpret_cast<float4*>(part_s + warp * d + dim) = acc;
    }
    __syncthreads();
    for (int dim = tid; dim < d; dim += kMergeThreads) {
        float acc = part_s[dim];
#pragma unroll
        for (int w = 1; w < kMergeWarps; ++w) acc += part_s[w * d + dim];
        out[(((size_t)seq * ar.rps + row) * n_q + hq) * d + dim] = float_to_bf16_bits(acc / L);
    }
}

// The same for at most MC chunks: one warp a (row, query head), lane = chunk for the statistics, then four dims a lane with all
// chunks requested at once.  Every sum is formed in the order of k_attn_merge (eight interleaved chains, added in turn), so
// the bits are the same.  A CTA of 8 warps and three barriers a pair, most of it idle, took 13.5 us for 4096 pairs.
template <int MC>
__global__ void __launch_bounds__(kMergeThreads) k_attn_merge_few(AttnScratch sc, int chunk_tokens, AttnRows ar, int n_pairs, int n_q, int d,
                                                                  const DevState* __restrict__ st, int draft_mode, int draft_units,
                                                                  uint16_t* __restrict__ out) {
    pdl_wait();
    pdl_early<3>();
    const int pair = blockIdx.x * kMergeWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (pair >= n_pairs) return;
    const int r = pair / n_q, hq = pair % n_q, sub = ar.hi - ar.lo, seq = r / sub, row = ar.lo + r % sub;
    const int vis = st->len[seq] + (draft_mode ? st->inflight[seq] + 1 : row + 1);
    if (draft_units < 0) chunk_tokens = tc_run_tokens(vis, -draft_units);
    const int n_ch = ceil_div(vis, chunk_tokens);
    const size_t base = (size_t)pair * ar.chunks;
    const float* op = sc.o + base * d;
    const float m = lane < n_ch ? __ldcg(sc.m + base + lane) : -INFINITY, l = lane < n_ch ? __ldcg(sc.l + base + lane) : 0.f;
    float M = 0.f, L = 0.f, w = 0.f;
    for (int d0 = 0; d0 < d; d0 += 128) {
        const int dim = min(d0 + lane * 4, d - 4);                        // lanes beyond the head repeat its last dims
        float4 o[MC];
#pragma unroll
        for (int c = 0; c < MC; ++c) o[c] = __ldcg(reinterpret_cast<const float4*>(op + (size_t)min(c, n_ch - 1) * d + dim));
        if (d0 == 0) {
            M = warp_max(m);
            w = lane < n_ch ? expf(m - M) : 0.f;
            L = warp_sum(w * l);
        }
        float4 total = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c0 = 0; c0 < kMergeWarps; ++c0) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = c0; c < MC; c += kMergeWarps) {
                const float wc = __shfl_sync(0xffffffffu, w, c);
                if (c < n_ch) {
                    acc.x = fmaf(wc, o[c].x, acc.x); acc.y = fmaf(wc, o[c].y, acc.y);
                    acc.z = fmaf(wc, o[c].z, acc.z); acc.w = fmaf(wc, o[c].w, acc.w);
                }
            }
            total.x = c0 ? total.x + acc.x : acc.x; total.y = c0 ? total.y + acc.y : acc.y;
            total.z = c0 ? total.z + acc.z : acc.z; total.w = c0 ? total.w + acc.w : acc.w;
        }
        const uint32_t b[4] = {float_to_bf16_bits(total.x / L), float_to_bf16_bits(total.y / L), float_to_bf16_bits(total.z / L),
                               float_to_bf16_bits(total.w / L)};
        *reinterpret_cast<uint2*>(out + (((size_t)seq * ar.rps + row) * n_q + hq) * d + dim) = make_uint2(b[0] | (b[1] << 16), b[2] | (b[3] << 16));
    }
}

int launch_attn_merge(const AttnScratch& sc, int chunk_tokens, int n_seq, const AttnRows& ar, int n_q, int d,
                      const DevState* st, int draft_mode, int draft_units, uint16_t* out, cudaStream_t s) {
    if (d % 4) return CASS_ERR_UNSUPPORTED;
    dim3 grid(n_q, n_seq * (ar.hi - ar.lo));
    const int pairs = n_q * n_seq * (ar.hi - ar.lo);
    // a warp a pair where few chunks are possible (by the cache's size, not by what is visible now), or where pairs abound: with up
    // to 32 chunks a CTA a pair is 0.3 to 0.4 us faster for 32 to 128 pairs (a drafted token of four 8B-shaped sequences) and up to 1 us
    // for 320; a warp a pair gains 1 us for 640 pairs and 3 us for 1792 (8 x 7 rows), 2 % of a prompt of 2500 tokens
#define CASS_MERGE_FEW(MC)                                                                                                              \
    do {                                                                                                                                \
        CASS_PDL_LAUNCH(k_attn_merge_few<MC>, dim3(ceil_div(pairs, kMergeWarps)), dim3(kMergeThreads), 0, s, sc, chunk_tokens, ar, pairs, n_q, \
                        d, st, draft_mode, draft_units, out);                                                                           \
        return CASS_OK;                                                                                                                 \
    } while (0)
    if (ar.chunks <= 8) CASS_MERGE_FEW(8);
    if (ar.chunks <= 16 && pairs >= 1024) CASS_MERGE_FEW(16);
    if (ar.chunks <= 32 && pairs >= 1024) CASS_MERGE_FEW(32);
#undef CASS_MERGE_FEW
    const size_t smem = ((size_t)((ar.chunks + 3) & ~3) + (size_t)kMergeWarps * d) * 4;
    if (smem > 200 * 1024) return CASS_ERR_CAPACITY;
    CASS_ALLOW_SMEM(k_attn_merge);
    CASS_PDL_LAUNCH(k_attn_merge, grid, dim3(kMergeThreads), smem, s, sc, chunk_tokens, ar, n_q, d, st, draft_mode,
                    draft_units, out);
    return CASS_OK;
}

bool draft_attn_tc_supported(const KvGeom& g, int n_q);
int launch_draft_attn_tc(const KvGeom& g, const KvComp& ck, const KvComp& cv, const uint16_t* qkv, int qkv_stride, int n_q,
                         int n_seq, const DevState* st, const AttnScratch& sc, uint16_t* out, cudaStream_t s);

// Both record formats, truncations t = 0 and 4, up to 8 query heads per KV head, head sizes that are multiples of 32.
int launch_draft_attn(const KvGeom& g, const KvComp& ck, const KvComp& cv, const uint16_t* qkv, int qkv_stride, int n_q,
                      int n_seq, const DevState* st, const AttnScratch& sc, uint16_t* out, cudaStream_t s) {
    if (!draft_attn_tc_supported(g, n_q)) return CASS_ERR_UNSUPPORTED;
    return launch_draft_attn_tc(g, ck, cv, qkv, qkv_stride, n_q, n_seq, st, sc, out, s);
}

}  // namespace cass
