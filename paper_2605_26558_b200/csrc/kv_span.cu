// KV encoder for spans of tokens: a prompt (every layer and sequence in one go) or a long append.  The one-kernel encoder
// in kv.cu hands out arena offsets token by token inside one CTA per (head, K|V), which suits the few rows of a decode
// step; over a prompt it is 16 CTAs walking all tokens in sequence (2.6 ms for 2000 tokens of two 8B-shaped layers).
// Here every record is formed on its own and only the offsets are a scan:
//   k_kv_form      select, bitmap, fields (and the bf16 rows); with a frozen codebook also entry words and word counts,
//                  else the histogram of kept exponents
//   k_kv_rank      histogram -> codebook
//   k_kv_lengths   entry words and word counts, once the codebook is there
//   k_kv_scan      word counts -> arena offsets, in place
//   k_kv_codes     exponent words into the arena
// One warp a record throughout; a record's words sit 128 bytes apart (32-token blocks), so the 8 warps of a CTA take
// consecutive tokens and share sectors.  Bound: instruction issue (81 to 89 %): 725 warp instructions a record in k_kv_form, half of
// them the selection, 310 in k_kv_lengths, 400 in k_kv_codes; 57, 24 and 31 us under ncu for 2000 tokens of two 8B-shaped layers.
#include "kv_record.cuh"

namespace cass {

constexpr int kSpanWarps = 8;

// The objects of (layer, sequence) of a grid's z index: every layer's and every sequence's storage has the same layout.
struct KvSpan {
    int start, n_new;              // positions start .. start + n_new - 1
    int seq0, n_seq, n_layers;     // z = layer * n_seq + sequence - seq0
    size_t layer_stride;
};
__device__ __forceinline__ size_t span_shift(const KvGeom& g, const KvSpan& sp, int z) {
    return (size_t)(z / sp.n_seq) * sp.layer_stride + (size_t)(sp.seq0 + z % sp.n_seq) * g.seq_stride;
}

// grid ((tokens / 8, cut off), n_kv * 2, layers * sequences)
template <int NJ, int T, bool HIST>
__global__ void __launch_bounds__(32 * kSpanWarps) k_kv_form(KvGeom g, KvComp ck, KvComp cv, uint16_t* __restrict__ k_cache,
                                                             uint16_t* __restrict__ v_cache, const uint16_t* __restrict__ src_k,
                                                             const uint16_t* __restrict__ src_v, int row_stride, KvSpan sp, int flags) {
    constexpr int F = 8 - T, PER = 32 / F, FW = NJ * 32 / PER;
    __shared__ uint32_t s_rec[kSpanWarps][3 + NJ + FW + 2];
    __shared__ __align__(8) uint8_t s_fld[kSpanWarps][NJ * 32 + 8];
    __shared__ uint32_t s_len[256];                                     // code lengths (HIST: counts)
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    uint16_t* cache = of_seq(kind ? v_cache : k_cache, 1, shift);
    pdl_wait();
    s_len[threadIdx.x] = HIST || !(flags & CASS_KV_COMPRESSED) ? 0u : c.exp_to_rank[threadIdx.x] + 1u;
    __syncthreads();
    // HIST: the rows are those of the cache
    const uint16_t* src = HIST ? cache + (size_t)sp.start * g.n_kv * g.d : (kind ? src_v : src_k) + (size_t)(blockIdx.z % sp.n_seq) * sp.n_new * row_stride;
    const size_t stride = HIST ? (size_t)g.n_kv * g.d : (size_t)row_stride;
    const int nj = g.d / 32;
    uint32_t* rec = s_rec[warp];
    for (int i = blockIdx.x * kSpanWarps + warp; i < sp.n_new; i += gridDim.x * kSpanWarps) {
        const int pos = sp.start + i;
        if (pos >= g.max_seq) break;
        const uint16_t* row = src + (size_t)i * stride + (size_t)head * g.d;
        uint32_t bits[NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) bits[j] = j < nj ? row[lane + 32 * j] : 0u;
        if (flags & CASS_KV_BF16) {
            uint16_t* dst = cache + ((size_t)pos * g.n_kv + head) * g.d;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (j < nj) dst[lane + 32 * j] = (uint16_t)bits[j];
        }
        if (!(flags & CASS_KV_COMPRESSED)) continue;
        uint32_t bm[NJ];
        kv_select<NJ>(bits, nj, g.n_prune, lane, bm);
        const bool mx = g.mode == 2;
        const int bm0 = g.e_words;                                      // the bitmap's place in the record
        uint32_t len[NJ], kbase = 0, xw[2] = {0, 0};
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            len[j] = 0;
            if (j >= nj) break;
            const bool keep = (bm[j] >> lane) & 1u;
            const uint32_t e = (bits[j] >> 7) & 0xFFu, k = kbase + __popc(bm[j] & lanemask_lt());
            uint32_t E;
            const uint32_t field = kv_field<T>(bits[j], keep, mx, E);
            xw[j / 4] |= E << (24 - 8 * (j % 4));
            if (keep) {
                s_fld[warp][k] = (uint8_t)field;
                if (HIST) atomicAdd(&s_len[e], 1u);
                else len[j] = s_len[e];
            }
            if (lane == j) rec[bm0 + j] = __brev(bm[j]);                // channel c at bit 31 - c%32
            kbase += __popc(bm[j]);
        }
        if (!HIST) {
            uint32_t entry[3], nw = 0;
            if (!mx) {
                nw = kv_entries<NJ>(g, len, nj, entry);
                if (lane < g.e_words) rec[lane] = lane == 0 ? entry[0] : lane == 1 ? entry[1] : entry[2];
            }
            if (lane == 0) c.off[(size_t)head * (g.max_seq + 1) + pos + 1] = nw;       // k_kv_scan makes it an offset
        } else if (mx && lane == 0) {
            c.off[(size_t)head * (g.max_seq + 1) + pos + 1] = 0;        // no exponent stream
        }
        if (mx && lane < g.x_words) rec[bm0 + nj + g.f_words + lane] = lane ? xw[1] : xw[0];
        __syncwarp();
        kv_field_words<T>(g, s_fld[warp], rec + bm0 + nj, lane);
        __syncwarp();
        uint32_t* blk = c.fixed + ((size_t)head * g.n_blocks + pos / 32) * g.wpt * 32 + pos % 32;
        for (int w = (HIST ? g.e_words : 0) + lane; w < g.wpt; w += 32) blk[w * 32] = rec[w];
        __syncwarp();
    }
    if (HIST) {
        __syncthreads();
        if (s_len[threadIdx.x]) atomicAdd(&c.hist[threadIdx.x], (unsigned long long)s_len[threadIdx.x]);
    }
}

// grid (K|V, layers * sequences): codebook from the histogram, which is left zero for the next time
__global__ void __launch_bounds__(256) k_kv_rank(KvGeom g, KvComp ck, KvComp cv, KvSpan sp) {
    __shared__ unsigned long long s[256];
    const KvComp c = of_seq(blockIdx.x ? cv : ck, 1, span_shift(g, sp, blockIdx.y));
    const int e = threadIdx.x;
    pdl_wait();
    const unsigned long long mine = c.hist[e];
    s[e] = mine;
    c.hist[e] = 0;
    __syncthreads();
    int rank = 0;
#pragma unroll 16
    for (int o = 0; o < 256; ++o) rank += (s[o] > mine) || (s[o] == mine && o < e);
    c.rank_to_exp[rank] = (uint8_t)e;
    c.exp_to_rank[e] = (uint8_t)rank;
}

// grid as k_kv_form: entry words and word counts of records whose bitmaps are there
template <int NJ>
__global__ void __launch_bounds__(32 * kSpanWarps) k_kv_lengths(KvGeom g, KvComp ck, KvComp cv, const uint16_t* __restrict__ k_cache,
                                                                const uint16_t* __restrict__ v_cache, KvSpan sp) {
    __shared__ uint32_t s_len[256];
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    const uint16_t* cache = of_seq(kind ? v_cache : k_cache, 1, shift);
    pdl_wait();
    s_len[threadIdx.x] = c.exp_to_rank[threadIdx.x] + 1u;
    __syncthreads();
    const int nj = g.d / 32;
    for (int i = blockIdx.x * kSpanWarps + warp; i < sp.n_new; i += gridDim.x * kSpanWarps) {
        const int pos = sp.start + i;
        if (pos >= g.max_seq) break;
        uint32_t* blk = c.fixed + ((size_t)head * g.n_blocks + pos / 32) * g.wpt * 32 + pos % 32;
        const uint16_t* row = cache + ((size_t)pos * g.n_kv + head) * g.d;
        uint32_t len[NJ], bits[NJ], bm[NJ], entry[3], nw;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            bm[j] = j < nj ? blk[(g.e_words + j) * 32] : 0u;
            bits[j] = j < nj ? row[lane + 32 * j] : 0u;
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) len[j] = (bm[j] << lane) >> 31 ? s_len[(bits[j] >> 7) & 0xFFu] : 0u;
        nw = kv_entries<NJ>(g, len, nj, entry);
        if (lane < g.e_words) blk[lane * 32] = lane == 0 ? entry[0] : lane == 1 ? entry[1] : entry[2];
        if (lane == 0) c.off[(size_t)head * (g.max_seq + 1) + pos + 1] = nw;
    }
}

// grid (n_kv * 2, layers * sequences): the word counts at off[start + 1 ...] become offsets behind off[start]
__global__ void __launch_bounds__(1024) k_kv_scan(KvGeom g, KvComp ck, KvComp cv, KvSpan sp, DevState* st) {
    __shared__ uint32_t s_sum[32];
    const int head = blockIdx.x % g.n_kv, kind = blockIdx.x / g.n_kv;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const KvComp c = of_seq(kind ? cv : ck, 1, span_shift(g, sp, blockIdx.y));
    uint32_t* off = c.off + (size_t)head * (g.max_seq + 1) + sp.start;
    const int n = min(sp.n_new, g.max_seq - sp.start);
    pdl_wait();
    uint32_t carry = off[0];
    for (int base = 1; base <= n; base += 1024) {
        const int i = base + tid;
        const uint32_t v = i <= n ? off[i] : 0u;
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        const uint32_t below = __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u);
        const uint32_t all = __reduce_add_sync(0xffffffffu, s_sum[lane]);
        // past the arena's end (its size covers every record that fits the cache): offsets stay valid, the codes are dropped
        const uint32_t o = carry + below + incl;
        if (i <= n) off[i] = min(o, (uint32_t)g.arena_words);
        if (o > (uint32_t)g.arena_words && i <= n) atomicCAS(&st->status, 0, CASS_ERR_CAPACITY);
        carry += all;
        __syncthreads();
    }
}

// grid as k_kv_form: the exponent words of every record at its offset
template <int NJ>
__global__ void __launch_bounds__(32 * kSpanWarps) k_kv_codes(KvGeom g, KvComp ck, KvComp cv, const uint16_t* __restrict__ k_cache,
                                                              const uint16_t* __restrict__ v_cache, const uint16_t* __restrict__ src_k,
                                                              const uint16_t* __restrict__ src_v, int row_stride, KvSpan sp) {
    __shared__ uint32_t s_len[256];
    __shared__ uint32_t s_una[kSpanWarps][64];                          // 1023 code bits, or 256 raw bytes
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    pdl_wait();
    s_len[threadIdx.x] = c.exp_to_rank[threadIdx.x] + 1u;
    __syncthreads();
    const uint16_t* src = src_k ? (kind ? src_v : src_k) + (size_t)(blockIdx.z % sp.n_seq) * sp.n_new * row_stride
                                : of_seq(kind ? v_cache : k_cache, 1, shift) + (size_t)sp.start * g.n_kv * g.d;
    const size_t stride = src_k ? (size_t)row_stride : (size_t)g.n_kv * g.d;
    const uint32_t* off = c.off + (size_t)head * (g.max_seq + 1);
    uint32_t* arena = c.arena + (size_t)head * g.arena_words;
    const int nj = g.d / 32;
    uint32_t* una = s_una[warp];
    for (int i = blockIdx.x * kSpanWarps + warp; i < sp.n_new; i += gridDim.x * kSpanWarps) {
        const int pos = sp.start + i;
        if (pos >= g.max_seq) break;
        const uint32_t* blk = c.fixed + ((size_t)head * g.n_blocks + pos / 32) * g.wpt * 32 + pos % 32;
        const uint16_t* row = src + (size_t)i * stride + (size_t)head * g.d;
        uint32_t bits[NJ], bm[NJ];
        const uint32_t o0 = off[pos], nw = off[pos + 1] - o0, first = blk[0];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            bm[j] = j < nj ? blk[(g.e_words + j) * 32] : 0u;
            bits[j] = j < nj ? row[lane + 32 * j] : 0u;
        }
        una[lane] = 0;
        una[lane + 32] = 0;
        __syncwarp();
        if (first & kKvRawFlag) {                                       // the kept exponents as bytes
            uint32_t base = 0;                                          // kept values of the slices before
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                if (j >= nj) break;
                const uint32_t k = base + (lane ? __popc(bm[j] >> (32 - lane)) : 0u);
                if ((bm[j] << lane) >> 31) atomicOr(&una[(k >> 2) & 63u], ((bits[j] >> 7) & 0xFFu) << (24 - 8 * (k & 3)));
                base += __popc(bm[j]);
            }
        } else {
            uint32_t len[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) len[j] = (bm[j] << lane) >> 31 ? s_len[(bits[j] >> 7) & 0xFFu] : 0u;
            kv_code_bits<NJ>(len, nj, lane, una);
        }
        __syncwarp();
        for (uint32_t w = lane; w < nw && w < 64u; w += 32) arena[o0 + w] = una[w];
        __syncwarp();
    }
}

template <int NJ, int T>
static int span_encode(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, const uint16_t* src_k,
                       const uint16_t* src_v, int row_stride, const KvSpan& sp, int flags, bool codebook, DevState* st, cudaStream_t s) {
    const int z = sp.n_layers * sp.n_seq, blocks = ceil_div(sp.n_new, kSpanWarps);
    const dim3 heads(g.n_kv * 2, z), threads(32 * kSpanWarps);
    if (codebook) {
        // a CTA adds its counts to the histogram once: some 2000 CTAs over all heads, each with its share of the tokens
        int bx = ceil_div(2048, g.n_kv * 2 * z);
        if (bx < 4) bx = 4;
        if (bx > blocks) bx = blocks;
        if (bx > 0)
            CASS_PDL_LAUNCH((k_kv_form<NJ, T, true>), dim3(bx, g.n_kv * 2, z), threads, 0, s, g, ck, cv, k_cache, v_cache,
                            (const uint16_t*)nullptr, (const uint16_t*)nullptr, 0, sp, flags);
        CASS_PDL_LAUNCH(k_kv_rank, dim3(2, z), dim3(256), 0, s, g, ck, cv, sp);
        if (bx == 0) return CASS_OK;
        if (g.mode == 1)
            CASS_PDL_LAUNCH(k_kv_lengths<NJ>, dim3(blocks, g.n_kv * 2, z), threads, 0, s, g, ck, cv, (const uint16_t*)k_cache,
                            (const uint16_t*)v_cache, sp);
    } else {
        CASS_PDL_LAUNCH((k_kv_form<NJ, T, false>), dim3(blocks, g.n_kv * 2, z), threads, 0, s, g, ck, cv, k_cache, v_cache, src_k, src_v,
                        row_stride, sp, flags);
        if (!(flags & CASS_KV_COMPRESSED)) return CASS_OK;
    }
    CASS_PDL_LAUNCH(k_kv_scan, heads, dim3(1024), 0, s, g, ck, cv, sp, st);
    if (g.mode == 1)
        CASS_PDL_LAUNCH(k_kv_codes<NJ>, dim3(blocks, g.n_kv * 2, z), threads, 0, s, g, ck, cv, (const uint16_t*)k_cache, (const uint16_t*)v_cache,
                        codebook ? (const uint16_t*)nullptr : src_k, codebook ? (const uint16_t*)nullptr : src_v, row_stride, sp);
    return CASS_OK;
}

template <int NJ>
static int span_encode_t(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, const uint16_t* src_k,
                         const uint16_t* src_v, int row_stride, const KvSpan& sp, int flags, bool codebook, DevState* st, cudaStream_t s) {
    if (g.t == 4) return span_encode<NJ, 4>(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, codebook, st, s);
    if (g.t == 0) return span_encode<NJ, 0>(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, codebook, st, s);
    return CASS_ERR_UNSUPPORTED;                                        // sessions take no other truncation
}

static int span_encode_any(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, const uint16_t* src_k,
                           const uint16_t* src_v, int row_stride, const KvSpan& sp, int flags, bool codebook, DevState* st, cudaStream_t s) {
    if (g.d <= 64) return span_encode_t<2>(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, codebook, st, s);
    if (g.d <= 128) return span_encode_t<4>(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, codebook, st, s);
    return span_encode_t<8>(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, codebook, st, s);
}

int launch_kv_span(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, const uint16_t* src_k,
                   const uint16_t* src_v, int row_stride, int start_pos, int n_new, int flags, DevState* st, int seq0, int n_seq, cudaStream_t s) {
    const KvSpan sp{start_pos, n_new, seq0, n_seq, 1, 0};
    return span_encode_any(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags, false, st, s);
}

int launch_kv_codebook(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, int n_layers,
                       size_t layer_stride, int n_seq, int n_tokens, DevState* st, cudaStream_t s) {
    const KvSpan sp{0, n_tokens, 0, n_seq, n_layers, layer_stride};
    return span_encode_any(g, ck, cv, k_cache, v_cache, nullptr, nullptr, 0, sp, CASS_KV_COMPRESSED, true, st, s);
}

}  // namespace cass
