// KV encoder for spans of tokens: a prompt (every layer and sequence in one go) or a long append.  The one-kernel encoder
// in kv.cu hands out arena offsets token by token inside one CTA per (head, K|V), which suits the few rows of a decode
// step; over a prompt it is 16 CTAs walking all tokens in sequence (2.6 ms for 2000 tokens of two 8B-shaped layers).
// Here every record is formed on its own and only the offsets are a scan (below; many records take the same steps with a lane each):
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

// grid (K|V, layers * sequences): codebook from the histogram, which is left zero for the next time.  A count and its exponent are one
// number, so that a comparison is one.  Lanes an exponent, us a call, 1 / 2 / 4 (and with two comparisons, one lane): 2000 tokens of two
// 8B-shaped layers 52.7 / 52.6 / 53.6 (54.4 with four), three layers of two sequences of 234 tokens (head size 64) 16.4 / 16.3 / 17.3 (17.8).
constexpr int kRankLanes = 2;
__global__ void __launch_bounds__(256 * kRankLanes) k_kv_rank(KvGeom g, KvComp ck, KvComp cv, KvSpan sp) {
    __shared__ __align__(16) unsigned long long s[256];
    const KvComp c = of_seq(blockIdx.x ? cv : ck, 1, span_shift(g, sp, blockIdx.y));
    const int e = threadIdx.x / kRankLanes, part = threadIdx.x % kRankLanes;
    pdl_wait();
    if (threadIdx.x < 256) {
        s[threadIdx.x] = c.hist[threadIdx.x] << 8 | (255u - threadIdx.x);      // of equal counts the smaller exponent first
        c.hist[threadIdx.x] = 0;
    }
    __syncthreads();
    const unsigned long long mine = s[e];
    int rank = 0;
#pragma unroll 16
    for (int i = 0; i < 128 / kRankLanes; ++i) {
        const ulonglong2 o = reinterpret_cast<const ulonglong2*>(s)[i * kRankLanes + part];
        rank += (o.x > mine ? 1 : 0) + (o.y > mine ? 1 : 0);
    }
#pragma unroll
    for (int i = 1; i < kRankLanes; i *= 2) rank += __shfl_xor_sync(0xffffffffu, rank, i);
    if (part == 0) {
        c.rank_to_exp[rank] = (uint8_t)e;
        c.exp_to_rank[e] = (uint8_t)rank;
    }
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

// ---- the same with a lane a record, where there are many -------------------------------------------------------------
// A warp takes 32 positions that share a block of the cache, a lane one of them: the rows are copied into shared memory (16 bytes
// beyond a multiple of 64 apart, so that lanes read 16 bytes of their own rows without conflicts), and the search, the bitmap, the
// fields and the code bits are then a lane's own work: no reductions, scans or ballots, which are most of what a warp on one record
// of four values a lane executes.  Record words are 32 tokens side by side, so a warp's stores are whole lines.
// Bound: the integer pipe (61 %) and latency, 235 instructions a record to form it (725 with a warp).  2000 tokens of two 8B-shaped layers
// 104 -> 53 us (form 30, lengths 11, codes 20 under ncu), Cassandra-2 64 -> 41, four layers of four sequences of 1000 tokens 369 -> 160.
// A warp's chain is long, 25 to 38 us for all the kernels whatever the size, against 8 to 20 where a warp a record leaves the chip idle:
// 512 warps 36 (warps) and 38 us, 640 warps of head size 64 35 and 28.  Releasing the successors early: 54 -> 64 us, their waiting CTAs
// take this one's place.
constexpr int kLaneWarps(int nj) { return nj <= 4 ? 4 : 2; }
constexpr int kLaneMin = 600;                        // warps (32 positions of a head, K or V) from which on lanes are faster
constexpr int kLaneCopies = 8;                       // of the histogram: lanes that share one meet less often

template <int NJ>
struct LaneRows {
    static constexpr int kStride = NJ * 64 + 16;     // bytes between two rows
    // The 32 rows of head `head` at positions 32 blk .. 32 blk + 31 of which lo .. hi - 1 exist; row(pos) in 16-byte pieces.  copy: the
    // same pieces of the cache, or null.
    template <class Row>
    static __device__ __forceinline__ void fetch(uint8_t* s, int nj, int blk, int lo, int hi, int lane, Row row, uint4* copy, size_t copy_stride) {
        const int ch = nj * 4;                       // pieces of a row
#pragma unroll 1
        for (int i0 = lane; i0 < 32 * ch; i0 += 32 * 8) {
            uint4 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = i0 + 32 * k, r = nj == NJ ? i / (NJ * 4) : i / ch, c = i - r * ch, pos = blk * 32 + r;
                v[k] = i < 32 * ch && pos >= lo && pos < hi ? __ldcg(row(pos) + c) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = i0 + 32 * k, r = nj == NJ ? i / (NJ * 4) : i / ch, c = i - r * ch, pos = blk * 32 + r;
                if (i < 32 * ch) {
                    *reinterpret_cast<uint4*>(s + r * kStride + c * 16) = v[k];
                    if (copy && pos >= lo && pos < hi) copy[(size_t)pos * copy_stride + c] = v[k];
                }
            }
        }
        __syncwarp();
    }
};

// Eight values of a lane's row: words of two, the lower channel in the lower half.
__device__ __forceinline__ void lane_get8(const uint8_t* row, int g, uint32_t (&x)[4]) {
    const uint4 v = *reinterpret_cast<const uint4*>(row + g * 16);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}

// The lane's kept set, as kv_select gives it: bit 31 - c % 32 of word c / 32, 32 words apart at bm.  A threshold with at most n_prune
// keys |x| below it and more below the next is searched by halving, near the largest value first; a packed addition leaves "not
// less" in bits 15 and 31.  Of the keys that equal it the first ones go.
// Loops over slices stay loops, and the values stay in shared memory: a warp runs through this once, and unrolled over 128
// channels the time went into fetching instructions (10 to 20 us whatever the size).
__device__ __forceinline__ void lane_select(const uint8_t* row, int nj, int n_prune, uint32_t* bm) {
    uint32_t lo = 0, ne = 0;
    if (n_prune > 0) {
        uint32_t big2 = 0, x[4];
#pragma unroll 4
        for (int q = 0; q < nj * 4; ++q) {
            lane_get8(row, q, x);
#pragma unroll
            for (int i = 0; i < 4; ++i) big2 = __vmaxu2(big2, x[i] & 0x7FFF7FFFu);
        }
        uint32_t hi = max(big2 >> 16, big2 & 0xFFFFu) + 1u;
        int under = 0;                                               // keys below lo
        uint32_t mid = hi > 6u * 128u ? hi - 6u * 128u : 0u;         // six binades below the largest
#pragma unroll 1
        for (;;) {
            const uint32_t add = (0x8000u - mid) * 0x10001u;
            int n = 0;
#pragma unroll 1
            for (int j = 0; j < nj; ++j) {
                uint32_t acc = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    lane_get8(row, j * 4 + q, x);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc = (acc >> 1) | (((x[i] & 0x7FFF7FFFu) + add) & 0x80008000u);
                }
                n += 32 - __popc(acc);
            }
            if (n <= n_prune) { lo = mid; under = n; }
            else hi = mid;
            if (under == n_prune) hi = lo + 1u;                      // nothing between: any threshold here will do
            if (!__any_sync(0xffffffffu, hi - lo > 1u)) break;
            mid = (lo + hi) / 2u;
        }
        ne = (uint32_t)(n_prune - under);
    }
    const uint32_t add = (0x8000u - lo) * 0x10001u;
    const bool ties = __any_sync(0xffffffffu, ne > 0);
#pragma unroll 1
    for (int j = 0; j < nj; ++j) {
        uint32_t keep = 0, more = 0, x[4];                           // not less than the threshold; than the one after it
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            lane_get8(row, j * 4 + q, x);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t v = (x[i] & 0x7FFF7FFFu) + add, u = v - 0x10001u;      // v >= 0x10001 in each half: lo <= 0x7FFF
                keep = __funnelshift_l(v, __funnelshift_l(v << 16, keep, 1), 1);
                more = __funnelshift_l(u, __funnelshift_l(u << 16, more, 1), 1);
            }
        }
        if (ties) {
            uint32_t eq = keep & ~more;
            const uint32_t here = __popc(eq);
            if (ne >= here) { keep &= ~eq; ne -= here; }
            else
                for (; ne > 0; --ne) {
                    const uint32_t b = 0x80000000u >> __clz(eq);
                    keep ^= b;
                    eq ^= b;
                }
        }
        bm[j * 32] = keep;
    }
}

__device__ __forceinline__ uint32_t lane_half(const uint32_t (&x)[4], int i) { return (i & 1) ? x[i / 2] >> 16 : x[i / 2] & 0xFFFFu; }
__device__ __forceinline__ uint32_t lane_exp(const uint32_t (&x)[4], int i) { return ((i & 1) ? x[i / 2] >> 23 : x[i / 2] >> 7) & 0xFFu; }

// A slice's first code bit into the entry words; the words and the word count of a record that ends at code bit `ub`.
__device__ __forceinline__ void lane_entry(int j, uint32_t ub, uint32_t (&entry)[3]) {
    const uint32_t v = j > 0 ? (ub & 0x3FFu) << (20 - 10 * ((j - 1) % 3)) : 0u;
    if (j <= 3) entry[0] |= v;
    else if (j <= 6) entry[1] |= v;
    else entry[2] |= v;
}
__device__ __forceinline__ uint32_t lane_entries(const KvGeom& g, uint32_t ub, uint32_t (&entry)[3], uint32_t* rec) {
    const bool raw = ub > (uint32_t)kv_code_budget(g.kept);
    for (int w = 0; w < g.e_words; ++w) rec[w * 32] = raw ? (w == 0 ? kKvRawFlag : 0u) : w == 0 ? entry[0] : w == 1 ? entry[1] : entry[2];
    return raw ? (uint32_t)ceil_div(g.kept, 4) : (ub + 31) / 32;
}

// grid (blocks of 32 positions / warps, n_kv * 2, layers * sequences), HIST and flags as for k_kv_form
template <int NJ, int T, bool HIST>
__global__ void __launch_bounds__(32 * kLaneWarps(NJ)) k_kv_form_lanes(KvGeom g, KvComp ck, KvComp cv, uint16_t* __restrict__ k_cache,
                                                                       uint16_t* __restrict__ v_cache, const uint16_t* __restrict__ src_k,
                                                                       const uint16_t* __restrict__ src_v, int row_stride, KvSpan sp, int flags) {
    constexpr int F = 8 - T, PER = 32 / F, W = kLaneWarps(NJ), S = LaneRows<NJ>::kStride;
    constexpr uint32_t MASK = 0x80000000u | (((1u << (7 - T)) - 1u) << (16 + T));
    __shared__ __align__(16) uint8_t s_rows[W][32 * S];
    __shared__ uint32_t s_bm[W][NJ * 32];
    __shared__ uint32_t s_tab[HIST ? 256 * kLaneCopies : 256];         // counts, or code lengths
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv, nj = g.d / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    uint16_t* cache = of_seq(kind ? v_cache : k_cache, 1, shift);
    const bool mx = g.mode == 2;
    pdl_wait();
    for (int i = tid; i < (HIST ? 256 * kLaneCopies : 256); i += 32 * W) s_tab[i] = HIST ? 0u : c.exp_to_rank[i] + 1u;
    __syncthreads();
    const int lo = sp.start, hi = min(sp.start + sp.n_new, g.max_seq), blk = lo / 32 + (int)blockIdx.x * W + warp;
    if (blk * 32 < hi) {
        const int pos = blk * 32 + lane;
        const bool active = pos >= lo && pos < hi;
        const size_t cache_stride = (size_t)g.n_kv * g.d / 8;          // pieces of 16 bytes
        uint4* cache16 = reinterpret_cast<uint4*>(cache) + (size_t)head * nj * 4;
        const uint4* src16 = reinterpret_cast<const uint4*>((kind ? src_v : src_k)) + (size_t)head * nj * 4;
        uint8_t* rows = s_rows[warp];
        LaneRows<NJ>::fetch(rows, nj, blk, lo, hi, lane, [&](int p) {
            if (HIST) return (const uint4*)(cache16 + (size_t)p * cache_stride);
            return src16 + ((size_t)(blockIdx.z % sp.n_seq) * sp.n_new + (p - lo)) * (row_stride / 8);
        }, !HIST && (flags & CASS_KV_BF16) ? cache16 : nullptr, cache_stride);
        uint8_t* row = rows + lane * S;
        uint32_t* bm = s_bm[warp] + lane;
        uint32_t x[4];
        lane_select(row, nj, g.n_prune, bm);
        // the kept values move to the front of the row: as they are, or (mx) as fields, a byte each
        uint32_t* rec = c.fixed + ((size_t)head * g.n_blocks + blk) * g.wpt * 32 + lane;
        uint32_t* tab = s_tab + (HIST ? lane % kLaneCopies : 0);
        auto note = [&](uint32_t e) { if (active) atomicAdd(&tab[e * kLaneCopies], 1u); };
        uint32_t ub = 0, xw[2] = {0, 0}, entry[3] = {0, 0, 0};
        uint8_t* to = row;
#pragma unroll 1
        for (int j = 0; j < nj; ++j) {
            const uint32_t bmj = bm[j * 32];
            lane_entry(j, ub, entry);
            uint32_t E = 0;
            if (mx) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    lane_get8(row, j * 4 + q, x);
#pragma unroll
                    for (int i = 0; i < 8; ++i) E = max(E, bmj & (0x80000000u >> (q * 8 + i)) ? lane_exp(x, i) : 0u);
                }
                if (j < 4) xw[0] |= E << (24 - 8 * j);
                else xw[1] |= E << (56 - 8 * j);
            }
            // no branches: a value is stored whether kept or not, at a place at or before its own, and the next one takes its
            // place if it was not
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                const uint32_t b8 = bmj << (8 * q);
                lane_get8(row, j * 4 + q, x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const bool keep = b8 & (0x80000000u >> i);
                    const uint32_t v = lane_half(x, i), e = lane_exp(x, i);
                    if (mx) {
                        const uint32_t m7 = e > 0u && E >= 7u ? (0x80u | (v & 0x7Fu)) >> min(1u + E - e, 8u) : 0u;
                        *to = (uint8_t)(((v >> 15) << (7 - T)) | (m7 >> T));
                        to += keep ? 1 : 0;
                        if (HIST && keep) note(e);
                    } else {
                        *reinterpret_cast<uint16_t*>(to) = (uint16_t)v;
                        to += keep ? 2 : 0;
                        if (!HIST) ub += keep ? s_tab[e] : 0u;
                    }
                }
            }
            if (active) rec[(g.e_words + j) * 32] = bmj;
        }
        __syncwarp();
        // every record has as many kept values: from here on the lanes are in step, eight values at a time
        uint32_t* fl = rec + (g.e_words + nj) * 32;
#pragma unroll 1
        for (int k = 0; k < g.kept; k += 8) {
            uint32_t word[2] = {0, 0};
            const int left = g.kept - k;
            if (mx) {
                const uint2 b = *reinterpret_cast<const uint2*>(row + k);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t f = ((i < 4 ? b.x : b.y) >> (8 * (i & 3))) & 0xFFu;
                    if (i < left) word[i / PER] |= f << (32 - F * (i % PER + 1));
                }
            } else {
                lane_get8(row, k / 8, x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t canon = i < left ? ((i & 1) ? x[i / 2] : x[i / 2] << 16) & MASK : 0u;
                    word[i / PER] |= __funnelshift_r(canon, canon, (F * (i % PER)) & 31);
                    if (HIST && i < left) note(lane_exp(x, i));
                }
            }
            if (active) {
                fl[k / PER * 32] = word[0];
                if (PER == 4 && left > 4) fl[(k / 4 + 1) * 32] = word[1];
            }
        }
        if (active) {
            if (mx)
                for (int w = 0; w < g.x_words; ++w) rec[(g.e_words + nj + g.f_words + w) * 32] = xw[w & 1];
            uint32_t* off = c.off + (size_t)head * (g.max_seq + 1) + pos + 1;
            if (!HIST) {
                const uint32_t nw = mx ? 0u : lane_entries(g, ub, entry, rec);
                *off = nw;
            } else if (mx) {
                *off = 0;                                                    // no exponent stream
            }
        }
    }
    if (HIST) {
        __syncthreads();
        for (int e = tid; e < 256; e += 32 * W) {
            uint32_t n = 0;
#pragma unroll
            for (int i = 0; i < kLaneCopies; ++i) n += s_tab[e * kLaneCopies + i];
            if (n) atomicAdd(&c.hist[e], (unsigned long long)n);
        }
    }
}

// grid as k_kv_form_lanes: what k_kv_lengths does
template <int NJ>
__global__ void __launch_bounds__(32 * kLaneWarps(NJ)) k_kv_lengths_lanes(KvGeom g, KvComp ck, KvComp cv, const uint16_t* __restrict__ k_cache,
                                                                          const uint16_t* __restrict__ v_cache, KvSpan sp) {
    constexpr int W = kLaneWarps(NJ), S = LaneRows<NJ>::kStride;
    __shared__ __align__(16) uint8_t s_rows[W][32 * S];
    __shared__ uint32_t s_len[256];
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv, nj = g.d / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    const uint4* cache16 = reinterpret_cast<const uint4*>(of_seq(kind ? v_cache : k_cache, 1, shift)) + (size_t)head * nj * 4;
    const int lo = sp.start, hi = min(sp.start + sp.n_new, g.max_seq), blk = lo / 32 + (int)blockIdx.x * W + warp, pos = blk * 32 + lane;
    const size_t cache_stride = (size_t)g.n_kv * g.d / 8;
    pdl_wait();
    for (int i = tid; i < 256; i += 32 * W) s_len[i] = c.exp_to_rank[i] + 1u;
    __syncthreads();
    if (blk * 32 >= hi) return;
    LaneRows<NJ>::fetch(s_rows[warp], nj, blk, lo, hi, lane, [&](int p) { return cache16 + (size_t)p * cache_stride; }, nullptr, 0);
    if (pos < lo || pos >= hi) return;
    const uint8_t* row = s_rows[warp] + lane * S;
    uint32_t* rec = c.fixed + ((size_t)head * g.n_blocks + blk) * g.wpt * 32 + lane;
    uint32_t ub = 0, x[4], entry[3] = {0, 0, 0};
#pragma unroll 1
    for (int j = 0; j < nj; ++j) {
        const uint32_t bmj = rec[(g.e_words + j) * 32];
        lane_entry(j, ub, entry);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            lane_get8(row, j * 4 + q, x);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t len = s_len[lane_exp(x, i)];
                ub += bmj & (0x80000000u >> (q * 8 + i)) ? len : 0u;
            }
        }
    }
    const uint32_t nw = lane_entries(g, ub, entry, rec);
    c.off[(size_t)head * (g.max_seq + 1) + pos + 1] = nw;
}

// grid as k_kv_form_lanes: what k_kv_codes does.  The 32 records' words are one run of the arena: they are put together in shared
// memory and leave as whole lines.
template <int NJ>
__global__ void __launch_bounds__(32 * kLaneWarps(NJ)) k_kv_codes_lanes(KvGeom g, KvComp ck, KvComp cv, const uint16_t* __restrict__ k_cache,
                                                                        const uint16_t* __restrict__ v_cache, const uint16_t* __restrict__ src_k,
                                                                        const uint16_t* __restrict__ src_v, int row_stride, KvSpan sp) {
    constexpr int W = kLaneWarps(NJ), S = LaneRows<NJ>::kStride, RUN = NJ * 8 * 32;      // at most a byte a value
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_len[256];
    const int head = blockIdx.y % g.n_kv, kind = blockIdx.y / g.n_kv, nj = g.d / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t shift = span_shift(g, sp, blockIdx.z);
    const KvComp c = of_seq(kind ? cv : ck, 1, shift);
    const uint4* cache16 = reinterpret_cast<const uint4*>(of_seq(kind ? v_cache : k_cache, 1, shift)) + (size_t)head * nj * 4;
    const uint4* src16 = src_k ? reinterpret_cast<const uint4*>(kind ? src_v : src_k) + (size_t)head * nj * 4 : nullptr;
    const int lo = sp.start, hi = min(sp.start + sp.n_new, g.max_seq), blk = lo / 32 + (int)blockIdx.x * W + warp, pos = blk * 32 + lane;
    const size_t cache_stride = (size_t)g.n_kv * g.d / 8;
    pdl_wait();
    for (int i = tid; i < 256; i += 32 * W) s_len[i] = c.exp_to_rank[i] + 1u;
    __syncthreads();
    if (blk * 32 >= hi) return;
    uint8_t* rows = smem + warp * (32 * S + RUN * 4);
    uint32_t* run = reinterpret_cast<uint32_t*>(rows + 32 * S);
    const bool active = pos >= lo && pos < hi;
    const uint32_t* off = c.off + (size_t)head * (g.max_seq + 1);
    const int first = max(blk * 32, lo), end = min(blk * 32 + 32, hi);
    const uint32_t base = off[first], n_run = min(off[end] - base, (uint32_t)RUN);
    const uint32_t o0 = active ? off[pos] - base : 0u, nw = active ? min(off[pos + 1] - base - o0, (uint32_t)(NJ * 8)) : 0u;
    for (uint32_t i = lane; i < n_run; i += 32) run[i] = 0;
    LaneRows<NJ>::fetch(rows, nj, blk, lo, hi, lane, [&](int p) {
        return src16 ? src16 + ((size_t)(blockIdx.z % sp.n_seq) * sp.n_new + (p - lo)) * (row_stride / 8) : cache16 + (size_t)p * cache_stride;
    }, nullptr, 0);
    if (active && nw > 0) {
        const uint8_t* row = rows + lane * S;
        const uint32_t* rec = c.fixed + ((size_t)head * g.n_blocks + blk) * g.wpt * 32 + lane;
        const bool raw = rec[0] & kKvRawFlag;
        const uint32_t w_end = min(o0 + nw, n_run);
        uint32_t x[4], p = o0 * 32u + (raw ? 0u : 0xFFFFFFFFu);              // bit of the run: of the next byte, or of the last code's end
#pragma unroll 1
        for (int j = 0; j < nj; ++j) {
            const uint32_t bmj = rec[(g.e_words + j) * 32];
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                const uint32_t b8 = bmj << (8 * q);
                lane_get8(row, j * 4 + q, x);
                if (raw) {
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t e = (x[0] >> 7) & 0xFFu;
                        x[0] = (x[0] >> 16) | (x[1] << 16); x[1] = (x[1] >> 16) | (x[2] << 16); x[2] = (x[2] >> 16) | (x[3] << 16); x[3] >>= 16;
                        if (!(b8 & (0x80000000u >> i))) continue;
                        if (p >> 5 < w_end) atomicOr(&run[p >> 5], e << (24u - (p & 31u)));
                        p += 8u;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const bool keep = b8 & (0x80000000u >> i);
                        const uint32_t len = s_len[lane_exp(x, i)];
                        p += keep ? len : 0u;
                        if (keep && p >> 5 < w_end) atomicOr(&run[p >> 5], 0x80000000u >> (p & 31u));
                    }
                }
            }
        }
    }
    __syncwarp();
    uint32_t* to = c.arena + (size_t)head * g.arena_words + base;
    for (uint32_t i = lane; i < n_run; i += 32) to[i] = run[i];
}

static bool span_by_lanes(const KvGeom& g, const uint16_t* src_k, const uint16_t* src_v, int row_stride, const KvSpan& sp, int flags, bool codebook) {
    if (!(flags & CASS_KV_COMPRESSED)) return false;
    if (!codebook && ((((uintptr_t)src_k | (uintptr_t)src_v) & 15) || row_stride % 8)) return false;      // rows are copied 16 bytes at a time
    const int warps = ceil_div(sp.start % 32 + sp.n_new, 32) * g.n_kv * 2 * sp.n_layers * sp.n_seq;
    return warps >= kLaneMin;
}

template <int NJ, int T>
static int span_encode(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache, const uint16_t* src_k,
                       const uint16_t* src_v, int row_stride, const KvSpan& sp, int flags, bool codebook, DevState* st, cudaStream_t s) {
    const int z = sp.n_layers * sp.n_seq, blocks = ceil_div(sp.n_new, kSpanWarps);
    const dim3 heads(g.n_kv * 2, z), threads(32 * kSpanWarps);
    if (span_by_lanes(g, src_k, src_v, row_stride, sp, flags, codebook)) {
        constexpr int W = kLaneWarps(NJ), codes_smem = W * (32 * LaneRows<NJ>::kStride + NJ * 8 * 32 * 4);
        const dim3 grid(ceil_div(ceil_div(sp.start % 32 + sp.n_new, 32), W), g.n_kv * 2, z), lanes(32 * W);
        if (codebook) {
            CASS_PDL_LAUNCH((k_kv_form_lanes<NJ, T, true>), grid, lanes, 0, s, g, ck, cv, k_cache, v_cache, (const uint16_t*)nullptr,
                            (const uint16_t*)nullptr, 0, sp, flags);
            CASS_PDL_LAUNCH(k_kv_rank, dim3(2, z), dim3(256 * kRankLanes), 0, s, g, ck, cv, sp);
            if (g.mode == 1)
                CASS_PDL_LAUNCH(k_kv_lengths_lanes<NJ>, grid, lanes, 0, s, g, ck, cv, (const uint16_t*)k_cache, (const uint16_t*)v_cache, sp);
        } else {
            CASS_PDL_LAUNCH((k_kv_form_lanes<NJ, T, false>), grid, lanes, 0, s, g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, sp, flags);
        }
        CASS_PDL_LAUNCH(k_kv_scan, heads, dim3(1024), 0, s, g, ck, cv, sp, st);
        if (g.mode == 1) {
            CASS_ALLOW_SMEM(k_kv_codes_lanes<NJ>);
            CASS_PDL_LAUNCH(k_kv_codes_lanes<NJ>, grid, lanes, (size_t)codes_smem, s, g, ck, cv, (const uint16_t*)k_cache, (const uint16_t*)v_cache,
                            codebook ? (const uint16_t*)nullptr : src_k, codebook ? (const uint16_t*)nullptr : src_v, row_stride, sp);
        }
        return CASS_OK;
    }
    if (codebook) {
        // a CTA adds its counts to the histogram once: some 2000 CTAs over all heads, each with its share of the tokens
        int bx = ceil_div(2048, g.n_kv * 2 * z);
        if (bx < 4) bx = 4;
        if (bx > blocks) bx = blocks;
        if (bx > 0)
            CASS_PDL_LAUNCH((k_kv_form<NJ, T, true>), dim3(bx, g.n_kv * 2, z), threads, 0, s, g, ck, cv, k_cache, v_cache,
                            (const uint16_t*)nullptr, (const uint16_t*)nullptr, 0, sp, flags);
        CASS_PDL_LAUNCH(k_kv_rank, dim3(2, z), dim3(256 * kRankLanes), 0, s, g, ck, cv, sp);
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
