// Online KV encoder (Sec. 4.2: per-token magnitude pruning of K and V, mantissa truncation, unary exponent
// code; Sec. 5.1 encoder) for the rows of a decode step (kv_span.cu: for prompts): one warp formats one (token, KV head, K|V)
// record; records are appended to the compressed cache and, on request, the raw bf16 rows go to the target's cache.
// Bound: a chain of latencies (the projection's parts from L2, the threshold search, the code positions, the stores), which a
// decode step pays once a layer.  Everything that does not depend on something fetched is fetched together, the search starts
// near its answer and ends with the first threshold that fits, the code positions of two slices are scanned in one word, and
// every warp finds its own arena offset: 8.1 -> 5.2 us for one new token a sequence, 11.5 -> 6.5 us for five of four sequences.
#include "kv_record.cuh"

namespace cass {

constexpr int kKvWarps = 8;

// What the fused form of the encoder needs on top: the projection's fp32 split-K parts (the q, k, v features of every
// row), the rotary tables and the bf16 qkv rows to write.
struct RopeSrc {
    Partials pp;
    const float *cos_t, *sin_t;
    uint16_t* qkv;          // [rows][(n_q + 2 n_kv) d]
    int n_q;
};

// Sums of N elements of the parts, added in part order; the loads of a batch of parts travel together.
template <int N>
struct PartSums {
    static constexpr int B = N >= 8 ? 4 : 8;
    float v[N][B];
    __device__ __forceinline__ void fetch(const Partials& pp, const size_t (&off)[N], int s0) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float* p = pp.p + (size_t)(s0 + i) * pp.seg_stride;
#pragma unroll
            for (int j = 0; j < N; ++j) v[j][i] = s0 + i < pp.n_seg ? __ldcg(p + off[j]) : 0.f;
        }
    }
    __device__ __forceinline__ void add(const Partials& pp, int s0, float (&acc)[N]) const {
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (s0 + i < pp.n_seg) {
#pragma unroll
                for (int j = 0; j < N; ++j) acc[j] += v[j][i];
            }
    }
    __device__ __forceinline__ void finish(const Partials& pp, const size_t (&off)[N], float (&acc)[N]) {        // after fetch(.., 0)
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] = 0.f;
        add(pp, 0, acc);
        for (int s0 = B; s0 < pp.n_seg; s0 += B) {
            fetch(pp, off, s0);
            add(pp, s0, acc);
        }
    }
};

// grid (n_kv, 2, sequences of the call); a sequence's rows start at row blockIdx.z * n_new of the source.  A CTA's 8 warps take
// its tokens in rounds of 8.
// FUSED: the source is the qkv projection's split-K parts: this kernel adds them, rounds to bf16, rotates q and k
// (RoPE, Sec. 2.1) and writes the qkv rows; the K and V records are then formed from the rotated values as in the
// plain form.  Blocks with blockIdx.x >= n_kv rotate the query heads; head_dim is 32 NJ with NJ even, so that a
// rotation pair (c, c + d/2) sits in one lane.  Not FUSED: head_dim <= 32 NJ.
template <bool FUSED, int NJ, int T>
__global__ void __launch_bounds__(32 * kKvWarps) k_kv_append(KvGeom g, KvComp ck, KvComp cv, uint16_t* __restrict__ k_cache,
                                                             uint16_t* __restrict__ v_cache, const uint16_t* __restrict__ src_k,
                                                             const uint16_t* __restrict__ src_v, int row_stride, int start_pos_arg,
                                                             int use_inflight, int n_new, int flags, DevState* st, int seq0, RopeSrc rs) {
    constexpr int FW = NJ * 32 / (32 / (8 - T));
    __shared__ uint32_t s_rec[kKvWarps][3 + NJ + FW + 2];    // entry words | bitmap | fields | slice exponents
    __shared__ __align__(8) uint8_t s_fld[kKvWarps][NJ * 32 + 8];
    __shared__ uint32_t s_una[kKvWarps][64];                 // exponent stream: 1023 code bits, or 256 raw bytes
    __shared__ __align__(16) uint32_t s_nw[2][kKvWarps];
    __shared__ uint32_t s_len[256];                          // code length of an exponent: frozen with the codebook
    const int head = blockIdx.x, kind = blockIdx.y, seq = seq0 + blockIdx.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nj = FUSED ? NJ : g.d / 32;
    const bool coded = (flags & CASS_KV_COMPRESSED) != 0;
    auto code_lengths = [&]() {
        if (coded && g.mode == 1 && (!FUSED || head < g.n_kv)) s_len[threadIdx.x] = of_seq((kind ? cv : ck).exp_to_rank, seq, g.seq_stride)[threadIdx.x] + 1u;
    };
    // FUSED: the predecessor is a projection, and the codebook tables were written before that: read ahead of the wait, they cost
    // no time.  A stand-alone append may follow their writer (k_kv_rank ends a codebook of no tokens).  Cassandra-2 records have no
    // codes, and what is looked up for them is not used.
    if (FUSED) code_lengths();
    pdl_wait();
    pdl_early<1>();
    if (!FUSED) code_lengths();
    int start_pos = start_pos_arg;
    if (FUSED || start_pos < 0) start_pos = st->len[seq] + (use_inflight ? st->inflight[seq] : 0);
    if (FUSED && head >= g.n_kv) {
        // ---- query heads: q[r][h][j], q[r][h][j + d/2] rotated by the row's position ----
        constexpr int half = NJ * 16;
        const int qkv_dim = (rs.n_q + 2 * g.n_kv) * g.d;
        const int per_row = rs.n_q * half, n_items = n_new * per_row;
        const Partials& pp = rs.pp;
        for (int it = ((head - g.n_kv) * 2 + kind) * blockDim.x + threadIdx.x; it < n_items; it += (gridDim.x - g.n_kv) * 2 * blockDim.x) {
            const int i = it / per_row, e = it % per_row, hq = e / half, j = e % half;
            const size_t r = (size_t)blockIdx.z * n_new + i;
            const int ia = hq * g.d + j, ib = ia + half;
            const size_t offs[2] = {r * pp.row_stride + ia, r * pp.row_stride + ib};
            PartSums<2> parts;
            parts.fetch(pp, offs, 0);
            const size_t ti = (size_t)(start_pos + i) * half + j;
            const float c = __ldg(rs.cos_t + ti), sn = __ldg(rs.sin_t + ti);      // travel together with the parts
            float ab[2];
            parts.finish(pp, offs, ab);
            const float2 rot = rope_pair(round_bf16(ab[0]), round_bf16(ab[1]), c, sn);
            rs.qkv[r * qkv_dim + ia] = float_to_bf16_bits(rot.x);
            rs.qkv[r * qkv_dim + ib] = float_to_bf16_bits(rot.y);
        }
        return;
    }
    const KvComp& c0 = kind ? cv : ck;                       // sequence 0's; shifted to this sequence below
    const uint16_t* src = (kind ? src_v : src_k) + (size_t)blockIdx.z * n_new * row_stride;
    uint16_t* cache = of_seq(kind ? v_cache : k_cache, seq, g.seq_stride);
    uint32_t* off = of_seq(c0.off, seq, g.seq_stride) + (size_t)head * (g.max_seq + 1);
    uint32_t* arena = of_seq(c0.arena, seq, g.seq_stride) + (size_t)head * g.arena_words;
    uint32_t* fixed = of_seq(c0.fixed, seq, g.seq_stride) + (size_t)head * g.n_blocks * g.wpt * 32;
    uint32_t* rec = s_rec[warp];
    uint32_t* una = s_una[warp];
    const bool mx = g.mode == 2;
    uint32_t off_round = 0;                                  // arena offset of the round's first token (in warps that have a token)

    for (int base = 0, round = 0; base < n_new; base += kKvWarps, ++round) {
        const int i = base + warp, pos = start_pos + i;
        const bool active = i < n_new && pos < g.max_seq;
        uint32_t bits[NJ];
        if (active) {
            if (FUSED) {
                constexpr int half = NJ * 16, hj = NJ / 2;
                const int qkv_dim = (rs.n_q + 2 * g.n_kv) * g.d;
                const size_t r = (size_t)blockIdx.z * n_new + i;
                const int feat = (rs.n_q + (kind ? g.n_kv : 0) + head) * g.d + lane;
                size_t offs[NJ];
#pragma unroll
                for (int j = 0; j < NJ; ++j) offs[j] = r * rs.pp.row_stride + feat + 32 * j;
                PartSums<NJ> parts;
                parts.fetch(rs.pp, offs, 0);
                float rc[hj], rsn[hj], val[NJ];              // the position's rotation, fetched while the parts travel
#pragma unroll
                for (int j = 0; j < hj; ++j) {
                    const size_t ti = (size_t)pos * half + lane + 32 * j;
                    rc[j] = __ldg(rs.cos_t + ti);
                    rsn[j] = __ldg(rs.sin_t + ti);
                }
                if (base == 0 && coded) off_round = off[start_pos];
                parts.finish(rs.pp, offs, val);
#pragma unroll
                for (int j = 0; j < NJ; ++j) val[j] = round_bf16(val[j]);
                if (kind == 0) {                             // K: rotate the pairs (c, c + d/2), both held by this lane
#pragma unroll
                    for (int j = 0; j < hj; ++j) {
                        const float2 rot = rope_pair(val[j], val[j + hj], rc[j], rsn[j]);
                        val[j] = rot.x;
                        val[j + hj] = rot.y;
                    }
                }
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    bits[j] = float_to_bf16_bits(val[j]);
                    rs.qkv[r * qkv_dim + feat + 32 * j] = (uint16_t)bits[j];
                }
            } else {
                const uint16_t* row = src + (size_t)i * row_stride + (size_t)head * g.d;
#pragma unroll
                for (int j = 0; j < NJ; ++j) bits[j] = j < nj ? row[lane + 32 * j] : 0u;
                if (base == 0 && coded) off_round = off[start_pos];
            }
            if (flags & CASS_KV_BF16) {
                uint16_t* dst = cache + ((size_t)pos * g.n_kv + head) * g.d;
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    if (j < nj) dst[lane + 32 * j] = (uint16_t)bits[j];
            }
        }
        if (!coded) continue;
        if (round == 0) __syncthreads();                     // the code lengths are there
        uint32_t n_words = 0;
        if (active) {
            uint32_t bm[NJ];
            kv_select<NJ>(bits, nj, g.n_prune, lane, bm);
            una[lane] = 0;
            una[lane + 32] = 0;
            uint32_t len[NJ], kbase = 0, xw[2] = {0, 0};
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                len[j] = 0;
                if (j >= nj) break;
                const bool keep = (bm[j] >> lane) & 1u;
                uint32_t E;
                const uint32_t field = kv_field<T>(bits[j], keep, mx, E);
                xw[j / 4] |= E << (24 - 8 * (j % 4));
                if (keep) {
                    s_fld[warp][kbase + __popc(bm[j] & lanemask_lt())] = (uint8_t)field;
                    len[j] = s_len[(bits[j] >> 7) & 0xFFu];
                }
                if (lane == j) rec[g.e_words + j] = __brev(bm[j]);           // channel c at bit 31 - c%32
                kbase += __popc(bm[j]);
            }
            if (mx) {
                if (lane < g.x_words) rec[g.bm_words + g.f_words + lane] = lane ? xw[1] : xw[0];
            } else {
                uint32_t entry[3];
                n_words = kv_entries<NJ>(g, len, nj, entry);
                if (lane < g.e_words) rec[lane] = lane == 0 ? entry[0] : lane == 1 ? entry[1] : entry[2];
                __syncwarp();
                if (entry[0] & kKvRawFlag) {                 // the kept exponents as bytes
                    uint32_t k0 = 0;
#pragma unroll
                    for (int j = 0; j < NJ; ++j) {
                        if (j >= nj) break;
                        const uint32_t k = k0 + __popc(bm[j] & lanemask_lt());
                        if ((bm[j] >> lane) & 1u) atomicOr(&una[(k >> 2) & 63u], ((bits[j] >> 7) & 0xFFu) << (24 - 8 * (k & 3)));
                        k0 += __popc(bm[j]);
                    }
                } else {
                    kv_code_bits<NJ>(len, nj, lane, una);
                }
            }
            __syncwarp();
            kv_field_words<T>(g, s_fld[warp], rec + g.e_words + g.bm_words, lane);
            __syncwarp();
            uint32_t* blk = fixed + (size_t)(pos / 32) * g.wpt * 32 + (pos % 32);
            for (int w = lane; w < g.wpt; w += 32) blk[w * 32] = rec[w];
        }
        uint32_t* nws = s_nw[round & 1];
        if (lane == 0) nws[warp] = n_words;
        __syncthreads();
        // offsets in token order, from the offset behind the last token that is there; every warp adds up for itself
        const uint4 lo = *reinterpret_cast<const uint4*>(nws), hi = *reinterpret_cast<const uint4*>(nws + 4);
        const uint32_t nw8[kKvWarps] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        uint32_t o = off_round, mine = 0, nw = 0;
#pragma unroll
        for (int w = 0; w < kKvWarps; ++w) {
            const bool fits = o + nw8[w] <= (uint32_t)g.arena_words;     // arena full: keep offsets valid, drop the codes
            if (w == warp) { mine = o; nw = fits ? nw8[w] : 0u; if (!fits && active && lane == 0) atomicCAS(&st->status, 0, CASS_ERR_CAPACITY); }
            o += fits ? nw8[w] : 0u;
        }
        off_round = o;
        if (active) {
            if (lane == 0) off[pos + 1] = mine + nw;
            for (uint32_t w = lane; w < nw; w += 32) arena[mine + w] = una[w];
            __syncwarp();
        }
    }
}

int launch_kv_append(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache,
                     const uint16_t* src_k, const uint16_t* src_v, int row_stride, int start_pos, int use_inflight,
                     int n_new, int flags, DevState* st, int seq0, int n_seq, cudaStream_t s) {
    if (n_new <= 0 || n_seq <= 0) return CASS_OK;
    // two rounds of 8 tokens inside one CTA per head cost less than the span encoder's three launches; more do not
    if (n_new > 2 * kKvWarps && start_pos >= 0)
        return launch_kv_span(g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, start_pos, n_new, flags, st, seq0, n_seq, s);
    const dim3 grid(g.n_kv, 2, n_seq);
#define CASS_KV_APPEND(NJ, T)                                                                                                  \
    CASS_PDL_LAUNCH((k_kv_append<false, NJ, T>), grid, dim3(32 * kKvWarps), 0, s, g, ck, cv, k_cache, v_cache, src_k, src_v, row_stride, \
                    start_pos, use_inflight, n_new, flags, st, seq0, RopeSrc{})
    if (g.t != 4 && g.t != 0) return CASS_ERR_UNSUPPORTED;                    // sessions take no other truncation
    if (g.t == 4) {
        if (g.d <= 64) CASS_KV_APPEND(2, 4);
        else if (g.d <= 128) CASS_KV_APPEND(4, 4);
        else CASS_KV_APPEND(8, 4);
    } else {
        if (g.d <= 64) CASS_KV_APPEND(2, 0);
        else if (g.d <= 128) CASS_KV_APPEND(4, 0);
        else CASS_KV_APPEND(8, 0);
    }
#undef CASS_KV_APPEND
    return CASS_OK;
}

bool rope_kv_fusable(const KvGeom& g) { return g.d % 64 == 0; }

int launch_rope_kv_append(const KvGeom& g, const KvComp& ck, const KvComp& cv, uint16_t* k_cache, uint16_t* v_cache,
                          Partials pp, const float* cos_t, const float* sin_t, uint16_t* qkv, int n_q, int use_inflight,
                          int rps, int flags, DevState* st, int n_seq, cudaStream_t s) {
    if (rps <= 0 || n_seq <= 0) return CASS_OK;
    if (!rope_kv_fusable(g) || !pp.p) return CASS_ERR_UNSUPPORTED;
    if (g.t != 4 && g.t != 0) return CASS_ERR_UNSUPPORTED;
    // one rotation a thread in two CTAs (K's and V's) per 512 of them: with the rows of a verification taken one after another
    // by the CTAs of one row, the query heads were the longest chain of the kernel
    const int q_blocks = ceil_div(n_q * (g.d / 2) * rps, 512);
    const dim3 grid(g.n_kv + q_blocks, 2, n_seq);
    const RopeSrc rs{pp, cos_t, sin_t, qkv, n_q};
#define CASS_KV_APPEND(NJ, T)                                                                                                  \
    CASS_PDL_LAUNCH((k_kv_append<true, NJ, T>), grid, dim3(32 * kKvWarps), 0, s, g, ck, cv, k_cache, v_cache, (const uint16_t*)nullptr, \
                    (const uint16_t*)nullptr, 0, -1, use_inflight, rps, flags, st, 0, rs)
    if (g.t == 4) {
        if (g.d == 64) CASS_KV_APPEND(2, 4);
        else if (g.d == 128) CASS_KV_APPEND(4, 4);
        else if (g.d == 192) CASS_KV_APPEND(6, 4);
        else CASS_KV_APPEND(8, 4);
    } else {
        if (g.d == 64) CASS_KV_APPEND(2, 0);
        else if (g.d == 128) CASS_KV_APPEND(4, 0);
        else if (g.d == 192) CASS_KV_APPEND(6, 0);
        else CASS_KV_APPEND(8, 0);
    }
#undef CASS_KV_APPEND
    return CASS_OK;
}

}  // namespace cass
