// Offline weight encoder: Wanda-scored per-row pruning, mantissa truncation, unary exponent coding,
// superblock packing (Sec. 4.2, 5.1, 5.3).  Bit-exact counterpart of the CPU oracle's blob.
#include <type_traits>

#include "wblob.cuh"

namespace cass {

// Workspace carve-up (all offsets 256-byte aligned).
struct EncWs {
    uint32_t* keepbm;        // [n][k_pad/32], or (by lanes) [n_rb][k_pad/32][32]
    uint2* sb_size;          // [n_rb * n_seg]  of each superblock's rows: most kept values, most code words
    unsigned long long* hist;   // [256] exponents of the kept values; zeroed by the caller, as is abort_flag behind it
    uint32_t* abort_flag;    // [1]
    uint8_t* exp_to_rank;    // [256]
    uint32_t* blk_size;      // [n_rb * n_seg][16][32]  code bits | kept values << 16 of a superblock's rows in each 128 columns
    size_t zero_bytes;       // hist and abort_flag
    size_t bytes;
};

static EncWs carve(void* base, int n_pad, int k_pad, int n_seg) {
    EncWs w;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b, 256); return (char*)base + o; };
    w.hist = (unsigned long long*)take(256 * 8);
    w.abort_flag = (uint32_t*)take(256);
    w.zero_bytes = off;
    w.exp_to_rank = (uint8_t*)take(256);
    w.keepbm = (uint32_t*)take((size_t)n_pad * (k_pad / 32) * 4);
    w.sb_size = (uint2*)take((size_t)(n_pad / kRowsPerBlock) * n_seg * 8);
    w.blk_size = (uint32_t*)take((size_t)(n_pad / kRowsPerBlock) * n_seg * 16 * 32 * 4);
    w.bytes = off;
    return w;
}

struct EncGeom {
    int n, k, k_pad, n_pad, n_rb, n_seg, seg_cols, chunk_cols, p, t, n_prune;
    int mx;          // 1: Cassandra-2 (shared exponents), 0: Cassandra-1 (unary code)
    int lanes;       // sizes and packing by lanes: the bitmaps' words lie 32 rows side by side
};

static int make_geom(const cass_format* fmt, int rows, int cols, EncGeom* g) {
    if (!fmt || rows <= 0 || cols <= 0) return CASS_ERR_INVALID_ARG;
    if (fmt->mode != 1 && fmt->mode != 2) return CASS_ERR_UNSUPPORTED;
    g->mx = fmt->mode == 2;
    int p = fmt->w_prune_permille, t = fmt->w_trunc_bits;
    if (p < 0 || p > 999 || t < 0 || t > 7) return CASS_ERR_INVALID_ARG;
    int chunk = fmt->w_chunk_cols ? fmt->w_chunk_cols : 256;
    int seg = fmt->w_seg_cols ? fmt->w_seg_cols : 2048;
    if (chunk % 32 || chunk <= 0 || seg % chunk || seg > 2048 || seg <= 0) return CASS_ERR_INVALID_ARG;
    if (cols > (1 << 20)) return CASS_ERR_UNSUPPORTED;
    g->n = rows; g->k = cols; g->p = p; g->t = t;
    g->k_pad = ceil_div(cols, 32) * 32;
    g->chunk_cols = chunk;
    int seg_lim = ceil_div(g->k_pad, chunk) * chunk;
    g->seg_cols = seg < seg_lim ? seg : seg_lim;
    g->n_seg = ceil_div(g->k_pad, g->seg_cols);
    g->n_rb = ceil_div(rows, kRowsPerBlock);
    g->n_pad = g->n_rb * kRowsPerBlock;
    g->n_prune = (int)(((long long)cols * p) / 1000);
    // Sizes and packing by lanes or by warps, measured both ways (us by warps / by lanes).  By warps a superblock is a CTA's, up to one an SM with
    // 1024 threads, then two with 512; by lanes a CTA has 2 to 16 warps, a warp's chain is long and longer for rows off 16- and 4-byte boundaries.
    //   up to one superblock an SM: 256 x 2048 55.3 / 48.8, 1000 x 1000 38.9 / 38.9, 900 x 8190 79.8 / 73.8, but with odd columns 4700 x 1001 53.2 /
    //     57.4, 900 x 8191 79.8 / 86.0, and in short segments 3000 x 768 38.5 / 38.9, 3000 x 512 32.8 / 34.8, 1376 x 256 26.6 / 30.7
    //   up to two: 5000 x 512 45.0 / 38.9, 5000 x 515 55.3 / 53.2, 5200 x 641 59.4 / 57.3, 4800 x 1185 86 / 84, but 6000 x 128 36.9 / 38.9, 9000 x 257 49.2 / 53.2
    //   more: 9600 x 64 47.1 / 40.7, 9500 x 501 65.5 / 57.3, 20000 x 512 92.2 / 69.7, 12000 x 513 88.1 / 73.7, 32000 x 512 125 / 96
    // Rows that keep more have longer chains still: unpruned 1000 x 1024 38.9 / 49.2, 5000 x 512 43.0 / 49.2, 4096 x 4096 114.7 / 104.4, at 30 % 38.9 / 38.9,
    // 46 / 40 and 120.6 / 100.3.  There it takes as many blocks of 128 columns as it did when lanes shared them out worse.
    const long long n_sb = (long long)g->n_rb * g->n_seg, blocks = (long long)g->n_rb * ceil_div(g->k_pad, 128);
    const bool many = n_sb > 2 * kSms || (n_sb > kSms ? g->seg_cols > 512 || (g->seg_cols > 256 && cols % 8 == 0) : g->seg_cols > 768 && cols % 2 == 0);
    const bool chains = p >= 300 || (blocks >= (g->seg_cols > 512 ? 1400 : 2600) && (cols % 8 == 0 || n_sb > kSms * (g->seg_cols > 768 ? 1 : 2)));
    g->lanes = !g->mx && t == 4 && many && chains;
    return CASS_OK;
}

// Eight columns a lane: byte `lane` of 8 bitmap words that lanes j0 .. j0 + 7 hold, and the row's 8 values from p on (two a
// word), of which those without a bit may be anything.
__device__ __forceinline__ uint32_t row_byte(uint32_t bm_lane, int j0, int lane) {
    return (__shfl_sync(0xffffffffu, bm_lane, j0 + (lane >> 2)) >> (24 - 8 * (lane & 3))) & 0xFFu;
}
__device__ __forceinline__ void row_load8(const uint16_t* __restrict__ p, uint32_t byte, bool vec, uint32_t (&v)[4]) {
    v[0] = v[1] = v[2] = v[3] = 0;
    if (vec) {                                                             // rows of whole 16-byte groups: one load
        if (byte) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(p));
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = byte & (0x80u >> (2 * i)) ? __ldg(p + 2 * i) : 0u, hi = byte & (0x40u >> (2 * i)) ? __ldg(p + 2 * i + 1) : 0u;
        v[i] = lo | (hi << 16);
    }
}

// ---- E1: per-row selection of the kept set -------------------------------------------------------------
// Keys (score bits, column) are unique and scores are non-negative floats, whose integer order is the float order, so
// "prune the n_prune smallest keys" is the rule "lowest score first, lower column first among equals".  The smallest
// kept key is found in two steps: the top 16 bits of its score by a bitwise search that counts smaller ones two at a time
// (packed bf16 compare and add: the scores' upper halves order as bf16 numbers), then the handful of keys that share
// those bits are ranked against each other.  A score that is no number (a NaN weight, an infinite one times a norm of 0) counts
// as infinite in the first step, which compares numbers, and as its bits in the second: it ranks above all others, as in an
// integer order, and every row keeps the same count, on which the layout of the verification data rests.
// A row is read once, 8 columns a lane, and its scores' upper halves stay in registers, NV values a lane; the few values
// of which more is needed are read again.  Up to 2048 columns a warp holds a row and no barrier is needed (WIDE: false, four rows
// a CTA); a longer row is a CTA's, of as many warps as it takes.
// The search starts from the row before: the threshold lies within a quarter of it in an ordinary matrix, which leaves 7 rounds
// of 15 (and 6 meetings of the row's warps).
// Bound: the integer pipe, which starts a warp instruction every other cycle (packed compare and add: 1.4 cycles a value
// and round), and the latency of those meetings, hence 64 values a lane and not 128: 14 to 24 warps an SM and, at 14336
// columns, no idle eighth.  Loads have to be issued well ahead of their use, hence the clamped, unconditional ones.
// 4096 x 14336: 219 -> 136 us.
constexpr int kSelList = 512;
constexpr int kSelWarps = 16, kSelWarps64 = 14;                          // most warps a row: 128 and 64 values a lane

__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t v) {
    __nv_bfloat162 r;
    *reinterpret_cast<uint32_t*>(&r) = v;
    return r;
}

// LANES: the bitmap goes to 32 rows' words side by side (decided at run time it took a value's address two multiplications: 15000 x 512 72.7
// us instead of 70.7, 9000 x 641 at 60 % 64.5 instead of 62.5, 12000 x 513 by lanes 78.8 instead of 76.9).  Rows of several warps wait for one
// another instead, and are faster so (4096 x 14336 140.8 us, as a constant 142.9): WIDE asks the geometry.
template <int NV, bool WIDE, bool LANES>
__global__ void __launch_bounds__(!WIDE ? 128 : NV == 128 ? 32 * kSelWarps : 32 * kSelWarps64, !WIDE ? 6 : NV == 128 ? 1 : 2)
    k_select(const uint16_t* __restrict__ W, const float* __restrict__ act, EncGeom g, uint32_t* __restrict__ keepbm,
             unsigned long long* __restrict__ hist) {
    constexpr int ROWS = WIDE ? 1 : 4, NG = NV / 8, LG = NV == 128 ? 4 : 2, HW = NV >= 32 ? NV / 32 : 1;
    __shared__ unsigned int s_exp[256];
    __shared__ unsigned long long s_list[ROWS][kSelList], s_thr[ROWS];
    __shared__ uint2 s_cnt[2][kSelWarps];
    __shared__ uint32_t s_m[ROWS];
    const int NT = WIDE ? (int)blockDim.x : 128, WPR = WIDE ? NT / 32 : 1;     // threads; warps a row
    const int tid = threadIdx.x, lane = tid & 31, warp = WIDE ? tid >> 5 : 0, slot = WIDE ? 0 : tid >> 5;
    auto row_sync = [&]() {
        if (WIDE) __syncthreads();
        else __syncwarp();
    };
    int turn = 0;
    auto row_sum2 = [&](uint32_t v, uint32_t w) {                        // sums over the row's lanes; two buffers in turn, one barrier
        uint2 r = make_uint2(__reduce_add_sync(0xffffffffu, v), __reduce_add_sync(0xffffffffu, w));
        if (!WIDE) return r;
        turn ^= 1;
        if (lane == 0) s_cnt[turn][warp] = r;
        row_sync();
        r = lane < WPR ? s_cnt[turn][lane] : make_uint2(0u, 0u);
        return make_uint2(__reduce_add_sync(0xffffffffu, r.x), __reduce_add_sync(0xffffffffu, r.y));
    };
    auto row_sum = [&](uint32_t v) {
        v = __reduce_add_sync(0xffffffffu, v);
        if (!WIDE) return v;
        turn ^= 1;
        if (lane == 0) s_cnt[turn][warp].x = v;
        row_sync();
        return __reduce_add_sync(0xffffffffu, lane < WPR ? s_cnt[turn][lane].x : 0u);
    };
    uint32_t guess = 0;                                                  // the row before's threshold, upper half
    for (int i = tid; i < 256; i += NT) s_exp[i] = 0;
    pdl_wait();
    __syncthreads();
    const int step = (int)gridDim.x * ROWS, row_bytes = g.k_pad / 8;
    const bool vec = g.k % 8 == 0 && (((uintptr_t)W | (uintptr_t)act) & 15) == 0;
    const int k_last = vec ? g.k - 8 : 0;
    for (int row = (int)blockIdx.x * ROWS + slot; row < g.n; row += step) {     // the same row for all of its warps
        const uint16_t* wr = W + (size_t)row * g.k;
        auto score_of = [&](int c) { return __float_as_uint(__fmul_rn(bf16_bits_to_float(wr[c] & 0x7FFFu), act ? __ldg(act + c) : 1.0f)); };
        auto col_of = [&](int i) { return ((warp + (i / 8) * WPR) * 32 + lane) * 8 + (i & 7); };       // column of the lane's value i
        auto hit_value = [](int h, uint32_t b) { const int i = __ffs(b) - 1; return h * 32 + 2 * (i & 15) + (i >> 4); };
        uint32_t x[NV / 2];                                              // upper halves of scores 2 i (low) and 2 i + 1
        int later = 0;
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            // LG groups' loads at a time: all of them at once would not fit the registers
            if (q > 0 && q % LG == 0) {
                if (LG == 4) asm volatile("" : "+r"(later) : "r"(x[q * 4 - 1]), "r"(x[q * 4 - 5]), "r"(x[q * 4 - 9]), "r"(x[q * 4 - 13]));
                else asm volatile("" : "+r"(later) : "r"(x[q * 4 - 1]), "r"(x[q * 4 - 5]));
            }
            const int c = col_of(q * 8) + later;
            uint32_t w[4];
            float a[8];
            if (vec) {
                const int cc = min(c, k_last);
                const uint4 wv = __ldg(reinterpret_cast<const uint4*>(wr + cc));
                w[0] = wv.x; w[1] = wv.y; w[2] = wv.z; w[3] = wv.w;
#pragma unroll
                for (int i = 0; i < 8; ++i) a[i] = 1.0f;
                if (act) {
                    const float4 lo = __ldg(reinterpret_cast<const float4*>(act + cc)), hi = __ldg(reinterpret_cast<const float4*>(act + cc + 4));
                    a[0] = lo.x; a[1] = lo.y; a[2] = lo.z; a[3] = lo.w; a[4] = hi.x; a[5] = hi.y; a[6] = hi.z; a[7] = hi.w;
                }
            } else {
                uint32_t h[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int ci = min(c + i, g.k - 1);
                    h[i] = __ldg(wr + ci);
                    a[i] = act ? __ldg(act + ci) : 1.0f;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = h[2 * i] | (h[2 * i + 1] << 16);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t lo = __float_as_uint(__fmul_rn(__uint_as_float((w[i] << 16) & 0x7FFF0000u), a[2 * i]));
                const uint32_t hi = __float_as_uint(__fmul_rn(__uint_as_float(w[i] & 0x7FFF0000u), a[2 * i + 1]));
                x[q * 4 + i] = __vminu2(__byte_perm(lo, hi, 0x7632), 0x7F807F80u);
            }
            if (c + 8 > g.k) {                                           // beyond the row: NaNs, which are neither below nor above anything
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (c + 2 * i >= g.k) x[q * 4 + i] |= 0x7FFFu;
                    if (c + 2 * i + 1 >= g.k) x[q * 4 + i] |= 0x7FFF0000u;
                }
            }
        }
        uint32_t top = 0, below = 0;                                     // upper half of the smallest kept score; scores below it
        uint32_t hit[HW] = {};                                           // which of the lane's values share it
        unsigned long long thr = 0;                                      // smallest kept key
        if (g.n_prune > 0) {
            if (lane == 0 && warp == 0) s_m[slot] = 0;
            auto below_of = [&](uint32_t cand) {                         // the lane's scores whose upper half is less
                const __nv_bfloat162 c2 = as_bf162(cand | (cand << 16));
                __nv_bfloat162 n[2] = {as_bf162(0), as_bf162(0)};
#pragma unroll
                for (int i = 0; i < NV / 2; ++i) n[i & 1] = __hadd2(n[i & 1], __hlt2(as_bf162(x[i]), c2));     // at most 32 in a counter: exact
                const __nv_bfloat162 sum = __hadd2(n[0], n[1]);
                return (uint32_t)(int)(__low2float(sum) + __high2float(sum));
            };
            // the largest candidate with at most n_prune scores below it: in [top, hi).  Below the normal numbers the packed
            // compare may flush: those scores are one bin (0); beyond infinity there is none
            uint32_t hi = 0x7F81u;
            if (guess > 0x00A0u && guess < 0x7F60u) {
                const uint2 c = row_sum2(below_of(guess - 32u), below_of(guess + 32u));
                if (c.x <= (uint32_t)g.n_prune) { top = guess - 32u; below = c.x; } else { hi = guess - 32u; }
                if (c.y <= (uint32_t)g.n_prune) { top = guess + 32u; below = c.y; } else { hi = min(hi, guess + 32u); }
            }
#pragma unroll 1
            while (hi - top > 1u && hi > 0x0080u) {
                const uint32_t cand = max((top + hi) / 2u, 0x0080u), cnt = row_sum(below_of(cand));
                if (cnt <= (uint32_t)g.n_prune) { top = cand; below = cnt; } else { hi = cand; }
            }
            guess = top;
            // bit i (low half) or 16 + i of hit[h]: value 2 (16 h + i) or the one after it
            const __nv_bfloat162 top2 = as_bf162(top ? top | (top << 16) : 0x00800080u);
#pragma unroll
            for (int i = 0; i < NV / 2; ++i)
                hit[i / 16] |= (top ? __heq2_mask(as_bf162(x[i]), top2) : __hlt2_mask(as_bf162(x[i]), top2)) & (0x00010001u << (i % 16));
            row_sync();                                                  // s_m is zero
#pragma unroll
            for (int h = 0; h < HW; ++h)
                for (uint32_t b = hit[h]; b; b &= b - 1) {
                    const int c = col_of(hit_value(h, b));
                    const uint32_t at = atomicAdd(&s_m[slot], 1u);
                    if (at < (uint32_t)kSelList) s_list[slot][at] = ((unsigned long long)score_of(c) << 20) | (unsigned)c;
                }
            const uint32_t want = (uint32_t)g.n_prune - below;           // rank of the smallest kept key among them
            row_sync();                                                  // the list is complete
            const int m = (int)s_m[slot];
            if (m <= kSelList) {
                for (int i = warp * 32 + lane; i < m; i += 32 * WPR) {
                    const unsigned long long mine = s_list[slot][i];
                    uint32_t less = 0;
                    for (int j = 0; j < m; ++j) less += s_list[slot][j] < mine;
                    if (less == want) s_thr[slot] = mine;
                }
                row_sync();
                thr = s_thr[slot];
            } else {
                // many equal scores (a constant row): bit by bit over the keys that share the upper half
                for (int bit = 51; bit >= 0; --bit) {
                    const unsigned long long cand = thr | (1ull << bit);
                    uint32_t less = 0;
#pragma unroll
                    for (int h = 0; h < HW; ++h)
                        for (uint32_t b = hit[h]; b; b &= b - 1) {
                            const int c = col_of(hit_value(h, b));
                            less += (((unsigned long long)score_of(c) << 20) | (unsigned)c) < cand;
                        }
                    if (row_sum(less) <= want) thr = cand;
                }
            }
            row_sync();                                                  // the list and s_thr are free again
        }
        // kept: the values above the shared upper half, and those of the list from the threshold on
        const __nv_bfloat162 t2 = as_bf162(top ? top | (top << 16) : 0x007F007Fu);
        const bool lanes = WIDE ? g.lanes != 0 : LANES;
        const size_t row_at = lanes ? (size_t)(row / kRowsPerBlock) * kRowsPerBlock * row_bytes + (size_t)(row % kRowsPerBlock) * 4 : (size_t)row * row_bytes;
        uint8_t* keep_row = reinterpret_cast<uint8_t*>(keepbm) + row_at;
        const int word_at = lanes ? 4 * kRowsPerBlock : 4;               // bytes between a row's words
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            const int c = col_of(q * 8);
            uint32_t kb = 0;                                             // column c + i at bit 7 - i
            if (g.n_prune > 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) kb |= __hgt2_mask(as_bf162(x[q * 4 + i]), t2) & (0x00400080u >> (2 * i));
                kb = (kb | (kb >> 16)) & 0xFFu;
                for (uint32_t b = (hit[q / 4] >> (4 * (q & 3))) & 0x000F000Fu; b; b &= b - 1) {
                    const int i = hit_value(0, b);
                    if ((((unsigned long long)score_of(c + i) << 20) | (unsigned)(c + i)) >= thr) kb |= 0x80u >> i;
                }
            } else {
                kb = c + 8 <= g.k ? 0xFFu : c < g.k ? (0xFF00u >> (g.k - c)) & 0xFFu : 0u;
            }
            // byte of column c in its word: the first column at the most significant end
            if (c / 8 < row_bytes) keep_row[(size_t)(c / 32) * word_at + ((c / 8 & 3) ^ 3)] = (uint8_t)kb;
            if (!g.mx) {
                uint32_t v[4];
                row_load8(wr + c, kb, vec, v);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (kb & (0x80u >> i)) atomicAdd(&s_exp[((i & 1) ? v[i / 2] >> 23 : v[i / 2] >> 7) & 0xFF], 1u);
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < 256; e += NT)
        if (s_exp[e]) atomicAdd(&hist[e], (unsigned long long)s_exp[e]);
}

// ---- E3: codebook: rank exponents by (count desc, exponent asc) -----------------------------------------
__global__ void k_codebook(const unsigned long long* __restrict__ hist, uint8_t* __restrict__ rank_to_exp,
                           uint8_t* __restrict__ exp_to_rank) {
    __shared__ unsigned long long s[256];
    int e = threadIdx.x;
    pdl_wait();
    s[e] = hist[e];
    __syncthreads();
    unsigned long long mine = s[e];
    int rank = 0;
#pragma unroll 16
    for (int o = 0; o < 256; ++o) rank += (s[o] > mine) || (s[o] == mine && o < e);
    rank_to_exp[rank] = (uint8_t)e;
    exp_to_rank[e] = (uint8_t)rank;
}

// ---- E4: superblock sizes: the most kept values and code words among its 32 rows (one CTA a superblock, a warp a row) ----
__global__ void __launch_bounds__(1024) k_sizes(const uint16_t* __restrict__ W, EncGeom g, const uint32_t* __restrict__ keepbm,
                                                const uint8_t* __restrict__ exp_to_rank, uint2* __restrict__ sb_size) {
    __shared__ uint32_t s_len[512], s_kept[kRowsPerBlock], s_words[kRowsPerBlock];
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
    const int rb = blockIdx.x / g.n_seg, seg = blockIdx.x % g.n_seg, row = rb * kRowsPerBlock + r;
    pdl_wait();
    if (!g.mx && threadIdx.x < 512) s_len[threadIdx.x] = exp_to_rank[threadIdx.x & 255] + 1u;     // by sign and exponent
    __syncthreads();
    uint32_t kept = 0, bits = 0;
    if (row < g.n) {
        const int w0 = seg * (g.seg_cols / 32), nw = seg_cols_of(g.k_pad, g.seg_cols, seg) / 32;       // at most 64 words
        const uint32_t* bmr = keepbm + (size_t)row * (g.k_pad / 32) + w0;
        const uint32_t bm0 = lane < nw ? bmr[lane] : 0u, bm1 = lane + 32 < nw ? bmr[lane + 32] : 0u;
        kept = __reduce_add_sync(0xffffffffu, __popc(bm0) + __popc(bm1));
        if (!g.mx) {
            const uint16_t* wr = W + (size_t)row * g.k + w0 * 32;
            const bool vec = g.k % 8 == 0 && ((uintptr_t)W & 15) == 0;
            for (int j0 = 0; j0 < nw; j0 += 8) {                         // 256 columns, 8 a lane
                const uint32_t byte = row_byte(j0 < 32 ? bm0 : bm1, j0 & 31, lane);
                uint32_t v[4];
                row_load8(wr + (j0 * 32 + lane * 8), byte, vec, v);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (byte & (0x80u >> i)) bits += s_len[(i & 1) ? v[i / 2] >> 23 : (v[i / 2] >> 7) & 0x1FFu];
            }
            bits = __reduce_add_sync(0xffffffffu, bits);
        } else {
            bits = 8u * ((kept + kMxBlock - 1) / kMxBlock);              // one exponent byte per block of 32 kept values
        }
    }
    if (lane == 0) { s_kept[r] = kept; s_words[r] = (bits + 31u) / 32u; }
    __syncthreads();
    if (r == 0) {
        const uint32_t mk = __reduce_max_sync(0xffffffffu, s_kept[lane]), mw = __reduce_max_sync(0xffffffffu, s_words[lane]);
        if (lane == 0) sb_size[blockIdx.x] = make_uint2(mk, mw);
    }
}

// ---- E4 and E6 for unary blobs by lanes: a warp takes 32 rows of some columns, a lane a row -------------------------------
// The weights come 64 columns of 32 rows at a time into shared memory with whole-line reads (rows 16 bytes beyond a multiple of
// 32 apart: lanes read 16 bytes of their own rows without conflicts); from there on a lane works on its own row, with no scans,
// shuffles or ballots.  Blocks of 128 columns are the unit of sizes and splits: k_sizes_lanes leaves the code bits and kept values of
// every row and block, so that k_pack_lanes can start anywhere.
// Bound: memory latency and issue.  4096 x 14336, t = 4: packing 154 -> 83 us (111 M -> 45 M warp instructions), sizes 39 -> 33 (HBM alone: 18),
// the whole encoder 332 -> 258.  Bitmaps in rows (each lane's word in a line of its own): packing 125, sizes 52; tiles of 128 columns, three
// CTAs an SM for two and a bit rounds: 97 and 43; sizes without the next tile's loads under way 43.
constexpr int kBlkCols = 128, kSegBlks = 2048 / kBlkCols;
template <int N>
using Int = std::integral_constant<int, N>;
constexpr int kTileCols = 64, kTileWords = kTileCols / 32, kBlkTiles = kBlkCols / kTileCols;
constexpr int kLaneRow = 16 + 2 * kTileCols;             // bytes of a row: up to 7 values left of the tile before, and the tile's
constexpr int kLaneTile = 32 * kLaneRow;

// Columns c0 .. c0 + 63 of rows row0 .. row0 + 31 on their way to s + 16, in pieces of the size that the rows' boundaries allow (V); zero
// beyond the matrix.  ask: the loads, ahead of work on the tile before; put: into shared memory.
template <class V>
struct LanesTile {
    static constexpr int NB = (int)sizeof(V), LR = kTileCols * 2 / NB < 32 ? kTileCols * 2 / NB : 32, RS = 32 / LR;      // bytes, lanes a row, rows at a time
    static constexpr int NC = kTileCols * 2 / NB / LR, N = 32 / RS * NC;                                       // pieces a lane and row; in all
    V v[N];
    __device__ __forceinline__ void ask(const uint16_t* __restrict__ W, int n, int k, int row0, int c0, int lane) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int r = row0 + i / NC * RS + lane / LR, c = c0 + (lane % LR + i % NC * LR) * (NB / 2);
            v[i] = r < n && c < k ? __ldg(reinterpret_cast<const V*>(W + (size_t)r * k + c)) : V{};
        }
    }
    __device__ __forceinline__ void put(int lane, uint8_t* s) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            *reinterpret_cast<V*>(s + (i / NC * RS + lane / LR) * kLaneRow + 16 + (lane % LR + i % NC * LR) * NB) = v[i];
        __syncwarp();
    }
};
// Two bytes a load would take 64 registers: the values are read when they are put, 8 rows at a time.
template <>
struct LanesTile<uint16_t> {
    const uint16_t* from;
    int rows, cols, pitch;
    __device__ __forceinline__ void ask(const uint16_t* __restrict__ W, int n, int k, int row0, int c0, int lane) {
        from = W + (size_t)row0 * k + c0 + lane;
        rows = n - row0;
        cols = k - c0 - lane;
        pitch = k;
    }
    __device__ __forceinline__ void put(int lane, uint8_t* s) {
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 8) {
            uint16_t h[8][kTileWords];
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int i = 0; i < kTileWords; ++i) h[r][i] = r0 + r < rows && i * 32 < cols ? __ldg(from + (size_t)(r0 + r) * pitch + i * 32) : (uint16_t)0;
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int i = 0; i < kTileWords; ++i) *reinterpret_cast<uint16_t*>(s + (r0 + r) * kLaneRow + 16 + (i * 32 + lane) * 2) = h[r][i];
        }
        __syncwarp();
    }
};
// Sign and exponent of value i of eight (words of two, the lower column in the lower half): index of the rank table.
__device__ __forceinline__ uint32_t lanes_code(const uint32_t (&x)[4], int i) { return (i & 1) ? x[i / 2] >> 23 : (x[i / 2] >> 7) & 0x1FFu; }
__device__ __forceinline__ void lanes_get8(const uint8_t* p, uint32_t (&x)[4]) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}

// One CTA a superblock: its sizes, and those of its blocks.
constexpr int kSizeWarps = 8;
template <class V>
__global__ void __launch_bounds__(32 * kSizeWarps) k_sizes_lanes(const uint16_t* __restrict__ W, EncGeom g, const uint32_t* __restrict__ keepbm,
                                                                 const uint8_t* __restrict__ exp_to_rank, uint2* __restrict__ sb_size,
                                                                 uint32_t* __restrict__ blk_size) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint8_t s_rank[512];
    __shared__ uint32_t s_kept[32], s_bits[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sb = blockIdx.x, rb = sb / g.n_seg, seg = sb % g.n_seg, row0 = rb * kRowsPerBlock, row = row0 + lane;
    pdl_wait();
    const int nw = seg_cols_of(g.k_pad, g.seg_cols, seg) / 32, w0 = seg * (g.seg_cols / 32);
    uint8_t* s = smem + warp * kLaneTile;
    // the warp's tiles: of block `warp`, then of block warp + kSizeWarps
    LanesTile<V> t;
    uint32_t bm[kTileWords];
    auto ask = [&](int w) {
        t.ask(W, g.n, g.k, row0, (w0 + w) * 32, lane);
#pragma unroll
        for (int j = 0; j < kTileWords; ++j)
            bm[j] = row < g.n && w + j < nw ? __ldg(keepbm + ((size_t)rb * (g.k_pad / 32) + w0 + w + j) * 32 + lane) : 0u;
    };
    constexpr int kBlk = kBlkCols / 32;                                  // words of a block
    uint32_t bits = 0, kept = 0;
    int w = warp * kBlk;
    if (w < nw) ask(w);
    // (the rank table is filled and the sums are zero behind the first loads)
    for (int i = tid; i < 512; i += 32 * kSizeWarps) s_rank[i] = exp_to_rank[i & 255];
    if (tid < 32) s_kept[tid] = s_bits[tid] = 0;
    __syncthreads();
#pragma unroll 1
    while (w < nw) {
        t.put(lane, s);
        uint32_t now[kTileWords];
#pragma unroll
        for (int j = 0; j < kTileWords; ++j) now[j] = bm[j];
        const int b = w / kBlk;
        int next = w + kTileWords;
        const bool block_end = next % kBlk == 0 || next >= nw;
        if (block_end) next = (b + kSizeWarps) * kBlk;
        if (next < nw) ask(next);
#pragma unroll
        for (int j = 0; j < kTileWords; ++j) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t x[4];
                lanes_get8(s + lane * kLaneRow + 16 + j * 64 + q * 16, x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t rank = s_rank[lanes_code(x, i)];
                    bits += now[j] & (0x80000000u >> (q * 8 + i)) ? rank : 0u;
                }
            }
            kept += __popc(now[j]);
        }
        if (block_end) {
            bits += kept;                                                // a code is as long as its rank and one
            blk_size[((size_t)sb * kSegBlks + b) * 32 + lane] = bits | (kept << 16);
            atomicAdd(&s_kept[lane], kept);
            atomicAdd(&s_bits[lane], bits);
            bits = kept = 0;
        }
        __syncwarp();
        w = next;
    }
    __syncthreads();
    if (warp == 0) {
        const uint32_t mk = __reduce_max_sync(0xffffffffu, s_kept[lane]), mw = __reduce_max_sync(0xffffffffu, (s_bits[lane] + 31u) / 32u);
        if (lane == 0) sb_size[sb] = make_uint2(mk, mw);
    }
}

// One CTA a superblock of t = 4, NW warps of PER blocks each.  A block's kept values move to the front of the row, behind those
// that were left over (no branches: every value is stored, the next one takes its place if it is pruned), and leave as groups of 8: a field word,
// and code bits in one word that goes to the row's code stream.  A word that two warps fill is zero before either adds to it.
template <int NW, int PER, class V>
__global__ void __launch_bounds__(32 * NW) k_pack_lanes(const uint16_t* __restrict__ W, EncGeom g, const uint32_t* __restrict__ keepbm,
                                                        const uint8_t* __restrict__ exp_to_rank, const uint32_t* __restrict__ blk_size,
                                                        uint32_t* __restrict__ blob, const uint32_t* __restrict__ abort_flag) {
    constexpr uint32_t kMask = 0x80700000u;                              // sign and kept mantissa bits of a binary32
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint8_t s_rank[512];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    if (*abort_flag) return;
    const int sb = blockIdx.x, rb = sb / g.n_seg, seg = sb % g.n_seg, row0 = rb * kRowsPerBlock, row = row0 + lane;
    const uint4 dir = reinterpret_cast<const uint4*>(blob + kBlobDirOffset / 4)[sb];
    const int scols = seg_cols_of(g.k_pad, g.seg_cols, seg), n_ch = dir_n_ch(dir.w), nw = scols / 32, w0 = seg * (g.seg_cols / 32);
    const uint32_t E = (uint32_t)dir_chunk_elems(dir.w);
    const SbGeom sg = SbGeom::make(n_ch, scols, (int)dir.y, (int)dir.z);
    uint32_t* body = blob + (size_t)dir.x * 4 + lane;                    // this row's words, 32 apart
    uint32_t *tab = body + sg.tab, *bmo = body + sg.bm, *fl = body + sg.fl, *un = body + sg.un;
    for (int i = tid; i < 512; i += 32 * NW) s_rank[i] = exp_to_rank[i & 255];
    const uint32_t* bmr = keepbm + ((size_t)rb * (g.k_pad / 32) + w0) * 32 + lane;
    auto bm_word = [&](int j) { return row < g.n && j < nw ? __ldg(bmr + j * 32) : 0u; };
    // where the warp's blocks begin: kept values and code bits of the row before them
    const int b0 = warp * PER, b1 = b0 + PER;
    uint32_t k = 0, pos = 0, all_k = 0, all_bits = 0;
#pragma unroll
    for (int b = 0; b < NW * PER; ++b) {
        const uint32_t v = b * (kBlkCols / 32) < nw ? __ldg(blk_size + ((size_t)sb * kSegBlks + b) * 32 + lane) : 0u;
        all_k += v >> 16;
        all_bits += v & 0xFFFFu;
        k += b < b0 ? v >> 16 : 0u;
        pos += b < b0 ? v & 0xFFFFu : 0u;
    }
    // words that more than one warp may add to, and what a row leaves of its sections
    if ((int)(k >> 3) < sg.w_f) fl[(k >> 3) * 32] = 0;
    if ((int)(pos >> 5) < sg.w_u) un[(pos >> 5) * 32] = 0;
    if (warp == NW - 1) {
        for (int j = (int)(all_k >> 3); j < sg.w_f; ++j) fl[j * 32] = 0;
        for (int j = (int)(all_bits >> 5); j < sg.w_u; ++j) un[j * 32] = 0;
        for (int c = 0; c <= n_ch; ++c)                                  // the totals, and chunks the row has no value for
            if (c == n_ch) tab[c * 32] = (all_k << 20) | all_bits;
            else if ((uint32_t)c * E >= all_k) tab[c * 32] = ((uint32_t)scols << 20) | all_bits;
    }
    __syncthreads();
    uint8_t* tile = smem + warp * kLaneTile;
    uint8_t* mine = tile + lane * kLaneRow;
    uint32_t skip = k & 7u, acc = 0;                                     // of the first group: values of the warp before; the code word in hand
    uint32_t k_grp = k & ~7u, k_next = (k + E - 1) / E * E;              // first value of the next group; of the next chunk
    bool un_shared = true, fl_shared = true;
    auto flush = [&]() {                                                 // the code word in hand is full
        if (un_shared) atomicOr(&un[(pos >> 5) * 32], acc);
        else un[(pos >> 5) * 32] = acc;
        un_shared = false;
    };
    auto append = [&](uint32_t bits, uint32_t len) {                     // len <= 32 bits from the top of `bits`
        const uint32_t s = pos & 31u;
        acc |= bits >> s;
        if (s + len >= 32u) {
            flush();
            acc = s ? bits << (32u - s) : 0u;
        }
        pos += len;
    };
    auto group = [&](uint32_t at, uint32_t first, uint32_t last, auto whole_c) {      // values first .. last - 1 of the eight at `at`
        constexpr bool whole = decltype(whole_c)::value;
        uint32_t x[4], f = 0, off = 0, bits = 0;
        lanes_get8(mine + at, x);
        if (first == 0 && k_grp % E == 0) atomicOr(&tab[k_grp / E * 32], pos);          // a chunk's first code bit
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool in = whole || ((uint32_t)i >= first && (uint32_t)i < last);
            const uint32_t canon = ((i & 1) ? x[i / 2] : x[i / 2] << 16) & kMask, rank = s_rank[lanes_code(x, i)];
            f = __funnelshift_l(f, f, 4) | (in ? canon : 0u);
            off += in ? rank + 1u : 0u;
            bits |= in && off <= 32u ? 0x80000000u >> (off - 1u) : 0u;
        }
        f = __funnelshift_l(f, f, 4);
        if (!whole || fl_shared) atomicOr(&fl[(k_grp >> 3) * 32], f);
        else fl[(k_grp >> 3) * 32] = f;
        fl_shared = false;
        if (off <= 32u) {
            append(bits, off);
        } else {
#pragma unroll 1
            for (uint32_t i = first; i < last; ++i) {
                uint32_t len = s_rank[(uint32_t)(*reinterpret_cast<const uint16_t*>(mine + at + i * 2)) >> 7] + 1u;
                for (; len > 32u; len -= 32u) append(0u, 32u);
                append(0x80000000u >> (len - 1u), len);
            }
        }
        k_grp += 8;
    };
    const int w_end = min(nw, b1 * (kBlkCols / 32));
    LanesTile<V> t;
#pragma unroll 1
    for (int w = b0 * (kBlkCols / 32); w < w_end; w += kTileWords) {
        uint32_t bm[kTileWords];
#pragma unroll
        for (int j = 0; j < kTileWords; ++j) {
            bm[j] = bm_word(w + j);
            if (w + j < nw) bmo[(w + j) * 32] = bm[j];
        }
        t.ask(W, g.n, g.k, row0, (w0 + w) * 32, lane);      // (a tile ahead: 88 registers instead of 60, 83 -> 88 us)
        t.put(lane, tile);
        uint32_t to = k - k_grp;                                         // place in the list: behind the values left (or skipped)
        uint8_t* p = mine + to * 2;
#pragma unroll
        for (int j = 0; j < kTileWords; ++j) {
            const uint32_t pc = __popc(bm[j]);
            while (k_next < k + pc) {                                    // a chunk begins in these columns
                uint32_t m = bm[j];
                for (uint32_t i = k_next - k; i > 0; --i) m &= ~(0x80000000u >> __clz(m));
                tab[k_next / E * 32] = (uint32_t)((w + j) * 32 + __clz(m)) << 20;
                k_next += E;
            }
            k += pc;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t x[4];
                lanes_get8(mine + 16 + j * 64 + q * 16, x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    *reinterpret_cast<uint16_t*>(p) = (uint16_t)((i & 1) ? x[i / 2] >> 16 : x[i / 2]);
                    p += bm[j] & (0x80000000u >> (q * 8 + i)) ? 2 : 0;
                }
            }
        }
        __syncwarp();
        uint32_t at = 0;
        if (skip > 0 && k - k_grp >= 8u) {                               // the group that the warp before began
            group(0, skip, 8, std::false_type{});
            skip = 0;
            at = 16;
        }
        for (; skip == 0 && k - k_grp >= 8u; at += 16) group(at, 0, 8, std::true_type{});
        if (at > 0) *reinterpret_cast<uint4*>(mine) = *reinterpret_cast<const uint4*>(mine + at);      // up to 7 values left
        __syncwarp();
    }
    if (k > k_grp + skip) group(0, skip, k - k_grp, std::false_type{});
    if (pos & 31u) atomicOr(&un[(pos >> 5) * 32], acc);
}

// ---- E5: directory (exclusive scan of superblock sizes) and header -------------------------------------
__global__ void __launch_bounds__(1024) k_directory(EncGeom g, const uint2* __restrict__ sb_size, uint32_t* __restrict__ blob,
                                                    unsigned long long blob_cap, uint32_t* abort_flag, int32_t* d_status) {
    __shared__ unsigned long long s_sum[32];
    __shared__ unsigned int s_maxsb;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_sb = g.n_rb * g.n_seg;
    const unsigned long long body_off = align_up((size_t)kBlobDirOffset + 16ull * n_sb, 128);
    if (tid == 0) s_maxsb = 0;
    pdl_wait();
    __syncthreads();
    uint32_t* dir = blob + kBlobDirOffset / 4;
    unsigned long long carry = body_off;
    unsigned int max_bytes = 0;
    for (int base = 0; base < n_sb; base += 1024) {
        const int sb = base + tid;
        unsigned long long bytes = 0;
        uint32_t wf = 0, wu = 0, max_kept = 0;
        int n_ch = 0;
        if (sb < n_sb) {
            const uint32_t per = 32u / (8u - (uint32_t)g.t);
            const uint2 mx = sb_size[sb];
            max_kept = mx.x;
            wu = mx.y;
            wf = (max_kept + per - 1) / per;
            const int scols = seg_cols_of(g.k_pad, g.seg_cols, sb % g.n_seg);
            n_ch = ceil_div(scols, g.chunk_cols);
            bytes = (unsigned long long)SbGeom::make(n_ch, scols, (int)wf, (int)wu).total * 4ull;
            max_bytes = max(max_bytes, (unsigned int)bytes);
        }
        unsigned long long incl = bytes;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        unsigned long long below = lane < warp ? s_sum[lane] : 0ull, all = s_sum[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            below += __shfl_xor_sync(0xffffffffu, below, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (sb < n_sb) {
            const int e_chunk = g.mx ? mx_chunk_elems_for((int)max_kept, n_ch) : chunk_elems_for((int)max_kept, n_ch);
            reinterpret_cast<uint4*>(dir)[sb] = make_uint4((uint32_t)((carry + below + incl - bytes) / 16), wf, wu,
                                                           (uint32_t)n_ch | ((uint32_t)e_chunk << 8));
        }
        carry += all;
        __syncthreads();
    }
    atomicMax(&s_maxsb, max_bytes);
    __syncthreads();
    if (tid < kBlobHeaderBytes / 4) blob[tid] = 0;
    // the padding between directory and first body
    for (unsigned long long o = kBlobDirOffset + 16ull * n_sb + 4ull * tid; o < body_off; o += 4096) blob[o / 4] = 0;
    __syncthreads();
    if (tid == 0) {
        uint32_t* h = blob;
        h[H_MAGIC] = kBlobMagic; h[H_VERSION] = kBlobVersion; h[H_ROWS] = g.n; h[H_COLS] = g.k; h[H_P] = g.p; h[H_T] = g.t;
        h[H_SEG] = g.seg_cols; h[H_CHUNK] = g.chunk_cols; h[H_NSEG] = g.n_seg; h[H_NRB] = g.n_rb;
        h[H_KEPT] = g.k - g.n_prune; h[H_DIROFF] = kBlobDirOffset; h[H_BODYOFF] = (uint32_t)body_off;
        h[H_TOTLO] = (uint32_t)carry; h[H_TOTHI] = (uint32_t)(carry >> 32); h[H_MAXSB] = s_maxsb;
        h[H_MODE] = g.mx ? kBlobModeMx : kBlobModeUnary;
        if (carry > blob_cap) {
            *abort_flag = 1;
            if (d_status) *d_status = CASS_ERR_CAPACITY;
        }
    }
}

// ---- E6: pack one superblock (a CTA of 16 or 32 warps, two or one of the 32 rows a warp) -------------------------------------------
// A warp takes 256 columns of its row at a time, 8 a lane, and compacts the kept values into a ring in shared memory;
// whenever 256 are there it packs them, 8 consecutive ones a lane: a lane forms whole field words (t = 4: one; t = 0:
// two), and its code bits in one word of its own that is then shifted to where a warp scan of the lengths puts it, so
// that a lane needs two atomics for 8 codewords.
// The body is built in shared memory, its 32-word lines one word apart (a row's words would share a bank otherwise), and
// leaves as contiguous stores; one that does not fit (code words of 5 bits a value and more at p = 0) is built in place.
// Cassandra-2 (MX): four lanes hold a block of 32 values, whose largest exponent is their shared one.
// T: truncated bits, or -1: any (from the geometry).
// Bound: instruction issue.  Two atomics a kept value on global memory, as before, took 0.6 ms of a 4096 x 14336 matrix.
constexpr int kPackRing = 512;
constexpr int kPackBodyBytes = 92 * 1024;
constexpr int pack_ring_bytes(int threads) { return threads / 32 * kPackRing * 2; }

// NT = 512: two CTAs an SM, one's stores overlap the other's packing.  NT = 1024: a row a warp, where an SM has one superblock
// at most and the time is that of a warp's rows (300 x 1500: 26.6 -> 18.4 us).
template <bool MX, int T, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_pack(const uint16_t* __restrict__ W, EncGeom g, const uint32_t* __restrict__ keepbm,
                                                          const uint8_t* __restrict__ exp_to_rank, uint32_t* __restrict__ blob,
                                                          const uint32_t* __restrict__ abort_flag) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_len[MX ? 1 : 512];                               // code length by sign and exponent
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    if (*abort_flag) return;
    const int sb = blockIdx.x, rb = sb / g.n_seg, seg = sb % g.n_seg;
    const uint4 dir = reinterpret_cast<const uint4*>(blob + kBlobDirOffset / 4)[sb];
    const int scols = seg_cols_of(g.k_pad, g.seg_cols, seg);
    const int n_ch = dir_n_ch(dir.w);
    const uint32_t E = (uint32_t)dir_chunk_elems(dir.w);
    const SbGeom sg = SbGeom::make(n_ch, scols, (int)dir.y, (int)dir.z);
    uint32_t* gbody = blob + (size_t)dir.x * 4;
    uint16_t* ring = reinterpret_cast<uint16_t*>(smem) + warp * kPackRing;
    const bool staged = sg.total / 32 * 33 * 4 <= kPackBodyBytes;
    const int ls = staged ? 33 : 32;                                       // words between two lines of the body
    uint32_t* body = staged ? reinterpret_cast<uint32_t*>(smem + pack_ring_bytes(NT)) : gbody;
    if (!MX && tid < 512) s_len[tid] = exp_to_rank[tid & 255] + 1u;
    for (int i = tid; i < sg.total / 32 * ls; i += NT) body[i] = 0;
    __syncthreads();

    const int t = T >= 0 ? T : g.t, F = 8 - t;
    const uint32_t per = 32u / (uint32_t)F;
    const int w0 = seg * (g.seg_cols / 32);
    const bool vec = g.k % 8 == 0 && ((uintptr_t)W & 15) == 0;
#pragma unroll 1
    for (int r = warp; r < kRowsPerBlock; r += NT / 32) {
        const int row = rb * kRowsPerBlock + r;
        const uint16_t* wr = W + (size_t)row * g.k + w0 * 32;
        const uint32_t* bmr = keepbm + (size_t)row * (g.k_pad / 32) + w0;
        uint32_t* tab_r = body + sg.tab / 32 * ls + r;
        uint32_t* bm_r = body + sg.bm / 32 * ls + r;
        uint32_t* fl_r = body + sg.fl / 32 * ls + r;
        uint32_t* un_r = body + sg.un / 32 * ls + r;
        uint32_t ub = 0, k_cnt = 0, k_done = 0, next_ch = 0, done_ch = 0;  // code bits packed; values compacted; packed; chunks whose column, whose entry is written

        const int n_blk = row < g.n ? ceil_div(sg.bm_words, 8) : 0;
        uint32_t bm8 = 0, v[4], byte = 0;
        auto fetch = [&](int blk) {                                        // bitmap words and values of the blk-th 256 columns
            bm8 = lane < 8 && blk * 8 + lane < sg.bm_words ? __ldg(bmr + blk * 8 + lane) : 0u;
            byte = row_byte(bm8, 0, lane);
            row_load8(wr + blk * 256 + lane * 8, byte, vec, v);
        };
        if (n_blk > 0) fetch(0);
#pragma unroll 1
        for (int blk = 0; blk < n_blk || k_cnt > k_done; ++blk) {
            if (blk < n_blk) {
                if (lane < 8 && blk * 8 + lane < sg.bm_words) bm_r[(blk * 8 + lane) * ls] = bm8;
                const uint32_t cnt = __popc(byte);
                uint32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                uint32_t k = k_cnt + incl - cnt;                           // index of the lane's first kept value
                k_cnt += __shfl_sync(0xffffffffu, incl, 31);
                while (next_ch < (uint32_t)n_ch && next_ch * E < k_cnt) {  // a chunk starts in these columns: where
                    const uint32_t nth = next_ch * E - k;                  // of the lane's kept values
                    if (nth < cnt) {
                        uint32_t b = byte;
                        for (uint32_t i = 0; i < nth; ++i) b &= ~(0x80000000u >> __clz(b));
                        tab_r[next_ch * ls] = (uint32_t)(blk * 256 + lane * 8 + __clz(b) - 24) << 20;
                    }
                    ++next_ch;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (byte & (0x80u >> i)) {
                        ring[k & (kPackRing - 1)] = (uint16_t)((i & 1) ? v[i / 2] >> 16 : v[i / 2]);
                        ++k;
                    }
                if (blk + 1 < n_blk) fetch(blk + 1);                       // the next columns travel while these are packed
                __syncwarp();
                if (k_cnt - k_done < 256u && blk + 1 < n_blk) continue;
            }
            // ---- pack the values k_done .. k_done + n - 1, 8 a lane ----
            const uint32_t n = min(256u, k_cnt - k_done);
            const uint32_t kk = k_done + (uint32_t)lane * 8u;
            const uint4 raw = *reinterpret_cast<const uint4*>(ring + (kk & (kPackRing - 1)));
            const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
            const int nv = min(8, max(0, (int)n - lane * 8));
            uint32_t e[8], entry = 0;                                      // values; the lane's first code bit or 8 x its block
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = (i & 1) ? rw[i / 2] >> 16 : rw[i / 2] & 0xFFFFu;
            if (MX) {
                uint32_t e_blk = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) if (i < nv) e_blk = max(e_blk, (e[i] >> 7) & 0xFFu);
                e_blk = max(e_blk, __shfl_xor_sync(0xffffffffu, e_blk, 1));
                e_blk = max(e_blk, __shfl_xor_sync(0xffffffffu, e_blk, 2));
                const uint32_t b = kk / kMxBlock;
                if ((lane & 3) == 0 && nv > 0) atomicOr(&un_r[(b / 4) * ls], e_blk << (24 - 8 * (b % 4)));
#pragma unroll
                for (int i = 0; i < 8; ++i) {                              // field: sign, magnitude in the block's unit
                    const uint32_t ex = (e[i] >> 7) & 0xFFu, shift = 1u + e_blk - ex;
                    const uint32_t m7 = (shift < 8u && ex > 0u && e_blk >= 7u) ? (0x80u | (e[i] & 0x7Fu)) >> shift : 0u;
                    e[i] = ((e[i] >> 15) << (7 - t)) | (m7 >> t);
                }
                entry = 8u * b;
            } else {
                uint32_t off = 0, bits = 0;                                // the lane's codewords from bit 31 of a word of its own
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i < nv) {
                        off += s_len[e[i] >> 7];
                        bits |= off <= 32u ? 0x80000000u >> (off - 1u) : 0u;
                    }
                uint32_t incl = off;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                uint32_t pos = ub + incl - off;
                entry = pos;
                if (off <= 32u) {
                    const uint32_t hi = bits >> (pos & 31u), lo = __funnelshift_r(0u, bits, pos & 31u);
                    if (hi) atomicOr(&un_r[(pos >> 5) * ls], hi);
                    if (lo) atomicOr(&un_r[((pos >> 5) + 1) * ls], lo);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (i < nv) {
                            pos += s_len[e[i] >> 7];
                            atomicOr(&un_r[((pos - 1) >> 5) * ls], 0x80000000u >> ((pos - 1) & 31));
                        }
                }
                ub += __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
                for (int i = 0; i < 8; ++i) e[i] = ((e[i] >> 15) << (7 - t)) | ((e[i] & 0x7Fu) >> t);
            }
            while (done_ch < (uint32_t)n_ch && done_ch * E < k_done + n) { // chunks that start here (a multiple of 8: some lane's first value)
                if (kk == done_ch * E) tab_r[done_ch * ls] |= entry;
                ++done_ch;
            }
            if (nv > 0) {
                if (per == 8 || per == 4) {                                // the lane's own words
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        uint32_t acc = 0;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int j = per == 8 ? h + i : i;
                            if (h + i < nv) acc |= MX ? e[h + i] << (32 - F * (j + 1)) : field_bits_in_word(e[h + i], j, t);
                        }
                        if (h < nv) fl_r[((kk + h) / per) * ls] |= acc;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (i < nv) {
                            const uint32_t k = kk + i;
                            atomicOr(&fl_r[(k / per) * ls], MX ? e[i] << (32 - F * (k % per + 1)) : field_bits_in_word(e[i], k % per, t));
                        }
                }
            }
            k_done += n;
            __syncwarp();
        }
        // chunks the row has no value for, and the totals
        const uint32_t end = MX ? 8u * ((k_cnt + kMxBlock - 1) / kMxBlock) : ub;
        for (int c = lane; c <= n_ch; c += 32) {
            if (c == n_ch) tab_r[c * ls] = (k_cnt << 20) | end;
            else if ((uint32_t)c * E >= k_cnt) tab_r[c * ls] = ((uint32_t)scols << 20) | end;
        }
    }
    if (!staged) return;
    __syncthreads();
    for (int i = tid; i < sg.total; i += NT) gbody[i] = body[i / 32 * 33 + i % 32];
}

// CTAs of k_select: as many as run at once (each takes rows in turn, so that the counts of kept exponents reach global
// memory once per CTA).
template <int NV, bool WIDE, bool LANES>
static int launch_select_as(const uint16_t* W, const float* act, const EncGeom& g, const EncWs& ws, cudaStream_t stream) {
    const int warps = WIDE ? ceil_div(g.k, 32 * NV) : 4, rows = WIDE ? 1 : 4;
    int per_sm = 1;
    CASS_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (k_select<NV, WIDE, LANES>), 32 * warps, 0));
    const int most = kSms * (per_sm < 1 ? 1 : per_sm), need = ceil_div(g.n, rows);
    CASS_PDL_LAUNCH((k_select<NV, WIDE, LANES>), dim3(need < most ? need : most), dim3(32 * warps), 0, stream, W, act, g, ws.keepbm, ws.hist);
    return CASS_OK;
}
// One warp a row while its lanes' registers hold it (64 values a lane), then as many warps as it takes; 128 values a lane where
// 14 warps of 64 do not reach.
template <bool LANES>
static int launch_select(const uint16_t* W, const float* act, const EncGeom& g, const EncWs& ws, cudaStream_t stream) {
    const int k = g.k;
    if (k <= 512) return launch_select_as<16, false, LANES>(W, act, g, ws, stream);
    if (k <= 1024) return launch_select_as<32, false, LANES>(W, act, g, ws, stream);
    if (k <= 2048) return launch_select_as<64, false, LANES>(W, act, g, ws, stream);
    if (k <= 2048 * kSelWarps64) return launch_select_as<64, true, false>(W, act, g, ws, stream);
    return launch_select_as<128, true, false>(W, act, g, ws, stream);
}

// ---- test hook: zero-padded reconstruction of the whole blob ---------------------------------------------
__global__ void k_decode(const uint32_t* __restrict__ blob, uint16_t* __restrict__ out) {
    const uint32_t* h = blob;
    const int n = h[H_ROWS], k = h[H_COLS], t = h[H_T], seg_cols = h[H_SEG], chunk_cols = h[H_CHUNK], n_seg = h[H_NSEG];
    const int k_pad = ceil_div(k, 32) * 32;
    const int sb = blockIdx.x, rb = sb / n_seg, seg = sb % n_seg;
    const uint32_t* dir = blob + kBlobDirOffset / 4 + sb * 4;
    const SbGeom sg = SbGeom::make(dir_n_ch(dir[3]), seg_cols_of(k_pad, seg_cols, seg), (int)dir[1], (int)dir[2]);
    const int chunk_elems = dir_chunk_elems(dir[3]);
    const uint32_t* body = blob + (size_t)dir[0] * 4;
    const uint8_t* cb = reinterpret_cast<const uint8_t*>(blob) + kBlobHeaderBytes;
    for (int item = threadIdx.x; item < sg.n_ch * 32; item += blockDim.x) {
        int ch = item >> 5, r = item & 31, row = rb * kRowsPerBlock + r;
        if (row >= n) continue;
        auto emit = [&](int col, uint16_t bits) {
            int c = seg * seg_cols + col;
            if (c < k) out[(size_t)row * k + c] = bits;
        };
        if (h[H_MODE] == kBlobModeMx) decode_chunk_generic_mx(body, sg, chunk_elems, ch, r, t, emit);
        else decode_chunk_generic(body, sg, chunk_elems, ch, r, t, cb, emit);
    }
}

// ---- content accounting: sum of the codeword lengths recorded in the chunk tables ------------------------
__global__ void k_code_bits(const uint32_t* __restrict__ blob, unsigned long long* __restrict__ out) {
    const uint32_t* h = blob;
    const int k = h[H_COLS], seg_cols = h[H_SEG], n_seg = h[H_NSEG];
    const int k_pad = ceil_div(k, 32) * 32;
    const int sb = blockIdx.x, seg = sb % n_seg;
    const uint32_t* dir = blob + kBlobDirOffset / 4 + sb * 4;
    const SbGeom sg = SbGeom::make(dir_n_ch(dir[3]), seg_cols_of(k_pad, seg_cols, seg), (int)dir[1], (int)dir[2]);
    const uint32_t* body = blob + (size_t)dir[0] * 4;
    unsigned int bits = body[sg.tab + sg.n_ch * 32 + threadIdx.x] & 0xFFFFFu;       // segment total of row threadIdx.x
    bits = __reduce_add_sync(0xffffffffu, bits);
    if (threadIdx.x == 0) atomicAdd(out, (unsigned long long)bits);
}

}  // namespace cass

using namespace cass;

extern "C" int cass_weight_blob_stats(const void* blob, const cass_blob_info* bi, void* d_scratch, cass_blob_stats* st,
                                      void* stream_) {
    if (!blob || !bi || !d_scratch || !st || ((uintptr_t)d_scratch & 7)) return CASS_ERR_INVALID_ARG;
    cudaStream_t stream = (cudaStream_t)stream_;
    CASS_CUDA_CHECK(cudaMemsetAsync(d_scratch, 0, 8, stream));
    k_code_bits<<<bi->n_rowblocks * bi->n_seg, 32, 0, stream>>>((const uint32_t*)blob, (unsigned long long*)d_scratch);
    CASS_LAUNCH_CHECK();
    unsigned long long code = 0;
    CASS_CUDA_CHECK(cudaMemcpyAsync(&code, d_scratch, 8, cudaMemcpyDeviceToHost, stream));
    CASS_CUDA_CHECK(cudaStreamSynchronize(stream));
    st->bitmap_bits = (uint64_t)bi->rows * bi->cols;
    st->field_bits = (uint64_t)bi->rows * bi->kept_per_row * (8 - bi->trunc_bits);
    st->code_bits = code;
    st->total_bits = bi->total_bytes * 8;
    return CASS_OK;
}

extern "C" int cass_encoded_weight_bytes(const cass_format* fmt, int rows, int cols, size_t* h_blob_bound,
                                         size_t* h_workspace_bytes) {
    EncGeom g;
    int rc = make_geom(fmt, rows, cols, &g);
    if (rc) return rc;
    const int F = 8 - g.t, per = 32 / F;
    size_t n_sb = (size_t)g.n_rb * g.n_seg;
    int n_ch = ceil_div(g.seg_cols, g.chunk_cols);
    // per superblock: table + bitmap + fields (kept values + one padding word per chunk) + codes at a
    // mean of 8 bits per kept value (+1 word of row padding)
    size_t kept_seg = (size_t)g.seg_cols;
    size_t words_row = (size_t)(n_ch + 1) + g.seg_cols / 32 + (kept_seg + per - 1) / per + n_ch + kept_seg * 8 / 32 + 1;
    size_t sb_bytes = words_row * 32 * 4;
    if (h_blob_bound) *h_blob_bound = align_up((size_t)kBlobDirOffset + 16 * n_sb, 128) + n_sb * sb_bytes;
    if (h_workspace_bytes) *h_workspace_bytes = carve(nullptr, g.n_pad, g.k_pad, g.n_seg).bytes;
    return CASS_OK;
}

extern "C" int cass_encode_weights(const cass_format* fmt, const void* W_bf16, const float* act_norm, int rows,
                                   int cols, void* blob, size_t blob_cap, void* workspace, size_t workspace_bytes,
                                   int32_t* d_status, void* stream_) {
    EncGeom g;
    int rc = make_geom(fmt, rows, cols, &g);
    if (rc) return rc;
    if (!W_bf16 || !blob || !workspace || ((uintptr_t)blob & 127)) return CASS_ERR_INVALID_ARG;
    EncWs ws = carve(workspace, g.n_pad, g.k_pad, g.n_seg);
    if (workspace_bytes < ws.bytes) return CASS_ERR_CAPACITY;
    size_t n_sb = (size_t)g.n_rb * g.n_seg;
    size_t body_off = align_up((size_t)kBlobDirOffset + 16 * n_sb, 128);
    if (blob_cap < body_off) return CASS_ERR_CAPACITY;
    if ((size_t)g.k * 4 > 200 * 1024) return CASS_ERR_UNSUPPORTED;
    cudaStream_t stream = (cudaStream_t)stream_;
    const uint16_t* W = (const uint16_t*)W_bf16;
    uint32_t* b32 = (uint32_t*)blob;

    CASS_CUDA_CHECK(cudaMemsetAsync(workspace, 0, ws.zero_bytes, stream));
    rc = g.lanes ? launch_select<true>(W, act_norm, g, ws, stream) : launch_select<false>(W, act_norm, g, ws, stream);
    if (rc) return rc;
    if (g.mx) {
        CASS_CUDA_CHECK(cudaMemsetAsync((uint8_t*)blob + kBlobHeaderBytes, 0, kBlobCodebookBytes, stream));    // no codebook
    } else {
        CASS_PDL_LAUNCH(k_codebook, dim3(1), dim3(256), 0, stream, (const unsigned long long*)ws.hist, (uint8_t*)blob + kBlobHeaderBytes,
                        ws.exp_to_rank);
    }
    // rows on 16-byte, 4-byte or 2-byte boundaries
    const uintptr_t ends = (uintptr_t)W | ((uintptr_t)g.k * 2);
    if (g.lanes) {
        auto sizes = [&](auto piece) -> int {
            using V = decltype(piece);
            CASS_ALLOW_SMEM(k_sizes_lanes<V>);
            CASS_PDL_LAUNCH(k_sizes_lanes<V>, dim3((unsigned)n_sb), dim3(32 * kSizeWarps), (size_t)(kSizeWarps * kLaneTile), stream, W, g,
                            (const uint32_t*)ws.keepbm, (const uint8_t*)ws.exp_to_rank, ws.sb_size, ws.blk_size);
            return CASS_OK;
        };
        rc = ends % 16 == 0 ? sizes(uint4{}) : ends % 4 == 0 ? sizes(uint32_t{}) : sizes(uint16_t{});
        if (rc) return rc;
    } else {
        CASS_PDL_LAUNCH(k_sizes, dim3((unsigned)n_sb), dim3(1024), 0, stream, W, g, (const uint32_t*)ws.keepbm, (const uint8_t*)ws.exp_to_rank,
                        ws.sb_size);
    }
    CASS_PDL_LAUNCH(k_directory, dim3(1), dim3(1024), 0, stream, g, (const uint2*)ws.sb_size, b32, (unsigned long long)blob_cap,
                    ws.abort_flag, d_status);
    auto launch_pack = [&](auto pack, int threads) -> int {
        const int smem = pack_ring_bytes(threads) + kPackBodyBytes;
        CASS_CUDA_CHECK(cudaFuncSetAttribute(pack, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        CASS_PDL_LAUNCH(pack, dim3((unsigned)n_sb), dim3((unsigned)threads), (size_t)smem, stream, W, g, (const uint32_t*)ws.keepbm,
                        (const uint8_t*)ws.exp_to_rank, b32, (const uint32_t*)ws.abort_flag);
        return CASS_OK;
    };
    if (g.lanes) {
        // warps a superblock: some 3000 of them in all, no more than it has blocks.  The blocks that it has are what they share: of the 16 of
        // 2048 columns each, half or more of the warps of a shorter segment had none (45000 x 256 112.6 -> 104.4 us, 30000 x 301 110.6 -> 99.0,
        // 32000 x 512 108.6 -> 96.3, 20000 x 640 106.5 -> 92.1, 12000 x 520 65.6 -> 61.2)
        const int blks = ceil_div(g.seg_cols, kBlkCols);
        auto pack_as = [&](auto warps, auto blocks, auto piece) -> int {
            constexpr int NW = decltype(warps)::value, PER = decltype(blocks)::value;
            using V = decltype(piece);
            CASS_ALLOW_SMEM(k_pack_lanes<NW, PER, V>);
            CASS_PDL_LAUNCH((k_pack_lanes<NW, PER, V>), dim3((unsigned)n_sb), dim3(32 * NW), (size_t)(NW * kLaneTile), stream, W, g, (const uint32_t*)ws.keepbm,
                            (const uint8_t*)ws.exp_to_rank, (const uint32_t*)ws.blk_size, b32, (const uint32_t*)ws.abort_flag);
            return CASS_OK;
        };
        auto pack = [&](auto piece) {
            if (blks <= 2) return pack_as(Int<2>{}, Int<1>{}, piece);
            if (blks <= 4) return pack_as(Int<4>{}, Int<1>{}, piece);
            if (n_sb >= 750) return blks <= 8 ? pack_as(Int<4>{}, Int<2>{}, piece) : blks <= 12 ? pack_as(Int<4>{}, Int<3>{}, piece) : pack_as(Int<4>{}, Int<4>{}, piece);
            if (blks <= 8) return pack_as(Int<8>{}, Int<1>{}, piece);
            return n_sb >= 375 ? pack_as(Int<8>{}, Int<2>{}, piece) : pack_as(Int<16>{}, Int<1>{}, piece);
        };
        return ends % 16 == 0 ? pack(uint4{}) : ends % 4 == 0 ? pack(uint32_t{}) : pack(uint16_t{});
    }
    // (t = 4 without lanes: see make_geom; with field places computed at run time 5000 x 512 took 44 us by warps instead of 40, 20000 x 501 107
    // instead of 98, 9000 x 641 69 instead of 65)
    if (n_sb <= kSms) rc = g.mx ? (g.t == 4 ? launch_pack(k_pack<true, 4, 1024>, 1024) : launch_pack(k_pack<true, -1, 1024>, 1024))
                               : (g.t == 4 ? launch_pack(k_pack<false, 4, 1024>, 1024) : launch_pack(k_pack<false, -1, 1024>, 1024));
    else rc = g.mx ? (g.t == 4 ? launch_pack(k_pack<true, 4, 512>, 512) : launch_pack(k_pack<true, -1, 512>, 512))
                   : (g.t == 4 ? launch_pack(k_pack<false, 4, 512>, 512) : launch_pack(k_pack<false, -1, 512>, 512));
    if (rc) return rc;
    return CASS_OK;
}

extern "C" int cass_weight_blob_info(const void* blob, cass_blob_info* h_info, void* stream_) {
    if (!blob || !h_info) return CASS_ERR_INVALID_ARG;
    uint32_t h[kBlobHeaderBytes / 4];
    cudaStream_t stream = (cudaStream_t)stream_;
    CASS_CUDA_CHECK(cudaMemcpyAsync(h, blob, sizeof(h), cudaMemcpyDeviceToHost, stream));
    CASS_CUDA_CHECK(cudaStreamSynchronize(stream));
    if (h[H_MAGIC] != kBlobMagic || h[H_VERSION] != kBlobVersion) return CASS_ERR_INVALID_ARG;
    h_info->rows = h[H_ROWS]; h_info->cols = h[H_COLS]; h_info->prune_permille = h[H_P]; h_info->trunc_bits = h[H_T];
    h_info->seg_cols = h[H_SEG]; h_info->chunk_cols = h[H_CHUNK]; h_info->n_seg = h[H_NSEG]; h_info->n_rowblocks = h[H_NRB];
    h_info->kept_per_row = h[H_KEPT]; h_info->max_superblock_bytes = h[H_MAXSB];
    h_info->mode = h[H_MODE] == kBlobModeMx ? 2 : 1; h_info->reserved = 0;
    h_info->total_bytes = (uint64_t)h[H_TOTLO] | ((uint64_t)h[H_TOTHI] << 32);
    return CASS_OK;
}

extern "C" int cass_decode_weights(const void* blob, const cass_blob_info* h_info, void* W_bf16_out, void* stream_) {
    if (!blob || !h_info || !W_bf16_out) return CASS_ERR_INVALID_ARG;
    cudaStream_t stream = (cudaStream_t)stream_;
    CASS_CUDA_CHECK(cudaMemsetAsync(W_bf16_out, 0, (size_t)h_info->rows * h_info->cols * 2, stream));
    k_decode<<<h_info->n_rowblocks * h_info->n_seg, 256, 0, stream>>>((const uint32_t*)blob, (uint16_t*)W_bf16_out);
    CASS_LAUNCH_CHECK();
    return CASS_OK;
}
