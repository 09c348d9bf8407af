// Verification data (Sec. 4.1 target inference, Sec. 5.1 encoder): what the Cassandra-1 speculation data leaves out
// -- the low t mantissa bits of the kept values and the pruned values as they are -- and the exact reconstruction
// of the bf16 matrix from the two parts (k_join).  A session told to verify from the two parts
// (cass_session_verify_from_parts) rebuilds every matrix with it right before the verification GEMM reads it.
//
// Layout: header of 8 words {magic 'CASV', 1, rows, cols, kept per row, t, words per row, 0}; per row
// ceil(kept*t/32) words of t-bit groups (kept values in column order, MSB first), then the pruned values in column
// order as 16-bit halfwords (little endian, padded to a word).  Every row has the same kept count, so rows are
// equally long.  The bitmap is the one in the speculation data.
#include <type_traits>

#include "wblob.cuh"

namespace cass {

constexpr uint32_t kVdataMagic = 0x56534143u;
constexpr int kVdataHeaderWords = 8;

__host__ __device__ inline int vdata_lo_words(int kept, int t) { return (kept * t + 31) / 32; }
__host__ __device__ inline int vdata_row_words(int cols, int kept, int t) { return vdata_lo_words(kept, t) + (cols - kept + 1) / 2; }

// Verification data of a row by one warp, 256 columns at a time, 8 a lane.  Pruned values go straight to their places; the
// low bits of kept values are collected in a ring and leave 8 values (t bytes) a lane.  Bound: latency and issue (about 80
// instructions a lane and 8 columns); one column a lane with two global atomics a kept value took 307 us for a
// 2825 x 11733 matrix.
constexpr int kSplitWarps = 8;
constexpr int kSplitRing = 512;

__global__ void __launch_bounds__(32 * kSplitWarps) k_split(const uint32_t* __restrict__ blob, const uint16_t* __restrict__ W,
                                                            uint32_t* __restrict__ vdata, int n, int k, int kept, int t, int seg_cols,
                                                            int n_seg) {
    __shared__ __align__(8) uint8_t s_low[kSplitWarps][kSplitRing];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * kSplitWarps + warp, k_pad = ceil_div(k, 32) * 32;
    pdl_wait();
    if (row >= n) return;
    const int lo_words = vdata_lo_words(kept, t), row_words = vdata_row_words(k, kept, t);
    uint32_t* lo = vdata + kVdataHeaderWords + (size_t)row * row_words;
    uint16_t* raw = reinterpret_cast<uint16_t*>(lo + lo_words);
    const uint16_t* wr = W + (size_t)row * k;
    const bool vec = k % 8 == 0 && ((uintptr_t)W & 15) == 0;
    const uint32_t low_mask = (1u << t) - 1u;
    uint8_t* ring = s_low[warp];
    uint32_t k_cnt = 0, k_done = 0;                                     // kept values met; written
    // the n values from k_done on, 8 a lane (n = 256, or what is left at the row's end): 8 t bits, the first at the top
    auto put = [&](uint32_t nv) {
        const uint32_t kk = k_done + (uint32_t)lane * 8u;
        if (t > 0 && (uint32_t)lane * 8u < nv) {
            const uint2 two = *reinterpret_cast<const uint2*>(ring + (kk & (kSplitRing - 1)));
            unsigned long long bits = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t v = (i < 4 ? two.x >> (8 * i) : two.y >> (8 * (i - 4))) & 0xFFu;
                bits = (bits << t) | ((uint32_t)lane * 8u + i < nv ? v : 0u);
            }
            const uint32_t byte0 = kk / 8u * (uint32_t)t;
            if (t == 4) {
                lo[byte0 / 4] = (uint32_t)bits;
            } else {
                for (int i = 0; i < t; ++i)                             // byte b of the stream sits at b ^ 3
                    if (byte0 + i < (uint32_t)lo_words * 4u) reinterpret_cast<uint8_t*>(lo)[(byte0 + i) ^ 3u] = (uint8_t)(bits >> (8 * (t - 1 - i)));
            }
        }
        k_done += nv;
        __syncwarp();
    };
    for (int seg = 0; seg < n_seg; ++seg) {
        const uint4 dir = __ldg(reinterpret_cast<const uint4*>(blob + kBlobDirOffset / 4) + (row / kRowsPerBlock) * n_seg + seg);
        const int scols = seg_cols_of(k_pad, seg_cols, seg), c_base = seg * seg_cols;
        const SbGeom sg = SbGeom::make(dir_n_ch(dir.w), scols, (int)dir.y, (int)dir.z);
        const uint32_t* bmr = blob + (size_t)dir.x * 4 + sg.bm + row % kRowsPerBlock;
        uint32_t byte = 0, v[4];
        auto fetch = [&](int j0) {                                      // 8 bitmap words and their values
            const uint32_t bm8 = lane < 8 && j0 + lane < sg.bm_words ? __ldg(bmr + (j0 + lane) * 32) : 0u;
            const int c = c_base + j0 * 32 + lane * 8;
            byte = (__shfl_sync(0xffffffffu, bm8, lane >> 2) >> (24 - 8 * (lane & 3))) & 0xFFu;
            if (vec) {
                const uint4 q = __ldg(reinterpret_cast<const uint4*>(wr + min(c, k - 8)));
                v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
            } else {
                uint32_t h[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) h[i] = __ldg(wr + min(c + i, k - 1));
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = h[2 * i] | (h[2 * i + 1] << 16);
            }
        };
        fetch(0);
        for (int j0 = 0; j0 < sg.bm_words; j0 += 8) {
            const int c = c_base + j0 * 32 + lane * 8, valid = max(0, min(8, min(k, c_base + scols) - c));
            const uint32_t cnt = __popc(byte);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            uint32_t kx = k_cnt + incl - cnt;                           // kept values before the lane's columns
            uint32_t px = (uint32_t)c - kx;                             // pruned ones
            k_cnt += __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t x = (i & 1) ? v[i / 2] >> 16 : v[i / 2] & 0xFFFFu;
                if (byte & (0x80u >> i)) { ring[kx & (kSplitRing - 1)] = (uint8_t)(x & low_mask); ++kx; }
                else if (i < valid) { raw[px] = (uint16_t)x; ++px; }
            }
            if (j0 + 8 < sg.bm_words) fetch(j0 + 8);
            __syncwarp();
            if (k_cnt - k_done >= 256u) put(256u);
        }
    }
    while (k_cnt > k_done) put(min(256u, k_cnt - k_done));
    // what the last value leaves of its words
    for (uint32_t b = (uint32_t)(ceil_div((int)k_cnt, 8) * t) + lane; b < (uint32_t)lo_words * 4u; b += 32) reinterpret_cast<uint8_t*>(lo)[b ^ 3u] = 0;
    if (lane == 0 && ((k - kept) & 1)) raw[k - kept] = 0;
    if (row == 0 && lane < kVdataHeaderWords)
        vdata[lane] = lane == 0 ? kVdataMagic : lane == 1 ? 1u : lane == 2 ? (uint32_t)n : lane == 3 ? (uint32_t)k : lane == 4 ? (uint32_t)kept
                      : lane == 5 ? (uint32_t)t : lane == 6 ? (uint32_t)row_words : 0u;
}

// Exact reconstruction (Sec. 4.1 target inference: speculation and verification data are loaded and the original values
// rebuilt; Sec. 5.1 mantissa concatenator).  One warp takes one (superblock, chunk), 64 columns (two bitmap words) of its 32 rows at a
// time, in two steps over a buffer in shared memory:
//   lane = row: the codewords, fields and low mantissa bits of the window's kept values become complete bf16 values, 8 at a time
//     as in the draft GEMV, in a list; groups of 8 do not end where windows do, so up to 7 values stay for the next window.  Behind
//     the list the window's pruned values, copied from the verification data meanwhile, half a warp a row;
//   lane = 8 columns, four rows at a time: a prefix count of the bitmap says where in the list and among the pruned values the
//     columns begin; each then takes the next of either, and the eight leave in one store, but for a chunk's first and last columns.
// Kept and pruned values of a window are 64 together, so the buffer is 82 halfwords a row, whatever the matrix looks like, and 28 warps
// fit an SM (72 registers; with 80 and 24 warps 20000 x 1528 takes 71 us instead of 64, with 64 and 32 28672 x 4096 258 instead of 217).
// Bound: instruction issue (62 %) and the latency of a window's steps: 31 M warp instructions for 6144 x 4096 (49 M with a list of a
// whole chunk's values, which 20 warps an SM had room for, and one row after the other with its loads).  6144 x 4096 at 40 %
// pruning 130 -> 56 us, at 30 % 243 -> 60 (a chunk took a second turn), at 60 % 129 -> 57; 28672 x 4096 374 -> 199.
constexpr int kJoinWarps = 4;
// Chunks up to which teams: as long as all have a place at once, seven CTAs an SM.  26 and 35 us with and without for 3908 x 1528 (738 chunks), 22 and 28
// for 9000 x 600 (846), 26 and 32 for 33000 x 256 (1032), but 45 and 40 for 640 x 14336 (1120), 43 and 36 for 2171 x 4088 (1088), 74 and 55 for 5979 x 4088 (2976).
constexpr int kJoinTeamMax = 7 * kSms;
// Halfwords: a row's windows begin where its output is on a 16-byte boundary, so that whatever the width eight columns leave in one store.
// With windows from bitmap words on and one store width for the whole matrix 8987 x 4089 took 139 us instead of 86, 19995 x 4090 171 instead of 160, and
// 4096 x 13823 210 instead of 122.  On 32-, 64- and 128-byte boundaries a chunk takes more windows: 20000 x 1528 66.5, then 67.8, 68.7 and 73.7.
constexpr int kJoinAlign = 8;
constexpr int kJoinRow = 82;                                            // halfwords: 7 + 64 + 7 + 2 for odd places; an odd number of words, rows in different banks

struct JoinGeom {
    int n, k, k_pad, seg_cols, n_seg, n_ch, n_tasks, lo_words, row_words, n_raw;
};

__device__ __forceinline__ uint32_t join_lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}

// Decoder of one row's kept values in a chunk, 8 at a time and in order: code words by bit searches as in the draft GEMV, then fields and low
// bits.  T, the truncated bits, is a constant, and with it every value's place: fields that do not fill a word (t = 2, 3, 5) are first
// joined into one stream of 8 F bits, the low bits into one of 8 t.  With a place computed for every value 8987 x 4088 took 116 us at t = 2 and 117
// at t = 5 instead of 93 and 95, 2171 x 4088 63 and 59 instead of 43 (t = 2, 5); fields and low bits of t = 4 by bytes: 6144 x 4096
// 60.0 -> 57.8, 28672 x 4096 219 -> 210.
template <int T>
struct JoinGroups {
    static constexpr int F = 8 - T, PER = 32 / F;
    static constexpr int NFW = T == 4 || T >= 6 ? 1 : T == 2 || T == 3 ? 3 : 2, NLW = T == 0 ? 0 : T <= 4 ? 2 : 3;      // words a group can touch
    static constexpr uint32_t kLow = (1u << T) - 1u, kKeep = 0x8000u | (0x7Fu & ~kLow);
    const uint32_t* rows;                                               // the superblock's words of this row
    int bm, un, last;                                                   // where in the superblock bitmap and codes begin, and its last words
    int f_at, f_in, k_first;                                            // field word of the next group and its first field there; values of the segment before the chunk's
    int row;                                                            // whose low bits
    uint32_t lo_bit, upos, lut_top;                                     // next low bit of the row; next code bit; table of exponents
    uint32_t u0, u1, u2, fn[NFW], ln[NLW > 0 ? NLW : 1];                // the word of bit upos and two more

    __device__ __forceinline__ uint32_t word(int at) const { return __ldg(rows + min(at, last)); }
    // field and low words of the next group, asked for a group ahead
    __device__ __forceinline__ void fetch(const uint32_t* vdata, const JoinGeom& jg, bool first) {
#pragma unroll
        for (int i = 0; i < NFW; ++i) fn[i] = word(f_at + i * 32);
        if constexpr (NLW > 0) {
            const uint32_t* lo = vdata + kVdataHeaderWords + (size_t)row * jg.row_words;
            const int li = (int)(lo_bit >> 5), lo_last = jg.lo_words - 1;
            if (T == 4 && !first) {                                     // one word a group
                ln[0] = ln[1];
                ln[1] = __ldg(lo + min(li + 1, lo_last));
            } else {
#pragma unroll
                for (int i = 0; i < NLW; ++i) ln[i] = __ldg(lo + min(li + i, lo_last));
            }
        }
    }
    // k: values of the segment, k_row: of the row, before the chunk's
    __device__ __forceinline__ void begin(const uint32_t* body, const SbGeom& sg, int lane, int row_, int k, int k_row, uint32_t bit, const uint16_t* lut,
                                          const uint32_t* vdata, const JoinGeom& jg) {
        rows = body + lane;
        bm = sg.bm;
        un = sg.un;
        last = sg.total - 32;
        f_at = sg.fl + k / PER * 32;
        f_in = k % PER;
        k_first = k;
        row = min(row_, jg.n - 1);
        lo_bit = (uint32_t)k_row * (uint32_t)T;
        upos = bit;
        lut_top = smem_u32(lut) + 62u;
        const int at = un + (int)(upos >> 5) * 32;
        u0 = word(at);
        u1 = word(at + 32);
        u2 = word(at + 64);
        fetch(vdata, jg, true);
    }
    // the values g .. g + 7 of the chunk, packed in pairs; those beyond its last are anything
    __device__ __forceinline__ void next(int g, const uint16_t* lut, const uint32_t* vdata, const JoinGeom& jg, uint32_t (&out)[4]) {
        // the group's fields from bit 31 of f0 on, its low bits from bit 31 of l0 on
        uint32_t f0 = fn[0], f1 = fn[NFW > 1 ? 1 : 0], l0 = 0, l1 = 0;
        if constexpr (T >= 6) {
            f0 = __funnelshift_l(f0, f0, F * f_in);
        } else if constexpr (T == 2 || T == 3 || T == 5) {              // a word's last two bits are none of a field's
            const uint32_t s0 = fn[0] | (fn[1] >> 30), s1 = (fn[1] << 2) | (NFW > 2 ? fn[NFW - 1] >> 28 : 0u);
            f0 = __funnelshift_l(s1, s0, F * f_in);
            f1 = NFW > 2 ? __funnelshift_l(fn[NFW - 1] << 4, s1, F * f_in) : 0u;
        }
        if constexpr (NLW > 0) {
            l0 = __funnelshift_l(ln[1], ln[0], lo_bit);
            if constexpr (NLW > 2) l1 = __funnelshift_l(ln[2], ln[1], lo_bit);
            lo_bit += 8 * T;
        }
        f_at += 8 / PER * 32;
        if constexpr (8 % PER != 0) {
            f_in += 8 % PER;
            if (f_in >= PER) {
                f_in -= PER;
                f_at += 32;
            }
        }
        fetch(vdata, jg, false);
        uint32_t uv = __funnelshift_l(u1, u0, upos), used = 8u * 32u, q = 0, v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {                                   // shifting the found one out leaves the next code at the top
            asm("bfind.u32 %0, %1;" : "=r"(q) : "r"(uv));
            uint32_t a;
            asm("mad.lo.u32 %0, %1, 0xFFFFFFFE, %2;" : "=r"(a) : "r"(q), "r"(lut_top));
            v[i] = join_lds16(a);
            used -= q;
            uv = __funnelshift_r(0u, uv, q);
        }
        if ((int32_t)q < 0) {                                           // eight codes did not fit the window
            // Kept values of the segment from this group on.  The last group's may be fewer than eight, and their codes there: one by one all the
            // same, the last group of every row and segment took 4 us of a small matrix (512 x 512 19.1 -> 15.7, 256 x 4096 22.9 -> 16.8), and
            // 6144 x 4096 62 instead of 56
            const int cnt = (int)(__ldg(rows + (bm - 32)) >> 20) - k_first - g;
            if (__popc(__funnelshift_l(u1, u0, upos)) < min(cnt, 8)) {  // one by one
                uint32_t ub = upos;
#pragma unroll 1
                for (int i = 0; i < 8; ++i) {
                    uint32_t x = 0;
                    if (i < cnt) x = lut[read_unary(rows + un, ub, (uint32_t)(last + 32 - un)) & 255];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = i == j ? x : v[j];
                }
                used = ub - upos;
            }
        }
        const int was = (int)(upos >> 5);
        upos += used;
        const int now = (int)(upos >> 5), at = un + now * 32;
        if (now == was + 1) {
            u0 = u1; u1 = u2;
            u2 = word(at + 64);
        } else if (now > was) {
            u0 = word(at);
            u1 = word(at + 32);
            u2 = word(at + 64);
        }
        // A pair of values: exponents | the rest.  F = 4: bytes 3 - j / 2 and 2 - j / 2 of the word have an even value's sign and mantissa (an odd one's
        // once it is rotated by 4), and the low bits go beside the mantissa.
        auto pair = [&](int i, uint32_t rest) { out[i] = __byte_perm(v[2 * i], v[2 * i + 1], 0x5410) | (rest & 0x807F807Fu); };
        if constexpr (T == 4) {
            const uint32_t fo = __funnelshift_l(f0, f0, 4), le = __funnelshift_r(l0, l0, 12), lo = __funnelshift_r(l0, l0, 8);
            const uint32_t xe = (f0 & 0xF0F0F0F0u) | (le & 0x0F0F0F0Fu), xo = (fo & 0xF0F0F0F0u) | (lo & 0x0F0F0F0Fu);      // even, odd values
            pair(0, __byte_perm(xe, xo, 0x7632));
            pair(1, __byte_perm(xe, xo, 0x6521));
            pair(2, __byte_perm(xe, xo, 0x5410));
            pair(3, __byte_perm(xe, xo, 0x4703));
        } else if constexpr (T == 0) {                                  // F = 8: bytes 3 - j and 2 - j
            pair(0, __byte_perm(f0, 0u, 0x2132));
            pair(1, __byte_perm(f0, 0u, 0x0310));
            pair(2, __byte_perm(f1, 0u, 0x2132));
            pair(3, __byte_perm(f1, 0u, 0x0310));
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if constexpr (32 % F == 0) {                            // rotated fields: one rotation puts both parts in place
                    v[i] |= __funnelshift_l(f0, f0, (F * i + 16) & 31) & kKeep;
                } else {                                                // packed ones: sign and mantissa both out of the top byte
                    const int b = T == 1 ? F * (i & 3) : F * i;
                    const uint32_t x = T == 1 ? (i < 4 ? f0 : f1) << b : b + F <= 32 ? f0 << b : b < 32 ? __funnelshift_l(f1, f0, b) : f1 << (b & 31);
                    v[i] |= __byte_perm(x, 0u, 0x4433) & kKeep;
                }
                const int b = T * i;
                const uint32_t x = b + T <= 32 ? l0 >> ((32 - b - T) & 31) : b < 32 ? __funnelshift_l(l1, l0, b) >> (32 - T) : l1 >> ((64 - b - T) & 31);
                v[i] |= x & kLow;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] = __byte_perm(v[2 * i], v[2 * i + 1], 0x5410);
        }
    }
};

// T: truncated bits.  TEAM: the CTA's four warps share one chunk, the first decoding and all of them copying and writing: the latency of a small
// matrix.
template <int T, bool TEAM>
__global__ void __launch_bounds__(32 * kJoinWarps, 7) k_join(const uint32_t* __restrict__ blob, const uint32_t* __restrict__ vdata,
                                                          uint16_t* __restrict__ out, JoinGeom jg) {
    // a window's first and last eight columns may reach up to 7 beyond it: what they read there is not stored
    constexpr int kTasks = TEAM ? 1 : kJoinWarps, kSteps = TEAM ? kJoinWarps : 1;      // chunks a CTA; warps a chunk
    __shared__ __align__(16) uint16_t s_buf[8 + kTasks * 32 * kJoinRow + 8];
    __shared__ uint4 s_row[kTasks][32];                                 // a row's window: its bits, places and ends, where it begins | kept values in the first half
    __shared__ uint2 s_copy[kTasks][32];                                // its pruned values: words from, how many | to
    __shared__ uint16_t s_lut[256];                                     // rank -> exponent at its bf16 position
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint8_t* cb = reinterpret_cast<const uint8_t*>(blob) + kBlobHeaderBytes;
    pdl_wait();
    for (int i = threadIdx.x; i < 256; i += 32 * kJoinWarps) s_lut[i] = (uint16_t)cb[i] << 7;
    __syncthreads();
    const int slot = TEAM ? 0 : warp, share = TEAM ? warp : 0, task = (int)blockIdx.x * kTasks + slot;
    auto sync = [&]() {
        if (TEAM) __syncthreads();
        else __syncwarp();
    };
    if (task >= jg.n_tasks) return;
    const int sb = task / jg.n_ch, ch = task % jg.n_ch, rb = sb / jg.n_seg, seg = sb % jg.n_seg;
    const uint4 dir = __ldg(reinterpret_cast<const uint4*>(blob + kBlobDirOffset / 4) + sb);
    const int scols = seg_cols_of(jg.k_pad, jg.seg_cols, seg), n_ch = dir_n_ch(dir.w), E = dir_chunk_elems(dir.w);
    if (ch >= n_ch) return;                                             // a shorter last segment
    const SbGeom sg = SbGeom::make(n_ch, scols, (int)dir.y, (int)dir.z);
    const uint32_t* body = blob + (size_t)dir.x * 4;
    const int c_base = seg * jg.seg_cols, row = rb * kRowsPerBlock + lane;
    const uint32_t e0 = __ldg(body + sg.tab + ch * 32 + lane);
    int col = ch == 0 ? 0 : (int)(e0 >> 20);                            // this lane's row: first column not yet written
    int col_end = ch + 1 < n_ch ? (int)(__ldg(body + sg.tab + (ch + 1) * 32 + lane) >> 20) : scols;
    col_end = row < jg.n ? min(col_end, jg.k - c_base) : col;
    int k_row = ch * E;                                                 // kept values of the row before this chunk
    for (int i = 0; i < seg; ++i) {
        const uint4 dp = __ldg(reinterpret_cast<const uint4*>(blob + kBlobDirOffset / 4) + rb * jg.n_seg + i);
        k_row += (int)(__ldg(blob + (size_t)dp.x * 4 + dir_n_ch(dp.w) * 32 + lane) >> 20);
    }
    JoinGroups<T> dec;
    dec.begin(body, sg, lane, row, ch * E, k_row, e0 & 0xFFFFFu, s_lut, vdata, jg);
    uint16_t* buf = s_buf + 8 + slot * 32 * kJoinRow;
    uint16_t* mine = buf + lane * kJoinRow;
    const uint32_t buf_a = smem_u32(buf);

    // The row's windows begin where its output is on a 16-byte boundary, up to 7 columns before the chunk's first (and before the segment)
    const uint32_t phase = (uint32_t)(reinterpret_cast<uintptr_t>(out) >> 1) + (uint32_t)row * (uint32_t)jg.k + (uint32_t)(c_base + col);
    int b0 = col - (int)(phase & (uint32_t)(kJoinAlign - 1)), ks = 0;   // the window's first column; values taken (decoded: whole groups of them)
    int raw_at = c_base + col - k_row;                                  // pruned values of the row before the window's
    auto bm_word = [&](int j) { return (uint32_t)j < (uint32_t)sg.bm_words ? __ldg(dec.rows + (dec.bm + j * 32)) : 0u; };
    uint32_t wa = bm_word(b0 >> 5), wb = bm_word((b0 >> 5) + 1), wc = bm_word((b0 >> 5) + 2);

#pragma unroll 1
    while (__any_sync(0xffffffffu, col < col_end)) {
        // ---- the window: columns col .. b0 + hi - 1 of this lane's row, bits of others cleared ----
        const bool more = col < col_end;
        const int off = more ? col - b0 : 64, hi = more ? min(64, col_end - b0) : 64;
        uint32_t w0 = __funnelshift_l(wb, wa, b0), w1 = __funnelshift_l(wc, wb, b0);
        wa = wc;
        wb = bm_word((b0 >> 5) + 3);
        wc = bm_word((b0 >> 5) + 4);
        {
            unsigned long long m = off < 64 ? ~0ull >> off : 0ull;
            if (hi < 64) m &= ~(~0ull >> hi);
            w0 &= (uint32_t)(m >> 32);
            w1 &= (uint32_t)m;
        }
        const int n0 = __popc(w0), kw = n0 + __popc(w1), base8 = ks & ~7, ke = ks + kw, done_to = (ke + 7) & ~7;
        // ---- its pruned values, behind the list ----
        const int n_raw = hi - off - kw;
        const uint32_t rw = (uint32_t)(jg.lo_words + (raw_at >> 1));
        const int n_w = n_raw > 0 ? ((raw_at & 1) + n_raw + 1) >> 1 : 0, to_w = (lane * kJoinRow + done_to - base8) >> 1;
        const uint32_t place = (uint32_t)(ks - base8) | ((uint32_t)(done_to - base8 + (raw_at & 1)) << 8) | ((uint32_t)off << 16) | ((uint32_t)hi << 24);
        if (share == 0) {
            s_copy[slot][lane] = make_uint2(rw, (uint32_t)n_w | ((uint32_t)to_w << 16));
            s_row[slot][lane] = make_uint4(w0, w1, place, (uint32_t)(b0 + kJoinAlign) | ((uint32_t)n0 << 16));
        }
        const bool whole = __all_sync(0xffffffffu, off == 0 && hi == 64);
        sync();
        auto copy = [&](uint32_t to, const uint32_t* from) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(from) : "memory"); };
#pragma unroll 4
        for (int r = share * 2 + (lane >> 4); r < kRowsPerBlock; r += 2 * kSteps) {        // half a warp a row
            const uint2 cp = s_copy[slot][r];
            const uint32_t n = cp.y & 0xFFFFu, to = buf_a + (cp.y >> 16) * 4u + (uint32_t)(lane & 15) * 4u;
            const uint32_t* from = vdata + kVdataHeaderWords + (size_t)(rb * kRowsPerBlock + r) * jg.row_words + (cp.x + (uint32_t)(lane & 15));
            if ((uint32_t)(lane & 15) < n) copy(to, from);
            if (n > 16u)                                                // up to 33 words
                for (uint32_t w = 16; w + (uint32_t)(lane & 15) < n; w += 16) copy(to + w * 4u, from + w);
        }
        // ---- lane = row: values up to ke, whole groups ----
        for (int done = (ks + 7) & ~7; share == 0 && done < done_to; done += 8) {
            uint32_t v[4];
            dec.next(done, s_lut, vdata, jg, v);
            uint32_t* to = reinterpret_cast<uint32_t*>(mine + done - base8);
#pragma unroll
            for (int i = 0; i < 4; ++i) to[i] = v[i];
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        sync();
        // ---- lane = 8 columns of one of four rows ----
        auto write = [&](auto whole_c) {
            constexpr bool W = decltype(whole_c)::value;                // every row has the whole window: nothing to leave out
            const int o = lane & 7, c = o * 8, r_first = share * 4 + (lane >> 3);
            const uint32_t sh = 8u * (uint32_t)(o & 3);
            uint16_t* to_row = out + (size_t)(rb * kRowsPerBlock + r_first) * jg.k + (c_base + c) - kJoinAlign;
            uint32_t row_a = buf_a + (uint32_t)(r_first * kJoinRow) * 2u;
#pragma unroll 1
            for (int r = r_first; r < kRowsPerBlock; r += 4 * kSteps, to_row += (size_t)(4 * kSteps) * jg.k, row_a += 4 * kSteps * kJoinRow * 2) {
                const uint4 p = s_row[slot][r];
                const int r_off = W ? 0 : (int)((p.z >> 16) & 0xFFu), r_hi = W ? 64 : (int)(p.z >> 24);
                if (!W && (c + 8 <= r_off || c >= r_hi)) continue;      // none of the window's columns
                const uint32_t w = o < 4 ? p.x : p.y, b = w << sh;
                const uint32_t before = (uint32_t)__popc(__funnelshift_rc(w, 0u, 32u - sh)) + (o < 4 ? 0u : p.w >> 16);      // kept values of the window before these columns
                uint32_t ak = row_a + ((p.z & 0xFFu) + before) * 2u;
                uint32_t ar = row_a + (((p.z >> 8) & 0xFFu) + (uint32_t)(c - r_off) - before) * 2u;
                uint32_t x[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const bool keep = b & (0x80000000u >> i);
                    x[i] = join_lds16(keep ? ak : ar);
                    ak += keep ? 2u : 0u;
                    ar += keep ? 0u : 2u;
                }
                uint16_t* to = to_row + (p.w & 0xFFFFu);
                if (W || (c >= r_off && c + 8 <= r_hi)) {
                    *reinterpret_cast<uint4*>(to) = make_uint4(x[0] | (x[1] << 16), x[2] | (x[3] << 16), x[4] | (x[5] << 16), x[6] | (x[7] << 16));
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (c + i >= r_off && c + i < r_hi) to[i] = (uint16_t)x[i];
                }
            }
        };
        if (whole) write(std::true_type{});
        else write(std::false_type{});
        sync();
        // ---- values decoded ahead move to the front ----
        if (share == 0 && (ke & 7) && (ke & ~7) != base8) {
            const uint32_t* from = reinterpret_cast<const uint32_t*>(mine + (ke & ~7) - base8);
            const uint32_t m[4] = {from[0], from[1], from[2], from[3]};
            uint32_t* to = reinterpret_cast<uint32_t*>(mine);
#pragma unroll
            for (int i = 0; i < 4; ++i) to[i] = m[i];
        }
        ks = ke;
        raw_at += n_raw;
        if (more) col = b0 + hi;
        b0 += 64;
    }
}

}  // namespace cass

using namespace cass;

extern "C" int cass_verification_data_bytes(const cass_blob_info* bi, size_t* h_bytes) {
    if (!bi || !h_bytes || bi->rows <= 0 || bi->cols <= 0) return CASS_ERR_INVALID_ARG;
    if (bi->mode != 1) return CASS_ERR_UNSUPPORTED;
    *h_bytes = ((size_t)kVdataHeaderWords + (size_t)bi->rows * vdata_row_words(bi->cols, bi->kept_per_row, bi->trunc_bits)) * 4;
    return CASS_OK;
}

extern "C" int cass_encode_verification_data(const void* blob, const cass_blob_info* bi, const void* W_bf16, void* vdata,
                                             size_t vdata_bytes, void* stream_) {
    size_t need = 0;
    int rc = cass_verification_data_bytes(bi, &need);
    if (rc) return rc;
    if (!blob || !W_bf16 || !vdata || ((uintptr_t)vdata & 3)) return CASS_ERR_INVALID_ARG;
    if (vdata_bytes < need) return CASS_ERR_CAPACITY;
    CASS_PDL_LAUNCH(k_split, dim3(ceil_div(bi->rows, kSplitWarps)), dim3(32 * kSplitWarps), 0, (cudaStream_t)stream_, (const uint32_t*)blob,
                    (const uint16_t*)W_bf16, (uint32_t*)vdata, (int)bi->rows, (int)bi->cols, (int)bi->kept_per_row, (int)bi->trunc_bits,
                    (int)bi->seg_cols, (int)bi->n_seg);
    return CASS_OK;
}

extern "C" int cass_decode_full(const void* blob, const cass_blob_info* bi, const void* vdata, void* W_bf16_out, void* stream_) {
    if (!blob || !bi || !vdata || !W_bf16_out) return CASS_ERR_INVALID_ARG;
    if (bi->mode != 1) return CASS_ERR_UNSUPPORTED;
    const int n_ch = ceil_div(bi->seg_cols, bi->chunk_cols);
    if (n_ch > 32) return CASS_ERR_UNSUPPORTED;
    cudaStream_t stream = (cudaStream_t)stream_;
    const uint32_t *b32 = (const uint32_t*)blob, *v32 = (const uint32_t*)vdata;
    uint16_t* o16 = (uint16_t*)W_bf16_out;
    const JoinGeom jg{bi->rows, bi->cols, ceil_div(bi->cols, 32) * 32, bi->seg_cols, bi->n_seg, n_ch,
                      bi->n_rowblocks * bi->n_seg * n_ch, vdata_lo_words(bi->kept_per_row, bi->trunc_bits),
                      vdata_row_words(bi->cols, bi->kept_per_row, bi->trunc_bits), bi->cols - bi->kept_per_row};
    const bool team = jg.n_tasks <= kJoinTeamMax;
#define CASS_JOIN(T_)                                                                                                               \
    do {                                                                                                                            \
        if (team) CASS_PDL_LAUNCH((k_join<T_, true>), dim3(jg.n_tasks), dim3(32 * kJoinWarps), 0, stream, b32, v32, o16, jg);        \
        else CASS_PDL_LAUNCH((k_join<T_, false>), dim3(ceil_div(jg.n_tasks, kJoinWarps)), dim3(32 * kJoinWarps), 0, stream, b32, v32, o16, jg); \
    } while (0)
    switch (bi->trunc_bits) {
        case 0: CASS_JOIN(0); break;
        case 1: CASS_JOIN(1); break;
        case 2: CASS_JOIN(2); break;
        case 3: CASS_JOIN(3); break;
        case 4: CASS_JOIN(4); break;
        case 5: CASS_JOIN(5); break;
        case 6: CASS_JOIN(6); break;
        case 7: CASS_JOIN(7); break;
        default: return CASS_ERR_INVALID_ARG;
    }
#undef CASS_JOIN
    return CASS_OK;
}
