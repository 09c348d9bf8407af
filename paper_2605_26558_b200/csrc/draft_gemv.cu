// Draft GEMV: y = decode(speculation data) * x with the decode done in registers (Sec. 4.1 draft inference;
// the software form of the decoder dataflow of Sec. 5.1: bitmap de-sparsification, unary exponent decode
// through a rank->exponent table, sign/mantissa concatenation).
//
// Work unit = one superblock (32 rows x one column segment).  A CTA owns one column segment (its slice of x
// stays in shared memory as fp32) and walks the row blocks assigned to it; a superblock arrives by one bulk
// asynchronous copy (contiguous reads, as Sec. 5.3 asks) into the CTA's single stage; the CTAs that share an SM
// overlap each other's copies and decodes.  Warp c decodes chunk c with lane = row: every lane
// walks its own bitmap, field and unary streams, which are interleaved word by word over the 32 rows so that
// all shared-memory reads of the streams are conflict free.
#include <cooperative_groups.h>

#include <type_traits>

#include "wblob.cuh"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace cass {

constexpr int kGemvStages = 1;         // stages of the copy ring per CTA; several CTAs share an SM, so their copies and decodes overlap
constexpr int kXSlack = 288;           // a window walk may look up to 8 x 32 + 8 columns past its start: what lies behind the x slice there is not used

// Bytes per column of the x slice in shared memory: one vector is kept as fp32, several as packed bf16 [col][nb].
__host__ __device__ constexpr int x_col_bytes(int nb) { return nb == 1 ? 4 : 2 * nb; }
__host__ __device__ constexpr uint32_t x_slice_bytes(int seg_cols, int nb) { return (uint32_t)(seg_cols * x_col_bytes(nb) + 511) / 512 * 512; }

// Shared memory, up to two vectors: superblock, x slice and slack, table, the chunks' sums (twice).  More: x slice, superblock, table; the
// slack is the superblock, and the sums take its place once it has been read: slack and sums (4.6 and 8 KB of 8 vectors) are the room of a
// third CTA on an SM (5120 x 13824, eight Cassandra-2 vectors: 96 -> 82 us with it and the paired multiply-adds).
__host__ __device__ constexpr bool gemv_compact(int nb) { return nb >= 4; }
static size_t gemv_stage_bytes(const cass_blob_info& bi, int nb) {
    const size_t sums = !gemv_compact(nb) ? 0 : (size_t)nb * ceil_div(bi.seg_cols, bi.chunk_cols) * 32 * 4, body = (size_t)bi.max_superblock_bytes + 384;
    return align_up(body > sums ? body : sums, 512);
}
static size_t gemv_smem_bytes(const cass_blob_info& bi, int nb) {
    const int n_ch = ceil_div(bi.seg_cols, bi.chunk_cols);
    const size_t stage = kGemvStages * gemv_stage_bytes(bi, nb), table = 256 * 4 + 64, slack = (size_t)kXSlack * x_col_bytes(nb);
    if (!gemv_compact(nb)) return stage + (size_t)bi.seg_cols * x_col_bytes(nb) + slack + table + (size_t)2 * n_ch * 32 * 4;
    return x_slice_bytes(bi.seg_cols, nb) + (stage + table > slack ? stage + table : slack);
}

// What the kernel declares itself: a segment's sums, the tile's sizes and flags, up to where the dynamic part may begin.
static size_t gemv_smem_static(int nb) { return align_up((size_t)nb * 32 * 4 + 32, 512); }

// What counts against a CTA's limit: every part side by side, whatever the layout, so that it does not decide which blobs are taken.
size_t gemv_smem_total(const cass_blob_info& bi, int nb) {
    const size_t stage = kGemvStages * align_up((size_t)bi.max_superblock_bytes + 384, 512);
    const size_t sums = (size_t)(nb < 2 ? 2 : nb) * ceil_div(bi.seg_cols, bi.chunk_cols) * 32 * 4;
    return stage + (size_t)(bi.seg_cols + kXSlack) * x_col_bytes(nb) + 256 * 4 + 64 + sums + gemv_smem_static(nb);
}

__device__ __forceinline__ uint32_t bfind_u32(uint32_t v) {         // index of the most significant one, -1 if none
    uint32_t r;
    asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t mad_lo(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// Sign and kept mantissa bits of a field at their binary32 positions, for truncations whose fields do not tile a
// word (8 - t = 7, 6, 5, 3): the field is packed from the most significant end, floor(32 / (8 - t)) per word.
template <int T>
__device__ __forceinline__ uint32_t packed_field_f32(uint32_t word, uint32_t j) {
    constexpr int F = 8 - T;
    const uint32_t f = (word >> (32u - (uint32_t)F * (j + 1u))) & ((1u << F) - 1u);
    return ((f >> (F - 1)) << 31) | ((f & ((1u << (F - 1)) - 1u)) << (16 + T));
}

template <int NB>
struct WalkState {
    float acc[NB];
    uint32_t bpos, upos;
};

// The NB values of x at one column: raw words as they sit in shared memory, and their use in the accumulators.
template <int NB>
struct XRaw { uint32_t w[NB == 1 ? 1 : NB / 2]; };

template <int NB, int OFF = 0>
__device__ __forceinline__ XRaw<NB> x_load(uint32_t addr) {
    XRaw<NB> r;
    if constexpr (NB <= 2) asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(r.w[0]) : "r"(addr), "n"(OFF));
    else if constexpr (NB == 4) asm volatile("ld.shared.v2.u32 {%0,%1}, [%2+%3];" : "=r"(r.w[0]), "=r"(r.w[1]) : "r"(addr), "n"(OFF));
    else asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4+%5];" : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]) : "r"(addr), "n"(OFF));
    return r;
}

// PAIRS: two multiply-adds an instruction, each rounded as one by itself.  28672 x 4096: four vectors 77 -> 69 us, two 60 -> 57, but two
// Cassandra-2 vectors, whose CTAs then take more registers than five an SM leave, 46.7 -> 49.5; and where latency is all, two vectors
// 7.1 -> 8.0 for 1376 x 256 and 10.4 -> 11.4 for 700 x 3000.
template <int NB, bool PAIRS>
__device__ __forceinline__ void x_fma(const XRaw<NB>& r, uint32_t wb, float (&acc)[NB]) {
    if constexpr (NB == 1) {
        acc[0] = fmaf(__uint_as_float(wb), __uint_as_float(r.w[0]), acc[0]);
    } else if constexpr (!PAIRS) {
        const float w = __uint_as_float(wb);
#pragma unroll
        for (int i = 0; i < NB / 2; ++i) {
            acc[2 * i] = fmaf(w, __uint_as_float(r.w[i] << 16), acc[2 * i]);
            acc[2 * i + 1] = fmaf(w, __uint_as_float(r.w[i] & 0xFFFF0000u), acc[2 * i + 1]);
        }
    } else {
        unsigned long long ww;
        asm("mov.b64 %0, {%1, %1};" : "=l"(ww) : "r"(wb));
#pragma unroll
        for (int i = 0; i < NB / 2; ++i)
            asm("{\n\t.reg .b64 a, x;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 x, {%3, %4};\n\tfma.rn.f32x2 a, %2, x, a;\n\tmov.b64 {%0, %1}, a;\n\t}"
                : "+f"(acc[2 * i]), "+f"(acc[2 * i + 1])
                : "l"(ww), "r"(r.w[i] << 16), "r"(r.w[i] & 0xFFFF0000u));
    }
}

// Careful walk of `count` (<= 8) kept values of one row from column bpos / code bit upos on: any gap between
// kept columns, any codeword length.  Used for the rare groups that do not fit the 32-bit windows.
// flC: the segment's first field word of this row; k0: index (inside the segment) of the group's first value.
template <int T, int NB, bool PAIRS>
__device__ __noinline__ WalkState<NB> group_slow(const uint32_t* bmS, const uint32_t* unS, const uint32_t* flC, uint32_t k0, int count,
                                                 WalkState<NB> st, uint32_t bpos_lim, uint32_t upos_lim, const float* xs,
                                                 const uint32_t* lut) {
    constexpr int F = 8 - T, PER = 32 / F;
    constexpr uint32_t MASK = 0x80000000u | (((1u << (7 - T)) - 1u) << (16 + T));
    for (int e = 0; e < count; ++e) {
        bool found = false;
        while (st.bpos < bpos_lim) {
            uint32_t w = bmS[(st.bpos >> 5) * 32] << (st.bpos & 31);
            if (w) { st.bpos += __clz(w); found = true; break; }
            st.bpos = (st.bpos | 31u) + 1u;
        }
        if (!found) break;                                   // corrupt stream: stop inside the buffers
        const XRaw<NB> xv = x_load<NB>(smem_u32(xs) + st.bpos * (uint32_t)x_col_bytes(NB));
        st.bpos += 1;
        const int rank = read_unary(unS, st.upos, upos_lim);
        const uint32_t k = k0 + (uint32_t)e;
        const uint32_t fword = flC[(k / PER) * 32];
        uint32_t a;
        if constexpr (32 % F == 0) a = __funnelshift_l(fword, fword, (F * (k % PER)) & 31) & MASK;
        else a = packed_field_f32<T>(fword, k % PER);
        x_fma<NB, PAIRS>(xv, a | lut[rank & 255], st.acc);
    }
    return st;
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {         // shared-space byte address
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t lds_u32_off(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}

// Dot product of one chunk (32 rows, lane = row) with x.  T = truncated mantissa bits (0 to 5).  Every lane walks its row in
// groups of 8 kept values: 32 bitmap bits and 64 code bits from its cursors on.  The highest set bit of the bitmap window is
// the next kept column, the highest one of the code window the next terminator; one funnel shift by its position drops it
// and everything above, so the next search starts at the top again and a search gives a distance: the running address of x
// moves by the columns skipped, and the position itself indexes the rank -> exponent table.
// A group whose 8 kept columns span more than 32 columns (wide: four of them), or four of whose codewords take more than 32
// bits, shows up as a window that ran dry (nothing left to find); that lane then redoes the group with the careful walk while
// the others wait.
// Bound: 17.5 warp instructions a kept value and lane with the kernel around them, of which 7 on the integer pipe (one every other
// cycle), two bit searches (one every 8 cycles) and 3 shared-memory loads (the gather of x meets a bank two to three times): issue
// slots 73 %, searches 70 %, shared memory 64 %, integer pipe 55 % busy.  Clearing the used bit with a shift and a mask, positions kept
// absolute and a code window for every 4 values took 19: 58.6 -> 53.0 us on 28672 x 4096 with the results added in the kernel.
// Finding some terminators by a conversion to float instead of a search: 54.5 to 56 us.
template <int T, int NB, bool WIDE, bool PAIRS>
__device__ __forceinline__ void chunk_dot_fast(const uint32_t* __restrict__ sb, const SbGeom& g, int ch, int lane,
                                               int chunk_elems, const float* __restrict__ xs,
                                               const uint32_t* __restrict__ lut, float (&acc)[NB]) {
    constexpr int F = 8 - T, PER = 32 / F;
    constexpr bool ROT = 32 % F == 0;                                    // fields tile a word: float-aligned and rotated
    constexpr int NFW = ROT ? kGroupCols / PER : 3;                      // field words a group of 8 can touch
    constexpr uint32_t MASK = 0x80000000u | (((1u << (7 - T)) - 1u) << (16 + T));   // sign + kept mantissa of a binary32
    static_assert(ROT ? (PER == 4 || PER == 8) : (PER >= 4 && PER <= 10), "fast path: 4 to 10 fields per word");
    constexpr uint32_t XS = (uint32_t)x_col_bytes(NB);            // bytes per column of the x slice
    constexpr uint32_t XL = XS == 4 ? 2 : XS == 8 ? 3 : 4;
    const uint32_t e0 = sb[g.tab + ch * 32 + lane];            // where this row's value ch * chunk_elems sits
    const uint32_t fw = (uint32_t)(ch * chunk_elems) / PER;    // the word of the chunk's first field (fields are numbered through the segment)
    uint32_t upos = e0 & 0xFFFFFu;
    const uint32_t* bmS = sb + g.bm + lane;
    const uint32_t* flS = sb + g.fl + lane;
    const uint32_t* unS = sb + g.un + lane;
    const uint32_t bm_a = smem_u32(bmS), un_a = smem_u32(unS), xs_a = smem_u32(xs), lut_a = smem_u32(lut);
    uint32_t fl_a = smem_u32(flS + fw * 32);
    uint32_t j0 = (uint32_t)(ch * chunk_elems) % PER;           // packed fields: place of the group's first field in its word
    // every row has chunk_elems values in each chunk except its last ones, so the lanes of a warp stay in step
    const int kept = (int)(sb[g.tab + g.n_ch * 32 + lane] >> 20);
    const int m = max(0, min(chunk_elems, kept - ch * chunk_elems));
    const int n_full = __reduce_min_sync(0xffffffffu, m) / kGroupCols;
    const int n_groups = ceil_div(__reduce_max_sync(0xffffffffu, m), kGroupCols);
    uint32_t xc = xs_a + (e0 >> 20) * XS;                       // address of the cursor's column in the x slice
    const uint32_t xc_lim = xs_a + (uint32_t)(g.bm_words * 32) * XS, upos_lim = (uint32_t)(g.w_u * 32);
    const uint32_t bm_x = bm_a - xs_a;

    auto group = [&](int grp, auto tail_c) {
        constexpr bool tail = decltype(tail_c)::value;         // two specialisations: full groups carry no per-value tests
        WalkState<NB> st0;
#pragma unroll
        for (int b = 0; b < NB; ++b) st0.acc[b] = acc[b];
        st0.upos = upos;
        // the x slice starts at a multiple of 512 bytes, so that the address itself gives the bit (modulo 32) and the word
        const uint32_t xc0 = xc, bpos = xc >> XL;
        const uint32_t ba = XL == 2 ? (xc & ~127u) + bm_x : (((xc - xs_a) >> (XL - 2)) & ~127u) + bm_a;
        const uint32_t bw1 = lds_u32_off<128>(ba), bv0 = __funnelshift_l(bw1, lds_u32(ba), bpos);      // 32 columns from the cursor on
        uint32_t bv = bv0;
        const uint32_t ua = un_a + (upos & ~31u) * 4u;
        const uint32_t u1 = lds_u32_off<128>(ua);
        const uint32_t uv0 = __funnelshift_l(u1, lds_u32(ua), upos);                       // 64 code bits from the cursor on
        const uint32_t uv1 = __funnelshift_l(lds_u32_off<256>(ua), u1, upos);
        uint32_t uv = uv0;
        uint32_t fwd[NFW];
        fwd[0] = lds_u32(fl_a);
        if (NFW > 1) fwd[1] = lds_u32_off<128>(fl_a);
        if (NFW > 2) fwd[2] = lds_u32_off<256>(fl_a);
        const int rem = m - grp * kGroupCols;
        uint32_t dry = 0;                           // sign bit set: a window ran dry under a value that counts
        uint32_t p = 0, xg = xc;                    // the cursor's column, less XS * 32 for every value found
        auto take = [&](auto e_c) {
            constexpr int e = decltype(e_c)::value, j = e % kGroupCodes;
            p = bfind_u32(bv);                                       // next kept column: 31 - p columns on
            xg = mad_lo(p, 0u - XS, xg);
            const XRaw<NB> xv = x_load<NB, (32 * (e + 1) - 1) * (int)XS>(xg);
            bv = __funnelshift_r(0u, bv, p);
            const uint32_t q = bfind_u32(uv);                        // next terminator: the code's rank is 31 - q
            const uint32_t eb = lds_u32(mad_lo(q, 0xFFFFFFFCu, lut_a + 124u));
            uv = __funnelshift_r(0u, uv, q);
            upos -= q;
            uint32_t wb;
            if constexpr (ROT) {
                const uint32_t fword = fwd[e / PER];
                const uint32_t a = __funnelshift_l(fword, fword, (F * (e % PER)) & 31);
                wb = (a & MASK) | eb;
            } else {
                const uint32_t jj = j0 + (uint32_t)e;                 // field jj of the group's (up to three) words
                const uint32_t wsel = jj >= 2u * PER ? 2u : (jj >= (uint32_t)PER ? 1u : 0u);
                const uint32_t fword = wsel == 2u ? fwd[NFW - 1] : (wsel == 1u ? fwd[1] : fwd[0]);
                wb = packed_field_f32<T>(fword, jj - wsel * PER) | eb;
            }
            if constexpr (!tail) {
                x_fma<NB, PAIRS>(xv, wb, acc);
                if (j == kGroupCodes - 1) dry |= WIDE ? p | q : q;
            } else if (e < rem) {
                x_fma<NB, PAIRS>(xv, wb, acc);
                dry |= p | q;
            }
        };
        take(std::integral_constant<int, 0>{}); take(std::integral_constant<int, 1>{});
        take(std::integral_constant<int, 2>{}); take(std::integral_constant<int, 3>{});
        const uint32_t used = upos + 4u * 32u - st0.upos;            // bits up to and including the fourth terminator: at most 32
        uv = __funnelshift_lc(uv1, uv0, used);
        if constexpr (WIDE) {                                                  // and the columns up to the fourth value's: the next 32 from there
            const uint32_t cols = (uint32_t)((int32_t)(xg - xc0) >> XL) + 4u * 32u;
            bv = __funnelshift_lc(__funnelshift_l(lds_u32_off<256>(ba), bw1, bpos), bv0, cols);
        }
        take(std::integral_constant<int, 4>{}); take(std::integral_constant<int, 5>{});
        take(std::integral_constant<int, 6>{}); take(std::integral_constant<int, 7>{});
        upos += 8u * 32u;                                            // 32 - q bits a code
        xc = xg + 8u * 32u * XS;
        if (tail) {                                                  // rows that ran out of values stay inside the buffers
            upos = min(upos, upos_lim);
            xc = min(xc, xc_lim);
        } else {
            dry |= p;
        }
        if ((int32_t)dry < 0) {
            st0.bpos = (xc0 - xs_a) >> XL;
            const WalkState<NB> r = group_slow<T, NB, PAIRS>(bmS, unS, flS, (uint32_t)(ch * chunk_elems + grp * kGroupCols), min(rem, kGroupCols),
                                                      st0, (xc_lim - xs_a) >> XL, upos_lim, xs, lut);
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[b] = r.acc[b];
            xc = xs_a + (r.bpos << XL); upos = r.upos;
        }
        if constexpr (ROT) {
            fl_a += NFW * 128u;
        } else {
            const uint32_t jn = j0 + (uint32_t)kGroupCols;
            const uint32_t adv = jn >= 2u * PER ? 2u : (jn >= (uint32_t)PER ? 1u : 0u);
            fl_a += adv * 128u;
            j0 = jn - adv * PER;
        }
    };

    int grp = 0;
    for (; grp < n_full; ++grp) group(grp, std::false_type{});
    for (; grp < n_groups; ++grp) group(grp, std::true_type{});
}

// ---- Cassandra-2 (MX) chunk: 4-bit fields (sign + 3 magnitude bits, t = 4), one exponent byte per 32 values ------
// Same bitmap walk as above; the unary parse is replaced by a 16-entry table look-up of the signed magnitude, and a
// block's 32 products are summed first and scaled by the block's power of two once (Sec. 5.1, MX decoder: the shared
// exponent is broadcast to the elements of its block).
template <int NB, bool PAIRS>
__device__ __noinline__ WalkState<NB> group_slow_mx(const uint32_t* bmS, uint32_t fword, int count, WalkState<NB> st,
                                                    uint32_t bpos_lim, const float* xs, const float* nlut) {
    for (int e = 0; e < count; ++e) {
        bool found = false;
        while (st.bpos < bpos_lim) {
            uint32_t w = bmS[(st.bpos >> 5) * 32] << (st.bpos & 31);
            if (w) { st.bpos += __clz(w); found = true; break; }
            st.bpos = (st.bpos | 31u) + 1u;
        }
        if (!found) break;
        const XRaw<NB> xv = x_load<NB>(smem_u32(xs) + st.bpos * (uint32_t)x_col_bytes(NB));
        st.bpos += 1;
        x_fma<NB, PAIRS>(xv, __float_as_uint(nlut[(fword >> (28 - 4 * e)) & 15u]), st.acc);
    }
    return st;
}

template <int NB, bool WIDE, bool PAIRS>
__device__ __forceinline__ void chunk_dot_mx4(const uint32_t* __restrict__ sb, const SbGeom& g, int ch, int lane,
                                              int chunk_elems, const float* __restrict__ xs,
                                              const float* __restrict__ nlut, float (&acc)[NB]) {
    constexpr uint32_t XS = (uint32_t)x_col_bytes(NB);
    constexpr uint32_t XL = XS == 4 ? 2 : XS == 8 ? 3 : 4;
    const uint32_t e0 = sb[g.tab + ch * 32 + lane];
    const uint32_t* bmS = sb + g.bm + lane;
    const uint32_t bm_a = smem_u32(bmS), xs_a = smem_u32(xs), nl_a = smem_u32(nlut);      // nlut is 64-byte aligned
    uint32_t fl_a = smem_u32(sb + g.fl + lane) + (uint32_t)(ch * chunk_elems / 8) * 128u;
    const uint32_t ex_a = smem_u32(sb + g.un + lane);
    const int kept = (int)(sb[g.tab + g.n_ch * 32 + lane] >> 20);
    const int m = max(0, min(chunk_elems, kept - ch * chunk_elems));
    const int n_full = __reduce_min_sync(0xffffffffu, m) / kGroupCols;
    const int n_groups = ceil_div(__reduce_max_sync(0xffffffffu, m), kGroupCols);
    uint32_t xc = xs_a + (e0 >> 20) * XS;                       // address of the cursor's column in the x slice
    const uint32_t blk0 = (e0 & 0xFFFFFu) >> 3;                 // index of the chunk's first exponent byte
    const uint32_t xc_lim = xs_a + (uint32_t)(g.bm_words * 32) * XS, bm_x = bm_a - xs_a;
    float blk[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) blk[b] = 0.f;

    auto group = [&](int grp, auto tail_c) {
        constexpr bool tail = decltype(tail_c)::value;
        WalkState<NB> st0;
#pragma unroll
        for (int b = 0; b < NB; ++b) st0.acc[b] = blk[b];
        st0.upos = 0;
        // the x slice starts at a multiple of 512 bytes, so that the address itself gives the bit (modulo 32) and the word
        const uint32_t xc0 = xc, bpos = xc >> XL;
        const uint32_t ba = XL == 2 ? (xc & ~127u) + bm_x : (((xc - xs_a) >> (XL - 2)) & ~127u) + bm_a;
        const uint32_t bw1 = lds_u32_off<128>(ba), bv0 = __funnelshift_l(bw1, lds_u32(ba), bpos);
        uint32_t bv = bv0;
        const uint32_t fword = lds_u32(fl_a);
        const int rem = m - grp * kGroupCols;
        uint32_t dry = 0, p = 0, xg = xc;
        auto take = [&](auto e_c) {
            constexpr int e = decltype(e_c)::value;
            p = bfind_u32(bv);                                       // next kept column: 31 - p columns on
            xg = mad_lo(p, 0u - XS, xg);
            const XRaw<NB> xv = x_load<NB, (32 * (e + 1) - 1) * (int)XS>(xg);
            bv = __funnelshift_r(0u, bv, p);
            const uint32_t off = e < 7 ? (fword >> (26 - 4 * e)) : (fword << 2);
            const uint32_t wb = lds_u32((off & 0x3Cu) | nl_a);                         // +-(magnitude << 4) as a float
            if constexpr (!tail) {
                x_fma<NB, PAIRS>(xv, wb, blk);
            } else if (e < rem) {
                x_fma<NB, PAIRS>(xv, wb, blk);
                dry |= p;
            }
        };
        take(std::integral_constant<int, 0>{}); take(std::integral_constant<int, 1>{});
        take(std::integral_constant<int, 2>{}); take(std::integral_constant<int, 3>{});
        if constexpr (WIDE) {                                                  // the next 32 columns from the fourth value's on
            if (!tail) dry |= p;
            const uint32_t cols = (uint32_t)((int32_t)(xg - xc0) >> XL) + 4u * 32u;
            bv = __funnelshift_lc(__funnelshift_l(lds_u32_off<256>(ba), bw1, bpos), bv0, cols);
        }
        take(std::integral_constant<int, 4>{}); take(std::integral_constant<int, 5>{});
        take(std::integral_constant<int, 6>{}); take(std::integral_constant<int, 7>{});
        xc = xg + 8u * 32u * XS;
        if (tail) xc = min(xc, xc_lim);
        else dry |= p;
        if ((int32_t)dry < 0) {
            st0.bpos = (xc0 - xs_a) >> XL;
            const WalkState<NB> r = group_slow_mx<NB, PAIRS>(bmS, fword, min(rem, kGroupCols), st0, (xc_lim - xs_a) >> XL, xs, nlut);
#pragma unroll
            for (int b = 0; b < NB; ++b) blk[b] = r.acc[b];
            xc = xs_a + (r.bpos << XL);
        }
        fl_a += 128u;
        if ((grp & 3) == 3 || grp == n_groups - 1) {              // a block of 32 values is complete: apply its scale
            const uint32_t bi = blk0 + (uint32_t)(grp >> 2);
            const uint32_t eb = (lds_u32(ex_a + (bi >> 2) * 128u) >> (24u - 8u * (bi & 3u))) & 0xFFu;
            const float scale = __uint_as_float(eb >= 7u ? (eb - 6u) << 23 : 0u);     // 2^(E - 133)
#pragma unroll
            for (int b = 0; b < NB; ++b) { acc[b] = fmaf(blk[b], scale, acc[b]); blk[b] = 0.f; }
        }
    };
    int grp = 0;
    for (; grp < n_full; ++grp) group(grp, std::false_type{});
    for (; grp < n_groups; ++grp) group(grp, std::true_type{});
}

// T >= 0: fast path for regular chunks, generic path otherwise.  T = -1: generic path only (any t).
// T = 104: Cassandra-2 blob with t = 4 (fast path); T = -2: Cassandra-2 blob, generic path (any t).
// grid = (n_seg, G): CTA (seg, j) handles the superblocks (rb, seg) for rb = j, j + G, ...
// NB vectors x[b] (bf16 [NB][k]) are multiplied in the same pass: every decoded weight is used NB times, and each
// vector's sums are formed in the same order as with NB = 1.
// out = 1: the matrix is one segment wide, a sum is the result.  out = 2: the n_seg CTAs of a row block are a cluster with one
// tile each, and the first adds the others' sums in segment order.  (A kernel of its own for these additions costs a launch,
// 2 us of the 10 us that a small matrix takes.)  out = 0: only `partial` is written.
// A thread whose wait for a copy runs out leaves the kernel: threads that have left hold up neither __syncthreads nor their
// warp's exchanges, and the others run out of their own waits in turn.  With out = 2 it must still meet its CTA and the cluster:
// its warp goes on through the one tile as one of no values (the results are then void, as the status says).
// Launch bounds: a blob may have chunks for 1024 threads, and the compiler then likes to fit two such CTAs, 32 registers a thread.
// Told that one is enough it takes 48 to 55 for two Cassandra-2 vectors, whose walk does not fit 32 without a spill (5120 x 13824:
// 37 to 39 us at 32 registers, as the rest of the kernel falls, 34.7 so).
template <int T, int NB, bool WIDE, bool PAIRS>
__global__ void __launch_bounds__(1024, T == 104 && NB == 2 ? 1 : 0) k_draft_gemv(const uint32_t* __restrict__ blob, const uint16_t* __restrict__ x,
                                                     float* __restrict__ partial, int32_t* __restrict__ d_status,
                                                     int stage_bytes, int max_sb, int n, int k, int t, int seg_cols,
                                                     int chunk_cols, int n_seg, int n_rb, unsigned long long blob_bytes,
                                                     int out, uint16_t* __restrict__ y_bf16, float* __restrict__ y_f32) {
    extern __shared__ __align__(512) uint8_t smem_raw[];
    __shared__ float s_sum[NB][32];                     // out = 2: this segment's sums
    const int lane = threadIdx.x & 31;
    auto store = [&](int b, int row, float sum) {
        if (y_f32) y_f32[(size_t)b * n + row] = sum;
        if (y_bf16) y_bf16[(size_t)b * n + row] = float_to_bf16_bits(sum);
    };
    auto result = [&](int b, int row, float sum) {      // a segment's sum of one row
        if (out == 1) store(b, row, sum);
        else if (out == 2) s_sum[b][lane] = sum;
    };
    auto tiles = [&]() -> bool {
        // The geometry comes from the host's copy of the header (the launch sized shared memory from it); the header
        // itself is fetched now and compared once it has arrived, so that its latency is off the critical path.
        const uint32_t* h = blob;
        uint32_t hw[9] = {};                                   // thread 32: what the header says, and what it should
        const uint32_t want[9] = {(uint32_t)n, (uint32_t)k, (uint32_t)t, (uint32_t)seg_cols, (uint32_t)chunk_cols, (uint32_t)n_seg, (uint32_t)n_rb,
                                  kBlobMagic, (T == 104 || T == -2) ? kBlobModeMx : kBlobModeUnary};
        const bool checks = threadIdx.x == (blockDim.x > 32 ? 32u : 0u);
        if (checks) {
            const int at[9] = {H_ROWS, H_COLS, H_T, H_SEG, H_CHUNK, H_NSEG, H_NRB, H_MAGIC, H_MODE};
#pragma unroll
            for (int i = 0; i < 9; ++i) hw[i] = __ldg(h + at[i]);
        }
        const int k_pad = ceil_div(k, 32) * 32;
        const int seg = blockIdx.x, rb0 = blockIdx.y, rb_step = gridDim.y;
        const int tid = threadIdx.x, warp = tid >> 5, n_warps = blockDim.x >> 5;

        constexpr bool kCompact = gemv_compact(NB);
        uint8_t* stage0 = smem_raw + (kCompact ? x_slice_bytes(seg_cols, NB) : 0u);
        float* xs = reinterpret_cast<float*>(kCompact ? smem_raw : smem_raw + (size_t)kGemvStages * stage_bytes);
        uint32_t* lut = reinterpret_cast<uint32_t*>(kCompact ? stage0 + (size_t)kGemvStages * stage_bytes
                                                             : reinterpret_cast<uint8_t*>(xs) + (size_t)(seg_cols + kXSlack) * x_col_bytes(NB));
        float* red = kCompact ? reinterpret_cast<float*>(stage0) : reinterpret_cast<float*>(lut + 256);      // NB = 1: [turn][n_warps][32], else [NB][n_warps][32]
        uint64_t* bar = reinterpret_cast<uint64_t*>(lut + 256 + (kCompact ? 0 : 2 * n_warps * 32));    // [kGemvStages]
        const int x_cols = kCompact ? seg_cols : seg_cols + kXSlack;
        __shared__ int s_skip[kGemvStages], s_bad;
        __shared__ uint32_t s_dir[kGemvStages][3];          // sizes of the tile in each stage

        const int scols = seg_cols_of(k_pad, seg_cols, seg);
        const int n_ch = scols == seg_cols ? (int)blockDim.x / 32 : ceil_div(scols, chunk_cols);
        // The launch sized shared memory from the host's copy of the header; a blob that does not match it is
        // refused instead of overrunning the buffers.
        if (seg >= n_seg || (int)blockDim.x < 32 * n_ch || n_ch > 32 || (T == 104 && (smem_u32(lut) & 63u)) ||
            (smem_u32(xs) & (32u * x_col_bytes(NB) - 1u))) {
            if (tid == 0 && d_status) atomicExch(d_status, CASS_ERR_INVALID_ARG);
            return false;
        }
        const int n_tiles = rb0 >= n_rb ? 0 : rb_step >= n_rb ? 1 : (n_rb - rb0 + rb_step - 1) / rb_step;

        if (tid == 0) {
            for (int s = 0; s < kGemvStages; ++s) mbar_init(&bar[s], 1);
            fence_mbar_init();
        }
        __syncthreads();

        // thread 0: start the copy of tile i into stage i % kGemvStages.  Nothing is read beyond blob + blob_bytes (the
        // size the caller's description gives): a directory entry that points outside is skipped and flagged.
        auto issue = [&](int i) {
            const int s = i % kGemvStages;
            const int sb_i = (rb0 + i * rb_step) * n_seg + seg;
            const uint32_t* dir = blob + kBlobDirOffset / 4 + sb_i * 4;
            const bool dir_ok = (unsigned long long)kBlobDirOffset + ((unsigned long long)sb_i + 1ull) * 16ull <= blob_bytes;
            const uint32_t d0 = dir_ok ? dir[0] : 0u, d1 = dir_ok ? dir[1] : 0u, d2 = dir_ok ? dir[2] : 0u, d3 = dir_ok ? dir[3] : 0u;
            const SbGeom g = SbGeom::make(dir_n_ch(d3), scols, (int)d1, (int)d2);
            const uint32_t bytes = (uint32_t)g.total * 4u;
            if (!dir_ok || bytes > (uint32_t)max_sb || dir_n_ch(d3) != n_ch || d1 > 0xFFFFu || d2 > 0xFFFFu ||
                (unsigned long long)d0 * 16ull + bytes > blob_bytes) {                // does not fit: skip the tile, flag it
                s_skip[s] = 1;
                if (d_status) atomicExch(d_status, CASS_ERR_INVALID_ARG);
                mbar_expect_tx(&bar[s], 0);
                return;
            }
            s_skip[s] = 0;
            s_dir[s][0] = d1; s_dir[s][1] = d2; s_dir[s][2] = d3;
            const uint8_t* src = reinterpret_cast<const uint8_t*>(blob) + (size_t)d0 * 16;
            uint8_t* dst = stage0 + (size_t)s * stage_bytes;
            mbar_expect_tx(&bar[s], bytes);
            for (uint32_t off = 0; off < bytes; off += 32768u) bulk_g2s(dst + off, src + off, min(32768u, bytes - off), &bar[s]);
        };
        if (tid == 0) {
            for (int i = 0; i < kGemvStages && i < n_tiles; ++i) issue(i);
        }
        // the rank -> exponent table, pre-shifted into place
        const uint8_t* cb = reinterpret_cast<const uint8_t*>(blob) + kBlobHeaderBytes;
        if (T == 104) {
            // signed magnitudes of the 16 field values, as floats: (+-) (m << 4)
            if (tid < 16) reinterpret_cast<float*>(lut)[tid] = (tid & 8 ? -16.f : 16.f) * (float)(tid & 7);
        } else {
            for (int i = tid; i < 256; i += blockDim.x) lut[i] = (uint32_t)cb[i] << 23;
        }
        if (checks) {
            bool bad = false;
#pragma unroll
            for (int i = 0; i < 9; ++i) bad = bad || hw[i] != want[i];
            s_bad = bad;
        }
        // Everything above reads only the blob, ahead of the wait for the predecessor: a blob is complete before it is multiplied
        // with.  Its writers are the encoder (k_directory and k_pack; its caller then asks for the blob's description, a call that
        // synchronises) and a caller's copy of it, which in a session lies behind the embedding and the norm before the first
        // projection.  x and the scratch `partial` are the predecessor's.
        pdl_wait();
        pdl_early<6>();
        // x of this segment, zero beyond the matrix: eight columns of one vector a thread and turn.  (One value a turn where rows are off
        // 16-byte boundaries, each turn a round trip: 17 us a call for 700 x 3000 and four vectors, 13 so; 28 and 17 for 2000 x 1500 and eight.)
        const int c0 = seg * seg_cols, n_items = x_cols / 8 * NB;
        auto put8 = [&](int it, const uint4& v) {
            const int i = it / NB * 8;
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            if constexpr (NB == 1) {                           // fp32
                *reinterpret_cast<float4*>(xs + i) = make_float4(__uint_as_float(w[0] << 16), __uint_as_float(w[0] & 0xFFFF0000u),
                                                                 __uint_as_float(w[1] << 16), __uint_as_float(w[1] & 0xFFFF0000u));
                *reinterpret_cast<float4*>(xs + i + 4) = make_float4(__uint_as_float(w[2] << 16), __uint_as_float(w[2] & 0xFFFF0000u),
                                                                     __uint_as_float(w[3] << 16), __uint_as_float(w[3] & 0xFFFF0000u));
            } else {                                           // packed bf16 [col][NB]: all vectors' values of one column side by side
                uint16_t* xs16 = reinterpret_cast<uint16_t*>(xs) + (size_t)i * NB + it % NB;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    xs16[2 * q * NB] = (uint16_t)(w[q] & 0xFFFFu);
                    xs16[(2 * q + 1) * NB] = (uint16_t)(w[q] >> 16);
                }
            }
        };
        const bool x_vec = (k & 7) == 0 && ((uintptr_t)x & 15) == 0;
        auto get8 = [&](int it, bool vec) {
            const int i = it / NB * 8, left = min(scols - i, k - c0 - i);
            const uint16_t* p = x + (size_t)(it % NB) * k + c0 + i;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (vec) {
                if (left > 0) v = __ldg(reinterpret_cast<const uint4*>(p));
            } else {
                uint32_t h[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) h[j] = j < left ? (uint32_t)__ldg(p + j) : 0u;
                v = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
            }
            return v;
        };
        if constexpr (NB == 1) {
            for (int it = tid; it < n_items; it += blockDim.x) put8(it, get8(it, x_vec));
        } else if (x_vec) {                                    // two turns' loads under way
            for (int it = tid; it < n_items; it += 2 * blockDim.x) {
                uint4 v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int at = it + u * blockDim.x, i = at / NB * 8;
                    v[u] = make_uint4(0u, 0u, 0u, 0u);
                    if (i < scols && c0 + i < k && at < n_items) v[u] = __ldg(reinterpret_cast<const uint4*>(x + (size_t)(at % NB) * k + c0 + i));
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (u == 0 || it + u * blockDim.x < n_items) put8(it + u * blockDim.x, v[u]);
            }
        } else {
#pragma unroll 1
            for (int it = tid; it < n_items; it += blockDim.x) put8(it, get8(it, false));
        }
        __syncthreads();
        if (s_bad) {
            // not the blob the caller described: flag it, let the copies already started land, produce nothing
            if (tid == 0 && d_status) atomicExch(d_status, CASS_ERR_INVALID_ARG);
            for (int j = 0; j < n_tiles && j < kGemvStages; ++j) mbar_wait_bounded(&bar[j % kGemvStages], 0u);
            return false;
        }

        for (int i = 0; i < n_tiles; ++i) {
            const int s = i % kGemvStages;
            const int rb = rb0 + i * rb_step;
            bool lost = false;
            if (!mbar_wait_bounded(&bar[s], (uint32_t)(i / kGemvStages) & 1u)) {
                // give up: flag the error, let the copies still in flight into this CTA's buffers land (bounded), leave
                if (d_status) atomicExch(d_status, CASS_ERR_TIMEOUT);
                for (int j = i; j < n_tiles && j < i + kGemvStages; ++j)
                    mbar_wait_bounded(&bar[j % kGemvStages], (uint32_t)(j / kGemvStages) & 1u);
                if (out != 2) return false;
                lost = true;
            }
            lost = __any_sync(0xffffffffu, lost);
            const uint32_t* sb = reinterpret_cast<const uint32_t*>(stage0 + (size_t)s * stage_bytes);
            float acc[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[b] = 0.f;
            if (warp < n_ch && !s_skip[s]) {
                const uint32_t* dir = s_dir[s] - 1;                   // written before the copy was started; its arrival orders the read
                const SbGeom g = SbGeom::make(n_ch, scols, (int)dir[1], (int)dir[2]);
                const int elems = lost ? 0 : dir_chunk_elems(dir[3]);
                if (T == 104) {
                    chunk_dot_mx4<NB, WIDE, PAIRS>(sb, g, warp, lane, elems, xs, reinterpret_cast<const float*>(lut), acc);
                } else if (T == -2) {
                    const uint32_t xs_a = smem_u32(xs);
                    decode_chunk_generic_mx(sb, g, elems, warp, lane, t, [&](int col, uint16_t bits) {
                        x_fma<NB, PAIRS>(x_load<NB>(xs_a + (uint32_t)col * (uint32_t)x_col_bytes(NB)), (uint32_t)bits << 16, acc);
                    });
                } else if (T >= 0) {
                    chunk_dot_fast<(T >= 0 && T <= 5 ? T : 0), NB, WIDE, PAIRS>(sb, g, warp, lane, elems, xs, lut, acc);
                } else {
                    const uint32_t xs_a = smem_u32(xs);
                    decode_chunk_generic(sb, g, elems, warp, lane, t, cb, [&](int col, uint16_t bits) {
                        x_fma<NB, PAIRS>(x_load<NB>(xs_a + (uint32_t)col * (uint32_t)x_col_bytes(NB)), (uint32_t)bits << 16, acc);
                    });
                }
            }
            const size_t n_pad = (size_t)n_rb * kRowsPerBlock;
            const int row = rb * kRowsPerBlock + lane;
            if constexpr (NB == 1) {
                float* red_i = red + (i & 1) * n_warps * 32;
                red_i[warp * 32 + lane] = acc[0];
                __syncthreads();                              // all reads of stage s are done; partial sums are visible
                if (tid == 0 && i + kGemvStages < n_tiles) {
                    fence_proxy_async();
                    issue(i + kGemvStages);
                }
                if (warp == 0) {
                    float sum = 0.f;
                    for (int w = 0; w < n_ch; ++w) sum += red_i[w * 32 + lane];
                    if (row < n) {
                        partial[(size_t)seg * n_pad + row] = sum;
                        result(0, row, sum);
                    }
                }
            } else {
                static_assert(kGemvStages == 1, "the sums take the place of the superblock that was read");
                if (kCompact) __syncthreads();                // all reads of it are done
#pragma unroll
                for (int b = 0; b < NB; ++b) red[(b * n_warps + warp) * 32 + lane] = acc[b];
                __syncthreads();
                if (!kCompact && tid == 0 && i + 1 < n_tiles) {
                    fence_proxy_async();
                    issue(i + 1);
                }
                for (int b = warp; b < NB; b += n_warps) {    // vector b's chunk sums, added in chunk order as with NB = 1
                    float sum = 0.f;
                    for (int w = 0; w < n_ch; ++w) sum += red[(b * n_warps + w) * 32 + lane];
                    if (row < n) {
                        partial[((size_t)b * n_seg + seg) * n_pad + row] = sum;
                        result(b, row, sum);
                    }
                }
                if (i + 1 < n_tiles) {
                    __syncthreads();                          // the sums are read before the next tile overwrites them
                    if (kCompact && tid == 0) {
                        fence_proxy_async();
                        issue(i + 1);
                    }
                }
            }
        }
        return true;
    };
    const bool done = tiles();
    if (out != 2) return;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();                                     // every CTA comes here, also one that gave up
    // Vector b by warp b, or the one vector by the first warp without a loop: the same additions, but the time of the whole kernel differs by more
    // than they take, and each instantiation has the faster one.  Loop / first warp, more than 52 % pruned: 512 x 512 at 53 % 6.2 / 4.6 us, 28672
    // x 4096 at 60 % 41.0 / 39.2; else 28672 x 4096 at t = 4 47.8 / 48.1, t = 0 49.8 / 50.3, t = 6 397 / 420, Cassandra-2 39.15 / 39.46, but
    // t = 1 73.7 / 69.3, t = 2 93.4 / 91.3, t = 5 (30 %) 101.8 / 100.1, and 4096 x 4096 at t = 3 24.8 / 24.5.
    constexpr bool kByWarps = NB > 1 || (!WIDE && T != 1 && T != 2 && T != 3 && T != 5);
    if (done && cluster.block_rank() == 0 && (kByWarps || threadIdx.x < 32)) {
        const int row = (int)blockIdx.y * kRowsPerBlock + lane;
        for (int b = kByWarps ? (int)threadIdx.x >> 5 : 0; b < NB; b += kByWarps ? (int)blockDim.x >> 5 : 1) {
            float part[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) part[s] = *cluster.map_shared_rank(&s_sum[b][lane], min(s, n_seg - 1));
            float sum = 0.f;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < n_seg) sum += part[s];
            if (row < n) store(b, row, sum);
        }
    }
    cluster.sync();                                     // nobody leaves while its sums may be read
}

// grid.y = vector b: partial [b][n_seg][n_pad] -> y [b][n]
__global__ void k_gemv_finish(const float* __restrict__ partial, int n, int n_pad, int n_seg,
                              uint16_t* __restrict__ y_bf16, float* __restrict__ y_f32) {
    pdl_launch_dependents();
    pdl_wait();
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int b = blockIdx.y;
    partial += (size_t)b * n_seg * n_pad;
    float acc = 0.f;
    for (int s = 0; s < n_seg; ++s) acc += partial[(size_t)s * n_pad + r];
    if (y_f32) y_f32[(size_t)b * n + r] = acc;
    if (y_bf16) y_bf16[(size_t)b * n + r] = float_to_bf16_bits(acc);
}

// y_bf16 / y_f32 (either may be null): [nb][rows] results.  Both null: only `partial`, which the caller's next kernel adds.
static int launch_gemv(const void* blob, const cass_blob_info& bi, const void* x_bf16, int nb, float* partial, uint16_t* y_bf16,
                       float* y_f32, int32_t* d_status, cudaStream_t stream) {
    const int n_ch = ceil_div(bi.seg_cols, bi.chunk_cols);
    if (n_ch > 32) return CASS_ERR_UNSUPPORTED;
    if (nb != 1 && nb != 2 && nb != 4 && nb != 8) return CASS_ERR_UNSUPPORTED;
    size_t smem = gemv_smem_bytes(bi, nb);
    const size_t total = smem + gemv_smem_static(nb);
    if (gemv_smem_total(bi, nb) > kSmemPerBlock) return CASS_ERR_CAPACITY;
    const int threads = 32 * n_ch;
    // One vector: one CTA per superblock -- the hardware hands out CTAs as shared memory frees, which balances the SMs to
    // within one superblock (a grid of as many CTAs as fit at once, each looping over its share, left SMs with 4 x 4
    // superblocks beside SMs with 4 x 3: 56.7 instead of 54.4 us on the 28672 x 4096 matrix).  Several vectors: the x
    // slice a CTA stages is nb times larger, so CTAs keep theirs and loop (one CTA per superblock: 52.3 instead of
    // 48.6 ms per step with 8 sequences).
    int g = bi.n_rowblocks, per_sm = (int)((228 * 1024) / (total + 1024));                 // CTAs an SM holds
    if (per_sm > 2048 / threads) per_sm = 2048 / threads;
    if (per_sm < 1) per_sm = 1;
    if (nb > 1) {
        g = ceil_div(kSms * per_sm, bi.n_seg);
        if (g > bi.n_rowblocks) g = bi.n_rowblocks;
    }
    if (g < 1) g = 1;
    // three of these CTAs fit an SM; a grid of up to two an SM is kept from sitting three on some: 4096 x 4096, eight Cassandra-2 vectors 24 and 32 us
    if (nb >= 4 && bi.n_seg * g > kSms && bi.n_seg * g <= 2 * kSms && smem < kSmemPerBlock / 3) smem = kSmemPerBlock / 3;
    // Results inside the kernel where the segments of a row block are one CTA, or a cluster of CTAs with one tile each and the
    // grid fills at most three quarters of the chip: a cluster starts only when all of its CTAs have room, which leaves SMs
    // idle where CTAs queue (12613 x 5686 at t = 0: 57.4 us, 47.0 with the finishing kernel; 4096 x 14336: 31.5 and 28.7;
    // against that 1000 x 3000: 8.6 and 8.9, 2000 x 11000: 17.9 and 18.4).
    const bool want = y_bf16 || y_f32;
    const bool room = 4ll * bi.n_seg * g <= 3ll * kSms * (nb >= 4 && per_sm > 2 ? 2 : per_sm);
    const int out = !want ? 0 : bi.n_seg == 1 ? 1 : (bi.n_seg <= 8 && g == bi.n_rowblocks && room) ? 2 : 0;
    // with q = 1 - p kept, 8 kept columns span 8 / q columns, give or take sqrt(8 p) / q: more than 32 about once in 10^4 groups
    // of a lane at p = 50 %, once in 40 at 60 %, and one lane's long gap costs its warp a careful walk (359 x 1467 at p = 60 %:
    // 26 us without the second window, 12.8 with it)
    const bool wide = bi.prune_permille > 520;
    const bool pairs2 = bi.n_seg * bi.n_rowblocks > 2 * kSms;
    dim3 grid(bi.n_seg, g), block(threads);
    const uint32_t* b = (const uint32_t*)blob;
    const uint16_t* x = (const uint16_t*)x_bf16;
    const int stage = (int)gemv_stage_bytes(bi, nb);
#define CASS_GEMV_LAUNCH(TT, NN, WW, PP)                                                                         \
    do {                                                                                                       \
        CASS_ALLOW_SMEM(k_draft_gemv<TT, NN, WW, PP>);                                                             \
        cudaLaunchConfig_t cfg = {};                                                                           \
        cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;            \
        cudaLaunchAttribute at[2];                                                                             \
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   /* prologue may overlap the predecessor */ \
        at[0].val.programmaticStreamSerializationAllowed = pdl_enabled();                                                  \
        at[1].id = cudaLaunchAttributeClusterDimension;                                                        \
        at[1].val.clusterDim.x = bi.n_seg; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;             \
        cfg.attrs = at; cfg.numAttrs = out == 2 ? 2 : 1;                                                       \
        CASS_CUDA_CHECK(cudaLaunchKernelEx(&cfg, k_draft_gemv<TT, NN, WW, PP>, b, x, partial, d_status, stage,         \
                                           (int)bi.max_superblock_bytes, (int)bi.rows, (int)bi.cols,           \
                                           (int)bi.trunc_bits, (int)bi.seg_cols, (int)bi.chunk_cols,           \
                                           (int)bi.n_seg, (int)bi.n_rowblocks,                                 \
                                           (unsigned long long)bi.total_bytes, out, y_bf16, y_f32));     \
    } while (0)
#define CASS_GEMV_LAUNCH_NB(TT)                                                                                \
    do {                                                                                                       \
        constexpr bool kHasWide = TT >= 0;          /* the generic decoders search any distance */               \
        constexpr bool kPairs2 = TT == 4;           /* two vectors: pairs where superblocks abound */            \
        if (wide && kHasWide) {                                                                                \
            if (nb == 1) CASS_GEMV_LAUNCH(TT, 1, kHasWide, false);                                             \
            else if (nb == 2 && pairs2 && kPairs2) CASS_GEMV_LAUNCH(TT, 2, kHasWide, kPairs2);                   \
            else if (nb == 2) CASS_GEMV_LAUNCH(TT, 2, kHasWide, false);                                        \
            else if (nb == 4) CASS_GEMV_LAUNCH(TT, 4, kHasWide, true);                                         \
            else CASS_GEMV_LAUNCH(TT, 8, kHasWide, true);                                                      \
        } else if (nb == 1) CASS_GEMV_LAUNCH(TT, 1, false, false);                                             \
        else if (nb == 2 && pairs2 && kPairs2) CASS_GEMV_LAUNCH(TT, 2, false, kPairs2);                          \
        else if (nb == 2) CASS_GEMV_LAUNCH(TT, 2, false, false);                                               \
        else if (nb == 4) CASS_GEMV_LAUNCH(TT, 4, false, true);                                                \
        else CASS_GEMV_LAUNCH(TT, 8, false, true);                                                             \
    } while (0)
    if (bi.mode == 2 && bi.trunc_bits == 4) CASS_GEMV_LAUNCH_NB(104);
    else if (bi.mode == 2) CASS_GEMV_LAUNCH_NB(-2);
    else if (bi.trunc_bits == 4) CASS_GEMV_LAUNCH_NB(4);
    else if (bi.trunc_bits == 0) CASS_GEMV_LAUNCH_NB(0);
    else if (bi.trunc_bits == 1) CASS_GEMV_LAUNCH_NB(1);          // fields that do not tile a word: the design-space sweep of Sec. 7.2
    else if (bi.trunc_bits == 2) CASS_GEMV_LAUNCH_NB(2);
    else if (bi.trunc_bits == 3) CASS_GEMV_LAUNCH_NB(3);
    else if (bi.trunc_bits == 5) CASS_GEMV_LAUNCH_NB(5);
    else CASS_GEMV_LAUNCH_NB(-1);
#undef CASS_GEMV_LAUNCH_NB
#undef CASS_GEMV_LAUNCH
    CASS_LAUNCH_CHECK();
    if (want && out == 0) {
        const int n_pad = bi.n_rowblocks * kRowsPerBlock;
        CASS_PDL_LAUNCH(k_gemv_finish, dim3(ceil_div(bi.rows, 256), nb), dim3(256), 0, stream, (const float*)partial, (int)bi.rows, n_pad,
                        (int)bi.n_seg, y_bf16, y_f32);
    }
    return CASS_OK;
}

int launch_draft_gemv(const void* blob, const cass_blob_info& bi, const void* x_bf16, int nb, float* partial,
                      int32_t* d_status, cudaStream_t stream) {
    return launch_gemv(blob, bi, x_bf16, nb, partial, nullptr, nullptr, d_status, stream);
}

}  // namespace cass

using namespace cass;

extern "C" int cass_draft_gemv(const void* blob, const cass_blob_info* h_info, const void* x_bf16, float* partial,
                               void* y_bf16, float* y_f32, int32_t* d_status, void* stream) {
    if (!blob || !h_info || !x_bf16 || !partial) return CASS_ERR_INVALID_ARG;
    return launch_gemv(blob, *h_info, x_bf16, 1, partial, (uint16_t*)y_bf16, y_f32, d_status, (cudaStream_t)stream);
}

extern "C" int cass_draft_gemv_batch(const void* blob, const cass_blob_info* h_info, const void* x_bf16, int n_vec,
                                     float* partial, void* y_bf16, float* y_f32, int32_t* d_status, void* stream) {
    if (!blob || !h_info || !x_bf16 || !partial) return CASS_ERR_INVALID_ARG;
    if (n_vec != 1 && n_vec != 2 && n_vec != 4 && n_vec != 8) return CASS_ERR_INVALID_ARG;
    return launch_gemv(blob, *h_info, x_bf16, n_vec, partial, (uint16_t*)y_bf16, y_f32, d_status, (cudaStream_t)stream);
}

// ---- variant with built-in scratch ------------------------------------------------------------------------
// The split-K partial sums of this variant live in a fixed array inside the library image, so the call needs no
// scratch buffer from its caller.  Every GPU that loads the library holds the array (2 MiB) until the process ends.
static __device__ __align__(256) float g_static_partial[CASS_STATIC_PARTIAL_FLOATS];

extern "C" int cass_draft_gemv_static(const void* blob, const cass_blob_info* h_info, const void* x_bf16, void* y_bf16,
                                      float* y_f32, int32_t* d_status, void* stream_) {
    if (!blob || !h_info || !x_bf16 || (!y_bf16 && !y_f32)) return CASS_ERR_INVALID_ARG;
    if (h_info->n_seg <= 0 || h_info->n_rowblocks <= 0) return CASS_ERR_INVALID_ARG;
    const size_t need = (size_t)h_info->n_seg * h_info->n_rowblocks * kRowsPerBlock;
    if (need > (size_t)CASS_STATIC_PARTIAL_FLOATS) return CASS_ERR_CAPACITY;     // matrix too large for the built-in scratch
    // In host code the array's name is only a handle; its device address is looked up once per device, with that
    // device current, and kept.
    constexpr int kMaxDevices = 64;
    static float* s_scratch[kMaxDevices] = {nullptr};
    int dev = -1;
    CASS_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return CASS_ERR_UNSUPPORTED;
    if (!s_scratch[dev]) {
        float* ptr = nullptr;
        if (cudaGetSymbolAddress((void**)&ptr, g_static_partial) != cudaSuccess || !ptr) return CASS_ERR_CUDA;
        s_scratch[dev] = ptr;
    }
    float* partial = s_scratch[dev];
    return launch_gemv(blob, *h_info, x_bf16, 1, partial, (uint16_t*)y_bf16, y_f32, d_status, (cudaStream_t)stream_);
}
