// Forming one record of the compressed KV cache with one warp: lane holds channels lane + 32 j of the token's row.  Shared by the
// encoder of a decode step's rows (kv.cu) and the one of spans of tokens (kv_span.cu).
#pragma once

#include "kernels.cuh"

namespace cass {

// lane holds elements lane + 32 j.  bm[j] (the same in every lane): bit `lane` set for the kept ones, the d - n_prune
// largest |x| (ties: the lower channel is pruned first).  Keys (|x| bits, channel) are unique; a threshold with exactly
// n_prune keys below it is searched two bits at a time (three counts packed into one reduction) and the search ends with
// the first one found.  It starts six binades below the largest value, where the threshold of an ordinary row lies, and
// from zero if too many keys lie below that.
template <int NJ>
__device__ __forceinline__ void kv_select(const uint32_t (&bits)[NJ], int nj, int n_prune, int lane, uint32_t (&bm)[NJ]) {
    uint32_t key[NJ], big = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        key[j] = j < nj ? (((bits[j] & 0x7FFFu) << 8) | (uint32_t)(lane + 32 * j)) : 0xFFFFFFFFu;
        big = j < nj ? max(big, key[j]) : big;
    }
    uint32_t thr = 0;
    if (n_prune > 0) {
        big = __reduce_max_sync(0xffffffffu, big);
        int bit = 20;                                                   // the next two bits to decide: bit + 1 and bit
        uint32_t base = 0;
        bool done = false;
        if (big >= (6u << 15)) {
            uint32_t c = 0;
            const uint32_t low = big - (6u << 15);
#pragma unroll
            for (int j = 0; j < NJ; ++j) c += key[j] < low;
            c = __reduce_add_sync(0xffffffffu, c);
            if ((int)c <= n_prune) { base = low; bit = 16; done = (int)c == n_prune; }      // within 6 x 2^15 < 2^18 of it
        }
        if (base == 0) {                                                // 23 key bits: the top one alone
            uint32_t c = 0;
#pragma unroll
            for (int j = 0; j < NJ; ++j) c += key[j] < (1u << 22);
            if ((int)__reduce_add_sync(0xffffffffu, c) <= n_prune) base = 1u << 22;
        }
        thr = base;
#pragma unroll 1
        for (; bit >= 0 && !done; bit -= 2) {
            const uint32_t c1 = thr + (1u << bit), c2 = thr + (2u << bit), c3 = thr + (3u << bit);
            uint32_t c = 0;                                             // three counts of at most 256 each in one word
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                c += (uint32_t)(key[j] < c1) + ((uint32_t)(key[j] < c2) << 10) + ((uint32_t)(key[j] < c3) << 20);
            c = __reduce_add_sync(0xffffffffu, c);
            const int n1 = (int)(c & 1023u), n2 = (int)((c >> 10) & 1023u), n3 = (int)(c >> 20);      // n1 <= n2 <= n3
            if (n3 <= n_prune) { thr = c3; done = n3 == n_prune; }
            else if (n2 <= n_prune) { thr = c2; done = n2 == n_prune; }
            else if (n1 <= n_prune) { thr = c1; done = n1 == n_prune; }
        }
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) bm[j] = __ballot_sync(0xffffffffu, j < nj && key[j] >= thr);
}

// Code lengths of a record's slices -> entry words and arena words (R: raw exponents where the codes take more room).
template <int NJ>
__device__ __forceinline__ uint32_t kv_entries(const KvGeom& g, const uint32_t (&len)[NJ], int nj, uint32_t (&entry)[3]) {
    uint32_t ub = 0;
    entry[0] = entry[1] = entry[2] = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        if (j >= nj) break;
        if (j > 0) entry[(j - 1) / 3] |= (ub & 0x3FFu) << (20 - 10 * ((j - 1) % 3));
        ub += __reduce_add_sync(0xffffffffu, len[j]);
    }
    if (ub > (uint32_t)kv_code_budget(g.kept)) {
        entry[0] = kKvRawFlag; entry[1] = entry[2] = 0;
        return (uint32_t)ceil_div(g.kept, 4);
    }
    return (ub + 31) / 32;
}

// The codewords' terminating ones into una (64 words, zero): a slice has at most 1023 code bits where codes are stored, so the
// scans of two slices share a word.
template <int NJ>
__device__ __forceinline__ void kv_code_bits(const uint32_t (&len)[NJ], int nj, int lane, uint32_t* una) {
    uint32_t base = 0;
#pragma unroll
    for (int j = 0; j < NJ; j += 2) {
        if (j >= nj) break;
        uint32_t incl = len[j] | (len[j + 1] << 16);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t p = base + (incl & 0xFFFFu) - 1u, q = base + (all & 0xFFFFu) + (incl >> 16) - 1u;
        if (len[j]) atomicOr(&una[(p >> 5) & 63u], 0x80000000u >> (p & 31));
        if (len[j + 1]) atomicOr(&una[(q >> 5) & 63u], 0x80000000u >> (q & 31));
        base += (all & 0xFFFFu) + (all >> 16);
    }
}

// Sign and kept mantissa bits of one value; MX (Cassandra-2): sign and magnitude in the unit of its 32-channel slice, whose shared
// exponent is E (0 otherwise).
template <int T>
__device__ __forceinline__ uint32_t kv_field(uint32_t bits, bool keep, bool mx, uint32_t& E) {
    E = 0;
    if (!mx) return ((bits >> 15) << (7 - T)) | ((bits & 0x7Fu) >> T);
    const uint32_t e = (bits >> 7) & 0xFFu;
    E = __reduce_max_sync(0xffffffffu, keep ? e : 0u);
    const uint32_t sh = 1u + E - e;
    const uint32_t m7 = (sh < 8u && e > 0u && E >= 7u) ? ((0x80u | (bits & 0x7Fu)) >> sh) : 0u;
    return ((bits >> 15) << (7 - T)) | (m7 >> T);
}

// The record's field words from its kept values' fields, one byte each (room up to the next multiple of 8).
template <int T>
__device__ __forceinline__ void kv_field_words(const KvGeom& g, const uint8_t* fld, uint32_t* words, int lane) {
    constexpr int F = 8 - T, PER = 32 / F;
    for (int w = lane; w < g.f_words; w += 32) {
        uint32_t acc = 0;
#pragma unroll
        for (int q = 0; q < PER; q += 4) {
            const uint32_t four = *reinterpret_cast<const uint32_t*>(&fld[w * PER + q]);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t f = (four >> (8 * b)) & 0xFFu;
                const uint32_t v = g.mode == 2 ? f << (32 - F * (q + b + 1)) : field_bits_in_word(f, q + b, T);
                acc |= w * PER + q + b < g.kept ? v : 0u;
            }
        }
        words[w] = acc;
    }
}

}  // namespace cass
