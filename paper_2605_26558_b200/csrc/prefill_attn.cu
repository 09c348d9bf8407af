// Causal attention of a prefill pass over the bf16 cache (Sec. 2.2) for head_dim 128, with the bits of the verification attention and
// its merge (verify_attn_tc.cu, draft_attn.cu): those cut the positions into chunks of 128, leave every chunk's maximum m, sum l and
// output o in memory, and add w_c o_c with w_c = exp(m_c - M) in a fixed order.  A pass of many rows needs no split over CTAs, so one
// CTA takes 128 (row, query head) pairs of a KV head through all of their chunks:
//   first   scores = Q K^T of every chunk -> m_c of every pair, hence M and all w_c
//   then    scores again, P = exp(scores - m_c) in bf16, l_c, o_c = P V, total += w_c o_c in the merge's order
// The scores are computed twice, which costs the tensor cores next to nothing, and no partial output leaves the SM.
// A pair is a lane of tensor memory and a thread: its 128 scores of a chunk are read 32 at a time, P goes back over them (the A
// operand of the second product comes from tensor memory), and no value crosses threads.  Two warpgroups take the chunks in turn and
// half of the output's dimensions each.  The sum l is formed in the order of the other kernel: four tokens 32 apart, then a tree.
// Bound: latency and issue (33 % of the slots with 8 warps at work): 1000 rows of 32 heads are 16 M exponentials, 28 instructions a score.
// 1000 rows of an 8B-shaped layer, cold: 62 us; the verification kernel and its merge took 210 (two launches of the scratch's
// room, 74 MB of partial outputs).  The heaviest CTAs first in the grid: 77 -> 62.
// 168 registers, what ten warps leave a thread; P in two terms spills 11 words.
#include "tc.cuh"
#include "kernels.cuh"

namespace cass {

constexpr int kPaTok = kPrefillChunk, kPaD = 128, kPaPairs = 128;
constexpr int kPaThreads = 320;                          // warp 0: TMA; warp 1: MMA issue and tensor memory; warps 2-5 and 6-9: softmax, output
constexpr int kPaTile = kPaTok * kPaD * 2;               // K, V or Q: two boxes of 128 x 64, 128-byte swizzle
constexpr int kPaSlots = 5;                              // tiles under way
constexpr int kPaSmem = (kPaSlots + 1) * kPaTile + 256 + 1024;
constexpr int kPaMaxChunks = 256;                        // the merge adds the sums of more in another order
constexpr uint32_t kPaS = 0, kPaO = 256;                 // tensor memory: two score (and P) buffers, two outputs, 128 columns each

__device__ __forceinline__ void pa_mma_tmem_a(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]),
                 "r"(v[13]), "r"(v[14]), "r"(v[15])
                 : "memory");
}
__device__ __forceinline__ void pa_arrive(uint64_t* bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory"); }

// What warp_sum gives for 32 lanes' values, in one thread.
__device__ __forceinline__ float tree_sum32(float (&v)[32]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) v[i] += v[i + o];
    return v[0];
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

struct PrefillAttn {
    int rps, n_q, n_kv, chunks, tile_rows, tiles, fine;     // rows a sequence; chunks the longest row sees; rows a CTA; CTAs a head and sequence
};

// grid: (KV heads, sequences, tiles), the last rows (most chunks) of all heads first.  stat_m, stat_l: [CTA][chunk][pair]; total_s (beyond 8 chunks):
// [CTA][dim][pair].  A role that gives up a wait flags the status and goes to the end; the others' waits run out in turn.
template <bool FINE>
__global__ void __launch_bounds__(kPaThreads, 1) k_prefill_attn(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                                                                const uint16_t* __restrict__ qkv, PrefillAttn pa, const DevState* __restrict__ st,
                                                                float* __restrict__ stat_m, float* __restrict__ stat_l, float* __restrict__ total_s,
                                                                uint16_t* __restrict__ out, int32_t* __restrict__ d_status) {
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    uint8_t *sQ = base, *sT = base + kPaTile;
    uint64_t* full = reinterpret_cast<uint64_t*>(sT + kPaSlots * kPaTile);
    uint64_t *empty = full + kPaSlots, *s_full = empty + kPaSlots;           // s_full: scores complete
    uint64_t *p_done = s_full + 2, *o_full = p_done + 2, *o_free = o_full + 2;      // p_done: scores read and (second time) P written
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(o_free + 2);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tile = pa.tiles - 1 - (int)blockIdx.z, head = blockIdx.x, seq = blockIdx.y;
    const int G = pa.n_q / pa.n_kv, first = tile * pa.tile_rows, rows = min(pa.tile_rows, pa.rps - first), P = rows * G;
    const int qkv_dim = (pa.n_q + 2 * pa.n_kv) * kPaD;
    if (tid == 0) {
        for (int i = 0; i < kPaSlots; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&s_full[b], 1); mbar_init(&p_done[b], 4); mbar_init(&o_full[b], 1); mbar_init(&o_free[b], 8); }
        fence_mbar_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    const int len = st->len[seq] + first;                                    // row r of the tile sits at position len + r
    const int n = ceil_div(len + rows, kPaTok);                              // chunks its last row sees
    if (warp >= 2) {
        // Q: pair p = row * G + head in the group, zero beyond P
        const uint16_t* q0 = qkv + ((size_t)seq * pa.rps + first) * qkv_dim + (size_t)head * G * kPaD;
        for (int i = tid - 64; i < kPaPairs * (kPaD / 8); i += kPaThreads - 64) {
            const int p = i / (kPaD / 8), c8 = i % (kPaD / 8);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (p < P) v = *reinterpret_cast<const uint4*>(q0 + (size_t)(p / G) * qkv_dim + (size_t)(p % G) * kPaD + c8 * 8);
            *reinterpret_cast<uint4*>(sQ + (c8 >> 3) * (kPaTile / 2) + p * 128 + (((c8 ^ p) & 7) << 4)) = v;
        }
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_early<4>();
    const uint32_t tmem = *tmem_slot;
    // The merge's order: chunk i of the second time is number i in the order c0, c0 + 8, c0 + 16, ... for c0 = 0 .. 7.
    const int chains = min(n, 8);
    auto next_chunk = [&](int c) { return c + 8 < n ? c + 8 : (c & 7) + 1; };

    if (warp == 0) {
        if (tc_elect()) {
            // tiles in the order of the MMAs: K of every chunk; then K of the first, and K of the next ahead of V of each
            int it = 0;
            bool ok = true;
            auto load = [&](const CUtensorMap* map, int c) {
                const int s = it % kPaSlots;
                ok = ok && mbar_wait_bounded(&empty[s], ((uint32_t)(it / kPaSlots) & 1u) ^ 1u);
                if (!ok) return;
                mbar_expect_tx(&full[s], kPaTile);
                tma_load_3d(sT + s * kPaTile, map, head * kPaD, c * kPaTok, seq, &full[s]);
                tma_load_3d(sT + s * kPaTile + kPaTile / 2, map, head * kPaD + 64, c * kPaTok, seq, &full[s]);
                ++it;
            };
            for (int c = 0; c < n; ++c) load(&map_k, c);
            for (int i = 0, c = 0; i <= n; ++i) {
                const int cn = i < n ? (i == 0 ? 0 : next_chunk(c)) : 0;
                if (i < n) load(&map_k, cn);
                if (i > 0) load(&map_v, c);
                c = cn;
            }
            if (!ok) atomicExch(d_status, CASS_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        if (tc_elect()) {
            int it = 0;
            bool ok = true;
            auto tile_in = [&]() -> uint8_t* {                               // the next tile, once it has arrived
                const int s = it % kPaSlots;
                ok = ok && mbar_wait_bounded(&full[s], (uint32_t)(it / kPaSlots) & 1u);
                tc_fence_after();
                return sT + s * kPaTile;
            };
            auto tile_out = [&]() { tc_commit(&empty[it % kPaSlots]); ++it; };
            auto scores = [&](int u) {
                const uint8_t* k = tile_in();
                if (!ok) return;
                constexpr uint32_t idesc = tc_idesc_mn(kPaPairs, kPaTok, false);
#pragma unroll
                for (int kb = 0; kb < 2; ++kb) {
                    const uint64_t ad = tc_smem_desc(sQ + kb * (kPaTile / 2)), bd = tc_smem_desc(k + kb * (kPaTile / 2));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma(tmem + kPaS + (u & 1) * 128, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc, (uint32_t)((kb | kk) != 0));
                }
                tile_out();
                tc_commit(&s_full[u & 1]);
            };
            auto output = [&](int i) {                                       // P of use n + i is in its buffer, the output buffer read
                const int u = n + i;
                ok = ok && mbar_wait_bounded(&p_done[u & 1], (uint32_t)(u >> 1) & 1u);
                if (i >= 2) ok = ok && mbar_wait_bounded(&o_free[i & 1], ((uint32_t)(i >> 1) & 1u) ^ 1u);
                const uint8_t* v = tile_in();
                if (!ok) return;
                constexpr uint32_t idesc = tc_idesc_mn(kPaPairs, kPaD, false) | (1u << 16);      // B: rows of tokens, contiguous along N
                const uint32_t d = tmem + kPaO + (i & 1) * 128, p = tmem + kPaS + (u & 1) * 128;
#pragma unroll
                for (int kk = 0; kk < kPaTok / 16; ++kk) {
                    const uint64_t bd = tc_smem_desc(v + kk * 2048, kPaTile / 2);
                    pa_mma_tmem_a(d, p + 32 * (kk >> 1) + 8 * (kk & 1), bd, idesc, (uint32_t)(kk != 0));
                    if (FINE) pa_mma_tmem_a(d, p + 32 * (kk >> 1) + 8 * (kk & 1) + 16, bd, idesc, 1u);
                }
                tile_out();
                tc_commit(&o_full[i & 1]);
            };
            for (int u = 0; u < 2 * n && ok; ++u) {
                // the buffer's use before is read: waited for with the output of that use the second time
                if (u >= 2 && u - 2 < n) ok = mbar_wait_bounded(&p_done[u & 1], (uint32_t)((u - 2) >> 1) & 1u);
                if (ok) scores(u);
                if (ok && u > n) output(u - 1 - n);
            }
            if (ok) output(n - 1);
            if (!ok) {
                atomicExch(d_status, CASS_ERR_TIMEOUT);
                for (int j = it; j < it + kPaSlots; ++j)                     // what is in flight lands before the CTA ends (bounded)
                    mbar_wait_bounded(&full[j % kPaSlots], (uint32_t)(j / kPaSlots) & 1u);
            }
        }
    } else {
        const int wg = (warp - 2) >> 2, q = warp & 3, p = q * 32 + lane;     // the thread's pair
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        const int row = p / G, lim = p < P ? len + row : -1;                 // the last position it sees
        const bool two_terms = first + row < pa.fine;
        const float scale = rsqrtf((float)kPaD);
        const size_t cta = ((size_t)seq * pa.n_kv + head) * pa.tiles + tile;
        float *sm = stat_m + cta * pa.chunks * kPaPairs + p, *sl = stat_l + cta * pa.chunks * kPaPairs + p;
        bool ok = true;
        auto wait = [&](uint64_t* bar, int use) {
            ok = __all_sync(0xffffffffu, ok && mbar_wait_bounded(bar, (uint32_t)use & 1u));
            tc_fence_after();
        };
        auto done = [&](uint64_t* bar) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) pa_arrive(bar);
        };
        // 32 scores from token t of chunk c on; those beyond the position `to` -inf, where some lane's chunk is cut
        auto load = [&](int u, int c, int t, int to, bool cut, float (&a)[32]) {
            uint32_t v[32];
            tmem_ld32(lanes + kPaS + (u & 1) * 128 + t, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) a[i] = __uint_as_float(v[i]);
            if (cut) {
                const int left = to - (c * kPaTok + t);                      // tokens 0 .. left are seen
#pragma unroll
                for (int i = 0; i < 32; ++i) a[i] = i <= left ? a[i] : -INFINITY;
            }
        };
        // ---- first: every chunk's maximum (the scale is positive and rounding keeps the order: it may come after) ----
        for (int u = wg; u < n && ok; u += 2) {
            wait(&s_full[u & 1], u >> 1);
            if (!ok) break;
            float m = __int_as_float(0x7FFFFFFF);                            // NaN: left only where all 128 are
#pragma unroll 1
            for (int t = 0; t < kPaTok; t += 32) {
                float a[32];
                load(u, u, t, lim, u * kPaTok + kPaTok - 1 > len, a);            // cut: the first row does not see the whole chunk
#pragma unroll
                for (int i = 0; i < 32; ++i) m = fmaxf(m, a[i]);
            }
            done(&p_done[u & 1]);
            sm[(size_t)u * kPaPairs] = __fmul_rn(m, scale);
        }
        asm volatile("bar.sync 2, 256;" ::: "memory");                       // the other warpgroup's chunks
        const int n_p = p < P ? ceil_div(lim + 1, kPaTok) : 0;               // chunks this pair sees
        float M = -INFINITY;
#pragma unroll 4
        for (int c = 0; c < n_p; ++c) M = fmaxf(M, __ldcg(sm + (size_t)c * kPaPairs));
        // ---- then: P of this warpgroup's uses; 64 dims of every chunk's output ----
        float r[64];                                                         // the total (up to 8 chunks), or a chain's sum
#pragma unroll
        for (int i = 0; i < 64; ++i) r[i] = 0.f;
        float* tot = total_s + (cta * kPaD + wg * 64) * kPaPairs + p;
        auto add = [&](int i, int c) {                                       // output of chunk c, i-th in order
            wait(&o_full[i & 1], i >> 1);
            if (!ok) return;
            const bool seen = c < n_p;
            const float w = seen ? expf(__ldcg(sm + (size_t)c * kPaPairs) - M) : 0.f;
            const bool all_see = __all_sync(0xffffffffu, seen);
#pragma unroll
            for (int d0 = 0; d0 < 64; d0 += 32) {
                uint32_t v[32];
                tmem_ld32(lanes + kPaO + (i & 1) * 128 + wg * 64 + d0, v);
                auto each = [&](auto f) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) f(r[d0 + j], __uint_as_float(v[j]));
                };
                if (n > 8) {
                    if (all_see) each([&](float& x, float o) { x = __fmaf_rn(w, o, x); });
                    else each([&](float& x, float o) { x = seen ? __fmaf_rn(w, o, x) : x; });
                } else if (c == 0) {                                         // every pair sees the first
                    each([&](float& x, float o) { x = __fmaf_rn(w, o, 0.f); });
                } else {
                    if (all_see) each([&](float& x, float o) { x = __fadd_rn(x, __fmaf_rn(w, o, 0.f)); });
                    else each([&](float& x, float o) { x = seen ? __fadd_rn(x, __fmaf_rn(w, o, 0.f)) : x; });
                }
            }
            done(&o_free[i & 1]);
            if (n > 8 && c + 8 >= n) {                                       // the chain's end
                const bool last = (c & 7) == chains - 1;
#pragma unroll
                for (int j = 0; j < 64; ++j) {
                    const float x = (c & 7) ? __fadd_rn(__ldcg(tot + (size_t)j * kPaPairs), r[j]) : r[j];
                    if (!last) __stcg(tot + (size_t)j * kPaPairs, x);
                    r[j] = last ? x : 0.f;
                }
            }
        };
        int c_prev = 0;
        for (int i = 0, c = 0; i < n && ok; ++i) {
            const int u = n + i;
            if (i > 0) c = next_chunk(c_prev);
            if ((u & 1) == wg) {
                // no maximum (nothing seen, or beside what is not seen NaN alone): numerators 0, as in the verification kernel
                const float mc = __ldcg(sm + (size_t)c * kPaPairs), m = mc == -INFINITY ? 0.f : mc;
                const int to = mc == -INFINITY ? -1 : lim;
                const bool cut = __any_sync(0xffffffffu, mc == -INFINITY) || c * kPaTok + kPaTok - 1 > len;
                wait(&s_full[u & 1], u >> 1);
                if (!ok) break;
                float l[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) l[j] = 0.f;
#pragma unroll 1
                for (int t = 0; t < kPaTok; t += 32) {
                    float a[32];
                    uint32_t hi[16], lo[16];
                    load(u, c, t, to, cut, a);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        float e[2], h[2];
#pragma unroll
                        for (int k = 0; k < 2; ++k) e[k] = expf(__fmul_rn(a[2 * j + k], scale) - m);
                        hi[j] = pack_bf16(e[0], e[1]);
                        h[0] = __uint_as_float(hi[j] << 16);
                        h[1] = __uint_as_float(hi[j] & 0xFFFF0000u);
                        if (FINE) {
                            lo[j] = two_terms ? pack_bf16(e[0] - h[0], e[1] - h[1]) : 0u;
                            h[0] += __uint_as_float(lo[j] << 16);
                            h[1] += __uint_as_float(lo[j] & 0xFFFF0000u);
                        }
                        l[2 * j] += h[0];                                    // the sum of what the MMA multiplies
                        l[2 * j + 1] += h[1];
                    }
                    tmem_st16(lanes + kPaS + (u & 1) * 128 + t, hi);
                    if (FINE) tmem_st16(lanes + kPaS + (u & 1) * 128 + t + 16, lo);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                done(&p_done[u & 1]);
                sl[(size_t)c * kPaPairs] = tree_sum32(l);
            }
            if (i > 0) add(i - 1, c_prev);
            c_prev = c;
        }
        if (ok) add(n - 1, c_prev);
        asm volatile("bar.sync 2, 256;" ::: "memory");                       // the other warpgroup's sums
        float L = 0.f;
        for (int c0 = 0; c0 < n_p; c0 += 32) {
            float x[32];
#pragma unroll
            for (int i = 0; i < 32; ++i)
                x[i] = c0 + i < n_p ? __fmul_rn(expf(__ldcg(sm + (size_t)(c0 + i) * kPaPairs) - M), __ldcg(sl + (size_t)(c0 + i) * kPaPairs)) : 0.f;
            const float t = tree_sum32(x);
            L = c0 ? L + t : t;
        }
        if (ok && p < P) {
            uint4* to = reinterpret_cast<uint4*>(out + (((size_t)seq * pa.rps + first + row) * pa.n_q + head * G + p % G) * kPaD + wg * 64);
#pragma unroll
            for (int d0 = 0; d0 < 64; d0 += 8) {
                uint32_t b[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) b[j] = float_to_bf16_bits((n_p < 8 ? r[d0 + j] + 0.f : r[d0 + j]) / L);      // + the empty chains' zeros
                to[d0 / 8] = make_uint4(b[0] | (b[1] << 16), b[2] | (b[3] << 16), b[4] | (b[5] << 16), b[6] | (b[7] << 16));
            }
        }
        if (!ok && lane == 0) atomicExch(d_status, CASS_ERR_TIMEOUT);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

static int prefill_tile_rows(int G) { return kPaPairs / G; }

bool prefill_attn_usable(const KvGeom& g, int n_q) {
    const int G = n_q / g.n_kv;
    return g.d == kPaD && G <= kPaPairs && ceil_div(g.max_seq, kPaTok) <= kPaMaxChunks;
}

size_t prefill_attn_stats(const KvGeom& g, int n_q, int n_seq, int rps, int positions) {
    return (size_t)n_seq * g.n_kv * ceil_div(rps, prefill_tile_rows(n_q / g.n_kv)) * kPaPairs * ceil_div(positions, kPaTok);
}

int launch_prefill_attn(const KvGeom& g, const uint16_t* k_cache, const uint16_t* v_cache, const uint16_t* qkv, int n_seq, int rps, int pos, int fine,
                        int n_q, const DevState* st, const AttnScratch& sc, uint16_t* out, int32_t* d_status, cudaStream_t s) {
    if (!prefill_attn_usable(g, n_q)) return CASS_ERR_UNSUPPORTED;
    CUtensorMap mk, mv;
    int rc = tc_cache_map(&mk, g, k_cache, n_seq);
    if (!rc) rc = tc_cache_map(&mv, g, v_cache, n_seq);
    if (rc) return rc;
    const int tile_rows = prefill_tile_rows(n_q / g.n_kv), tiles = ceil_div(rps, tile_rows);
    const PrefillAttn pa{rps, n_q, g.n_kv, ceil_div(pos + rps, kPaTok), tile_rows, tiles, fine};
#define CASS_PREFILL_ATTN(F_)                                                                                                                \
    do {                                                                                                                                   \
        CASS_ALLOW_SMEM(k_prefill_attn<F_>);                                                                                                \
        CASS_PDL_LAUNCH(k_prefill_attn<F_>, dim3(g.n_kv, n_seq, tiles), dim3(kPaThreads), (size_t)kPaSmem, s, mk, mv, qkv, pa, st, sc.m, sc.l, sc.o, \
                        out, d_status);                                                                                                    \
    } while (0)
    if (fine > 0) CASS_PREFILL_ATTN(true);
    else CASS_PREFILL_ATTN(false);
#undef CASS_PREFILL_ATTN
    return CASS_OK;
}

}  // namespace cass
