// Small per-token operators of the decoder layer (Sec. 2.1): embedding gather, RMSNorm, RoPE, SwiGLU, residual
// add, greedy argmax, and the greedy accept / rollback step (Sec. 2.2).  Activations are bf16 between
// operators; arithmetic inside an operator is fp32.
#include "kernels.cuh"

namespace cass {

__global__ void k_rope_table(float* __restrict__ cos_t, float* __restrict__ sin_t, int max_seq, int half, float theta) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)max_seq * half) return;
    int pos = (int)(i / half), j = (int)(i % half);
    double inv = pow((double)theta, -2.0 * (double)j / (double)(2 * half));
    double ang = (double)pos * inv;
    cos_t[i] = (float)cos(ang);
    sin_t[i] = (float)sin(ang);
}

__global__ void k_embed(const int32_t* __restrict__ toks, int rps, int seq_stride, const uint16_t* __restrict__ embed,
                        uint16_t* __restrict__ h, int hidden) {
    pdl_wait();
    pdl_early<0>();
    int r = blockIdx.x;
    const uint16_t* src = embed + (size_t)toks[(size_t)(r / rps) * seq_stride + r % rps] * hidden;
    uint16_t* dst = h + (size_t)r * hidden;
    if ((hidden & 7) == 0 && (((uintptr_t)src | (uintptr_t)dst) & 15) == 0) {
        // 16 bytes per load, two loads in flight per thread: the row costs one or two round trips
        const uint4* s4 = reinterpret_cast<const uint4*>(src);
        uint4* d4 = reinterpret_cast<uint4*>(dst);
        const int n16 = hidden / 8;
        for (int i = threadIdx.x; i < n16; i += 2 * blockDim.x) {
            const int j = i + blockDim.x;
            const uint4 a = s4[i];
            uint4 b = make_uint4(0u, 0u, 0u, 0u);
            if (j < n16) b = s4[j];
            d4[i] = a;
            if (j < n16) d4[j] = b;
        }
        return;
    }
    for (int i = threadIdx.x; i < hidden; i += blockDim.x) dst[i] = src[i];
}

__device__ __forceinline__ float block_sum(float v, float* s_red) {
    v = warp_sum(v);
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int i = 0; i < nw; ++i) t += s_red[i];
    return t;
}

// h (+= y) then out = h * rsqrt(mean(h^2) + eps) * gain, all rounded to bf16 where stored.  Four values per thread
// and iteration (16-byte loads of the fp32 partial sums); the updated values stay in registers for the second pass.
constexpr int kNormMaxIter = 8;          // hidden <= 8 * 4 * blockDim.x

template <int ITERS>          // rounds of 4 x blockDim.x values: hidden <= ITERS * 4 * blockDim.x
__global__ void __launch_bounds__(1024) k_residual_rmsnorm(uint16_t* __restrict__ h, const uint16_t* __restrict__ y_bf16,
                                                           Partials pp,
                                                           const uint16_t* __restrict__ gain, uint16_t* __restrict__ out,
                                                           int hidden, float eps) {
    __shared__ float s_red[32];
    // the gains are weights: they are requested ahead of the wait for the predecessor
    uint2 gvs[ITERS];
#pragma unroll
    for (int it = 0; it < ITERS; ++it) {
        const int i = threadIdx.x * 4 + it * (int)blockDim.x * 4;
        gvs[it] = (out && i < hidden) ? __ldg(reinterpret_cast<const uint2*>(gain + i)) : make_uint2(0u, 0u);
    }
    pdl_wait();
    pdl_early<0>();
    const int r = blockIdx.x;
    uint16_t* hr = h + (size_t)r * hidden;
    float vals[ITERS][4];
    float ss = 0.f;
    const int step = blockDim.x * 4;
#pragma unroll
    for (int it = 0; it < ITERS; ++it) {
        const int i = threadIdx.x * 4 + it * step;
        if (i < hidden) {
            const uint2 hv = *reinterpret_cast<const uint2*>(hr + i);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            if (pp.p) acc = parts_sum4(pp, (size_t)r * pp.row_stride + i);       // requested before hv is first used: one round trip for both
            float v[4] = {__uint_as_float(hv.x << 16), __uint_as_float(hv.x & 0xFFFF0000u), __uint_as_float(hv.y << 16),
                          __uint_as_float(hv.y & 0xFFFF0000u)};
            if (y_bf16 || pp.p) {
                float y[4];
                if (pp.p) {
                    y[0] = round_bf16(acc.x); y[1] = round_bf16(acc.y); y[2] = round_bf16(acc.z); y[3] = round_bf16(acc.w);
                } else {
                    const uint2 yv = *reinterpret_cast<const uint2*>(y_bf16 + (size_t)r * hidden + i);
                    y[0] = __uint_as_float(yv.x << 16); y[1] = __uint_as_float(yv.x & 0xFFFF0000u);
                    y[2] = __uint_as_float(yv.y << 16); y[3] = __uint_as_float(yv.y & 0xFFFF0000u);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = round_bf16(v[q] + y[q]);
                uint2 o;
                o.x = (uint32_t)float_to_bf16_bits(v[0]) | ((uint32_t)float_to_bf16_bits(v[1]) << 16);
                o.y = (uint32_t)float_to_bf16_bits(v[2]) | ((uint32_t)float_to_bf16_bits(v[3]) << 16);
                *reinterpret_cast<uint2*>(hr + i) = o;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) { vals[it][q] = v[q]; ss += v[q] * v[q]; }
        }
    }
    ss = block_sum(ss, s_red);
    const float inv = 1.0f / sqrtf(ss / (float)hidden + eps);
    if (out) {
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int i = threadIdx.x * 4 + it * step;
            if (i < hidden) {
                const uint2 gv = gvs[it];
                const float gq[4] = {__uint_as_float(gv.x << 16), __uint_as_float(gv.x & 0xFFFF0000u), __uint_as_float(gv.y << 16),
                                     __uint_as_float(gv.y & 0xFFFF0000u)};
                uint32_t ob[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) ob[q] = float_to_bf16_bits(vals[it][q] * inv * gq[q]);
                uint2 o;
                o.x = ob[0] | (ob[1] << 16);
                o.y = ob[2] | (ob[3] << 16);
                *reinterpret_cast<uint2*>(out + (size_t)r * hidden + i) = o;
            }
        }
    }
}

__device__ __forceinline__ void unpack4(uint2 v, float (&x)[4]) {
    x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xFFFF0000u);
    x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xFFFF0000u);
}

// The same for many rows (a prefill pass) whose projections come as bf16: a quarter of the threads, each in the place of four whose
// values lie `n_virt` / 4 warps apart, so that a row's sum is formed as above (lanes' sums of a warp by exchange, the warps' in order) and its bits
// are the same.  A row of 1024 threads with one quadruple each waits, two rows an SM, for one round trip after the other: 18.5 -> 9.8 us for 1000 rows of 4096.
template <int ITERS>
__global__ void __launch_bounds__(256) k_residual_rmsnorm_rows(uint16_t* __restrict__ h, const uint16_t* __restrict__ y, const uint16_t* __restrict__ gain,
                                                               uint16_t* __restrict__ out, int hidden, int n_virt, float eps) {
    __shared__ float s_red[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, step = n_virt * 128;      // virtual warps warp + nw * v
    pdl_wait();
    pdl_early<0>();
    uint16_t* hr = h + (size_t)blockIdx.x * hidden;
    const uint16_t* yr = y + (size_t)blockIdx.x * hidden;
    uint2 hv[4][ITERS], yv[4][ITERS];
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int w = warp + nw * v, i = (w * 32 + lane) * 4 + it * step;
            const bool in = w < n_virt && i < hidden;
            hv[v][it] = in ? *reinterpret_cast<const uint2*>(hr + i) : make_uint2(0u, 0u);
            yv[v][it] = in ? *reinterpret_cast<const uint2*>(yr + i) : make_uint2(0u, 0u);
        }
    float vals[4][ITERS][4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int w = warp + nw * v;
        float ss = 0.f;
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int i = (w * 32 + lane) * 4 + it * step;
            float a[4], b[4];
            unpack4(hv[v][it], a);
            unpack4(yv[v][it], b);
            if (w < n_virt && i < hidden) {
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = round_bf16(a[q] + b[q]);
                *reinterpret_cast<uint2*>(hr + i) = make_uint2((uint32_t)float_to_bf16_bits(a[0]) | ((uint32_t)float_to_bf16_bits(a[1]) << 16),
                                                               (uint32_t)float_to_bf16_bits(a[2]) | ((uint32_t)float_to_bf16_bits(a[3]) << 16));
#pragma unroll
                for (int q = 0; q < 4; ++q) ss += a[q] * a[q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) vals[v][it][q] = a[q];
        }
        ss = warp_sum(ss);
        if (lane == 0 && w < n_virt) s_red[w] = ss;
    }
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < n_virt; ++w) t += s_red[w];
    const float inv = 1.0f / sqrtf(t / (float)hidden + eps);
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int w = warp + nw * v, i = (w * 32 + lane) * 4 + it * step;
            if (w < n_virt && i < hidden) {
                float g[4];
                unpack4(__ldg(reinterpret_cast<const uint2*>(gain + i)), g);
                uint32_t o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) o[q] = float_to_bf16_bits(vals[v][it][q] * inv * g[q]);
                *reinterpret_cast<uint2*>(out + (size_t)blockIdx.x * hidden + i) = make_uint2(o[0] | (o[1] << 16), o[2] | (o[3] << 16));
            }
        }
}

// Four rotated pairs, or eight plain v elements, a thread (head sizes are multiples of 32): 16-byte loads of the parts.
__global__ void __launch_bounds__(128) k_qkv_rope(uint16_t* __restrict__ qkv, Partials pp,
                                                  const float* __restrict__ cos_t, const float* __restrict__ sin_t,
                                                  const DevState* __restrict__ st, int use_inflight, int rps, int n_q, int n_kv, int d) {
    pdl_wait();
    pdl_early<0>();
    const int r = blockIdx.y, half = d / 2;
    const int qkv_dim = (n_q + 2 * n_kv) * d;
    const int b = r / rps;
    const int pos = st->len[b] + (use_inflight ? st->inflight[b] : 0) + r % rps;
    uint16_t* row = qkv + (size_t)r * qkv_dim;
    const int n_rot = (n_q + n_kv) * half;             // rotated pairs
    const int n_items = n_rot + n_kv * half;           // + pairs of plain v elements
    auto load4 = [&](int ia, int ib, float (&x)[4], float (&y)[4]) {
        if (pp.p) {
            float4 s, t;
            parts_sum4_pair(pp, (size_t)r * pp.row_stride + ia, (size_t)r * pp.row_stride + ib, s, t);
            x[0] = round_bf16(s.x); x[1] = round_bf16(s.y); x[2] = round_bf16(s.z); x[3] = round_bf16(s.w);
            y[0] = round_bf16(t.x); y[1] = round_bf16(t.y); y[2] = round_bf16(t.z); y[3] = round_bf16(t.w);
        } else {
            unpack4(*reinterpret_cast<const uint2*>(row + ia), x);
            unpack4(*reinterpret_cast<const uint2*>(row + ib), y);
        }
    };
    auto store4 = [&](int i, const float (&x)[4]) {
        *reinterpret_cast<uint2*>(row + i) = make_uint2((uint32_t)float_to_bf16_bits(x[0]) | ((uint32_t)float_to_bf16_bits(x[1]) << 16),
                                                        (uint32_t)float_to_bf16_bits(x[2]) | ((uint32_t)float_to_bf16_bits(x[3]) << 16));
    };
    const int it = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (it >= n_items) return;
    const int head = it / half, j = it % half;         // v heads follow the k heads
    const int ia = head * d + j, ib = ia + half;
    float x[4], y[4];
    if (it < n_rot) {
        const float4 c4 = __ldg(reinterpret_cast<const float4*>(cos_t + (size_t)pos * half + j));
        const float4 s4 = __ldg(reinterpret_cast<const float4*>(sin_t + (size_t)pos * half + j));
        load4(ia, ib, x, y);
        const float c[4] = {c4.x, c4.y, c4.z, c4.w}, sn[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 rot = rope_pair(x[q], y[q], c[q], sn[q]);
            x[q] = rot.x;
            y[q] = rot.y;
        }
    } else {
        if (!pp.p) return;                             // v is there already
        load4(ia, ib, x, y);
    }
    store4(ia, x);
    store4(ib, y);
}

// Four features a thread: 16-byte loads of the parts, one address for four.  (One a thread was bound by instruction issue:
// 18.3 us for 128 rows of 14336, 29 MB of parts.)
__global__ void __launch_bounds__(128) k_swiglu(Partials pp, uint16_t* __restrict__ act, int ffn) {
    pdl_wait();
    pdl_early<0>();
    const int r = blockIdx.y;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) * 4; i < ffn; i += gridDim.x * blockDim.x * 4) {
        float g[4], u[4];
        float4 gs, us;
        parts_sum4_pair(pp, (size_t)r * pp.row_stride + i, (size_t)r * pp.row_stride + ffn + i, gs, us);
        g[0] = round_bf16(gs.x); g[1] = round_bf16(gs.y); g[2] = round_bf16(gs.z); g[3] = round_bf16(gs.w);
        u[0] = round_bf16(us.x); u[1] = round_bf16(us.y); u[2] = round_bf16(us.z); u[3] = round_bf16(us.w);
        uint32_t o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float silu = g[q] / (1.0f + expf(-g[q]));
            o[q] = float_to_bf16_bits(silu * u[q]);
        }
        *reinterpret_cast<uint2*>(act + (size_t)r * ffn + i) = make_uint2(o[0] | (o[1] << 16), o[2] | (o[3] << 16));
    }
}

// The same of bf16 projections (a prefill pass), eight features of one row a thread: two 16-byte loads under way and one store.  Four
// features a thread: 32 us for 1000 rows of 14336, 86 MB, 21 so.
__global__ void __launch_bounds__(256) k_swiglu_rows(const uint16_t* __restrict__ gu, uint16_t* __restrict__ act, int ffn, int n_items) {
    pdl_wait();
    pdl_early<0>();
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= n_items) return;
    const int per = ffn / 8, r = it / per, i = (it - r * per) * 8;
    const uint16_t* row = gu + (size_t)r * 2 * ffn + i;
    const uint4 gv = __ldcs(reinterpret_cast<const uint4*>(row)), uv = __ldcs(reinterpret_cast<const uint4*>(row + ffn));
    const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, uw[4] = {uv.x, uv.y, uv.z, uv.w};
    uint32_t o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float g0 = __uint_as_float(gw[q] << 16), g1 = __uint_as_float(gw[q] & 0xFFFF0000u);
        const float s0 = g0 / (1.0f + expf(-g0)), s1 = g1 / (1.0f + expf(-g1));
        o[q] = (uint32_t)float_to_bf16_bits(s0 * __uint_as_float(uw[q] << 16)) | ((uint32_t)float_to_bf16_bits(s1 * __uint_as_float(uw[q] & 0xFFFF0000u)) << 16);
    }
    *reinterpret_cast<uint4*>(act + (size_t)r * ffn + i) = make_uint4(o[0], o[1], o[2], o[3]);
}

// Greedy token of each row, lowest index on ties, in two levels: slices of the vocabulary, then the slices' winners.
constexpr int kArgmaxSlices = 128;

__device__ __forceinline__ void argmax_combine(float& best, int& best_i, float ov, int oi) {
    if (ov > best || (ov == best && oi < best_i)) { best = ov; best_i = oi; }
}

// Bound: the latency of the parts' loads (20 rows of 152064 logits, written out again: 24 MB of L2 traffic): two quadruples a
// thread travel together, 22.8 -> 8.7 us; one value at a time where the rows are no multiple of 16 bytes apart.
__global__ void __launch_bounds__(256) k_argmax_part(Partials pp, int vocab, int per, float* __restrict__ tmp_v,
                                                     int32_t* __restrict__ tmp_i, float* __restrict__ logits_copy) {
    __shared__ float s_v[8];
    __shared__ int s_i[8];
    pdl_wait();
    pdl_early<0>();
    const int r = blockIdx.y, nsl = gridDim.x;
    const int lo = blockIdx.x * per, hi = min(vocab, lo + per);                  // lo: a multiple of 4
    float best = -INFINITY;
    int best_i = 0x7fffffff;
    if (vocab % 4 == 0 && pp.row_stride % 4 == 0 && pp.seg_stride % 4 == 0 && (((uintptr_t)pp.p | (uintptr_t)logits_copy) & 15) == 0) {
        const size_t row = (size_t)r * pp.row_stride;
        for (int i = lo + (int)threadIdx.x * 4; i < hi; i += 2048) {
            const int j = i + 1024 < hi ? i + 1024 : i;                          // the same again changes nothing
            float4 a, b;
            parts_sum4_pair(pp, row + i, row + j, a, b);
            if (logits_copy) {
                float* to = logits_copy + (size_t)r * vocab;
                *reinterpret_cast<float4*>(to + i) = a;
                if (j != i) *reinterpret_cast<float4*>(to + j) = b;
            }
            argmax_combine(best, best_i, a.x, i); argmax_combine(best, best_i, a.y, i + 1);
            argmax_combine(best, best_i, a.z, i + 2); argmax_combine(best, best_i, a.w, i + 3);
            argmax_combine(best, best_i, b.x, j); argmax_combine(best, best_i, b.y, j + 1);
            argmax_combine(best, best_i, b.z, j + 2); argmax_combine(best, best_i, b.w, j + 3);
        }
    } else {
        for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const float v = parts_sum(pp, (size_t)r * pp.row_stride + i);
            if (logits_copy) logits_copy[(size_t)r * vocab + i] = v;
            argmax_combine(best, best_i, v, i);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        float ov = __shfl_xor_sync(0xffffffffu, best, o);
        int oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        argmax_combine(best, best_i, ov, oi);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_v[warp] = best; s_i[warp] = best_i; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) argmax_combine(best, best_i, s_v[w], s_i[w]);
        tmp_v[r * nsl + blockIdx.x] = best;
        tmp_i[r * nsl + blockIdx.x] = best_i;
    }
}

__global__ void __launch_bounds__(kArgmaxSlices) k_argmax_final(const float* __restrict__ tmp_v, const int32_t* __restrict__ tmp_i,
                                                                int nsl, int32_t* __restrict__ out, int out_stride, DevState* st,
                                                                int bump_inflight) {
    __shared__ float s_v[kArgmaxSlices / 32];
    __shared__ int s_i[kArgmaxSlices / 32];
    pdl_wait();
    pdl_early<0>();
    const int r = blockIdx.x;
    float best = -INFINITY;
    int best_i = 0x7fffffff;
    if ((int)threadIdx.x < nsl) { best = tmp_v[r * nsl + threadIdx.x]; best_i = tmp_i[r * nsl + threadIdx.x]; }
    for (int o = 16; o > 0; o >>= 1) {
        float ov = __shfl_xor_sync(0xffffffffu, best, o);
        int oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        argmax_combine(best, best_i, ov, oi);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_v[warp] = best; s_i[warp] = best_i; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kArgmaxSlices / 32; ++w) argmax_combine(best, best_i, s_v[w], s_i[w]);
        out[(size_t)r * out_stride] = best_i == 0x7fffffff ? 0 : best_i;
        if (bump_inflight && r < kMaxBatch) {
            // the draft counter never passes the margin kept free at the end of a cache (positions len .. len + 15)
            if (st->inflight[r] < kMaxVerifyRows - 1) st->inflight[r] += 1;
            else atomicCAS(&st->status, 0, CASS_ERR_INVALID_ARG);
        }
    }
}

// Greedy acceptance: a = min({i-1 : draft_i != target_{i-1}} U {g}); emit draft_1..draft_a and target_a.
// One block per sequence b: draft[b * draft_stride + i], target[b][g+1] -> n_acc[b], out_tokens[b][g+1],
// next_tok[b * next_stride].
__global__ void k_accept(DevState* st, const int32_t* __restrict__ draft, int draft_stride, const int32_t* __restrict__ target, int g,
                         int32_t* n_acc, int32_t* out_tokens, int32_t* next_tok, int next_stride) {
    pdl_wait();
    pdl_early<0>();
    if (threadIdx.x != 0) return;
    const int b = blockIdx.x;
    draft += (size_t)b * draft_stride;
    target += (size_t)b * (g + 1);
    out_tokens += (size_t)b * (g + 1);
    n_acc += b;
    if (next_tok) next_tok += (size_t)b * next_stride;
    int a = 0;
    while (a < g && draft[a] == target[a]) ++a;
    for (int i = 0; i < a; ++i) out_tokens[i] = draft[i];
    out_tokens[a] = target[a];
    for (int i = a + 1; i <= g; ++i) out_tokens[i] = -1;
    *n_acc = a;
    if (next_tok) *next_tok = target[a];
    // Every later call touches positions up to len + 15 at most; a sequence that would come closer than that to
    // the end of its cache stops growing and the status word says so.
    if (st->len[b] + a + 1 + kMaxVerifyRows > st->max_seq) atomicCAS(&st->status, 0, CASS_ERR_CAPACITY);
    else st->len[b] += a + 1;
    st->inflight[b] = 0;
}

__global__ void k_calib_accum(const uint16_t* __restrict__ x, int rows, int cols, float* __restrict__ sumsq,
                              const DevState* __restrict__ st) {
    pdl_wait();
    pdl_early<0>();
    if (!st->calib_on) return;
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols) return;
    float acc = sumsq[c];
#pragma unroll 8
    for (int r = 0; r < rows; ++r) {
        float v = bf16_bits_to_float(x[(size_t)r * cols + c]);
        acc += v * v;
    }
    sumsq[c] = acc;
}

__global__ void k_sqrt(const float* __restrict__ in, float* __restrict__ out, size_t n) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = sqrtf(in[i]);
}

int launch_rope_table(float* cos_t, float* sin_t, int max_seq, int d, float theta, cudaStream_t s) {
    size_t n = (size_t)max_seq * (d / 2);
    k_rope_table<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(cos_t, sin_t, max_seq, d / 2, theta);
    CASS_LAUNCH_CHECK();
    return CASS_OK;
}

int launch_embed(const int32_t* toks, int rps, int seq_stride, const uint16_t* embed, uint16_t* h, int rows, int hidden, cudaStream_t s) {
    CASS_PDL_LAUNCH(k_embed, dim3(rows), dim3(256), 0, s, toks, rps, seq_stride, embed, h, hidden);
    return CASS_OK;
}

static int norm_threads(int hidden) {
    int t = ceil_div(ceil_div(hidden, 4), 32) * 32;
    return t > 1024 ? 1024 : t;
}

static int norm_iters(int hidden, int threads) {
    const int it = ceil_div(hidden, 4 * threads);
    return it <= 1 ? 1 : (it <= 2 ? 2 : (it <= 4 ? 4 : 8));
}

int launch_residual_rmsnorm(uint16_t* h, const uint16_t* y_bf16, Partials pp,
                            const uint16_t* gain, uint16_t* out, int rows, int hidden, float eps, cudaStream_t s) {
    if (hidden % 4 || hidden > kNormMaxIter * 4 * 1024) return CASS_ERR_UNSUPPORTED;
    const int threads = norm_threads(hidden);
    if (y_bf16 && !pp.p && out && rows > 2 * kSms && norm_iters(hidden, threads) <= 2) {
        const int n_virt = threads / 32, quarter = ceil_div(n_virt, 4) * 32;
        if (norm_iters(hidden, threads) == 1) CASS_PDL_LAUNCH(k_residual_rmsnorm_rows<1>, dim3(rows), dim3(quarter), 0, s, h, y_bf16, gain, out, hidden, n_virt, eps);
        else CASS_PDL_LAUNCH(k_residual_rmsnorm_rows<2>, dim3(rows), dim3(quarter), 0, s, h, y_bf16, gain, out, hidden, n_virt, eps);
        return CASS_OK;
    }
    switch (norm_iters(hidden, threads)) {
        case 1: CASS_PDL_LAUNCH(k_residual_rmsnorm<1>, dim3(rows), dim3(threads), 0, s, h, y_bf16, pp, gain, out, hidden, eps); break;
        case 2: CASS_PDL_LAUNCH(k_residual_rmsnorm<2>, dim3(rows), dim3(threads), 0, s, h, y_bf16, pp, gain, out, hidden, eps); break;
        case 4: CASS_PDL_LAUNCH(k_residual_rmsnorm<4>, dim3(rows), dim3(threads), 0, s, h, y_bf16, pp, gain, out, hidden, eps); break;
        default: CASS_PDL_LAUNCH(k_residual_rmsnorm<8>, dim3(rows), dim3(threads), 0, s, h, y_bf16, pp, gain, out, hidden, eps); break;
    }
    return CASS_OK;
}

int launch_rmsnorm(const uint16_t* h, const uint16_t* gain, uint16_t* out, int rows, int hidden, float eps, cudaStream_t s) {
    return launch_residual_rmsnorm(const_cast<uint16_t*>(h), nullptr, Partials{nullptr, 0, 0, 0}, gain, out, rows, hidden, eps, s);
}

int launch_qkv_rope(uint16_t* qkv, Partials pp, const float* cos_t, const float* sin_t,
                    const DevState* st, int use_inflight, int rows, int rps, int n_q, int n_kv, int d, cudaStream_t s) {
    dim3 grid(ceil_div((n_q + 2 * n_kv) * (d / 2), 512), rows);
    CASS_PDL_LAUNCH(k_qkv_rope, grid, dim3(128), 0, s, qkv, pp, cos_t, sin_t, st, use_inflight, rps, n_q, n_kv, d);
    return CASS_OK;
}

int launch_swiglu(const uint16_t* gu_bf16, Partials pp, uint16_t* act, int rows, int ffn,
                  cudaStream_t s) {
    if (!pp.p) {                                             // ffn is a multiple of 8
        const int items = rows * (ffn / 8);
        CASS_PDL_LAUNCH(k_swiglu_rows, dim3(ceil_div(items, 256)), dim3(256), 0, s, gu_bf16, act, ffn, items);
        return CASS_OK;
    }
    dim3 grid(ceil_div(ffn, 512), rows);
    CASS_PDL_LAUNCH(k_swiglu, grid, dim3(128), 0, s, pp, act, ffn);
    return CASS_OK;
}

int launch_argmax(Partials pp, int rows, int vocab, int32_t* out, int out_stride,
                  float* logits_copy, float* tmp_v, int32_t* tmp_i, DevState* st, int bump_inflight, cudaStream_t s) {
    // few rows: as many CTAs as a quadruple a thread allows; many: two of them a thread
    int nsl = ceil_div(vocab, rows >= 4 ? 2048 : 1024);
    if (nsl > kArgmaxSlices) nsl = kArgmaxSlices;
    const int per = ceil_div(ceil_div(vocab, nsl), 4) * 4;
    dim3 grid(nsl, rows);
    CASS_PDL_LAUNCH(k_argmax_part, grid, dim3(256), 0, s, pp, vocab, per, tmp_v, tmp_i, logits_copy);
    CASS_PDL_LAUNCH(k_argmax_final, dim3(rows), dim3(kArgmaxSlices), 0, s, (const float*)tmp_v, (const int32_t*)tmp_i, nsl, out, out_stride, st, bump_inflight);
    return CASS_OK;
}

// Positions of a prefill pass: every sequence's length, its drafts forgotten.
__global__ void k_set_len(DevState* st, int len) {
    pdl_wait();
    st->len[threadIdx.x] = len;
    st->inflight[threadIdx.x] = 0;
}
int launch_set_len(DevState* st, int len, cudaStream_t s) {
    CASS_PDL_LAUNCH(k_set_len, dim3(1), dim3(kMaxBatch), 0, s, st, len);
    return CASS_OK;
}

// The last `take` of each sequence's rps rows: dst [n_seq][take][cols] (cols a multiple of 8).
__global__ void k_last_rows(const uint16_t* __restrict__ src, int rps, int take, int cols, uint16_t* __restrict__ dst) {
    pdl_wait();
    const int seq = blockIdx.x / take, i = blockIdx.x % take;
    const uint4* s4 = reinterpret_cast<const uint4*>(src + ((size_t)seq * rps + rps - take + i) * cols);
    uint4* d4 = reinterpret_cast<uint4*>(dst + (size_t)blockIdx.x * cols);
    for (int c = threadIdx.x; c < cols / 8; c += blockDim.x) d4[c] = s4[c];
}
int launch_last_rows(const uint16_t* src, int n_seq, int rps, int take, int cols, uint16_t* dst, cudaStream_t s) {
    CASS_PDL_LAUNCH(k_last_rows, dim3(n_seq * take), dim3(256), 0, s, src, rps, take, cols, dst);
    return CASS_OK;
}

int launch_accept(DevState* st, int n_seq, const int32_t* draft, int draft_stride, const int32_t* target, int g, int32_t* n_acc,
                  int32_t* out_tokens, int32_t* next_tok, int next_stride, cudaStream_t s) {
    CASS_PDL_LAUNCH(k_accept, dim3(n_seq), dim3(32), 0, s, st, draft, draft_stride, target, g, n_acc, out_tokens, next_tok, next_stride);
    return CASS_OK;
}

int launch_calib_accum(const uint16_t* x, int rows, int cols, float* sumsq, const DevState* st, cudaStream_t s) {
    CASS_PDL_LAUNCH(k_calib_accum, dim3(ceil_div(cols, 256)), dim3(256), 0, s, x, rows, cols, sumsq, st);
    return CASS_OK;
}

int launch_sqrt(const float* in, float* out, size_t n, cudaStream_t s) {
    k_sqrt<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, out, n);
    CASS_LAUNCH_CHECK();
    return CASS_OK;
}

}  // namespace cass
