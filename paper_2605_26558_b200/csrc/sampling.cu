// Sampling-based acceptance (Sec. 2.2, Eq. 1: rejection sampling against the draft's distribution) and the two
// small operators it needs around it: softmax of logits at a temperature and an inverse-CDF draw.  Random numbers
// are inputs (uniform in [0, 1)); nothing here generates them.
#include <cfloat>

#include <cooperative_groups.h>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace cass {

constexpr int kSampleThreads = 256;

__device__ __forceinline__ float block_reduce(float v, bool is_max, float* s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = is_max ? warp_max(v) : warp_sum(v);
    __syncthreads();                                      // s_red may still be read from a previous call
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    float r = s_red[0];
    for (int w = 1; w < nw; ++w) r = is_max ? fmaxf(r, s_red[w]) : r + s_red[w];      // fixed order
    return r;
}

// probs[r][v] = exp((logits[r][v] - max) / T) / sum.  A cluster of CTAs holds a row (NV values a thread, in registers up to 16; of
// 32 and 40, which vocabularies of 128256 and 152064 take, the compiler spills 27 and 52: two CTAs
// an SM leave 64 registers a thread), so that it is read and written once and only the two reductions cross CTAs, through distributed shared
// memory.  Bound: latency (one round trip to memory, two cluster barriers): 13.5 us for 20 rows of 128256, 18.2 for 20 of 152064;
// one CTA a row was 501 dependent rounds over a vocabulary of 128256, 200 us.
constexpr int kSoftmaxThreads = 512;

template <int NV>
__global__ void __launch_bounds__(kSoftmaxThreads, 2) k_softmax_rows(const float* __restrict__ logits, int vocab, int per, float inv_t,
                                                                  float* __restrict__ probs) {
    __shared__ float s_red[kSoftmaxThreads / 32], s_cta[2];
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), tid = threadIdx.x;
    pdl_wait();
    const size_t row = (size_t)(blockIdx.x / cs) * vocab;
    const int v0 = rank * per + tid, v1 = min(vocab, (rank + 1) * per);
    float x[NV], m = -FLT_MAX;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int v = v0 + i * kSoftmaxThreads;
        x[i] = __ldg(logits + row + min(v, vocab - 1));                    // unconditional: all of them travel at once
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if (v0 + i * kSoftmaxThreads >= v1) x[i] = -FLT_MAX;
        m = fmaxf(m, x[i]);
    }
    auto over_cluster = [&](float v, bool is_max, float* slot) {           // fixed order: CTAs by rank
        v = block_reduce(v, is_max, s_red);
        if (tid == 0) *slot = v;
        cluster.sync();
        // one lane a CTA, so that the remote reads are one round trip; then in the order of the ranks
        const float mine = *cluster.map_shared_rank(slot, min(tid & 31, cs - 1));
        float r = __shfl_sync(0xffffffffu, mine, 0);
#pragma unroll
        for (int c = 1; c < 8; ++c) {
            const float o = __shfl_sync(0xffffffffu, mine, c);
            if (c < cs) r = is_max ? fmaxf(r, o) : r + o;
        }
        return r;
    };
    m = over_cluster(m, true, &s_cta[0]);
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        x[i] = v0 + i * kSoftmaxThreads < v1 ? __expf((x[i] - m) * inv_t) : 0.f;
        sum += x[i];
    }
    const float inv = 1.f / over_cluster(sum, false, &s_cta[1]);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int v = v0 + i * kSoftmaxThreads;
        if (v < v1) probs[row + v] = x[i] * inv;
    }
    cluster.sync();                                                        // nobody leaves while its sums may be read
}

// The same by one CTA a row, for vocabularies that the registers of a cluster do not hold.
__global__ void __launch_bounds__(1024) k_softmax_rows_long(const float* __restrict__ logits, int vocab, float inv_t, float* __restrict__ probs) {
    __shared__ float s_red[32];
    pdl_wait();
    const float* in = logits + (size_t)blockIdx.x * vocab;
    float* out = probs + (size_t)blockIdx.x * vocab;
    float m = -FLT_MAX;
#pragma unroll 8
    for (int v = threadIdx.x; v < vocab; v += blockDim.x) m = fmaxf(m, in[v]);
    m = block_reduce(m, true, s_red);
    float sum = 0.f;
#pragma unroll 8
    for (int v = threadIdx.x; v < vocab; v += blockDim.x) {
        const float e = __expf((in[v] - m) * inv_t);
        out[v] = e;
        sum += e;
    }
    sum = block_reduce(sum, false, s_red);
    const float inv = 1.f / sum;
#pragma unroll 8
    for (int v = threadIdx.x; v < vocab; v += blockDim.x) out[v] *= inv;
}

// Inverse-CDF draw over weight(v), v in [0, vocab), by the CTAs of a cluster: the lowest index whose cumulative weight
// exceeds u * total.  The indices are cut into kSampleThreads segments of `per`; a segment is summed in index order by one
// thread and the segment sums are added in order, so the result depends on neither scheduling nor the cluster's size.
// A CTA brings its segments into shared memory with contiguous reads first (segments an odd number of floats apart: the
// summing threads then never share a bank).  Returns the index to every thread (vocab - 1 when the total is not positive).
// Bound: the chain of additions (`per` of a segment, then the 256 sums); reading each segment from global memory as it was
// summed took a dependent round trip for every few values, 350 us over a vocabulary of 128256; four draws now take 12.7 us, an
// acceptance of four sequences 14.1.
// The kernel arrives at the cluster's barrier when it starts (barrier_arrive), and the first draw waits for it here before it
// stores into rank 0's memory: a CTA's shared memory may be touched only once that CTA is known to run.
struct DrawShared {
    float seg[kSampleThreads + 1];         // this CTA's copy of all sums, then the sums before each segment; last: the total
    float all[kSampleThreads];             // rank 0: where the CTAs leave their sums
    int pick;                              // rank 0
};

__host__ __device__ inline int draw_stride(int vocab) { return ceil_div(vocab, kSampleThreads) | 1; }

// STAGED = false: a vocabulary whose segments do not fit shared memory is read where it is.
// first: the kernel's first draw.
template <bool STAGED, class W>
__device__ int cluster_inverse_cdf(cg::cluster_group& cluster, bool first, W weight, int vocab, float u, DrawShared& sh, float* w_s,
                                   float* total_out) {
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int per = ceil_div(vocab, kSampleThreads), stride = draw_stride(vocab), n_seg = kSampleThreads / cs, seg0 = rank * n_seg;
    if (rank == 0 && tid == 0) sh.pick = vocab - 1;
    if (STAGED) {
        // the CTA's segments are one contiguous range; segment s of it sits s * (stride - per) floats further in shared memory
        const int base = seg0 * per, n_el = min(vocab - base, n_seg * per);
        const uint32_t magic = stride == per ? 0u : 0xFFFFFFFFu / (uint32_t)per + 1u;      // e / per = high half of e x magic: e x per < 2^32
        for (int e0 = tid; e0 < n_el; e0 += kSampleThreads * 16) {
            float x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                x[k] = weight(base + min(e0 + k * kSampleThreads, n_el - 1));      // unconditional: all of them travel at once
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int e = e0 + k * kSampleThreads;
                if (e < n_el) w_s[e + (int)__umulhi((uint32_t)e, magic)] = x[k];
            }
        }
    }
    __syncthreads();
    const int v0 = (seg0 + tid) * per, n = tid < n_seg ? max(0, min(vocab - v0, per)) : 0;
    auto mine = [&](int i) { return STAGED ? w_s[tid * stride + i] : weight(v0 + i); };
    float sum = 0.f, x[8], nx[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = k < n ? mine(k) : 0.f;
    for (int i = 0; i < n; i += 8) {                                       // the next eight values travel while eight are added
#pragma unroll
        for (int k = 0; k < 8; ++k) nx[k] = i + 8 + k < n ? mine(i + 8 + k) : 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) { sum += x[k]; x[k] = nx[k]; }         // adding 0 at the end changes nothing
    }
    if (first) cluster.barrier_wait();
    if (tid < n_seg) *cluster.map_shared_rank(&sh.all[seg0 + tid], 0) = sum;
    cluster.sync();
    sh.seg[tid] = *cluster.map_shared_rank(&sh.all[tid], 0);
    __syncthreads();
    if (tid == 0) {                                                        // exclusive scan of the segment sums, in order
        float run = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = sh.seg[j];
        for (int k = 0; k < kSampleThreads; k += 8) {
#pragma unroll
            for (int j = 0; j < 8; ++j) nx[j] = k + 8 < kSampleThreads ? sh.seg[k + 8 + j] : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) { sh.seg[k + j] = run; run += x[j]; x[j] = nx[j]; }
        }
        sh.seg[kSampleThreads] = run;
    }
    __syncthreads();
    const float total = sh.seg[kSampleThreads], target = u * total;
    if (tid < n_seg) {
        const float before = sh.seg[seg0 + tid], after = sh.seg[seg0 + tid + 1];
        if (before <= target && target < after) {                          // exactly one thread: the segment sums are non-negative
            float run = before;
            int pick = v0 + n - 1;
            bool found = false;
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = j < n ? mine(j) : 0.f;
            for (int k = 0; k < n && !found; k += 8) {
#pragma unroll
                for (int j = 0; j < 8; ++j) nx[j] = k + 8 + j < n ? mine(k + 8 + j) : 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    run += x[j];
                    x[j] = nx[j];
                    if (!found && k + j < n && run > target) { pick = v0 + k + j; found = true; }
                }
            }
            *cluster.map_shared_rank(&sh.pick, 0) = pick;
        }
    }
    cluster.sync();
    const int pick = *cluster.map_shared_rank(&sh.pick, 0);
    if (total_out) *total_out = total;
    cluster.sync();                                                        // `pick` and `all` may be written again, or their CTA may leave
    return pick;
}

template <bool STAGED>
__global__ void __launch_bounds__(kSampleThreads) k_sample_rows(const float* __restrict__ probs, int vocab,
                                                                const float* __restrict__ u, int32_t* __restrict__ tokens,
                                                                int tok_stride) {
    extern __shared__ float w_s[];
    __shared__ DrawShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.barrier_arrive();
    pdl_wait();
    const int row = blockIdx.x / (int)cluster.num_blocks();
    const float* p = probs + (size_t)row * vocab;
    const int pick = cluster_inverse_cdf<STAGED>(cluster, true, [&](int v) { return __ldg(p + v); }, vocab, u[row], sh, w_s, nullptr);
    if (cluster.block_rank() == 0 && threadIdx.x == 0) tokens[(size_t)row * tok_stride] = pick;
}

// One cluster per sequence b.  Eq. 1: n = min({i-1 : r_i > p_i(x_i) / q_i(x_i)} U {g}); then one more token: from the
// normalised positive part of p_{n+1} - q_{n+1} after a rejection, from p_{g+1} after full acceptance.
template <bool STAGED>
__global__ void __launch_bounds__(kSampleThreads) k_accept_sampling(DevState* st, const int32_t* __restrict__ draft, int draft_stride,
                                                                    const float* __restrict__ p, const float* __restrict__ q, int vocab,
                                                                    const float* __restrict__ r, const float* __restrict__ u, int g,
                                                                    int32_t* n_acc, int32_t* out_tokens, int32_t* next_tok,
                                                                    int next_stride) {
    extern __shared__ float w_s[];
    __shared__ DrawShared sh;
    __shared__ int s_n;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.barrier_arrive();
    pdl_wait();
    const int b = blockIdx.x / (int)cluster.num_blocks();
    draft += (size_t)b * draft_stride;
    p += (size_t)b * (g + 1) * vocab;
    q += (size_t)b * g * vocab;
    r += (size_t)b * g;
    if (threadIdx.x < 32) {                                                // lane i: draft i (g < 16)
        const int i = threadIdx.x, x = i < g ? draft[i] : 0;
        const bool in_range = x >= 0 && x < vocab;
        // r > p/q, written without the division (q(x) = 0 cannot have been drawn; it rejects unless p(x) = 0 too)
        const bool reject = i >= g || !in_range || r[i] * q[(size_t)i * vocab + x] > p[(size_t)i * vocab + x];
        const unsigned m = __ballot_sync(0xffffffffu, reject);
        if (i == 0) s_n = __ffs(m) - 1;                                    // lane g rejects: n <= g
    }
    __syncthreads();
    const int n = s_n;
    const float* pn = p + (size_t)n * vocab;
    const float* qn = q + (size_t)n * vocab;                               // read only when n < g
    float total = 0.f;
    int extra = 0;
    if (n < g)
        extra = cluster_inverse_cdf<STAGED>(cluster, true, [&](int v) { return fmaxf(__ldg(pn + v) - __ldg(qn + v), 0.f); }, vocab, u[b], sh, w_s, &total);
    if (!(total > 0.f)) extra = cluster_inverse_cdf<STAGED>(cluster, n == g, [&](int v) { return __ldg(pn + v); }, vocab, u[b], sh, w_s, nullptr);
    if (cluster.block_rank() != 0 || threadIdx.x != 0) return;
    out_tokens += (size_t)b * (g + 1);
    for (int i = 0; i < n; ++i) out_tokens[i] = draft[i];
    out_tokens[n] = extra;
    for (int i = n + 1; i <= g; ++i) out_tokens[i] = -1;
    n_acc[b] = n;
    if (next_tok) next_tok[(size_t)b * next_stride] = extra;
    if (st && b < kMaxBatch) {                                             // the same length rule as the greedy accept
        if (st->len[b] + n + 1 + kMaxVerifyRows > st->max_seq) atomicCAS(&st->status, 0, CASS_ERR_CAPACITY);
        else st->len[b] += n + 1;
        st->inflight[b] = 0;
    }
}

// Launch of `units` clusters of cs CTAs.
template <class... P, class... A>
static int launch_clusters(void (*kernel)(P...), int units, int cs, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * cs)); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = pdl_enabled();
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cs; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) == cudaSuccess ? CASS_OK : CASS_ERR_CUDA;
}

int launch_softmax(const float* logits, int rows, int vocab, float temperature, float* probs, cudaStream_t s) {
    // CTAs a row: about 4096 values each, at most the portable 8
    int cs = 1;
    while (cs < 8 && cs * 4096 < vocab) cs *= 2;
    const int per = ceil_div(vocab, cs), nv = ceil_div(per, kSoftmaxThreads);
    const float inv_t = 1.f / temperature;
    if (nv <= 2) return launch_clusters(k_softmax_rows<2>, rows, cs, kSoftmaxThreads, 0, s, logits, vocab, per, inv_t, probs);
    if (nv <= 8) return launch_clusters(k_softmax_rows<8>, rows, cs, kSoftmaxThreads, 0, s, logits, vocab, per, inv_t, probs);
    if (nv <= 16) return launch_clusters(k_softmax_rows<16>, rows, cs, kSoftmaxThreads, 0, s, logits, vocab, per, inv_t, probs);
    if (nv <= 32) return launch_clusters(k_softmax_rows<32>, rows, cs, kSoftmaxThreads, 0, s, logits, vocab, per, inv_t, probs);
    if (nv <= 40) return launch_clusters(k_softmax_rows<40>, rows, cs, kSoftmaxThreads, 0, s, logits, vocab, per, inv_t, probs);
    CASS_PDL_LAUNCH(k_softmax_rows_long, dim3(rows), dim3(1024), 0, s, logits, vocab, inv_t, probs);
    return CASS_OK;
}

// CTAs a draw, and the shared memory each needs: its segments of the vocabulary (0: too many to stage)
static size_t draw_plan(int vocab, int* cs) {
    *cs = 1;
    while (*cs < 8 && *cs * 2048 < vocab) *cs *= 2;
    const size_t smem = (size_t)(kSampleThreads / *cs) * draw_stride(vocab) * 4;
    return smem <= 220 * 1024 ? smem : 0;                                  // vocabularies up to 450000
}

int launch_sample(const float* probs, int rows, int vocab, const float* u, int32_t* tokens, int tok_stride, cudaStream_t s) {
    int cs;
    const size_t smem = draw_plan(vocab, &cs);
    if (!smem) return launch_clusters(k_sample_rows<false>, rows, cs, kSampleThreads, 0, s, probs, vocab, u, tokens, tok_stride);
    CASS_ALLOW_SMEM(k_sample_rows<true>);
    return launch_clusters(k_sample_rows<true>, rows, cs, kSampleThreads, smem, s, probs, vocab, u, tokens, tok_stride);
}

int launch_accept_sampling(DevState* st, int n_seq, const int32_t* draft, int draft_stride, const float* p, const float* q,
                           int vocab, const float* r, const float* u, int g, int32_t* n_acc, int32_t* out_tokens,
                           int32_t* next_tok, int next_stride, cudaStream_t s) {
    int cs;
    const size_t smem = draw_plan(vocab, &cs);
    auto kernel = smem ? k_accept_sampling<true> : k_accept_sampling<false>;
    CASS_ALLOW_SMEM(k_accept_sampling<true>);
    return launch_clusters(kernel, n_seq, cs, kSampleThreads, smem, s, st, draft, draft_stride, p, q, vocab, r, u, g, n_acc, out_tokens,
                           next_tok, next_stride);
}

}  // namespace cass

using namespace cass;

extern "C" int cass_softmax(const float* logits, int rows, int vocab, float temperature, float* probs, void* stream) {
    if (!logits || !probs || rows < 0 || vocab <= 0 || !(temperature > 0.f)) return CASS_ERR_INVALID_ARG;
    if (rows == 0) return CASS_OK;
    return launch_softmax(logits, rows, vocab, temperature, probs, (cudaStream_t)stream);
}

extern "C" int cass_sample(const float* probs, int rows, int vocab, const float* u, int32_t* tokens, int tok_stride,
                           void* stream) {
    if (!probs || !u || !tokens || rows < 0 || vocab <= 0 || tok_stride < 1) return CASS_ERR_INVALID_ARG;
    if (rows == 0) return CASS_OK;
    return launch_sample(probs, rows, vocab, u, tokens, tok_stride, (cudaStream_t)stream);
}
