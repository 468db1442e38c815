// Group-lasso regularised momentum SGD over all conv weights (Eq. 1-2, Algorithm 1) and
// zero-group detection (Sec. 4.1 threshold, Sec. 4.2 max-abs per channel).
//
// All layers are processed by one launch per phase through a chunk table. A weight tensor [K][RS][C] is seen as K*RS "lines" of C
// contiguous floats, cut into column groups of up to 128 columns (of equal width: 143 columns are 96 + 47, not 128 + 15); a chunk is
// a run of lines of one column group. A warp takes a few lines of its chunk at a time: lane l owns the columns l, l + 32, l + 64,
// l + 96 of the group (four consecutive ones and 16-byte accesses where C is a multiple of 128), so that every access is a coalesced
// run of a line, per-column quantities stay in registers for the whole chunk, and a line's total is up to four values per lane away
// from a warp reduction: a third of a shuffle per element, where one column per lane had more than one (norms of 15.5 M parameters
// 29.7 -> 24 us, detection over 23.5 M 32.6 -> 23 us, finishing launch included).
//
// One kernel template walks the chunks:
//   group_kernel<UPD, SUM, MAX, FLAG>  UPD: g~, v, w, bf16 shadow (reads w, g, v; writes w, v, shadow)
//                         SUM: per line and per (chunk, column) sums of squares of the weights (the new ones with UPD)
//                         MAX: the same for the maxima of |w| (bit patterns: ordered like the values, a NaN sorts above +inf)
//                         FLAG: the same for "some |w| is not below the threshold" (a NaN is not below)
//   <0,1,0,0> group norms of W_i;  <1,0,0,0> the update;  <1,1,1,0> the carried update, which leaves the sums and maxima of
//   W_{i+1} so that the next step needs no pass over the weights of its own;  <0,0,0,1> zero-group detection.
//   finish   fixed-order combination to s_out[k], s_in[c], the 1/norm factors, the Eq. 2 sum (last block, by ticket), the
//            group maxima and, for the detection, the zero masks. (Finishing a layer in its last block, by ticket, instead of in a
//            launch of its own was slower: fence, ticket, fence and one block's loads in a row, 8 us behind the largest layers.)
// No floating-point atomics and fixed reduction orders: results are run-to-run identical.
#include "pt_internal.h"

namespace {

struct LayerDev {
    float *w; const float *g; float *v; __nv_bfloat16 *wb;
    float *sumsq_out, *sumsq_in;
    uint8_t *zero_out, *zero_in;
    int K, C, RS, ldw;
    int reg_in, reg_out;
    int n_cg, cgw;              // column groups and their width (a multiple of 32, at most 128)
    int n_lc;                   // line chunks
    int vec;                    // 16-byte accesses: C is a multiple of 128 and the tensors are aligned
    long long line_off;         // offset of this layer's per-line partials (lines * n_cg)
    long long col_off;          // offset of this layer's column partials (n_lc * C)
    long long k_off, c_off;     // offsets into the per-K / per-C arrays
};

// A chunk is a run of lines of one layer restricted to one column group, nsub * 32 lanes wide.
struct Chunk { int layer, line0, nlines, cg, lc, nsub, pad0, pad1; };

// kind 0: 32 output-channel groups from `start` (four per warp); kind 1: 32 input-channel groups from `start` (x 8 slices of the chunks)
struct FinishJob { int layer, kind, start, pad; };

struct WsLayout { size_t linesum, colpart, linemax, colmax, inv_out, inv_in, gmax_out, gmax_in, job_reg, ticket, total; };

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// Elements of a chunk, one block of a pass with per-chunk results: 16384 for models of 12 M parameters or more, else 4096 (never less
// than 64 lines). The plain update has no per-chunk results: several blocks share a chunk.
// (15.5 M parameters: 4096 / 8192 / 16384 take 25.7 / 25.8 / 24.1 us for the norms and 75 / 71 / 66 us for the update.)
constexpr int kChunk = 16384, kChunkSmall = 4096;
constexpr long long kSmallModel = 12ll << 20;
constexpr int kUpdateSplit = 4, kUpdateSplitSmall = 2;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// U per-lane values (one per line) are reduced over the 32 lanes: log2(U) halving exchanges leave lane l with the partial of line
// l / (32 / U) over its group of 32 / U lanes, the rest of the butterfly adds the lanes of a group (U = 8: 9 shuffles instead of
// 40). The tree is fixed, so the result is run-to-run identical. Returns the line's total in every lane of its group.
template <int U, typename T, typename Op>
__device__ __forceinline__ T warp_reduce(T (&v)[U], int lane, Op op)
{
#pragma unroll
    for (int half = U / 2, bit = 16; half >= 1; half >>= 1, bit >>= 1)
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const bool hi = lane & bit;
            const T send = hi ? v[i] : v[i + half], keep = hi ? v[i + half] : v[i];
            v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, bit));
        }
#pragma unroll
    for (int bit = 16 / U; bit >= 1; bit >>= 1) v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], bit));
    return v[0];
}
struct OpAdd { __device__ __forceinline__ float operator()(float a, float b) const { return a + b; } };
struct OpMax { __device__ __forceinline__ unsigned int operator()(unsigned int a, unsigned int b) const { return a > b ? a : b; } };

struct GroupP {
    const LayerDev *layers;
    const Chunk *chunks;
    float *inv_out, *inv_in;
    float *linesum, *colpart;
    unsigned *linemax, *colmax, *gmax_out, *gmax_in;
    double *job_reg;
    unsigned *ticket;           // arrivals of the finish launch's blocks; cleared by the sweep in front of it
    pt_sgd_hparams hp;
    float thr;
    int split;                  // blocks that share a chunk (the plain update)
    int reverse;                // chunks from the last to the first: the update finds the end of what the norms read in L2
};

// A thread's elements of one line: NS scalars 32 columns apart, or one 16-byte vector.
template <int NS, bool VEC>
__device__ __forceinline__ void line_load(const float *__restrict__ p, const bool (&on)[4], float (&o)[4])
{
    if (VEC) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    } else {
#pragma unroll
        for (int j = 0; j < NS; ++j)
            if (on[j]) o[j] = p[32 * j];
    }
}

template <bool UPD, bool SUM, bool MAX, bool FLAG, int NS, bool VEC>
__device__ __forceinline__ void chunk_body(const GroupP &p, const LayerDev &L, const Chunk &ch, int sub, float *s_col, unsigned *s_colm)
{
    constexpr bool RED = SUM || MAX || FLAG;
    // lines in flight: 8 to 16 elements of three tensors, or up to 32 elements of one, per thread
    constexpr int U = UPD ? (NS == 1 ? 8 : 4) : 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = ch.cg * L.cgw + (VEC ? lane * 4 : lane);
    bool on[4];
    float ci[4], cacc[4];
    unsigned cm[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        on[j] = VEC || (j < NS && c0 + 32 * j < L.C);
        ci[j] = 0.f; cacc[j] = 0.f; cm[j] = 0u;
        if (UPD && on[j]) ci[j] = p.inv_in[L.c_off + c0 + (VEC ? j : 32 * j)];
    }
    const float *io = p.inv_out + L.k_off;
    const int SPLIT = RED ? 1 : p.split;
    for (int l = (sub * kWarps + warp) * U; l < ch.nlines; l += SPLIT * kWarps * U) {
        float w[U][4], g[UPD ? U : 1][4], v[UPD ? U : 1][4], ko[UPD ? U : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool lv = l + u < ch.nlines;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[u][j] = 0.f;
            if (lv) {
                const int line = ch.line0 + l + u;
                const size_t i = (size_t)line * L.C + c0;
                line_load<NS, VEC>(L.w + i, on, w[u]);
                if (UPD) {
                    line_load<NS, VEC>(L.g + i, on, g[u]);
                    line_load<NS, VEC>(L.v + i, on, v[u]);
                    ko[u] = io[line / L.RS];
                }
            }
        }
        if (UPD) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (l + u >= ch.nlines) continue;
                const int line = ch.line0 + l + u;
                const size_t i = (size_t)line * L.C + c0;
                __nv_bfloat16 *wb = L.wb ? L.wb + (size_t)line * L.ldw + c0 : nullptr;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (!on[j]) continue;
                    const float gt = g[u][j] + p.hp.weight_decay * w[u][j] + p.hp.lambda * w[u][j] * (ko[u] + ci[j]);
                    v[u][j] = p.hp.momentum * v[u][j] + gt;
                    w[u][j] = w[u][j] - p.hp.lr * v[u][j];
                    if (!VEC) {
                        L.v[i + 32 * j] = v[u][j];
                        L.w[i + 32 * j] = w[u][j];
                        if (wb) wb[32 * j] = __float2bfloat16_rn(w[u][j]);
                    }
                }
                if (VEC) {
                    *reinterpret_cast<float4 *>(L.v + i) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
                    *reinterpret_cast<float4 *>(L.w + i) = make_float4(w[u][0], w[u][1], w[u][2], w[u][3]);
                    if (wb) {
                        const __nv_bfloat162 h0 = __floats2bfloat162_rn(w[u][0], w[u][1]), h1 = __floats2bfloat162_rn(w[u][2], w[u][3]);
                        *reinterpret_cast<uint2 *>(wb) = make_uint2(*reinterpret_cast<const unsigned *>(&h0), *reinterpret_cast<const unsigned *>(&h1));
                    }
                }
            }
        }
        if constexpr (RED) {
        const int lu = lane / (32 / U);                  // the line whose total a warp reduction leaves in this lane
        const bool writer = (lane & (32 / U - 1)) == 0 && l + lu < ch.nlines;
        const size_t o = (size_t)(L.line_off + (long long)(ch.line0 + l + lu) * L.n_cg + ch.cg);
        if (FLAG) {
            unsigned lf = 0u;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                bool any = false;
#pragma unroll
                for (int j = 0; j < NS; ++j) {
                    const bool alive = on[j] && l + u < ch.nlines && !(fabsf(w[u][j]) < p.thr);
                    cm[j] |= alive ? 1u : 0u;
                    any |= alive;
                }
                const bool r = __any_sync(0xffffffffu, any);
                if (u == lu) lf = r ? 1u : 0u;
            }
            if (writer) p.linemax[o] = lf;
        }
        if (MAX) {
            unsigned b[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                b[u] = 0u;
#pragma unroll
                for (int j = 0; j < NS; ++j) {
                    const unsigned m = on[j] ? __float_as_uint(w[u][j]) & 0x7fffffffu : 0u;
                    cm[j] = max(cm[j], m);
                    b[u] = max(b[u], m);
                }
            }
            const unsigned tot = warp_reduce<U>(b, lane, OpMax());
            if (writer) p.linemax[o] = tot;
        }
        if (SUM) {
            float q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                q[u] = 0.f;
#pragma unroll
                for (int j = 0; j < NS; ++j) {
                    const float t = w[u][j] * w[u][j];
                    cacc[j] += t;
                    q[u] += t;
                }
            }
            const float tot = warp_reduce<U>(q, lane, OpAdd());
            if (writer) p.linesum[o] = tot;
        }
        }
    }
    if constexpr (!RED) return;
    // the warps' column partials, to be added in order
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const int c = VEC ? lane * 4 + j : lane + 32 * j;
        if (SUM) s_col[warp * 128 + c] = cacc[j];
        if (MAX || FLAG) s_colm[warp * 128 + c] = cm[j];
    }
}

template <bool UPD, bool SUM, bool MAX, bool FLAG>
__global__ void __launch_bounds__(kThreads) group_kernel(const GroupP p)
{
    constexpr bool RED = SUM || MAX || FLAG;
    const int SPLIT = RED ? 1 : p.split;
    __shared__ float s_col[SUM ? kWarps * 128 : 1];
    __shared__ unsigned s_colm[(MAX || FLAG) ? kWarps * 128 : 1];
    const unsigned bi = p.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const Chunk ch = p.chunks[bi / SPLIT];
    const int sub = (int)(bi % SPLIT);
    const LayerDev L = p.layers[ch.layer];
    pdl_wait();
    // A sweep that writes the weights lets its dependents start only when it has completed: the convolution kernels' weight
    // producers do not wait for their predecessor (weights are never written by a kernel that releases its dependents early),
    // and a convolution may well be the next launch of the stream.
    if (!UPD) pdl_trigger();
    if (SUM && blockIdx.x == 0 && threadIdx.x == 0) *p.ticket = 0u;
    if (L.vec) chunk_body<UPD, SUM, MAX, FLAG, 4, true>(p, L, ch, sub, s_col, s_colm);
    else if (ch.nsub == 4) chunk_body<UPD, SUM, MAX, FLAG, 4, false>(p, L, ch, sub, s_col, s_colm);
    else if (ch.nsub == 3) chunk_body<UPD, SUM, MAX, FLAG, 3, false>(p, L, ch, sub, s_col, s_colm);
    else if (ch.nsub == 2) chunk_body<UPD, SUM, MAX, FLAG, 2, false>(p, L, ch, sub, s_col, s_colm);
    else chunk_body<UPD, SUM, MAX, FLAG, 1, false>(p, L, ch, sub, s_col, s_colm);
    if constexpr (!RED) return;
    __syncthreads();
    const int e = threadIdx.x, c = ch.cg * L.cgw + e;
    if (e >= 32 * ch.nsub || c >= L.C) return;
    const size_t o = (size_t)(L.col_off + (long long)ch.lc * L.C + c);
    if (SUM) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += s_col[w * 128 + e];
        p.colpart[o] = s;
    }
    if (MAX || FLAG) {
        unsigned m = 0u;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = max(m, s_colm[w * 128 + e]);
        p.colmax[o] = m;
    }
}

// ---- finish
template <bool SUM, bool MAX, bool FLAG>
__global__ void __launch_bounds__(kThreads) finish_kernel(const GroupP p, const FinishJob *__restrict__ jobs, double *reg_out)
{
    __shared__ double s_red[kWarps];
    __shared__ float s_ps[kWarps][32];
    __shared__ unsigned s_pm[kWarps][32];
    __shared__ unsigned s_last;
    const FinishJob J = jobs[blockIdx.x];
    const LayerDev L = p.layers[J.layer];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();
    pdl_trigger();
    double reg = 0.0;
    if (J.kind == 0) {
        // a group's partials, one per (line, column group), are consecutive: the lanes take them in turn, then a fixed butterfly
        const int np = L.RS * L.n_cg, k0 = J.start + warp * 4;
        float s[4];
        unsigned m[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            s[u] = 0.f; m[u] = 0u;
            if (k0 + u >= L.K) continue;
            const long long at = L.line_off + (long long)(k0 + u) * np;
            for (int e = lane; e < np; e += 32) {
                if (SUM) s[u] += p.linesum[at + e];
                if (MAX || FLAG) m[u] = max(m[u], p.linemax[at + e]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (SUM)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
            if (MAX || FLAG) m[u] = __reduce_max_sync(0xffffffffu, m[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u;
            if (lane != u || k >= L.K) continue;
            if (SUM) {
                L.sumsq_out[k] = s[u];
                p.inv_out[L.k_off + k] = (L.reg_out && s[u] > 1e-24f) ? rsqrtf(s[u]) : 0.f;
                if (L.reg_out) reg = (double)sqrtf(s[u]);
            }
            if (MAX) p.gmax_out[L.k_off + k] = m[u];
            if (FLAG) L.zero_out[k] = m[u] ? 0 : 1;
        }
    } else {
        const int c = J.start + lane;
        float s = 0.f;
        unsigned m = 0u;
        if (c < L.C)
#pragma unroll 4
            for (int e = warp; e < L.n_lc; e += kWarps) {                  // this slice in ascending order
                const size_t at = (size_t)(L.col_off + (long long)e * L.C + c);
                if (SUM) s += p.colpart[at];
                if (MAX || FLAG) m = max(m, p.colmax[at]);
            }
        s_ps[warp][lane] = s;
        s_pm[warp][lane] = m;
        __syncthreads();
        if (warp == 0 && c < L.C) {
            float t = 0.f;
            unsigned q = 0u;
#pragma unroll
            for (int y = 0; y < kWarps; ++y) { t += s_ps[y][lane]; q = max(q, s_pm[y][lane]); }     // the slices in ascending order
            if (SUM) {
                L.sumsq_in[c] = t;
                p.inv_in[L.c_off + c] = (L.reg_in && t > 1e-24f) ? rsqrtf(t) : 0.f;
                if (L.reg_in) reg = (double)sqrtf(t);
            }
            if (MAX) p.gmax_in[L.c_off + c] = q;
            if (FLAG) L.zero_in[c] = q ? 0 : 1;
        }
    }
    if constexpr (!SUM) return;
    if (!reg_out) return;
    // Eq. 2 without lambda: per-block sum by a fixed tree (shuffles inside a warp, then the eight warps in order), then the
    // last block to finish adds the blocks' sums in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) reg += __shfl_xor_sync(0xffffffffu, reg, o);
    if (lane == 0) s_red[warp] = reg;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) tot += s_red[w];
        p.job_reg[blockIdx.x] = tot;
        __threadfence();
        s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1u ? 1u : 0u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kThreads) t += __ldcg(p.job_reg + i);     // strided slices, ascending
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    __syncthreads();
    if (lane == 0) s_red[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) tot += s_red[w];
        *reg_out = tot;
    }
}

// ---- zero masks from the group maxima a carried update left in the workspace
__global__ void masks_kernel(const LayerDev *__restrict__ layers, const unsigned *__restrict__ gmax_out,
                             const unsigned *__restrict__ gmax_in, float thr)
{
    const LayerDev L = layers[blockIdx.x];
    pdl_wait();
    for (int k = threadIdx.x; k < L.K; k += blockDim.x) L.zero_out[k] = (__uint_as_float(gmax_out[L.k_off + k]) < thr) ? 1 : 0;
    for (int c = threadIdx.x; c < L.C; c += blockDim.x) L.zero_in[c] = (__uint_as_float(gmax_in[L.c_off + c]) < thr) ? 1 : 0;
}

// ---- in-place zeroing of the detected groups (weights, momentum, shadow)
__global__ void __launch_bounds__(kThreads) zero_groups_kernel(const LayerDev *__restrict__ layers, const Chunk *__restrict__ chunks)
{
    const Chunk ch = chunks[blockIdx.x];
    const LayerDev L = layers[ch.layer];
    const int e = threadIdx.x & 127, c = ch.cg * L.cgw + e;
    pdl_wait();
    if (e >= L.cgw || c >= L.C) return;
    const bool zc = L.zero_in[c] != 0;
    for (int l = threadIdx.x >> 7; l < ch.nlines; l += kThreads / 128) {
        const int line = ch.line0 + l;
        if (zc || L.zero_out[line / L.RS]) {
            L.w[(size_t)line * L.C + c] = 0.f;
            L.v[(size_t)line * L.C + c] = 0.f;
            if (L.wb) L.wb[(size_t)line * L.ldw + c] = __float2bfloat16_rn(0.f);
        }
    }
}

// ---------------------------------------------------------------------------------- host side
struct Tables {
    std::vector<LayerDev> layers;
    std::vector<Chunk> chunks;             // grouped by layer, layers in the caller's order
    std::vector<int> first_chunk;          // per layer
    std::vector<FinishJob> jobs;
    bool small;
    WsLayout ws;
};

bool vec_aligned(const void *p) { return ((uintptr_t)p & 15) == 0; }

pt_status build_tables(const pt_layer *layers, int n, Tables *t)
{
    if (!layers || n <= 0) return PT_ERR_INVALID_ARG;
    t->layers.resize(n);
    t->first_chunk.assign(n, 0);
    t->chunks.clear();
    t->jobs.clear();
    long long line_off = 0, col_off = 0, k_off = 0, c_off = 0;
    long long params = 0;
    for (int i = 0; i < n; ++i) params += (long long)layers[i].K * layers[i].RS * layers[i].C;
    t->small = params < kSmallModel;
    const int elems = t->small ? kChunkSmall : kChunk;
    for (int i = 0; i < n; ++i) {
        const pt_layer &s = layers[i];
        if (!s.w || !s.v || s.K <= 0 || s.C <= 0 || s.RS <= 0) return PT_ERR_INVALID_ARG;
        if (s.w_bf16 && (s.ldw < s.C || s.ldw % 8)) return PT_ERR_INVALID_ARG;
        if ((long long)s.K * s.RS * (long long)(s.ldw > s.C ? s.ldw : s.C) >= (1ll << 31)) return PT_ERR_UNSUPPORTED;
        LayerDev &d = t->layers[i];
        memset(&d, 0, sizeof(d));
        d.w = s.w; d.g = s.g; d.v = s.v; d.wb = (__nv_bfloat16 *)s.w_bf16;
        d.sumsq_out = s.sumsq_out; d.sumsq_in = s.sumsq_in; d.zero_out = s.zero_out; d.zero_in = s.zero_in;
        d.K = s.K; d.C = s.C; d.RS = s.RS; d.ldw = s.ldw;
        d.reg_in = s.reg_in; d.reg_out = s.reg_out;
        d.vec = s.C % 128 == 0 && vec_aligned(s.w) && vec_aligned(s.g) && vec_aligned(s.v) && vec_aligned(s.w_bf16) ? 1 : 0;
        const int lines = s.K * s.RS;
        d.n_cg = pt_ceil_div(s.C, 128);
        d.cgw = 32 * pt_ceil_div(pt_ceil_div(s.C, 32), d.n_cg);
        d.n_cg = pt_ceil_div(s.C, d.cgw);
        // lines of a chunk: `elems` elements at the width of the layer's widest column group, whole rounds of 8 lines per warp; more
        // for tall tensors so that no column has more than ~32 chunk partials to add up
        int lpc = elems / d.cgw / 64 * 64;
        if (lpc < 64) lpc = 64;
        while (lines > 32 * lpc) lpc *= 2;
        d.n_lc = pt_ceil_div(lines, lpc);
        t->first_chunk[i] = (int)t->chunks.size();
        for (int lc = 0; lc < d.n_lc; ++lc)
            for (int cg = 0; cg < d.n_cg; ++cg) {
                Chunk ch;
                ch.layer = i; ch.line0 = lc * lpc;
                ch.nlines = lines - ch.line0 < lpc ? lines - ch.line0 : lpc;
                ch.cg = cg; ch.lc = lc;
                ch.nsub = pt_ceil_div(s.C - cg * d.cgw < d.cgw ? s.C - cg * d.cgw : d.cgw, 32);
                ch.pad0 = ch.pad1 = 0;
                t->chunks.push_back(ch);
            }
        for (int k0 = 0; k0 < s.K; k0 += 32) t->jobs.push_back(FinishJob{i, 0, k0, 0});
        for (int c0 = 0; c0 < s.C; c0 += 32) t->jobs.push_back(FinishJob{i, 1, c0, 0});
        d.line_off = line_off; line_off += (long long)lines * d.n_cg;
        d.col_off = col_off;   col_off += (long long)d.n_lc * s.C;
        d.k_off = k_off;       k_off += s.K;
        d.c_off = c_off;       c_off += s.C;
    }
    WsLayout &w = t->ws;
    size_t o = 0;
    w.linesum = o;  o = pt_align_up(o + (size_t)line_off * 4, 256);
    w.colpart = o;  o = pt_align_up(o + (size_t)col_off * 4, 256);
    w.linemax = o;  o = pt_align_up(o + (size_t)line_off * 4, 256);
    w.colmax = o;   o = pt_align_up(o + (size_t)col_off * 4, 256);
    w.inv_out = o;  o = pt_align_up(o + (size_t)k_off * 4, 256);
    w.inv_in = o;   o = pt_align_up(o + (size_t)c_off * 4, 256);
    w.gmax_out = o; o = pt_align_up(o + (size_t)k_off * 4, 256);
    w.gmax_in = o;  o = pt_align_up(o + (size_t)c_off * 4, 256);
    w.job_reg = o;  o = pt_align_up(o + t->jobs.size() * 8, 256);
    w.ticket = o;   o += 256;
    w.total = o;
    return PT_OK;
}

// The tables of a set of layers on the device: [LayerDev * n][Chunk * m][FinishJob * j]. A set that one of the slots was last built from (the same
// array contents: shapes, pointers) costs a comparison of a few kilobytes; building and comparing the tables takes 30 us for a
// ResNet-50, more than the launches.
struct Bound {
    const LayerDev *dl; const Chunk *dc; const FinishJob *dj;
    const pt_group_slot *slot;
    GroupP p;
};

pt_status bind(pt_ctx *c, const pt_layer *layers, int n, bool detect, void *ws, size_t ws_bytes, cudaStream_t st, Bound *b)
{
    if (!layers || n <= 0) return PT_ERR_INVALID_ARG;
    pt_group_slot *slots = detect ? c->detect_tab : c->lasso_tab;
    const int n_slots = detect ? 2 : 3;
    pt_group_slot *s = nullptr;
    for (int i = 0; i < n_slots && !s; ++i)
        if (slots[i].reg.valid && slots[i].args.size() == (size_t)n * sizeof(pt_layer) && memcmp(slots[i].args.data(), layers, n * sizeof(pt_layer)) == 0)
            s = &slots[i];
    if (!s) {
        Tables t;
        pt_status r = build_tables(layers, n, &t);
        if (r != PT_OK) return r;
        const size_t lb = pt_align_up(t.layers.size() * sizeof(LayerDev), 256), cb = pt_align_up(t.chunks.size() * sizeof(Chunk), 256);
        std::vector<char> buf(lb + cb + t.jobs.size() * sizeof(FinishJob), 0);
        memcpy(buf.data(), t.layers.data(), t.layers.size() * sizeof(LayerDev));
        memcpy(buf.data() + lb, t.chunks.data(), t.chunks.size() * sizeof(Chunk));
        memcpy(buf.data() + lb + cb, t.jobs.data(), t.jobs.size() * sizeof(FinishJob));
        // a slot that already holds these bytes is reused, otherwise the oldest one is overwritten
        int *next = detect ? &c->detect_next : &c->lasso_next;
        for (int i = 0; i < n_slots && !s; ++i)
            if (slots[i].reg.valid && slots[i].reg.key.size() == buf.size() && memcmp(slots[i].reg.key.data(), buf.data(), buf.size()) == 0) s = &slots[i];
        if (!s) {
            s = &slots[*next % n_slots];
            *next = (*next + 1) % n_slots;
        }
        char *dev = nullptr;
        s->args.clear();
        r = pt_upload_table(c, &s->reg, buf.data(), buf.size(), st, &dev);
        if (r != PT_OK) return r;
        s->chunks_off = lb; s->n_chunks = (unsigned)t.chunks.size();
        s->small = t.small;
        s->jobs_off = lb + cb; s->n_jobs = (unsigned)t.jobs.size();
        s->first_chunk = t.first_chunk;
        static_assert(sizeof(WsLayout) == sizeof(s->ws), "layout of the workspace");
        memcpy(s->ws, &t.ws, sizeof(t.ws));
        s->args.assign((const char *)layers, (const char *)(layers + n));
    }
    WsLayout w;
    memcpy(&w, s->ws, sizeof(w));
    if (!ws || ws_bytes < w.total || ((uintptr_t)ws & 255)) return PT_ERR_WORKSPACE;
    b->slot = s;
    b->dl = (const LayerDev *)s->reg.dev;
    b->dc = (const Chunk *)(s->reg.dev + s->chunks_off);
    b->dj = (const FinishJob *)(s->reg.dev + s->jobs_off);
    char *a = (char *)ws;
    GroupP &p = b->p;
    memset(&p, 0, sizeof(p));
    p.layers = b->dl; p.chunks = b->dc;
    p.linesum = (float *)(a + w.linesum); p.colpart = (float *)(a + w.colpart);
    p.linemax = (unsigned *)(a + w.linemax); p.colmax = (unsigned *)(a + w.colmax);
    p.inv_out = (float *)(a + w.inv_out); p.inv_in = (float *)(a + w.inv_in);
    p.gmax_out = (unsigned *)(a + w.gmax_out); p.gmax_in = (unsigned *)(a + w.gmax_in);
    p.job_reg = (double *)(a + w.job_reg);
    p.ticket = (unsigned *)(a + w.ticket);
    return PT_OK;
}

template <bool SUM, bool MAX, bool FLAG>
pt_status launch_finish(pt_ctx *c, const Bound &b, double *reg_out, cudaStream_t st)
{
    PT_CUDA_OK(pt_launch_pdl(finish_kernel<SUM, MAX, FLAG>, dim3(b.slot->n_jobs), dim3(kThreads), 0, st, b.p, b.dj, reg_out));
    c->launches += 1;
    return PT_OK;
}

}  // namespace

extern "C" size_t pt_group_lasso_workspace_bytes(const pt_ctx *c, const pt_layer *layers, int32_t n)
{
    (void)c;
    Tables t;
    if (build_tables(layers, n, &t) != PT_OK) return 0;
    return t.ws.total;
}

// phases: 1 = group norms of the current weights (sweep + finish), 2 = parameter update from the factors in the workspace,
// 4 = the update also leaves the sums of squares of the new weights, and a finish follows it (carried form); 8 = and their
// maxima (for pt_find_zero_groups_carried).
// The update may be restricted to layers [first, first + count) (count < 0: all): the chunk table is ordered by layer.
static pt_status lasso_phases(pt_ctx *c, const pt_layer *layers, int32_t n, const pt_sgd_hparams *hp, double *reg_sum_out, void *ws,
                              size_t ws_bytes, void *stream, int phases, int first = 0, int count = -1)
{
    if (!c || ((phases & 2) && !hp)) return PT_ERR_INVALID_ARG;
    if (count >= 0 && (first < 0 || first + count > n)) return PT_ERR_INVALID_ARG;
    if (!layers || n <= 0) return PT_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i)
        if (((phases & 2) && !layers[i].g) || !layers[i].sumsq_out || !layers[i].sumsq_in) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    Bound b;
    pt_status s = bind(c, layers, n, false, ws, ws_bytes, st, &b);
    if (s != PT_OK) return s;
    const unsigned nch = b.slot->n_chunks;
    if (phases & 1) {
        PT_CUDA_OK(pt_launch_pdl(group_kernel<false, true, false, false>, dim3(nch), dim3(kThreads), 0, st, b.p));
        c->launches += 1;
        s = launch_finish<true, false, false>(c, b, reg_sum_out, st);
        if (s != PT_OK) return s;
    }
    if (phases & 2) {
        unsigned c0 = 0, c1 = nch;
        if (count >= 0) {
            const std::vector<int> &fc = b.slot->first_chunk;
            c0 = count > 0 ? (unsigned)fc[first] : 0;
            c1 = count > 0 ? (first + count < n ? (unsigned)fc[first + count] : nch) : 0;
        }
        if (c1 > c0) {
            GroupP p = b.p;
            p.hp = *hp;
            p.chunks = b.dc + c0;
            if ((phases & 4) && (phases & 8)) PT_CUDA_OK(pt_launch_pdl(group_kernel<true, true, true, false>, dim3(c1 - c0), dim3(kThreads), 0, st, p));
            else if (phases & 4) PT_CUDA_OK(pt_launch_pdl(group_kernel<true, true, false, false>, dim3(c1 - c0), dim3(kThreads), 0, st, p));
            else {
                p.reverse = (phases & 1) ? 1 : 0;
                p.split = b.slot->small ? kUpdateSplitSmall : kUpdateSplit;
                PT_CUDA_OK(pt_launch_pdl(group_kernel<true, false, false, false>, dim3((c1 - c0) * (unsigned)p.split), dim3(kThreads), 0, st, p));
            }
            c->launches += 1;
        }
        if (phases & 4) {
            s = (phases & 8) ? launch_finish<true, true, false>(c, b, reg_sum_out, st) : launch_finish<true, false, false>(c, b, reg_sum_out, st);
            if (s != PT_OK) return s;
        }
    }
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

extern "C" pt_status pt_group_lasso_sgd_step(pt_ctx *c, const pt_layer *layers, int32_t n, const pt_sgd_hparams *hp,
                                             double *reg_sum_out, void *ws, size_t ws_bytes, void *stream)
{
    return lasso_phases(c, layers, n, hp, reg_sum_out, ws, ws_bytes, stream, 3);
}

extern "C" pt_status pt_group_lasso_norms(pt_ctx *c, const pt_layer *layers, int32_t n, double *reg_sum_out, void *ws,
                                          size_t ws_bytes, void *stream)
{
    return lasso_phases(c, layers, n, nullptr, reg_sum_out, ws, ws_bytes, stream, 1);
}

extern "C" pt_status pt_group_lasso_sgd_apply(pt_ctx *c, const pt_layer *layers, int32_t n, const pt_sgd_hparams *hp, void *ws,
                                              size_t ws_bytes, void *stream)
{
    return lasso_phases(c, layers, n, hp, nullptr, ws, ws_bytes, stream, 2);
}

extern "C" pt_status pt_group_lasso_sgd_apply_layers(pt_ctx *c, const pt_layer *layers, int32_t n, int32_t first, int32_t count,
                                                     const pt_sgd_hparams *hp, void *ws, size_t ws_bytes, void *stream)
{
    if (count < 0) return PT_ERR_INVALID_ARG;
    return lasso_phases(c, layers, n, hp, nullptr, ws, ws_bytes, stream, 2, first, count);
}

extern "C" pt_status pt_group_lasso_sgd_step_carried(pt_ctx *c, const pt_layer *layers, int32_t n, const pt_sgd_hparams *hp,
                                                     int32_t with_maxima, double *reg_sum_next, void *ws, size_t ws_bytes, void *stream)
{
    return lasso_phases(c, layers, n, hp, reg_sum_next, ws, ws_bytes, stream, 2 | 4 | (with_maxima ? 8 : 0));
}

extern "C" pt_status pt_find_zero_groups(pt_ctx *c, const pt_layer *layers, int32_t n, float threshold,
                                         int32_t zero_in_place, void *ws, size_t ws_bytes, void *stream)
{
    if (!c || !(threshold >= 0.f) || !layers || n <= 0) return PT_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i)
        if (!layers[i].zero_out || !layers[i].zero_in) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    Bound b;
    pt_status s = bind(c, layers, n, true, ws, ws_bytes, st, &b);
    if (s != PT_OK) return s;
    const unsigned nch = b.slot->n_chunks;
    b.p.thr = threshold;
    PT_CUDA_OK(pt_launch_pdl(group_kernel<false, false, false, true>, dim3(nch), dim3(kThreads), 0, st, b.p));
    c->launches += 1;
    s = launch_finish<false, false, true>(c, b, nullptr, st);
    if (s != PT_OK) return s;
    if (zero_in_place) {
        PT_CUDA_OK(pt_launch_pdl(zero_groups_kernel, dim3(nch), dim3(kThreads), 0, st, b.dl, b.dc));
        c->launches += 1;
    }
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

extern "C" pt_status pt_find_zero_groups_carried(pt_ctx *c, const pt_layer *layers, int32_t n, float threshold, int32_t zero_in_place,
                                                 void *ws, size_t ws_bytes, void *stream)
{
    if (!c || !(threshold >= 0.f) || !layers || n <= 0) return PT_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i)
        if (!layers[i].zero_out || !layers[i].zero_in) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    Bound b;
    pt_status s = bind(c, layers, n, false, ws, ws_bytes, st, &b);          // the table of the step that left the maxima
    if (s != PT_OK) return s;
    const unsigned nch = b.slot->n_chunks;
    PT_CUDA_OK(pt_launch_pdl(masks_kernel, dim3((unsigned)n), dim3(256u), 0, st, b.dl, (const unsigned *)b.p.gmax_out, (const unsigned *)b.p.gmax_in, threshold));
    c->launches += 1;
    if (zero_in_place) {
        PT_CUDA_OK(pt_launch_pdl(zero_groups_kernel, dim3(nch), dim3(kThreads), 0, st, b.dl, b.dc));
        c->launches += 1;
    }
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}
