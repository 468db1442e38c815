// Channel gating (Sec. 4.2, the alternative to channel union): a residual branch reads only the dense input channels of
// its first convolution out of the shared node tensor (gather) and its last convolution's dense output channels are put
// back at their positions in the node where the residual add happens (scatter-add). Both are pure data movement over
// NHWC bf16 tensors -- the tensor reshaping whose memory traffic the paper measured -- plus the list of dense channels.
// The gradient of the gather is the scatter-add and vice versa, so the two kernels serve both passes.
#include "pt_internal.h"
#include "pt_sm100_ptx.cuh"

namespace {

constexpr int kGateMax = 4096;          // channels of a node / of a selection (index tables live in shared memory)
constexpr int kGateThreads = 256;

// An index outside the tensor is skipped (nothing is read or written there) and reported through the status word.
__device__ __forceinline__ void bad_index(unsigned int *status, unsigned int where)
{
    if (atomicCAS(&status[0], 0u, (unsigned)PT_DEV_BAD_INDEX) == 0u) status[1] = where;
}

// Ascending list of the indices whose flag is zero; one block, chunks of 1024 flags, ballot + warp totals.
__global__ void __launch_bounds__(1024) dense_list_kernel(const uint8_t *__restrict__ zero, int n, int *__restrict__ idx, int *__restrict__ count)
{
    __shared__ int warp_tot[32];
    __shared__ int base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) base = 0;
    __syncthreads();
    for (int start = 0; start < n; start += 1024) {
        const int i = start + tid;
        const bool keep = i < n && zero[i] == 0;
        const unsigned b = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) warp_tot[warp] = __popc(b);
        __syncthreads();
        int off = base;
        for (int w = 0; w < warp; ++w) off += warp_tot[w];
        if (keep) idx[off + __popc(b & ((1u << lane) - 1u))] = i;
        __syncthreads();
        if (tid == 0) {
            int t = 0;
            for (int w = 0; w < 32; ++w) t += warp_tot[w];
            base += t;
        }
        __syncthreads();
    }
    for (int i = base + tid; i < n; i += 1024) idx[i] = -1;
    if (tid == 0) *count = base;
}

// Both gates move whole pixel rows: a block takes every gridDim.x-th chunk of `pix` consecutive pixels, whose rows are one
// contiguous run of bytes in every tensor. A producer warp brings the runs into a ring of shared-memory stages with untiled bulk
// copies; the other warps move the channels out of shared memory into registers and store them.
//   Bound by HBM. Reading the selected channels of a row straight from global memory (eight 2-byte loads per 16-byte store)
// left it bound by the load units instead: 58 us to gather 211 of 222 channels of 64x56x56 pixels and 63 us to add them back,
// 2.9 and 4.2 TB/s. A thread keeps one pair of neighbouring output channels (one 4-byte store) and walks the pixels of the
// chunk: the lanes of a warp read consecutive words, free of bank conflicts, write 128 consecutive bytes, and the selection sits
// in registers. (One thread that issues the copies between two block-wide barriers, with bulk stores from a staging buffer,
// reached 5.5 TB/s in the gather but 4.1 in the sum: its ~250 cycles per copy were on every warp's path.)
struct GateP {
    long long npix;
    int pix;                    // pixels per chunk
    int in_ld, out_ld, node_ld; // channel pitches: rows picked from (source | branch), rows written, node_in rows (0: none)
    int n_in;                   // channels of the rows picked from
    int n_sel, c_out;           // selection length; channels of the output that exist
    unsigned long long chunks;
    int test_skip;              // test hook (pt_test_skip_next_arrive): the producers leave out their first stage
};
constexpr int kGateStages = 3;
constexpr int kGateBlock = 256;                  // most consumer threads of a block of the staged form
constexpr int kGatePerSm = 2;
// Bytes a chunk brings in. Few and large copies: 24 KB x 3 stages x 2 blocks per SM gathers in 30 us and adds in 43 us at the size
// above (5.6 and 6.2 TB/s); 12 KB x 4 x 3 takes 31 and 51 us, 8 KB x 4 x 5 takes 32 and 86 us.
constexpr size_t kGateChunk = 24 * 1024;
constexpr int kGateMaxRow = 24 * 1024;           // longest pixel row (all inputs together) the staged form takes

struct __align__(8) GateCtl {
    uint64_t full[kGateStages], empty[kGateStages];
    int abort_flag;
    unsigned none;                               // what a channel without a pick reads
};

// SCATTER = false: out[p][j] = in[p][idx[j]] (j < n_sel), 0 in the pad lanes.
// SCATTER = true : out[p][c] = act(node[p][c] + in[p][j] where idx[j] == c), fp32 add, one rounding; 0 in the pad lanes.
template <bool SCATTER, bool RELU>
__global__ void __launch_bounds__(kGateBlock + 32, kGatePerSm) gate_kernel(const GateP p, const unsigned short *in, const int *__restrict__ idx,
                                                                          const unsigned short *node, unsigned short *out, unsigned int *status)
{
    extern __shared__ __align__(128) uint8_t smem[];
    GateCtl *ctl = reinterpret_cast<GateCtl *>(smem);
    volatile int *abort_flag = &ctl->abort_flag;
    const uint32_t sbase = sm100::smem_u32(smem);
    // for every output channel the position picked from the row (0xffff: none)
    unsigned short *s_pick = reinterpret_cast<unsigned short *>(smem + 128);
    const uint32_t in_row = (uint32_t)p.in_ld * 2u, out_row = (uint32_t)p.out_ld * 2u, node_row = (uint32_t)p.node_ld * 2u;
    const uint32_t stage_bytes = (uint32_t)p.pix * (in_row + node_row);
    const uint32_t ring = sbase + 128u + (out_row + 127u) / 128u * 128u;
    const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x - 32, cons_warps = nthr >> 5;
    if (tid == 0) {
        for (int s = 0; s < kGateStages; ++s) {
            sm100::mbar_init(sm100::smem_u32(&ctl->full[s]), 1);
            sm100::mbar_init(sm100::smem_u32(&ctl->empty[s]), (uint32_t)cons_warps);
        }
        ctl->abort_flag = 0;
        ctl->none = SCATTER ? 0x80008000u : 0u;  // the gather writes zeros there; in the sum -0 changes nothing, a node value of -0 included
        sm100::fence_mbar_init();
    }
    if (SCATTER)
        for (int c = tid; c < p.out_ld; c += blockDim.x) s_pick[c] = 0xffffu;
    __syncthreads();
    if (tid >= nthr) {
        if (lane == 0) {
            int s = 0, ph = 0, issued = 0;
            for (long long ch = blockIdx.x; ch < (long long)p.chunks; ch += gridDim.x, ++issued) {
                const long long p0 = ch * p.pix;
                const uint32_t n = (uint32_t)(p.npix - p0 < p.pix ? p.npix - p0 : p.pix);
                if (!sm100::mbar_wait(sm100::smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, status, 43)) break;
                if (p.test_skip && issued == 0) {                        // test hook: this stage never becomes full
                    if (++s == kGateStages) { s = 0; ph ^= 1; }
                    continue;
                }
                const uint32_t bar = sm100::smem_u32(&ctl->full[s]), dst = ring + (uint32_t)s * stage_bytes;
                sm100::mbar_arrive_expect_tx(bar, n * (in_row + node_row));
                sm100::bulk_load(dst, in + (size_t)p0 * p.in_ld, n * in_row, bar);
                if (SCATTER && node_row) sm100::bulk_load(dst + (uint32_t)p.pix * in_row, node + (size_t)p0 * p.node_ld, n * node_row, bar);
                if (++s == kGateStages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) sm100::drain_ring(sm100::smem_u32(&ctl->full[0]), kGateStages, issued);
        }
        __syncwarp();
    } else {
        // the selection, checked once per block while the first chunks are on their way
        for (int j = tid; j < (SCATTER ? p.n_sel : p.out_ld); j += nthr) {
            int id = j < p.n_sel ? idx[j] : -1;
            if (j < p.n_sel && (id < 0 || id >= (SCATTER ? p.c_out : p.n_in))) { bad_index(status, SCATTER ? 41u : 40u); id = -1; }
            if (!SCATTER) s_pick[j] = id < 0 ? (unsigned short)0xffffu : (unsigned short)id;
            else if (id >= 0) s_pick[id] = (unsigned short)j;
        }
        sm100::named_barrier(1, nthr);
        const int pairs = p.out_ld >> 1;
        const int rows = pairs < nthr ? nthr / pairs : 1;                // pixels the block's threads cover at a time
        const int pr = pairs < nthr ? tid / pairs : 0, cp0 = tid - pr * pairs;
        const uint32_t none = sm100::smem_u32(&ctl->none);
        const uint32_t dn = SCATTER && node_row ? (uint32_t)rows * node_row : 0u;
        int s = 0, ph = 0;
        for (long long ch = blockIdx.x; ch < (long long)p.chunks; ch += gridDim.x) {
            const long long p0 = ch * p.pix;
            const int n = (int)(p.npix - p0 < p.pix ? p.npix - p0 : p.pix);
            if (!sm100::mbar_wait(sm100::smem_u32(&ctl->full[s]), ph, abort_flag, status, 42)) break;
            const uint32_t src = ring + (uint32_t)s * stage_bytes + (uint32_t)pr * in_row;
            const uint32_t nsrc = ring + (uint32_t)s * stage_bytes + (uint32_t)p.pix * in_row + (uint32_t)pr * node_row;
            for (int cp = cp0; cp < pairs && pr < rows; cp += nthr) {    // once, unless a row has more pairs than the block has threads
                const unsigned pick = *reinterpret_cast<const unsigned *>(s_pick + 2 * cp);
                const unsigned i0 = pick & 0xffffu, i1 = pick >> 16;
                const uint32_t d0 = i0 != 0xffffu ? (uint32_t)rows * in_row : 0u, d1 = i1 != 0xffffu ? (uint32_t)rows * in_row : 0u;
                uint32_t a0 = d0 ? src + 2u * i0 : none, a1 = d1 ? src + 2u * i1 : none;
                uint32_t an = dn ? nsrc + 4u * (uint32_t)cp : none;
                const unsigned keep = (2 * cp < p.c_out ? 0xffffu : 0u) | (2 * cp + 1 < p.c_out ? 0xffff0000u : 0u);
                unsigned *o = reinterpret_cast<unsigned *>(out + (size_t)(p0 + pr) * p.out_ld) + cp;
                const size_t do_ = (size_t)rows * (p.out_ld >> 1);
                // four pixels at a time: all their loads go out before the first result is stored
                for (int pp = pr; pp < n; pp += 4 * rows) {
                    unsigned short a[4], b[4];
                    unsigned w[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (pp + u * rows < n) {
                            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(a[u]) : "r"(a0 + u * d0));
                            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(b[u]) : "r"(a1 + u * d1));
                            w[u] = 0u;
                            if (SCATTER && dn) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[u]) : "r"(an + u * dn));
                        }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (pp + u * rows < n) {
                            unsigned r = (unsigned)a[u] | ((unsigned)b[u] << 16);
                            if (SCATTER) {
                                float v0 = __uint_as_float(w[u] << 16) + __uint_as_float(r << 16);
                                float v1 = __uint_as_float(w[u] & 0xffff0000u) + __uint_as_float(r & 0xffff0000u);
                                if (RELU) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
                                const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
                                r = *reinterpret_cast<const unsigned *>(&h) & keep;
                            }
                            o[u * do_] = r;
                        }
                    a0 += 4u * d0; a1 += 4u * d1; an += 4u * dn; o += 4 * do_;
                }
            }
            __syncwarp();
            if (lane == 0) sm100::mbar_arrive(sm100::smem_u32(&ctl->empty[s]));
            if (++s == kGateStages) { s = 0; ph ^= 1; }
        }
    }
}

// Rows that do not fit the staged form (more than kGateMaxRow bytes per pixel): straight from global memory.
// dst[p][j] = src[p][idx[j]] (j < n_sel), 0 in the pad lanes. A thread produces 8 consecutive output channels (one 16-byte
// store); the threads of a block walk a contiguous range of pixels, so a source row is fetched once and then hit in L1.
__global__ void __launch_bounds__(kGateThreads) gather_kernel(const unsigned short *__restrict__ src, int ld_src, int c_src,
                                                              const int *__restrict__ idx, int n_sel, unsigned short *__restrict__ dst,
                                                              int ld_dst, long long npix, long long pix_per_block, unsigned int *status)
{
    __shared__ int s_idx[kGateMax];
    for (int j = threadIdx.x; j < ld_dst; j += kGateThreads) {
        int id = j < n_sel ? idx[j] : -1;
        if (j < n_sel && (id < 0 || id >= c_src)) { bad_index(status, 40u); id = -1; }
        s_idx[j] = id;
    }
    __syncthreads();
    const long long p_beg = (long long)blockIdx.x * pix_per_block;
    const long long p_end = p_beg + pix_per_block < npix ? p_beg + pix_per_block : npix;
    if (p_beg >= p_end) return;
    const int groups = ld_dst >> 3;
    const int items = (int)(p_end - p_beg) * groups;
    const unsigned short *s0 = src + (size_t)p_beg * ld_src;
    unsigned short *d0 = dst + (size_t)p_beg * ld_dst;
    for (int it = threadIdx.x; it < items; it += kGateThreads) {
        const int p = it / groups, g = it - p * groups;
        const unsigned short *row = s0 + (size_t)p * ld_src;
        __align__(16) unsigned short o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int id = s_idx[g * 8 + e];
            o[e] = id >= 0 ? __ldg(row + id) : (unsigned short)0;
        }
        *reinterpret_cast<uint4 *>(d0 + (size_t)p * ld_dst + g * 8) = *reinterpret_cast<const uint4 *>(o);
    }
}

__device__ __forceinline__ float bf16_bits_to_float(unsigned short h) { return __uint_as_float((unsigned)h << 16); }

// node_out[p][c] = act(node_in[p][c] + branch[p][j] where idx[j] == c), fp32 add, one rounding to bf16; 0 in the pad lanes.
__global__ void __launch_bounds__(kGateThreads) scatter_add_kernel(const unsigned short *__restrict__ branch, int ld_b,
                                                                   const int *__restrict__ idx, int n_sel,
                                                                   const unsigned short *node_in,
                                                                   unsigned short *node_out, int ld_node, int c_node,
                                                                   long long npix, long long pix_per_block, int relu, unsigned int *status)
{
    __shared__ short s_inv[kGateMax];
    for (int c = threadIdx.x; c < ld_node; c += kGateThreads) s_inv[c] = -1;
    __syncthreads();
    for (int j = threadIdx.x; j < n_sel; j += kGateThreads) {
        const int id = idx[j];
        if (id < 0 || id >= c_node) bad_index(status, 41u);
        else s_inv[id] = (short)j;
    }
    __syncthreads();
    const long long p_beg = (long long)blockIdx.x * pix_per_block;
    const long long p_end = p_beg + pix_per_block < npix ? p_beg + pix_per_block : npix;
    if (p_beg >= p_end) return;
    const int groups = ld_node >> 3;
    const int items = (int)(p_end - p_beg) * groups;
    const unsigned short *b0 = branch + (size_t)p_beg * ld_b;
    const unsigned short *i0 = node_in ? node_in + (size_t)p_beg * ld_node : nullptr;
    unsigned short *o0 = node_out + (size_t)p_beg * ld_node;
    for (int it = threadIdx.x; it < items; it += kGateThreads) {
        const int p = it / groups, g = it - p * groups;
        uint4 in = make_uint4(0u, 0u, 0u, 0u);
        // node_in may be the tensor node_out (in-place merge): a plain load, not the read-only path, and no restrict
        if (i0) in = *reinterpret_cast<const uint4 *>(i0 + (size_t)p * ld_node + g * 8);
        const unsigned short *ie = reinterpret_cast<const unsigned short *>(&in);
        const unsigned short *brow = b0 + (size_t)p * ld_b;
        __align__(16) unsigned short o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int c = g * 8 + e;
            float v = bf16_bits_to_float(ie[e]);
            const int j = s_inv[c];
            if (j >= 0) v += bf16_bits_to_float(__ldg(brow + j));
            if (relu) v = v > 0.f ? v : 0.f;
            const __nv_bfloat16 r = __float2bfloat16_rn(v);
            o[e] = c < c_node ? *reinterpret_cast<const unsigned short *>(&r) : (unsigned short)0;
        }
        *reinterpret_cast<uint4 *>(o0 + (size_t)p * ld_node + g * 8) = *reinterpret_cast<const uint4 *>(o);
    }
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Blocks walk contiguous pixel ranges; a few blocks per SM, and no range so long that its item count overflows an int.
void gate_grid(const pt_ctx *c, long long npix, int groups, unsigned *blocks, long long *pix_per_block)
{
    long long nb = (long long)c->sm_count * 8;
    long long ppb = (npix + nb - 1) / nb;
    if (ppb < 8) ppb = 8;
    const long long cap = (long long)(1 << 30) / (groups > 0 ? groups : 1);
    if (ppb > cap) ppb = cap;
    *pix_per_block = ppb;
    *blocks = (unsigned)((npix + ppb - 1) / ppb);
}

// Staged form: chunks of about kGateChunk bytes, at most kGatePerSm blocks per SM.
template <bool SCATTER, bool RELU>
pt_status gate_launch(pt_ctx *ctx, GateP p, const void *in, const int *idx, const void *node, void *out, cudaStream_t st)
{
    const size_t row = (size_t)(p.in_ld + p.node_ld) * 2;
    if (ctx->test_skip == 4) { p.test_skip = 1; ctx->test_skip = 0; }
    p.pix = (int)(kGateChunk / row);
    if (p.pix < 1) p.pix = 1;
    // small tensors: chunks no larger than what gives every SM one
    const long long share = (p.npix + ctx->sm_count - 1) / ctx->sm_count;
    if (p.pix > share) p.pix = (int)share;
    if (p.pix > 8) p.pix &= ~7;                      // chunks then start on 128-byte lines whatever the pitch is
    p.chunks = (unsigned long long)((p.npix + p.pix - 1) / p.pix);
    const int pairs = p.out_ld / 2;
    const int threads = pairs >= kGateBlock ? kGateBlock : pt_ceil_div(kGateBlock / pairs * pairs, 32) * 32;
    const size_t smem = 128 + pt_align_up((size_t)p.out_ld * 2, 128) + kGateStages * (size_t)p.pix * row;
    const unsigned attr = kAttrGate << (SCATTER ? RELU ? 2 : 1 : 0);
    if (!(ctx->attr_done & attr)) {
        PT_CUDA_OK(cudaFuncSetAttribute(gate_kernel<SCATTER, RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        ctx->attr_done |= attr;
    }
    const unsigned long long cap = (unsigned long long)ctx->sm_count * kGatePerSm;
    gate_kernel<SCATTER, RELU><<<(unsigned)(p.chunks < cap ? p.chunks : cap), threads + 32, smem, st>>>(
        p, (const unsigned short *)in, idx, (const unsigned short *)node, (unsigned short *)out, ctx->d_status);
    ctx->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

}  // namespace

pt_status pt_gate_set_wait_limit_ns(unsigned long long ns)
{
    PT_CUDA_OK(cudaMemcpyToSymbol(sm100::g_wait_limit_ns, &ns, sizeof(ns)));
    return PT_OK;
}

extern "C" pt_status pt_dense_channel_list(pt_ctx *ctx, const uint8_t *zero_flags, int32_t n, int32_t *idx, int32_t *count, void *stream)
{
    if (!ctx || !zero_flags || !idx || !count || n < 0) return PT_ERR_INVALID_ARG;
    dense_list_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(zero_flags, n, idx, count);
    ctx->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

extern "C" pt_status pt_channel_gather(pt_ctx *ctx, const void *src, int32_t ld_src, int32_t c_src, const int32_t *idx, int32_t n_sel,
                                       void *dst, int32_t ld_dst, int64_t npix, void *stream)
{
    if (!ctx || !src || !dst || !idx || npix < 0 || n_sel < 0 || c_src < 1) return PT_ERR_INVALID_ARG;
    if (ld_src < c_src || ld_dst < n_sel || ld_dst < 8 || (ld_src & 7) || (ld_dst & 7) || !aligned16(src) || !aligned16(dst))
        return PT_ERR_INVALID_ARG;
    if (ld_dst > kGateMax) return PT_ERR_UNSUPPORTED;
    if (npix == 0) return PT_OK;
    if (ld_src * 2 <= kGateMaxRow) {
        GateP p{};
        p.npix = npix; p.in_ld = ld_src; p.out_ld = ld_dst; p.n_in = c_src; p.n_sel = n_sel; p.c_out = n_sel;
        return gate_launch<false, false>(ctx, p, src, idx, nullptr, dst, (cudaStream_t)stream);
    }
    unsigned blocks;
    long long ppb;
    gate_grid(ctx, npix, ld_dst >> 3, &blocks, &ppb);
    gather_kernel<<<blocks, kGateThreads, 0, (cudaStream_t)stream>>>((const unsigned short *)src, ld_src, c_src, idx, n_sel,
                                                                     (unsigned short *)dst, ld_dst, npix, ppb, ctx->d_status);
    ctx->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

extern "C" pt_status pt_channel_scatter_add(pt_ctx *ctx, const void *branch, int32_t ld_branch, const int32_t *idx, int32_t n_sel,
                                            const void *node_in, void *node_out, int32_t ld_node, int32_t c_node, int64_t npix,
                                            int32_t relu, void *stream)
{
    if (!ctx || !branch || !node_out || !idx || npix < 0 || n_sel < 0 || c_node < 1) return PT_ERR_INVALID_ARG;
    if (ld_node < c_node || ld_branch < n_sel || ld_branch < 8 || n_sel > c_node || (ld_node & 7) || (ld_branch & 7) ||
        !aligned16(branch) || !aligned16(node_out) || (node_in && !aligned16(node_in)))
        return PT_ERR_INVALID_ARG;
    if (ld_node > kGateMax || n_sel > 32767) return PT_ERR_UNSUPPORTED;
    if (npix == 0) return PT_OK;
    if ((ld_branch + ld_node) * 2 <= kGateMaxRow) {
        GateP p{};
        p.npix = npix; p.in_ld = ld_branch; p.out_ld = ld_node; p.node_ld = node_in ? ld_node : 0;
        p.n_in = n_sel; p.n_sel = n_sel; p.c_out = c_node;
        if (relu) return gate_launch<true, true>(ctx, p, branch, idx, node_in, node_out, (cudaStream_t)stream);
        return gate_launch<true, false>(ctx, p, branch, idx, node_in, node_out, (cudaStream_t)stream);
    }
    unsigned blocks;
    long long ppb;
    gate_grid(ctx, npix, ld_node >> 3, &blocks, &ppb);
    scatter_add_kernel<<<blocks, kGateThreads, 0, (cudaStream_t)stream>>>((const unsigned short *)branch, ld_branch, idx, n_sel,
                                                                          (const unsigned short *)node_in, (unsigned short *)node_out,
                                                                          ld_node, c_node, npix, ppb, relu ? 1 : 0, ctx->d_status);
    ctx->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}
