// Reconfiguration (Sec. 4.2): keep sets per channel space by the intersection / channel-union
// rule, ascending keep maps by a block-wide scan, and the gather of the surviving weights,
// momentum, bf16 shadow and BN vectors into the smaller dense model.
#include "pt_internal.h"
#include <atomic>
#include <chrono>

namespace {

struct SpaceDev {
    int size, fixed;
    int member0, n_members;     // range in the member table
    int map_off;                // start of this space's entries in new2old
    int pad_;
};
struct MemberDev { const uint8_t *mask; };   // a writer's zero_out or a reader's zero_in (length = space size)

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One block per space. keep[j] = fixed | OR_writers !zero_out[j] | OR_readers !zero_in[j].
// The counts go straight to pinned host memory; the last block to finish (device ticket) then raises the host flag, so the
// host learns the new sizes from one posted write instead of a copy and a stream synchronisation.
__global__ void __launch_bounds__(1024) keep_scan_kernel(const SpaceDev *__restrict__ spaces,
                                                         const MemberDev *__restrict__ members,
                                                         int32_t *__restrict__ new2old, volatile int32_t *host_counts,
                                                         volatile unsigned int *host_flag, unsigned int seq, unsigned int *ticket)
{
    __shared__ int s_warp[32];
    __shared__ int s_base, s_tile;
    const SpaceDev sp = spaces[blockIdx.x];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    pdl_wait();                                  // the masks are the previous kernel's output
    __syncthreads();
    for (int j0 = 0; j0 < sp.size; j0 += blockDim.x) {
        const int j = j0 + threadIdx.x;
        int keep = 0;
        if (j < sp.size) {
            keep = sp.fixed;
            // all members' flags are fetched side by side (no early exit: the loads would form a dependent chain)
            int dead = 1;
#pragma unroll 4
            for (int m = 0; m < sp.n_members; ++m) dead &= (members[sp.member0 + m].mask[j] != 0);
            keep |= !dead;
        }
        const unsigned ball = __ballot_sync(0xffffffffu, keep);
        const int in_warp = __popc(ball & ((1u << lane) - 1u));
        if (lane == 0) s_warp[wid] = __popc(ball);
        __syncthreads();
        if (wid == 0) {
            const int v = (lane < nwarps) ? s_warp[lane] : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            s_warp[lane] = incl - v;                 // exclusive prefix of the warp totals
            if (lane == 31) s_tile = incl;           // kept channels in this tile
        }
        __syncthreads();
        const int base = s_base;
        if (keep) new2old[sp.map_off + base + s_warp[wid] + in_warp] = j;   // ascending original index
        __syncthreads();
        if (threadIdx.x == 0) s_base = base + s_tile;
        __syncthreads();
    }
    const int total = s_base;
    for (int j = total + threadIdx.x; j < sp.size; j += blockDim.x) new2old[sp.map_off + j] = -1;
    __syncthreads();
    if (threadIdx.x == 0) {
        host_counts[blockIdx.x] = total;
        __threadfence_system();
        if (atomicAdd(ticket, 1u) == gridDim.x - 1u) {
            *ticket = 0u;
            __threadfence_system();
            *host_flag = seq;
        }
    }
}

// The gather walks the lines (k, rs) of the NEW tensors: a chunk is a run of lines of one tensor restricted to a group of up to 128
// columns. Lane l of a warp owns the new columns l, l + 32, l + 64, l + 96 of the group; their old columns sit in its registers, and
// the old lines of the warp's lines in the lanes' registers (handed round by shuffles), so that an element costs its loads and
// stores and little else. Reads are gathered, writes coalesced. (Walking the new tensor as one flat stream, with both tables in shared
// memory, took 30 instructions per element: 85 us for 15.5 M kept parameters.)
struct GatherJob {
    const float *ow, *ov; const __nv_bfloat16 *owb;
    float *nw, *nv; __nv_bfloat16 *nwb;
    const int32_t *mapK, *mapC;
    int Kn, Cn, RS, Co, ldwo, ldwn;
    int kind;                  // 0 = weight tensors, 1 = per-channel vector
    int Ko;                    // old number of output channels (range check of the map)
    int lines, cgw;            // new tensor: Kn*RS lines; width of its column groups
};
struct GatherChunk { int job, line0, n_lines, c0; };

constexpr int kGThreads = 256;
constexpr int kGWarps = kGThreads / 32;
constexpr int kGMaxC = 4096;
// Elements of a chunk (at most 32 lines per warp): a block's start is a chain of four loads (chunk, job, map, element), so large
// ones where they still give every SM eight, small ones for small models (15.5 M kept parameters: 4096 / 8192 / 16384 take 88 / 73
// / 70 us; 0.3 M: 5.3 / 7.4 / 10.3 us).
constexpr int kGElems = 16384, kGElemsSmall = 4096;

// A map entry outside the old tensor (a new graph larger than the plan's counts reads the -1 padding of the map) is skipped:
// nothing is read or written for it, and the status word reports it (PT_ERR_INVALID_ARG at the next poll).
__device__ __forceinline__ void bad_map_entry(unsigned int *status, unsigned int where)
{
    if (atomicCAS(&status[0], 0u, (unsigned)PT_DEV_BAD_INDEX) == 0u) status[1] = where;
}

// One batch of a warp: U lines x NS columns per lane of w, v and the shadow, all loads before the first store. ol: the lines' old
// lines (-1: skipped), the same in every lane; co: the lane's old columns (-1: skipped or past the end).
template <int U, int NS>
__device__ __forceinline__ void gather_lines(const GatherJob &J, int line, int n, const int (&ol)[U], const int (&co)[4], int c)
{
    // 32-bit element offsets (the host checks that the old tensors have fewer than 2^31 elements at their pitch, and the new w and v are
    // dense and no larger), except for the new shadow, whose pitch is the caller's choice
    float w[U][NS], v[U][NS];
    unsigned short h[U][NS];
    const unsigned short *ob = reinterpret_cast<const unsigned short *>(J.owb);
    unsigned short *nb = reinterpret_cast<unsigned short *>(J.nwb);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            if (u >= n || (ol[u] | co[j]) < 0) continue;
            const unsigned src = (unsigned)ol[u] * (unsigned)J.Co + (unsigned)co[j];
            w[u][j] = __ldg(J.ow + src);
            if (J.nv) v[u][j] = __ldg(J.ov + src);
            if (nb) h[u][j] = __ldg(ob + ((unsigned)ol[u] * (unsigned)J.ldwo + (unsigned)co[j]));
        }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            if (u >= n || (ol[u] | co[j]) < 0) continue;
            const unsigned dst = (unsigned)(line + u) * (unsigned)J.Cn + (unsigned)(c + 32 * j);
            J.nw[dst] = w[u][j];
            if (J.nv) J.nv[dst] = v[u][j];
            if (nb) nb[(size_t)(line + u) * (size_t)J.ldwn + (unsigned)(c + 32 * j)] = h[u][j];
        }
}

template <int U, int NS>
__device__ __forceinline__ void gather_warp(const GatherJob &J, int line, int n, int my_ol, const int (&co)[4], int c)
{
    for (int l = 0; l < n; l += U) {
        int ol[U];
#pragma unroll
        for (int u = 0; u < U; ++u) ol[u] = __shfl_sync(0xffffffffu, my_ol, (l + u) & 31);
        gather_lines<U, NS>(J, line + l, n - l, ol, co, c);
    }
}

__global__ void __launch_bounds__(kGThreads) gather_kernel(const GatherJob *__restrict__ jobs, const GatherChunk *__restrict__ chunks,
                                                           unsigned int *status)
{
    const GatherChunk ch = chunks[blockIdx.x];
    const GatherJob J = jobs[ch.job];
    if (J.kind == 1) {       // vector: nw[k'] = ow[mapK[k']]
        for (int k = threadIdx.x; k < J.Kn; k += kGThreads) {
            const int ko = J.mapK[k];
            if (ko < 0 || ko >= J.Ko) { bad_map_entry(status, 50u); continue; }
            J.nw[k] = J.ow[ko];
        }
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (ch.n_lines + kGWarps - 1) / kGWarps;               // lines of a warp, consecutive, at most 32
    const int line = ch.line0 + warp * per, n = min(per, ch.n_lines - warp * per);
    if (n <= 0) return;
    const int c = ch.c0 + lane;
    int co[4], my_ol = -1;
    int ns = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        co[j] = -1;
        if (ch.c0 + 32 * j < J.Cn && 32 * j < J.cgw) ns = j + 1;
        if (c + 32 * j < J.Cn && 32 * j < J.cgw) {
            const int o = J.mapC[c + 32 * j];
            if (o < 0 || o >= J.Co) bad_map_entry(status, 51u);
            else co[j] = o;
        }
    }
    if (lane < n) {
        const int kn = (line + lane) / J.RS, rs = (line + lane) - kn * J.RS, ko = J.mapK[kn];
        if (ko < 0 || ko >= J.Ko) bad_map_entry(status, 52u);
        else my_ol = ko * J.RS + rs;
    }
    __syncwarp();
    if (ns == 4) gather_warp<2, 4>(J, line, n, my_ol, co, c);
    else if (ns == 3) gather_warp<2, 3>(J, line, n, my_ol, co, c);
    else if (ns == 2) gather_warp<4, 2>(J, line, n, my_ol, co, c);
    else gather_warp<8, 1>(J, line, n, my_ol, co, c);
}

pt_status check_graph(const pt_graph *g)
{
    if (!g || !g->spaces || !g->layers || !g->links || g->n_spaces <= 0 || g->n_layers <= 0) return PT_ERR_INVALID_ARG;
    for (int i = 0; i < g->n_layers; ++i) {
        const pt_layer_link &k = g->links[i];
        if (k.in_space < 0 || k.in_space >= g->n_spaces || k.out_space < 0 || k.out_space >= g->n_spaces) return PT_ERR_INVALID_ARG;
        if (g->layers[i].C != g->spaces[k.in_space].size || g->layers[i].K != g->spaces[k.out_space].size) return PT_ERR_INVALID_ARG;
    }
    return PT_OK;
}

}  // namespace

extern "C" pt_status pt_reconfigure_plan_enqueue(pt_ctx *c, const pt_graph *g, int32_t *new2old, void *stream)
{
    if (!c || !new2old) return PT_ERR_INVALID_ARG;
    pt_status s = check_graph(g);
    if (s != PT_OK) return s;
    if (g->n_spaces > 65536) return PT_ERR_UNSUPPORTED;
    // The counts, their flag and its sequence number are the context's: a captured launch would raise the flag of its capture again on
    // every replay, and a plan on another stream could overwrite the counts of one that is still running.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    PT_CUDA_OK(cudaStreamIsCapturing((cudaStream_t)stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) return PT_ERR_UNSUPPORTED;
    if (c->plan_spaces && c->plan_stream != stream && *(volatile unsigned int *)c->h_counts != c->plan_seq) return PT_ERR_INVALID_ARG;
    std::vector<SpaceDev> sp(g->n_spaces);
    std::vector<MemberDev> mem;
    long long off = 0;
    for (int i = 0; i < g->n_spaces; ++i) {
        if (g->spaces[i].size < 0) return PT_ERR_INVALID_ARG;
        sp[i].size = g->spaces[i].size;
        sp[i].fixed = g->spaces[i].fixed ? 1 : 0;
        sp[i].member0 = (int)mem.size();
        for (int l = 0; l < g->n_layers; ++l) {
            if (g->links[l].out_space == i) {
                if (!g->layers[l].zero_out) return PT_ERR_INVALID_ARG;
                mem.push_back(MemberDev{g->layers[l].zero_out});
            }
            if (g->links[l].in_space == i) {
                if (!g->layers[l].zero_in) return PT_ERR_INVALID_ARG;
                mem.push_back(MemberDev{g->layers[l].zero_in});
            }
        }
        sp[i].n_members = (int)mem.size() - sp[i].member0;
        sp[i].map_off = (int)off;
        sp[i].pad_ = 0;
        off += sp[i].size;
        if (off >= (1ll << 31)) return PT_ERR_UNSUPPORTED;
    }
    size_t sb = pt_align_up(sp.size() * sizeof(SpaceDev), 256), mb = pt_align_up(mem.size() * sizeof(MemberDev) + 8, 256);
    std::vector<char> buf(sb + mb + (size_t)g->n_spaces * 4, 0);
    memcpy(buf.data(), sp.data(), sp.size() * sizeof(SpaceDev));
    if (!mem.empty()) memcpy(buf.data() + sb, mem.data(), mem.size() * sizeof(MemberDev));
    cudaStream_t st = (cudaStream_t)stream;
    char *dev = nullptr;
    s = pt_upload_table(c, &c->graph_tab, buf.data(), buf.size(), st, &dev);
    if (s != PT_OK) return s;
    // counts and flag live in pinned host memory the kernel writes directly: [0] = flag (sequence number), [16..] = counts
    volatile unsigned int *flag = (volatile unsigned int *)c->h_counts;
    volatile int32_t *counts = (volatile int32_t *)c->h_counts + 16;
    const unsigned int seq = ++c->plan_seq;
    PT_CUDA_OK(pt_launch_pdl(keep_scan_kernel, dim3((unsigned)g->n_spaces), dim3(1024), 0, st, (const SpaceDev *)dev,
                             (const MemberDev *)(dev + sb), new2old, (volatile int32_t *)counts, (volatile unsigned int *)flag, seq,
                             c->d_status + 2));
    c->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    c->plan_spaces = g->n_spaces;
    c->plan_stream = stream;
    return PT_OK;
}

// The documented synchronisation: the host needs the new sizes. It waits for the kernel's flag (bounded), looking at the
// stream now and then so that an error upstream ends the wait.
extern "C" pt_status pt_reconfigure_plan_wait(pt_ctx *c, int32_t n_spaces, int32_t *new_sizes, void *stream)
{
    if (!c || !new_sizes || n_spaces < 1 || c->plan_spaces != n_spaces) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const volatile unsigned int *flag = (const volatile unsigned int *)c->h_counts;
    const volatile int32_t *counts = (const volatile int32_t *)c->h_counts + 16;
    const unsigned int seq = c->plan_seq;
    const auto t0 = std::chrono::steady_clock::now();
    unsigned spins = 0;
    bool seen = false;
    while (!(seen = (*flag == seq))) {
        if ((++spins & 0x3fffu) == 0u) {
            const cudaError_t q = cudaStreamQuery(st);
            if (q == cudaSuccess) { seen = (*flag == seq); break; }
            if (q != cudaErrorNotReady) { (void)cudaGetLastError(); return PT_ERR_CUDA; }
            if (std::chrono::steady_clock::now() - t0 > std::chrono::seconds(30)) break;
        }
    }
    if (!seen) {
        PT_CUDA_OK(cudaStreamSynchronize(st));
        if (*flag != seq) return PT_ERR_CUDA;
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    for (int i = 0; i < n_spaces; ++i) new_sizes[i] = counts[i];
    return PT_OK;
}

extern "C" pt_status pt_reconfigure_plan(pt_ctx *c, const pt_graph *g, int32_t *new2old, int32_t *new_sizes, void *stream)
{
    if (!new_sizes) return PT_ERR_INVALID_ARG;
    const pt_status s = pt_reconfigure_plan_enqueue(c, g, new2old, stream);
    return s != PT_OK ? s : pt_reconfigure_plan_wait(c, g->n_spaces, new_sizes, stream);
}

extern "C" pt_status pt_reconfigure(pt_ctx *c, const pt_graph *og, const int32_t *new2old, const pt_graph *ng, void *stream)
{
    if (!c || !new2old || !og || !ng) return PT_ERR_INVALID_ARG;
    if (!og->spaces || !og->layers || !og->links || !ng->spaces || !ng->layers || !ng->links) return PT_ERR_INVALID_ARG;
    if (og->n_spaces <= 0 || og->n_layers <= 0 || og->n_spaces != ng->n_spaces || og->n_layers != ng->n_layers) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    // The table below depends on the arguments only (shapes, pointers, the map's address), not on what the buffers hold:
    // this call sits right behind the host synchronisation of the plan, so a repeated reconfiguration skips the rebuild.
    std::vector<char> args;
    {
        const size_t ns = (size_t)og->n_spaces * sizeof(pt_space), nl = (size_t)og->n_layers * sizeof(pt_layer);
        const size_t nk = (size_t)og->n_layers * sizeof(pt_layer_link);
        args.resize(2 * (ns + nl + nk) + sizeof(new2old));
        char *a = args.data();
        memcpy(a, og->spaces, ns); a += ns; memcpy(a, ng->spaces, ns); a += ns;
        memcpy(a, og->layers, nl); a += nl; memcpy(a, ng->layers, nl); a += nl;
        memcpy(a, og->links, nk); a += nk; memcpy(a, ng->links, nk); a += nk;
        memcpy(a, &new2old, sizeof(new2old));
    }
    for (int i = 0; i < 4; ++i) {
        pt_ctx::GatherSlot &gs = c->gather_slot[i];
        if (!(gs.reg.valid && gs.chunks && args == gs.args)) continue;
        const char *dev = gs.reg.dev;
        gather_kernel<<<gs.chunks, kGThreads, 0, st>>>((const GatherJob *)dev, (const GatherChunk *)(dev + gs.jobs_bytes), c->d_status);
        c->launches += 1;
        PT_CUDA_OK(cudaGetLastError());
        return PT_OK;
    }
    pt_status s = check_graph(og);
    if (s != PT_OK) return s;
    s = check_graph(ng);
    if (s != PT_OK) return s;
    std::vector<int> map_off(og->n_spaces);
    long long off = 0;
    for (int i = 0; i < og->n_spaces; ++i) {
        map_off[i] = (int)off;
        off += og->spaces[i].size;
        if (ng->spaces[i].size > og->spaces[i].size) return PT_ERR_INVALID_ARG;
    }
    std::vector<GatherJob> jobs;
    std::vector<GatherChunk> chunks;
    long long kept = 0;
    for (int l = 0; l < og->n_layers; ++l) kept += (long long)ng->layers[l].K * ng->layers[l].RS * ng->layers[l].C;
    const int elems = kept >= (long long)kGElems * 8 * c->sm_count * 3 / 4 ? kGElems : kGElemsSmall;
    for (int l = 0; l < og->n_layers; ++l) {
        const pt_layer &o = og->layers[l], &n = ng->layers[l];
        const pt_layer_link &ol = og->links[l], &nl = ng->links[l];
        if (ol.in_space != nl.in_space || ol.out_space != nl.out_space || o.RS != n.RS) return PT_ERR_INVALID_ARG;
        if (n.K == 0 || n.C == 0) continue;                 // a dead layer: nothing to carry over
        if (!o.w || !n.w || (n.v && !o.v) || (n.w_bf16 && !o.w_bf16)) return PT_ERR_INVALID_ARG;
        if (n.w_bf16 && (n.ldw < n.C || n.ldw % 8)) return PT_ERR_INVALID_ARG;
        if (n.C > kGMaxC) return PT_ERR_UNSUPPORTED;
        if ((long long)o.K * o.RS * (o.ldw > o.C ? o.ldw : o.C) >= (1ll << 31)) return PT_ERR_UNSUPPORTED;
        GatherJob J;
        memset(&J, 0, sizeof(J));
        J.ow = o.w; J.ov = o.v; J.owb = (const __nv_bfloat16 *)o.w_bf16;
        J.nw = n.w; J.nv = n.v; J.nwb = (__nv_bfloat16 *)n.w_bf16;
        J.mapK = new2old + map_off[ol.out_space];
        J.mapC = new2old + map_off[ol.in_space];
        J.Kn = n.K; J.Cn = n.C; J.RS = n.RS; J.Co = o.C; J.Ko = o.K; J.ldwo = o.ldw; J.ldwn = n.ldw;
        J.kind = 0;
        J.lines = n.K * n.RS;
        const int job = (int)jobs.size();
        const int n_cg = pt_ceil_div(n.C, 128);
        J.cgw = 32 * pt_ceil_div(pt_ceil_div(n.C, 32), n_cg);           // column groups of equal width
        jobs.push_back(J);
        int per = elems / J.cgw;                                       // lines of a chunk: at most 256, a warp's 32
        if (per > 32 * kGWarps) per = 32 * kGWarps;
        for (int l0 = 0; l0 < J.lines; l0 += per)
            for (int c0 = 0; c0 < n.C; c0 += J.cgw) chunks.push_back(GatherChunk{job, l0, J.lines - l0 < per ? J.lines - l0 : per, c0});
        for (int b = 0; b < 4; ++b) {
            if (!nl.bn[b]) continue;
            if (!ol.bn[b]) return PT_ERR_INVALID_ARG;
            GatherJob V;
            memset(&V, 0, sizeof(V));
            V.ow = ol.bn[b]; V.nw = nl.bn[b]; V.mapK = J.mapK; V.Kn = n.K; V.Ko = o.K; V.kind = 1;
            chunks.push_back(GatherChunk{(int)jobs.size(), 0, 0, 0});
            jobs.push_back(V);
        }
    }
    if (chunks.empty()) return PT_OK;
    const unsigned nchk = (unsigned)chunks.size();
    const size_t jb = pt_align_up(jobs.size() * sizeof(GatherJob), 256), cb = chunks.size() * sizeof(GatherChunk);
    std::vector<char> buf(jb + cb, 0);
    memcpy(buf.data(), jobs.data(), jobs.size() * sizeof(GatherJob));
    memcpy(buf.data() + jb, chunks.data(), chunks.size() * sizeof(GatherChunk));
    char *dev = nullptr;
    pt_ctx::GatherSlot &gs = c->gather_slot[c->gather_next];
    c->gather_next = (c->gather_next + 1) & 3;
    gs.chunks = 0;
    s = pt_upload_table(c, &gs.reg, buf.data(), buf.size(), st, &dev);
    if (s != PT_OK) return s;
    gather_kernel<<<nchk, kGThreads, 0, st>>>((const GatherJob *)dev, (const GatherChunk *)(dev + jb), c->d_status);
    c->launches += 1;
    PT_CUDA_OK(cudaGetLastError());
    gs.args.swap(args);
    gs.chunks = nchk;
    gs.jobs_bytes = jb;
    return PT_OK;
}
