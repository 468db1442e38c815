// Batch normalisation + residual add + ReLU on ragged channel counts, forward and backward (Sec. 2.1: the normalisation
// layers read their inputs several times and are bound by memory bandwidth). NHWC bf16 activations with channel pitch ld,
// fp32 statistics and parameters. Two passes per direction:
//   forward : reduce (per-channel sum and sum of squares about a pivot), apply (mean, 1/std, moving statistics, then
//             y = relu(gamma*xhat + beta + residual))
//   backward: reduce (dbeta = sum dz, dgamma = sum dz*xhat), apply (dx, dresidual)
// Partial sums are combined in a fixed order (run-to-run identical); no atomics.
//
// The passes are bound by HBM and, on the small maps, by what a launch costs. A block owns a slab of at most 64 channels and a
// share of the pixels. A producer warp brings chunks of the slab (2-D TMA boxes; where one slab is the whole pixel row, untiled
// bulk copies of consecutive rows) into a ring of shared-memory stages; the other warps keep one 16-byte vector column each and
// walk the chunk's pixels. What is in flight is the ring (up to 190 KB per SM), not what fits beside the sums in registers.
//   A slab also keeps the number of partial-sum rows a channel has at SMs / slabs, so that every block of the apply pass finishes
// the sums of its own channels itself, in fp64, while its first chunks are on their way. (A finishing kernel between the passes
// cost 5 to 9 us per call: a launch, a round trip for the rows, a launch.)
#include "pt_internal.h"
#include "pt_sm100_ptx.cuh"

namespace {

constexpr int kBnThreads = 512;             // most consumer threads of a block (a producer warp follows them)
constexpr int kBnMaxStages = 6;
constexpr int kBnSlab = 8;                  // most 16-byte vectors (8 channels) of a pixel a block owns
// Few and large copies: three blocks per SM with 12 KB stages took 63 us for the backward pass at 64x28x28x371 where one block with
// 48 KB stages took 55.
constexpr size_t kBnRing = 190 * 1024;
constexpr size_t kBnStage = 48 * 1024;      // bytes a stage brings in when the tensor is large

struct BnP {
    long long M;            // pixels
    int C, ld, LV;          // channels, pitch, vectors per pixel (ld / 8)
    int slabs, sv;          // channel slabs, vectors of a slab
    int ppb;                // pixel rows the consumer threads cover at a time
    int consumers;          // consumer threads: sv * ppb rounded up to whole warps
    int parts;              // blocks that share a slab's pixels
    int pix;                // pixels per chunk
    long long chunks;
    int stages, n_in;       // ring depth; input tensors of the pass
    int reverse;            // walk the chunks from the last to the first
    int rows, rows_vec;     // apply passes: rows of partial sums to finish; 1 = they may be read 16 bytes at a time
    int pairs;              // 1: every row is followed by one of what its rounding left (a reduce pass's rows; not a convolution's)
    int pivot;              // the forward sums are about the channel's value at pixel 0 (else about 0)
    float eps, momentum;
    int relu;
    int test_skip;          // test hook (pt_test_skip_next_arrive): the producers leave out their first stage
};

struct __align__(8) BnCtl {
    uint64_t full[kBnMaxStages], empty[kBnMaxStages];
    int abort_flag;
};
// shared memory: [BnCtl, 128 bytes][four tables of 64 floats][ring]; the apply passes' fp64 slices follow the ring
constexpr uint32_t kBnTab = 128u, kBnData = 128u + 4u * 64u * 4u + 128u;     // the ring starts at 1280 bytes

__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8])
{
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __bfloat1622float2(h[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8])
{
    uint4 v;
    __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    return v;
}

__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}

// PASS 0 (forward reduce):  a0 = sum(x - pivot), a1 = sum((x - pivot)^2), pivot = the channel's value at pixel 0 (keeps the variance
//                           free of the cancellation a large mean would cause in sum(x^2) - sum(x)^2/M).        in: x
// PASS 1 (backward reduce): a0 = sum(dz), a1 = sum(dz * xhat), dz = dy where y > 0 (ReLU) else 0.               in: x, dy (, y)
// PASS 2 (forward apply):   out = relu(x*scale + shift + residual), scale = gamma*invstd, shift = beta - mean*scale.  in: x (, residual)
//                           The pivot comes from the row pass 0 left: out may be x itself, whose pixel 0 another block may have written.
// PASS 3 (backward apply):  out2 = dz; out = gamma*invstd * (dz - dbeta/M - xhat*dgamma/M).                     in: x, dy (, y)
// A reduce pass leaves two rows [2][ld] of partial sums per part: the sums, and what their rounding to fp32 left. A thread adds a chunk's few rows in fp32 and the chunks'
// sums after that, a block its threads' in fp64: one fp32 chain per thread over all of its rows stagnates on the small terms of the
// squares (1/std off by 2.7e-7 at 256x56x56x64, now 3e-8: the rounding of the result). Pad lanes (channel >= C) of the outputs are written as zeros.
struct BnArgs {
    const uint4 *in[3];
    const float *gamma, *beta;
    float *mean, *invstd;                   // read by pass 1 and 3, written by pass 2
    float *rmean, *rvar;                    // moving statistics (pass 2, optional)
    float *dgamma, *dbeta;                  // written by pass 3
    float *partial;                         // rows of partial sums: written by the reduce passes, read by the apply passes
    float *pivots;                          // the channels' pivots: written by pass 0, read by pass 2 (p.pivot)
    uint4 *out, *out2;
    unsigned int *status;
};

template <int PASS>
__global__ void __launch_bounds__(kBnThreads + 32, 1)
bn_kernel(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1, const __grid_constant__ CUtensorMap tm2,
          const BnP p, const BnArgs g)
{
    constexpr bool REDUCE = PASS < 2, BWD = (PASS & 1) != 0;
    extern __shared__ __align__(128) uint8_t smem[];
    BnCtl *ctl = reinterpret_cast<BnCtl *>(smem);
    volatile int *abort_flag = &ctl->abort_flag;
    float *tab = reinterpret_cast<float *>(smem + kBnTab);                       // [4][64] constants of the slab's channels
    const uint32_t ring = sm100::smem_u32(smem) + kBnData;
    const uint32_t in_bytes = (uint32_t)p.pix * (uint32_t)p.sv * 16u;            // one input's share of a stage
    const uint32_t stage_bytes = in_bytes * (uint32_t)p.n_in;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int cons_warps = p.consumers >> 5;
    const int slab = blockIdx.x % p.slabs, part = blockIdx.x / p.slabs;
    const int v0 = slab * p.sv;                                                  // first vector of the slab
    if (t == 0) {
        for (int s = 0; s < p.stages; ++s) {
            sm100::mbar_init(sm100::smem_u32(&ctl->full[s]), 1);
            sm100::mbar_init(sm100::smem_u32(&ctl->empty[s]), (uint32_t)cons_warps);
        }
        ctl->abort_flag = 0;
        sm100::fence_mbar_init();
    }
    __syncthreads();
    // An apply pass behind a reduce pass of the same call reads nothing that pass writes except the sums, and that pass has waited
    // for everything before it: the producer starts at once and the ring fills while the sums are being finished. (Behind a
    // convolution, pt_bn_relu_fwd_stats, x is what the predecessor writes: p.pivot = 0 there.) Everybody else waits.
    const bool early = (PASS == 2 && p.pivot) || PASS == 3;
    if (!(early && warp == cons_warps)) sm100::grid_dependency_wait();
    sm100::grid_launch_dependents();
    if (warp == cons_warps) {
        if (lane == 0) {
            int s = 0, ph = 0, issued = 0;
            for (long long i = part; i < p.chunks; i += p.parts, ++issued) {
                const long long ch = p.reverse ? p.chunks - 1 - i : i, p0 = ch * p.pix;
                if (!sm100::mbar_wait(sm100::smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, g.status, 60)) break;
                if (p.test_skip && issued == 0) {                                // test hook: this stage never becomes full
                    if (++s == p.stages) { s = 0; ph ^= 1; }
                    continue;
                }
                const uint32_t bar = sm100::smem_u32(&ctl->full[s]), dst = ring + (uint32_t)s * stage_bytes;
                if (p.slabs == 1) {                                              // whole rows: consecutive bytes
                    const uint32_t bytes = (uint32_t)(p.M - p0 < p.pix ? p.M - p0 : p.pix) * (uint32_t)p.ld * 2u;
                    sm100::mbar_arrive_expect_tx(bar, bytes * (uint32_t)p.n_in);
                    sm100::bulk_load(dst, g.in[0] + (size_t)p0 * p.LV, bytes, bar);
                    if (p.n_in > 1) sm100::bulk_load(dst + in_bytes, g.in[1] + (size_t)p0 * p.LV, bytes, bar);
                    if (BWD && p.n_in > 2) sm100::bulk_load(dst + 2u * in_bytes, g.in[2] + (size_t)p0 * p.LV, bytes, bar);
                } else {                                                         // (what lies outside the tensor arrives as zeros)
                    sm100::mbar_arrive_expect_tx(bar, stage_bytes);
                    sm100::tma_load_2d(dst, &tm0, bar, v0 * 8, (int)p0);
                    if (p.n_in > 1) sm100::tma_load_2d(dst + in_bytes, &tm1, bar, v0 * 8, (int)p0);
                    if (BWD && p.n_in > 2) sm100::tma_load_2d(dst + 2u * in_bytes, &tm2, bar, v0 * 8, (int)p0);
                }
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) sm100::drain_ring(sm100::smem_u32(&ctl->full[0]), p.stages, issued);
        }
        return;
    }
    const int pr = t / p.sv, cv = t - pr * p.sv;
    const bool active = pr < p.ppb && v0 + cv < p.LV;
    const int cols = p.sv * 8, c0 = v0 * 8;                                      // the slab's channels
    // ---- the slab's constants: [0] = pivot | mean | scale | gamma*invstd, [1] = - | invstd | shift | mean, [2], [3] = those of pass 3
    if (REDUCE) {
        for (int e = t; e < cols; e += p.consumers) {
            const int c = c0 + e;
            tab[e] = c < p.C ? (PASS == 0 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(g.in[0])[c]) : g.mean[c]) : 0.f;
            tab[64 + e] = (PASS == 1 && c < p.C) ? g.invstd[c] : 0.f;
            if (PASS == 0 && part == 0 && c < p.C) g.pivots[c] = tab[e];
        }
    } else {
        // fp64 sums of the slab's columns of the partial rows: thread (quad of columns, slice) adds its rows in ascending order, eight
        // loads in flight, then one thread per value adds the slices in order
        double *sl = reinterpret_cast<double *>(smem + kBnData + (size_t)p.stages * stage_bytes);
        const int quads = cols / 4 * 2, slices = p.consumers / quads;            // the two halves of a row: sums, then sums of squares
        const int q = t % quads, z = t / quads, half = q >= quads / 2 ? 1 : 0, cq = (q - half * (quads / 2)) * 4;
        if (z < slices) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            float lo[4] = {0.f, 0.f, 0.f, 0.f};                                  // the roundings' rows: fp32 is plenty for their sum
            if (c0 + cq < p.ld) {
                const int pitch = p.pairs ? 4 * p.ld : 2 * p.ld;
                const float *src = g.partial + (size_t)half * p.ld + c0 + cq;
                const auto row = [&](int rr, int off) {
                    const float *a = src + (size_t)rr * pitch + off;
                    return rr >= p.rows ? make_float4(0.f, 0.f, 0.f, 0.f) : p.rows_vec ? *reinterpret_cast<const float4 *>(a) : make_float4(a[0], a[1], a[2], a[3]);
                };
                for (int r = z; r < p.rows; r += (p.pairs ? 4 : 8) * slices) {
                    float4 v[8];                                                 // eight rows, or four and what their rounding left
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = p.pairs ? row(r + (u & 3) * slices, u < 4 ? 0 : 2 * p.ld) : row(r + u * slices, 0);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (u >= 4 && p.pairs) { lo[0] += v[u].x; lo[1] += v[u].y; lo[2] += v[u].z; lo[3] += v[u].w; }
                        else { acc[0] += (double)v[u].x; acc[1] += (double)v[u].y; acc[2] += (double)v[u].z; acc[3] += (double)v[u].w; }
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) sl[(size_t)z * (quads * 4) + q * 4 + e] = acc[e] + (double)lo[e];
        }
        sm100::named_barrier(1, p.consumers);
        for (int e = t; e < cols; e += p.consumers) {
            const int c = c0 + e;
            double s0 = 0.0, s1 = 0.0;
            for (int k = 0; k < slices; ++k) { s0 += sl[(size_t)k * (quads * 4) + e]; s1 += sl[(size_t)k * (quads * 4) + cols + e]; }
            float k0 = 0.f, k1 = 0.f, k2 = 0.f, k3 = 0.f;
            if (c < p.C) {
                if (PASS == 2) {
                    const double M = (double)p.M, d = s0 / M;
                    double var = s1 / M - d * d;
                    if (var < 0.0) var = 0.0;
                    const double mean = (p.pivot ? (double)g.pivots[c] : 0.0) + d;
                    const float fm = (float)mean, fi = (float)(1.0 / sqrt(var + (double)p.eps));
                    k0 = g.gamma[c] * fi;
                    k1 = g.beta[c] - fm * k0;
                    if (part == 0) {
                        g.mean[c] = fm;
                        g.invstd[c] = fi;
                        if (g.rmean && g.rvar) {
                            const double mom = (double)p.momentum;
                            g.rmean[c] = (float)((1.0 - mom) * (double)g.rmean[c] + mom * mean);
                            g.rvar[c] = (float)((1.0 - mom) * (double)g.rvar[c] + mom * var * (p.M > 1 ? M / (M - 1.0) : 1.0));
                        }
                    }
                } else {
                    // dx = gamma*invstd * (dz - dbeta/M - (x - mean) * (invstd*dgamma/M)), the differences taken first: they cancel
                    const float is = g.invstd[c], db = (float)s0, dg = (float)s1;
                    k0 = g.gamma[c] * is;
                    k1 = g.mean[c];
                    k2 = -(is * dg / (float)p.M);
                    k3 = db / (float)p.M;
                    if (part == 0) { g.dbeta[c] = db; g.dgamma[c] = dg; }
                }
            }
            tab[e] = k0; tab[64 + e] = k1;
            if (PASS == 3) { tab[128 + e] = k2; tab[192 + e] = k3; }
        }
    }
    sm100::named_barrier(1, p.consumers);
    const bool masked = BWD && p.n_in > 2;
    const bool has_aux = p.n_in > 1;
    // per-channel constants of the thread's vector (0 past the true channel count) and, for the outputs, the bits to keep
    float k0[8], k1[8], k2[PASS == 3 ? 8 : 1], k3[PASS == 3 ? 8 : 1], t0[REDUCE ? 8 : 1], t1[REDUCE ? 8 : 1];
    unsigned keep[REDUCE ? 1 : 4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int e = active ? cv * 8 + j : 0;
        k0[j] = tab[e];
        k1[j] = tab[64 + e];
        if (PASS == 3) { k2[j] = tab[128 + e]; k3[j] = tab[192 + e]; }
        if (REDUCE) t0[j] = t1[j] = 0.f;
        if (!REDUCE && (j & 1) == 0) keep[j >> 1] = (c0 + e < p.C ? 0xffffu : 0u) | (c0 + e + 1 < p.C ? 0xffff0000u : 0u);
    }
    const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f);
    const uint32_t pitch = (uint32_t)p.sv * 16u;
    int s = 0, ph = 0;
    for (long long i = part; i < p.chunks; i += p.parts) {
        const long long ch = p.reverse ? p.chunks - 1 - i : i, p0 = ch * p.pix;
        const int n = (int)(p.M - p0 < p.pix ? p.M - p0 : p.pix);
        if (!sm100::mbar_wait(sm100::smem_u32(&ctl->full[s]), ph, abort_flag, g.status, 61)) break;
        if (active) {
            const uint32_t base = ring + (uint32_t)s * stage_bytes + (uint32_t)cv * 16u;
            const size_t row0 = (size_t)p0 * p.LV + v0 + cv;
            float a0[REDUCE ? 8 : 1], a1[REDUCE ? 8 : 1];                        // the chunk's sums
            if (REDUCE)
#pragma unroll
                for (int j = 0; j < 8; ++j) a0[j] = a1[j] = 0.f;
#pragma unroll 2
            for (int r = pr; r < n; r += p.ppb) {
                const uint32_t at = base + (uint32_t)r * pitch;
                float xv[8], av[8];
                unpack8(lds128(at), xv);
                if (PASS == 0) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) { const float dd = xv[j] - k0[j]; a0[j] += dd; a1[j] = fmaf(dd, dd, a1[j]); }
                } else if (PASS == 2) {
                    if (has_aux) unpack8(lds128(at + in_bytes), av);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        xv[j] = fmaf(xv[j], k0[j], k1[j]);
                        if (has_aux) xv[j] += av[j];
                    }
                    uint4 o = pack8(xv);
                    __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&o);
                    if (p.relu)
#pragma unroll
                        for (int j = 0; j < 4; ++j) h[j] = __hmax2(h[j], zero2);
                    g.out[row0 + (size_t)r * p.LV] = make_uint4(o.x & keep[0], o.y & keep[1], o.z & keep[2], o.w & keep[3]);
                } else {
                    // dz keeps dy's bits where y > 0 (a NaN does not count as above 0)
                    uint4 d = lds128(at + in_bytes);
                    if (masked) {
                        const uint4 m = lds128(at + 2u * in_bytes);
                        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&m);
                        d.x &= __hgt2_mask(h[0], zero2);
                        d.y &= __hgt2_mask(h[1], zero2);
                        d.z &= __hgt2_mask(h[2], zero2);
                        d.w &= __hgt2_mask(h[3], zero2);
                    }
                    if (PASS == 1) {
                        unpack8(d, av);
#pragma unroll
                        for (int j = 0; j < 8; ++j) { a0[j] += av[j]; a1[j] = fmaf(av[j], xv[j] - k0[j], a1[j]); }
                    } else {
                        // pad lanes may hold anything, NaN included: their bits never get through
                        d = make_uint4(d.x & keep[0], d.y & keep[1], d.z & keep[2], d.w & keep[3]);
                        unpack8(d, av);
#pragma unroll
                        for (int j = 0; j < 8; ++j) xv[j] = k0[j] * fmaf(xv[j] - k1[j], k2[j], av[j] - k3[j]);
                        const uint4 o = pack8(xv);
                        g.out[row0 + (size_t)r * p.LV] = make_uint4(o.x & keep[0], o.y & keep[1], o.z & keep[2], o.w & keep[3]);
                        if (g.out2) g.out2[row0 + (size_t)r * p.LV] = d;
                    }
                }
            }
            if (REDUCE)
#pragma unroll
                for (int j = 0; j < 8; ++j) { t0[j] += a0[j]; t1[j] += a1[j]; }
        }
        __syncwarp();
        if (lane == 0) sm100::mbar_arrive(sm100::smem_u32(&ctl->empty[s]));
        if (++s == p.stages) { s = 0; ph ^= 1; }
    }
    if (!REDUCE) return;
    // the slab's part of two rows of partial sums. The ring is idle by then (every chunk has been consumed) and takes the threads'
    // sums, 16 per thread at a pitch of 17 words; the 16 x sv values are then added in fp64 over the ppb pixel rows by all threads, in
    // `pieces` groups of rows, and the groups by one thread per value: a fixed order
    float *red = reinterpret_cast<float *>(smem + kBnData);
    double *red2 = reinterpret_cast<double *>(red + p.consumers * 17);           // (consumers is a multiple of 32)
    sm100::named_barrier(1, p.consumers);
    if (pr < p.ppb)
#pragma unroll
        for (int j = 0; j < 8; ++j) { red[t * 17 + j] = active ? t0[j] : 0.f; red[t * 17 + 8 + j] = active ? t1[j] : 0.f; }
    sm100::named_barrier(1, p.consumers);
    const int vals = p.sv * 16, pieces = p.consumers / vals;                     // (at least 2: a slab has at most 128 values)
    const int piece = t / vals, v = t - piece * vals, half = v >= cols ? 1 : 0, c = v - half * cols;
    if (piece < pieces) {
        const float *src = red + (c >> 3) * 17 + half * 8 + (c & 7);
        // (two rows at a time in fp32: half of the conversions to fp64, and what that rounds is lost among the many pairs)
        double acc[2] = {0.0, 0.0};
        const int step = pieces * p.sv * 17;
        src += piece * p.sv * 17;
        for (int r = piece; r < p.ppb; r += 8 * pieces, src += 8 * step) {
            float u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) u[i] = r + i * pieces < p.ppb ? src[i * step] : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i & 1] += (double)(u[2 * i] + u[2 * i + 1]);
        }
        red2[piece * vals + v] = acc[0] + acc[1];
    }
    sm100::named_barrier(1, p.consumers);
    if (piece == 0 && c0 + c < p.ld) {
        double sum = 0.0;
#pragma unroll 4
        for (int k = 0; k < pieces; ++k) sum += red2[k * vals + v];
        if (PASS == 1 && half) sum *= (double)tab[64 + c];                       // sum(dz * (x - mean)) -> sum(dz * xhat)
        const float hi = (float)sum;
        float *o = g.partial + ((size_t)part * 4 + half) * p.ld + c0 + c;
        *o = hi;
        o[2 * p.ld] = isfinite(hi) ? (float)(sum - (double)hi) : 0.f;
    }
}

pt_status bn_params(const pt_ctx *c, const pt_bn_desc *d, BnP *p)
{
    if (!c || !d) return PT_ERR_INVALID_ARG;
    if (d->N < 1 || d->H < 1 || d->W < 1 || d->C < 1 || d->ld < d->C || (d->ld & 7)) return PT_ERR_INVALID_ARG;
    if (!(d->eps >= 0.f) || !(d->momentum >= 0.f && d->momentum <= 1.f)) return PT_ERR_INVALID_ARG;
    if (d->ld > 2048) return PT_ERR_UNSUPPORTED;
    memset(p, 0, sizeof(*p));
    p->M = (long long)d->N * d->H * d->W;
    p->C = d->C; p->ld = d->ld; p->LV = d->ld / 8;
    // slabs of equal width (144 channels are three slabs of 48, not 64 + 64 + 16)
    p->slabs = pt_ceil_div(p->LV, kBnSlab);
    p->sv = pt_ceil_div(p->LV, p->slabs);
    p->slabs = pt_ceil_div(p->LV, p->sv);
    p->ppb = kBnThreads / p->sv;
    p->consumers = (p->sv * p->ppb + 31) / 32 * 32;
    p->eps = d->eps; p->momentum = d->momentum; p->relu = d->relu ? 1 : 0;
    // one block per SM; no more parts of a slab than it has rows of the consumer threads
    const long long most = c->sm_count / p->slabs > 0 ? c->sm_count / p->slabs : 1, need = (p->M + p->ppb - 1) / p->ppb;
    p->parts = (int)(need < most ? need : most);
    return PT_OK;
}

// bf16 tensor (channels, pixels) with pitch ld: boxes of one slab x `pix` pixels.
bool make_slab_map(const pt_ctx *c, CUtensorMap *tm, const void *base, const BnP &p)
{
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                               const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    if (!c->encode_tiled) return false;
    cuuint64_t dims[2] = {(cuuint64_t)p.ld, (cuuint64_t)p.M}, strides[1] = {(cuuint64_t)p.ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)p.sv * 8, (cuuint32_t)p.pix}, estr[2] = {1, 1};
    return ((Encode)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int PASS>
pt_status launch_bn(pt_ctx *c, BnP p, const BnArgs &g, int n_in, cudaStream_t st)
{
    p.n_in = n_in;
    // stages of about kBnStage bytes, smaller ones where that would leave blocks without a chunk (a tensor of 7x7 maps is a few
    // megabytes), at least one row of the consumer threads, at most the 256 rows of a TMA box
    const long long share = (p.M + p.parts - 1) / p.parts;
    long long pix = (long long)(kBnStage / ((size_t)n_in * p.sv * 16));
    if (pix > share) pix = share;
    pix = pix / p.ppb * p.ppb;
    if (pix < p.ppb) pix = p.ppb;
    if (pix > 256 && p.slabs > 1) pix = 256;
    pix &= ~7ll;                                                 // (at least 64 by then) TMA boxes start on 128-byte boundaries
    p.pix = (int)pix;
    p.chunks = (p.M + pix - 1) / pix;
    const long long per_block = (p.chunks + p.parts - 1) / p.parts;
    const size_t stage = (size_t)pix * n_in * p.sv * 16;
    p.stages = (int)(kBnRing / stage);
    if (p.stages > kBnMaxStages) p.stages = kBnMaxStages;
    if (p.stages > per_block) p.stages = (int)per_block;
    // an apply pass walks backwards: what the pass before it read (or wrote) last is still in L2
    p.reverse = PASS >= 2 ? 1 : 0;
    p.rows_vec = ((uintptr_t)g.partial & 15) == 0 ? 1 : 0;
    size_t smem = kBnData + (size_t)p.stages * stage;
    const size_t red = kBnData + (size_t)p.consumers * 17 * sizeof(float) + kBnThreads * sizeof(double);
    if (PASS < 2 && smem < red) smem = red;
    if (PASS >= 2) smem += (size_t)p.consumers * 4 * sizeof(double);             // the fp64 slices of the partial rows' sums
    if (!(c->attr_done & (kAttrBn << PASS))) {
        PT_CUDA_OK(cudaFuncSetAttribute(bn_kernel<PASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        c->attr_done |= kAttrBn << PASS;
    }
    if (c->test_skip == 3) { p.test_skip = 1; c->test_skip = 0; }
    CUtensorMap tm[3];
    memset(tm, 0, sizeof(tm));
    if (p.slabs > 1)
        for (int k = 0; k < n_in; ++k)
            if (!make_slab_map(c, &tm[k], g.in[k], p)) return PT_ERR_CUDA;
    PT_CUDA_OK(pt_launch_pdl(bn_kernel<PASS>, dim3((unsigned)(p.slabs * p.parts)), dim3((unsigned)p.consumers + 32u), smem, st, tm[0], tm[1],
                             tm[2], p, g));
    c->launches += 1;
    return PT_OK;
}

}  // namespace

pt_status pt_bn_set_wait_limit_ns(unsigned long long ns)
{
    PT_CUDA_OK(cudaMemcpyToSymbol(sm100::g_wait_limit_ns, &ns, sizeof(ns)));
    return PT_OK;
}

extern "C" size_t pt_bn_workspace_bytes(const pt_ctx *c, const pt_bn_desc *d)
{
    BnP p;
    if (bn_params(c, d, &p) != PT_OK) return 0;
    return ((size_t)p.parts * 4 + 1) * p.ld * sizeof(float);     // the reduce pass's rows of partial sums, the forward pass's pivots
}

static bool aligned16(const void *q) { return ((uintptr_t)q & 15) == 0; }

extern "C" pt_status pt_bn_relu_fwd(pt_ctx *c, const pt_bn_desc *d, const void *x, const void *residual, const float *gamma,
                                    const float *beta, float *running_mean, float *running_var, float *save_mean,
                                    float *save_invstd, void *y, void *ws, size_t ws_bytes, void *stream)
{
    BnP p;
    pt_status r = bn_params(c, d, &p);
    if (r != PT_OK) return r;
    if (!x || !gamma || !beta || !save_mean || !save_invstd || !y || (running_mean == nullptr) != (running_var == nullptr))
        return PT_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(y) || (residual && !aligned16(residual))) return PT_ERR_INVALID_ARG;
    if (!ws || ws_bytes < pt_bn_workspace_bytes(c, d)) return PT_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    BnArgs g{};
    g.in[0] = (const uint4 *)x; g.in[1] = (const uint4 *)residual;
    g.gamma = gamma; g.beta = beta; g.mean = save_mean; g.invstd = save_invstd; g.rmean = running_mean; g.rvar = running_var;
    g.partial = (float *)ws; g.pivots = g.partial + (size_t)p.parts * 4 * p.ld; g.out = (uint4 *)y; g.status = c->d_status;
    r = launch_bn<0>(c, p, g, 1, st);
    if (r != PT_OK) return r;
    p.rows = p.parts; p.pairs = 1; p.pivot = 1;
    r = launch_bn<2>(c, p, g, residual ? 2 : 1, st);
    if (r != PT_OK) return r;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

extern "C" pt_status pt_bn_relu_bwd(pt_ctx *c, const pt_bn_desc *d, const void *x, const void *y, const void *dy, const float *gamma,
                                    const float *save_mean, const float *save_invstd, void *dx, void *dresidual, float *dgamma,
                                    float *dbeta, void *ws, size_t ws_bytes, void *stream)
{
    BnP p;
    pt_status r = bn_params(c, d, &p);
    if (r != PT_OK) return r;
    if (!x || !dy || !gamma || !save_mean || !save_invstd || !dx || !dgamma || !dbeta || (p.relu && !y)) return PT_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(dy) || !aligned16(dx) || (y && !aligned16(y)) || (dresidual && !aligned16(dresidual)))
        return PT_ERR_INVALID_ARG;
    if (!ws || ws_bytes < pt_bn_workspace_bytes(c, d)) return PT_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    const int n_in = p.relu ? 3 : 2;                        // without ReLU there is no mask to read
    BnArgs g{};
    g.in[0] = (const uint4 *)x; g.in[1] = (const uint4 *)dy; g.in[2] = (const uint4 *)y;
    g.gamma = gamma; g.mean = const_cast<float *>(save_mean); g.invstd = const_cast<float *>(save_invstd); g.dgamma = dgamma; g.dbeta = dbeta;
    g.partial = (float *)ws; g.out = (uint4 *)dx; g.out2 = (uint4 *)dresidual; g.status = c->d_status;
    r = launch_bn<1>(c, p, g, n_in, st);
    if (r != PT_OK) return r;
    p.rows = p.parts; p.pairs = 1;
    r = launch_bn<3>(c, p, g, n_in, st);
    if (r != PT_OK) return r;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// The forward pass when the convolution that produced x already took the channel sums (pt_conv_fwd_stats): no reduction pass
// over x; the apply pass finishes the convolution's rows of partial sums.
extern "C" pt_status pt_bn_relu_fwd_stats(pt_ctx *c, const pt_bn_desc *d, const void *x, const void *residual, const float *gamma,
                                          const float *beta, float *running_mean, float *running_var, float *save_mean,
                                          float *save_invstd, void *y, const float *stats, int32_t n_parts, void *stream)
{
    BnP p;
    pt_status r = bn_params(c, d, &p);
    if (r != PT_OK) return r;
    if (!x || !gamma || !beta || !save_mean || !save_invstd || !y || !stats || n_parts < 1 ||
        (running_mean == nullptr) != (running_var == nullptr))
        return PT_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(y) || (residual && !aligned16(residual))) return PT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    // n_parts rows of [2][ld] partial sums, taken about 0
    p.rows = (int)n_parts;
    BnArgs g{};
    g.in[0] = (const uint4 *)x; g.in[1] = (const uint4 *)residual;
    g.gamma = gamma; g.beta = beta; g.mean = save_mean; g.invstd = save_invstd; g.rmean = running_mean; g.rvar = running_var;
    g.partial = const_cast<float *>(stats); g.out = (uint4 *)y; g.status = c->d_status;
    r = launch_bn<2>(c, p, g, residual ? 2 : 1, st);
    if (r != PT_OK) return r;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}
