// tcgen05 / TMEM / TMA implicit-GEMM convolutions for sm_100a.
//
//   conv_gemm_kernel   fwd and dgrad of 1x1 / strided layers: persistent CTAs, im2col-mode (or plain 2-D) TMA loads of
//                      128 pixels x 64 channels, K-major (fwd) or MN-major (dgrad) weight tiles from the same bf16 shadow,
//                      double/triple-buffered fp32 accumulators in TMEM, TMA-store epilogue.
//   conv_halo_kernel   stride-1 RxS fwd/dgrad, the parities of a stride-2 dgrad, stride-2 fwd by parity planes: one halo tile per 64-channel chunk,
//                      filter taps as row-shifted UMMA descriptors of that tile; a 32-byte-pixel mode (16 lanes per
//                      position, 32-byte swizzle, one MMA per tap) runs the space-to-depth stem where conv_stem_kernel does not.
//   conv_wgrad_kernel  weight gradient: both operands MN-major, reduction over pixels split across CTAs, partial tiles
//                      summed in-kernel in a fixed order.
//   conv_wgrad_taps_kernel  weight gradient by filter rows: the staged pixels of one serve all of its taps (stride 1 or 2, one tile of input channels: 160 for three
//                      columns, 256 for two, 64 for eight).
//   conv_wgrad_packed_kernel  weight gradient of narrow stride-1 layers: several pixels to a staged row.
//   conv_wgrad_rows_kernel  weight gradient of stride-1 layers with at most 64 input channels: row blocks of x staged
//                      once, taps as row-shifted descriptors, two or four taps per MMA on the M side; same finish phase.
//   conv_stem_kernel   forward pass of the few-channel stride-2 stem straight from the image.
//   stem_* kernels     space-to-depth layout kernels of its weight gradient (and of forward passes that conv_stem_kernel does not take).
// Ragged channel counts are handled by the TMA unit (true extents in the tensor maps: zero-fill on load, clipping on
// store) and by skipping the 16-wide k-steps past the last valid channel.
// Issue is spread over warps in all three kernels: one thread spends ~200 cycles per TMA instruction and 50-100 per
// tcgen05.mma, more than a narrow MMA takes to run, so operands are loaded by several producer warps and, where
// independent accumulators exist, MMAs are issued by up to four warps, each with its own ring and TMEM buffers.
// The kernels are launched with programmatic stream serialization (griddepcontrol.wait after the prologue).
// Every wait on a barrier or a counter is bounded; on expiry the CTA records PT_DEV_TIMEOUT in the status word, drains its copies and
// exits. (The cluster barriers of the weight gradients' exchange have no limit: every thread of every CTA reaches them, aborting ones
// too.)
#include "pt_internal.h"
#include "pt_sm100_ptx.cuh"
#include <cudaTypedefs.h>

using namespace sm100;

namespace {
// A tensor-map encode that the driver refused is kept, with its line, for pt_last_cuda_error.
bool map_ok(CUresult r, int line)
{
    if (r != CUDA_SUCCESS) pt_note_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncode* (refused by the driver)", __FILE__, line);
    return r == CUDA_SUCCESS;
}


constexpr int kBM = 128;            // output pixels per CTA tile
constexpr int kKC = 64;             // reduction channels per stage (one 128-byte swizzle row)
constexpr int kMaxStages = 8;
constexpr int kThreads = 288;           // wgrad kernel: dy producer, MMA issuer, 4 epilogue warps (x producers in the main loop), 3 more MMA issuers
constexpr int kGemmThreads = 512;       // fwd/dgrad kernel: A producer, MMA issuer, up to 12 epilogue warps, B producer, second MMA issuer
constexpr int kMaxTaps = 64;

struct GemmP {
    int M_total;        // output pixels of this launch's raster
    int n_cols;         // true number of output channels
    int BN;             // tile width (multiple of 16)
    int n_tiles;        // tiles along the channel dimension
    int c_red;          // true number of reduction channels
    int k_chunks;       // ceil(c_red / 64)
    int taps;           // filter taps visited by this launch (<= kMaxTaps)
    int Pd, Qd;         // raster of output pixels (rows, columns) per image
    int stride;         // traversal stride of the raster in the source tensor
    int lo_h, lo_w;     // source coordinate of raster position (0,0) for tap (0,0)
    int stages;
    int tmem_cols;
    // output pixel mapping: pixel (n, i, j) of the raster -> out[((n*oH + i*o_step + o_h0)*oW + j*o_step + o_w0)*ld_out]
    int oH, oW, o_step, o_h0, o_w0;
    int ld_out, out_f32;
    int vec_cols;       // strided bf16 outputs: channels covered by whole 16-byte vectors
    int zero_mask;      // stride-2 dgrad: bit (a*2+b) set => also write zeros to the pixel at parity (a,b) of each 2x2 cell
    int tma_store;      // 1: bf16 output rows are consecutive pixels -> staged in shared memory and written by TMA stores
    int m_tiles;        // ceil(M_total / 128)
    int epi_groups;     // 1..3 groups of four epilogue warps
    int n_a, n_b;       // producer warps of the activation tiles (two: one per issuer's ring), of streamed weight tiles (1 or 2)
    int tail_lanes;     // channel lanes the last activation chunk is staged with: 64, 32 or 16 (rows of 128, 64 or 32 bytes)
    int a_tiled;        // 1: 1x1 stride-1 problem, the A operand is a plain 2-D (channels, pixels) tiled map
    int resident;       // 1: every weight tile of the launch stays in shared memory (loaded once); the ring carries A only
    int n_issuers;      // 2 (resident weights only): two MMA issuer warps take alternate tiles, each with half of the ring's stages
    int acc_per;        // two issuers: accumulator buffers per issuer (1 or 2)
    int alias_staging;  // 1: the CTA has a single tile; the epilogue's staging slabs lie in the (then idle) ring
    int test_skip;      // test hook (pt_test_skip_next_arrive): the A producer leaves out the first stage of its first tile
    int stats_off;      // byte offset in shared memory of the epilogue warps' statistics accumulators (stats != nullptr)
    int stats_warp;     // bytes of one warp's accumulators: 512 per 64-channel chunk of the tile
    int stats_lo;       // 1: two rows of sums per row of CTAs
    float *stats;       // optional: rows [2][ld_out] of floats, one per n_tiles CTAs: per output channel, sum and sum of squares of
                        // the bf16 values they stored (the batch-normalisation statistics of the layer that follows)
    void *out;
    unsigned int *status;
    unsigned char tap_oh[kMaxTaps], tap_ow[kMaxTaps];   // im2col offsets of each visited tap
    unsigned short tap_wt[kMaxTaps];                    // index r*S+s of the weights the tap multiplies
};

struct __align__(8) Ctl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t accum;
    uint32_t tmem_base;
    int abort_flag;
};

// Control block of the persistent fwd/dgrad kernel.
struct __align__(8) PCtl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t acc_full[4];       // MMA issuer -> epilogue: accumulator buffer b holds a finished tile
    uint64_t acc_empty[4];      // epilogue -> MMA issuer: buffer b has been read out (4 arrivals, one per warp of its group)
    uint64_t w_full;            // resident weights have landed
    uint32_t tmem_base;
    int abort_flag;
#ifdef PT_DEVICE_TRACE
    unsigned int chain_seq;
#endif
};

constexpr uint32_t kSlabs = 2;                          // staging slabs per epilogue warp (TMA stores in flight)

// Batch-normalisation statistics of a staged output chunk: `rows` is a bit mask of the warp's 32 staged rows (128 bytes each,
// 128-byte swizzle, first row `row0` of the slab) that are real output pixels. Lane l owns channels 2l and 2l + 1 of the
// 64-channel chunk and adds the bf16 values exactly as they were stored, rows in ascending order: sum and sum of squares,
// accumulated in the warp's own shared-memory slots (acc: 128 floats per chunk of the tile, four per lane); stats_store_cta
// combines the warps of a CTA at the end. Feature normalisation (Sec. 2.1) reads its input twice; taking the sums here,
// from the tile that is still in shared memory, removes the first of the two passes.
// Fewer rows than this and the rounding of a CTA's sums (2^-25 over the square root of their number) shows in 1/std: 16x7x7x2000 has 18.
constexpr int kStatsFewRows = 64;
constexpr uint32_t kStatsChunkBytes = 128u * 4u;              // per 64-channel chunk: 32 lanes x (sum, sum of squares) x two channels

__device__ __forceinline__ void chunk_stats(uint32_t slab, int row0, uint32_t rows, int lane, uint32_t acc)
{
    float s0a = 0.f, s1a = 0.f, s0b = 0.f, s1b = 0.f;
    const uint32_t jj = (uint32_t)lane >> 2, wi = ((uint32_t)lane & 3u) << 2;
    // Eight loads are issued before the first is used (one at a time, each waits out the shared-memory latency: 1500 cycles
    // per chunk in the first version, more than the rest of the epilogue). Rows that are not output pixels (the halo tiles'
    // raster has some) are loaded too and count as zeros.
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 8) {
        uint32_t word[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t m = (uint32_t)(row0 + r0 + j);
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(word[j]) : "r"(slab + m * 128u + ((jj ^ (m & 7u)) << 4) + wi));
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const bool on = (rows >> (r0 + j)) & 1u;
            const float a = on ? __uint_as_float(word[j] << 16) : 0.f, b = on ? __uint_as_float(word[j] & 0xffff0000u) : 0.f;
            s0a += a; s1a = fmaf(a, a, s1a);
            s0b += b; s1b = fmaf(b, b, s1b);
        }
    }
    float4 t;
    const uint32_t slot = acc + (uint32_t)lane * 16u;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(slot) : "memory");
    t.x += s0a; t.y += s1a; t.z += s0b; t.w += s1b;
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(slot), "f"(t.x), "f"(t.y), "f"(t.z), "f"(t.w) : "memory");
}

__device__ __forceinline__ void stats_clear(uint32_t acc0, int lane, int n_chunks)
{
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        if (ch < n_chunks)
            asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(acc0 + (uint32_t)ch * 512u + (uint32_t)lane * 16u), "f"(0.f) : "memory");
}

// The sums of a CTA's epilogue warps (accumulators of `stride` bytes each, from `acc0` on) are added in the order of the warps, in fp64
// (two warps at a time in fp32: half of the conversions), and leave for a row of partial sums, [2][ld] floats, or for two (`lo`): the sums rounded, and what the rounding left. A CTA's tiles all have the same output channels n0 .. (its grid is a multiple of
// the number of channel tiles), so that it writes once, and the CTAs of a row, one per channel tile, write disjoint columns; the
// last one also writes the zeros up to ld. `tid` of `nthr` epilogue threads; a barrier of theirs comes before the call. (One row
// per epilogue warp made up to 1776 rows, a few megabytes, for the normalisation to add up.)
__device__ __forceinline__ void stats_store_cta(uint32_t acc0, uint32_t stride, int n_warps, int tid, int nthr, float *dst, int ld, int lo, int n_cols,
                                                int n0, int n_end)
{
    for (int c = n0 + tid; c < n_end; c += nthr) {
        double s0 = 0.0, s1 = 0.0;
        if (c < n_cols) {
            // a chunk is 64 channels: lane (c % 64) / 2 keeps (sum, sum of squares) of its two channels
            const int e = c - n0;
            const uint32_t a = acc0 + (uint32_t)(e >> 6) * 512u + (uint32_t)((e & 63) >> 1) * 16u + (uint32_t)(e & 1) * 8u;
            for (int w = 0; w < n_warps; w += 2) {               // (four, eight or twelve warps)
                float u0, u1, v0, v1;
                asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(u0), "=f"(u1) : "r"(a + (uint32_t)w * stride) : "memory");
                asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v0), "=f"(v1) : "r"(a + (uint32_t)(w + 1) * stride) : "memory");
                s0 += (double)(u0 + v0); s1 += (double)(u1 + v1);
            }
        }
        const float h0 = (float)s0, h1 = (float)s1;
        dst[c] = h0;
        dst[ld + c] = h1;
        if (lo) {
            dst[2 * ld + c] = isfinite(h0) ? (float)(s0 - (double)h0) : 0.f;
            dst[3 * ld + c] = isfinite(h1) ? (float)(s1 - (double)h1) : 0.f;
        }
    }
}

// Device-side timeline of CTA 0 (a build with -DPT_DEVICE_TRACE; read back with pt_debug_gemm_trace): per pipeline stage in
// issue order, when the A producer found it free / issued it, when the MMA issuer found it full / committed it; per tile, when
// the epilogue got the accumulator and when it had issued its stores.
#ifdef PT_DEVICE_TRACE
__device__ unsigned long long g_gemm_trace[8][64];
#define GTRACE(role, idx) do { if (blockIdx.x == 0 && (idx) < 64 && (threadIdx.x & 31) == 0) g_gemm_trace[role][idx] = globaltimer_ns(); } while (0)
// Timeline of a chain of launches: launch number seq (a device counter, taken by CTA 0 at entry) stamps its entry, the end of
// its prologue, the return of its dependency wait, its first activation load, its first full stage, its last commit, the end
// of its last epilogue and its exit.
__device__ unsigned long long g_chain_trace[256][12];
__device__ unsigned int g_chain_seq;
#define CTRACE(ev) do { if (blockIdx.x == 0 && (threadIdx.x & 31) == 0 && ctl->chain_seq < 256) g_chain_trace[ctl->chain_seq][ev] = globaltimer_ns(); } while (0)
#else
#define GTRACE(role, idx) do { } while (0)
#define CTRACE(ev) do { } while (0)
#endif

// Persistent: each CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... The TMA ring runs continuously across
// tiles. The accumulator has G = 2 or 3 buffers in TMEM and buffer b has its own group of four epilogue warps, so the
// loads and MMAs of the next tiles overlap the epilogues of the previous ones.
// STATS: the epilogue also takes the batch-normalisation statistics (a variant of its own: the plain kernels keep their registers).
// n / d for 0 <= n < 2^22 and a divisor known per kernel: float reciprocal plus one correction step (an integer division
// costs ~40 instructions, and the reduction below does two per 16-byte item).
__device__ __forceinline__ int fast_div(int n, int d, float inv_d)
{
    int q = __float2int_rz(__int2float_rn(n) * inv_d);
    if ((q + 1) * d <= n) ++q;
    if (q * d > n) --q;
    return q;
}

// Stores a warp's 32 staged rows (128 bytes each, 128-byte swizzle) of `pieces` 16-byte vectors to the pixels `pix` (one per lane) whose bit
// of `rows` is set: eight lanes to a pixel. (Every lane on the next vector whatever its row: 33.9 -> 35.9 us for 256 <- 512 channels at 56x56, batch 64.)
__device__ __forceinline__ void store_rows_apart(__nv_bfloat16 *out, int ld, uint32_t slab, int col, int pieces, uint32_t rows, int pix, int lane)
{
    const int j = lane & 7;
    uint4 t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t r = (uint32_t)(i * 4 + (lane >> 3));
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(t[i].x), "=r"(t[i].y), "=r"(t[i].z), "=r"(t[i].w)
                     : "r"(slab + r * 128u + (((uint32_t)j ^ (r & 7u)) << 4)) : "memory");
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = i * 4 + (lane >> 3);
        const int px = __shfl_sync(0xffffffffu, pix, r);
        if (j < pieces && ((rows >> r) & 1u)) *reinterpret_cast<uint4 *>(out + (size_t)px * (size_t)ld + col + j * 8) = t[i];
    }
}

// APART: bf16 output pixels two apart (a variant of its own: one kernel with both epilogues spills).
template <bool B_MN, bool STATS, bool APART>
__global__ void __launch_bounds__(kGemmThreads, 1) conv_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                 const __grid_constant__ CUtensorMap tmT /* last chunk of A */,
                                                                 const __grid_constant__ CUtensorMap tmB,
                                                                 const __grid_constant__ CUtensorMap tmC, const GemmP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    PCtl *ctl = reinterpret_cast<PCtl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t staging_base = (smem_base + (uint32_t)sizeof(PCtl) + 1023u) & ~1023u;
    const uint32_t a_bytes = kBM * kKC * 2;
    const uint32_t b_bytes = B_MN ? (uint32_t)((p.BN + 63) / 64) * 8192u : (uint32_t)p.BN * 128u;
    const uint32_t b_slot = (b_bytes + 1023u) & ~1023u;
    // resident weights: all taps x chunks sit in front of the ring, whose stages then hold an A tile only
    // a CTA with a single tile stages its output in the ring, which is idle by then: no separate staging area
    const uint32_t w_base = staging_base + (p.alias_staging ? 0u : (uint32_t)p.epi_groups * 4u * kSlabs * 4096u);
    const uint32_t stage_bytes = p.resident ? a_bytes : a_bytes + b_slot;
    const uint32_t data_base = w_base + (p.resident ? (uint32_t)(p.taps * p.k_chunks) * b_slot : 0u);
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int iters = p.taps * p.k_chunks;
    const int total_tiles = p.m_tiles * p.n_tiles;
    // Producers: warp 0 the activation tiles, warp 14 the weights; streamed MN-major weight tiles are one 8 KB box per 64 columns, every
    // other one of which warp 15 issues. With two issuers (resident weights) and several chunks per tile warp 14 feeds the second issuer's
    // ring: a thread issues a box only every 0.3 to 0.5 us (77 -> 19 at 56x56, batch 256: 41.6 -> 29.5 us; with a single chunk per tile
    // the output side is the longer one and the second producer costs up to 1 us). Halves of an activation or K-major weight tile from
    // two warps each were measured too: no faster, the deep layers wait for what is in flight.
    const int nb_b = (p.BN + 63) / 64;
    const bool ring2 = p.n_a == 2;
    const int a_id = warp == 0 ? 0 : (ring2 && warp == 14) ? 1 : -1;
    const int b_id = warp == 14 ? 0 : (!p.resident && warp == 15 && p.n_b > 1) ? 1 : -1;

#ifdef PT_DEVICE_TRACE
    if (threadIdx.x == 0) {
        ctl->chain_seq = blockIdx.x == 0 ? atomicAdd(&g_chain_seq, 1u) : 0xffffffffu;
        CTRACE(0);
    }
#endif
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), (uint32_t)(1 + (p.resident ? 0 : p.n_b)));
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        mbar_init(smem_u32(&ctl->w_full), 1);
        for (int b = 0; b < 4; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 4);
        }
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        if (p.tma_store) prefetch_tmap(&tmC);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    // The weights are not written by the kernels that precede a convolution in a stream (those that trigger their dependents
    // early are convolutions themselves), so the weight producers start loading at once; everybody else waits for the
    // previous kernel's results here.
    // The activation producer (warp 0) waits just before its first load instead: its set-up (tile coordinates, tap tables: a
    // few hundred cycles of divisions and first-touch parameter reads) then runs while the previous kernel drains.
    if (!(a_id >= 0 || b_id >= 0)) grid_dependency_wait();
    grid_launch_dependents();

    if (a_id >= 0 || b_id >= 0) {
        if (lane == 0) {
            // ---------------- TMA producers
            const bool is_a = a_id >= 0;                     // (warp 14 with two rings: the weights first, then activations)
            if (warp == 0) CTRACE(8);
            const uint32_t my_bytes = is_a ? a_bytes : B_MN ? (uint32_t)((nb_b - b_id + p.n_b - 1) / p.n_b) * 8192u : b_bytes;
            const uint32_t tail_bytes = is_a ? (uint32_t)(kBM * p.tail_lanes * 2) : my_bytes;
            int s = 0, ph = 0, issued = 0;   // stage-ring position, continuous across tiles; stages filled
            bool dep_waited = false;         // the activation producer has waited for the previous kernel's results
            const int SR = p.stages / p.n_issuers;
            const bool both = is_a && p.n_issuers == 2 && !ring2;      // this producer feeds two rings, a tile each in turn
            int ring = ring2 && a_id == 1 ? 1 : 0, s1 = 0, ph1 = 0;    // the ring it feeds now; its position in the other one
            if (b_id == 0 && p.resident) {
                // n_tiles == 1 here: every weight tile of the launch, once
                const uint32_t bar = smem_u32(&ctl->w_full);
                mbar_arrive_expect_tx(bar, (uint32_t)iters * b_bytes);
                for (int tap = 0; tap < p.taps; ++tap)
                    for (int kc = 0; kc < p.k_chunks; ++kc) {
                        const uint32_t dst = w_base + (uint32_t)(tap * p.k_chunks + kc) * b_slot;
                        const int wtap = p.tap_wt[tap];
                        if (!B_MN) tma_load_3d(dst, &tmB, bar, kc * kKC, wtap, 0);
                        else for (int nb = 0; nb < (p.BN + 63) / 64; ++nb) tma_load_3d(dst + (uint32_t)nb * 8192u, &tmB, bar, nb * 64, wtap, kc * kKC);
                    }
            }
            // every tile, or with a producer per ring every other one
            for (int tile = blockIdx.x + ring * (int)gridDim.x; tile < total_tiles && !*abort_flag && (is_a || !p.resident);
                 tile += (ring2 ? 2 : 1) * (int)gridDim.x) {
                const int sbase = ring * SR;
                const int n_tile = tile % p.n_tiles, m_tile = tile / p.n_tiles;
                const int n0 = n_tile * p.BN;
                const int m0 = m_tile * kBM;
                int w0 = 0, h0 = 0, n = 0;
                if (is_a && !p.a_tiled) {
                    const int q = m0 % p.Qd, t = m0 / p.Qd, pp = t % p.Pd;
                    n = t / p.Pd;
                    w0 = q * p.stride + p.lo_w; h0 = pp * p.stride + p.lo_h;
                }
                bool ok = true;
                for (int tap = 0; tap < p.taps && ok; ++tap) {
                    const int wtap = p.tap_wt[tap];
                    const uint16_t ow = (uint16_t)p.tap_ow[tap], oh = (uint16_t)p.tap_oh[tap];
                    for (int kc = 0; kc < p.k_chunks; ++kc) {
                        if (warp == 0 && issued == 0) CTRACE(9);
                        ok = mbar_wait(smem_u32(&ctl->empty[sbase + s]), ph ^ 1, abort_flag, p.status, 1);
                        if (!ok) break;
                        if (warp == 0 && issued == 0) CTRACE(10);
                        if (warp == 0) GTRACE(0, issued); else if (warp == 14) GTRACE(2, issued);
                        const uint32_t bar = smem_u32(&ctl->full[sbase + s]);
                        const uint32_t a_dst = data_base + (uint32_t)(sbase + s) * stage_bytes, b_dst = a_dst + a_bytes;
                        if (warp == 0 && p.test_skip && issued == 0) {    // test hook: this stage never becomes full
                            ++issued;
                            if (++s == SR) { s = 0; ph ^= 1; }
                            continue;
                        }
                        const bool tail = kc + 1 == p.k_chunks;
                        mbar_arrive_expect_tx(bar, tail ? tail_bytes : my_bytes);
                        if (is_a && !dep_waited) { CTRACE(1); grid_dependency_wait(); CTRACE(2); dep_waited = true; }
                        if (is_a) {
                            const CUtensorMap *tm = tail ? &tmT : &tmA;
                            if (p.a_tiled) tma_load_2d(a_dst, tm, bar, kc * kKC, m0);
                            else tma_load_im2col_4d(a_dst, tm, bar, kc * kKC, w0, h0, n, ow, oh);
                        } else if (!B_MN) {
                            tma_load_3d(b_dst, &tmB, bar, kc * kKC, wtap, n0);
                        } else {
                            for (int nb = b_id; nb < nb_b; nb += p.n_b)
                                tma_load_3d(b_dst + (uint32_t)nb * 8192u, &tmB, bar, n0 + nb * 64, wtap, kc * kKC);
                        }
                        if (warp == 0) GTRACE(1, issued); else if (warp == 14) GTRACE(3, issued);
                        if (warp == 0 && issued == 0) CTRACE(3);
                        ++issued;
                        if (++s == SR) { s = 0; ph ^= 1; }
                    }
                }
                if (!ok) break;
                if (both) { int t = s; s = s1; s1 = t; t = ph; ph = ph1; ph1 = t; ring ^= 1; }
            }
            if (*abort_flag) {       // the copies this thread issued: stages of one ring or of both, resident weights
                if (b_id == 0 && p.resident) drain_ring(smem_u32(&ctl->w_full), 1, 1);
                // (a producer of two rings fills a tile's stages in each in turn: how many of them each got follows from their number)
                const int tiles = issued / iters, rest = issued - tiles * iters;
                const int first = both ? (tiles + 1) / 2 * iters + (tiles & 1 ? 0 : rest) : issued;
                drain_ring(smem_u32(&ctl->full[(both ? 0 : ring) * SR]), SR, first);
                if (both) drain_ring(smem_u32(&ctl->full[SR]), SR, issued - first);
            }
        }
    } else if (warp == 1 || (warp == 15 && p.n_issuers == 2)) {
        // ---------------- MMA issuer(s): the warp walks the loops in lockstep, lane 0 issues. With two issuers, issuer i
        // takes the CTA's tiles i, i + 2, ..., reads ring i and owns the accumulator buffers i*acc_per .. + acc_per - 1.
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(kBM, p.BN, 0, B_MN ? 1 : 0);
        const uint64_t bstep = B_MN ? 128ull : 2ull;
        const uint64_t a_desc0 = make_desc_rows(0u, 128u), t_desc0 = make_desc_rows(0u, (uint32_t)p.tail_lanes * 2u);
        const uint64_t b_desc0 = make_desc(0u, B_MN ? 8192u : 16u, 1024u);
        const int last_steps = (p.c_red - (p.k_chunks - 1) * kKC + 15) / 16;      // k-steps of a tap's last chunk
        const int NI = p.n_issuers, issuer = warp == 1 ? 0 : 1;
        const int SR = p.stages / NI, sbase = issuer * SR;
        int s = 0, ph = 0, b = 0, aph = 0, nt = 0;
        int consumed = 0;
        (void)consumed;
        bool ok = true;
        if (p.resident) ok = mbar_wait(smem_u32(&ctl->w_full), 0, abort_flag, p.status, 8);
        for (int tile = blockIdx.x + issuer * (int)gridDim.x; tile < total_tiles && ok; tile += NI * (int)gridDim.x, ++nt) {
            if (NI == 2) { b = p.acc_per == 2 ? issuer * 2 + (nt & 1) : issuer; aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1; }
            ok = mbar_wait(smem_u32(&ctl->acc_empty[b]), aph ^ 1, abort_flag, p.status, 7);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(b * p.BN);
            uint32_t acc = 0u;
            for (int tap = 0; tap < p.taps && ok; ++tap) {
                for (int kc = 0; kc < p.k_chunks; ++kc) {
                    ok = mbar_wait(smem_u32(&ctl->full[sbase + s]), ph, abort_flag, p.status, 2);
                    if (!ok) break;
                    if (warp == 1) GTRACE(4, consumed);
                    if (warp == 1 && consumed == 0) CTRACE(4);
                    tc_fence_after();
                    const uint32_t a_src = data_base + (uint32_t)(sbase + s) * stage_bytes;
                    const uint32_t b_src = p.resident ? w_base + (uint32_t)(tap * p.k_chunks + kc) * b_slot : a_src + a_bytes;
                    // one descriptor per operand and stage; a k-step only moves the 14-bit start-address field
                    // (units of 16 bytes): +32 B inside a K-major row, +2048 B (16 rows) in an MN-major tile
                    const uint64_t ad0 = (kc + 1 < p.k_chunks ? a_desc0 : t_desc0) | desc_addr(a_src);
                    const uint64_t bd0 = b_desc0 | desc_addr(b_src);
                    if (kc + 1 < p.k_chunks || last_steps == 4) {
                        umma_bf16_lead(d_tmem, ad0, bd0, idesc, acc, leader);
#pragma unroll
                        for (int k = 1; k < 4; ++k) umma_bf16_lead(d_tmem, ad0 + 2ull * k, bd0 + bstep * k, idesc, 1u, leader);
                    } else {
                        for (int k = 0; k < last_steps; ++k) umma_bf16_lead(d_tmem, ad0 + 2ull * k, bd0 + bstep * k, idesc, k ? 1u : acc, leader);
                    }
                    acc = 1u;
                    umma_commit_lead(smem_u32(&ctl->empty[sbase + s]), leader);   // frees the stage when these MMAs have read it
                    if (warp == 1) GTRACE(5, consumed);
                    ++consumed;
                    if (++s == SR) { s = 0; ph ^= 1; }
                }
            }
            if (ok) umma_commit_lead(smem_u32(&ctl->acc_full[b]), leader);   // this tile's accumulator is complete
            if (NI == 1 && ++b == p.epi_groups) { b = 0; aph ^= 1; }
            if (warp == 1) CTRACE(5);
        }
    } else if (warp - 2 < 4 * p.epi_groups) {
        // ---------------- epilogue: warp w may touch TMEM lanes 32*(w%4) .. +31; group g drains accumulator buffer g,
        // i.e. the tiles tc = g, g + G, g + 2G, ... of this CTA
        const int quarter = warp & 3, group = (warp - 2) >> 2, G = p.epi_groups;
        const uint32_t slab0 = (p.alias_staging ? data_base : staging_base) + (uint32_t)(warp - 2) * (kSlabs * 4096u);
        // statistics: accumulated over the warp's tiles in shared memory, combined at the end
        const uint32_t st_acc = smem_base + (uint32_t)p.stats_off + (uint32_t)(warp - 2) * (uint32_t)p.stats_warp;
        if (STATS && p.stats) {
            stats_clear(st_acc, lane, (p.BN + 63) / 64);
            __syncwarp();
        }
        int tc = group, sl = 0;
        bool ok = true;
        for (int tile = blockIdx.x + group * gridDim.x; tile < total_tiles && ok; tile += G * gridDim.x, tc += G) {
            int b = group, aph = (tc / G) & 1;
            if (p.n_issuers == 2) {                     // G == 2: group g serves issuer g, whose nt-th tile this is
                const int nt = tc >> 1;
                b = p.acc_per == 2 ? group * 2 + (nt & 1) : group;
                aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1;
            }
            const int n_tile = tile % p.n_tiles, m_tile = tile / p.n_tiles;
            const int m0 = m_tile * kBM, n0 = n_tile * p.BN;
            // direct stores: this thread's raster pixel and where it lands in the output view
            const int m = m0 + quarter * 32 + lane;
            const bool row_ok = !p.tma_store && m < p.M_total;
            int pix = 0;
            if (row_ok) {
                const int j = m % p.Qd, t = m / p.Qd, i = t % p.Pd, img = t / p.Pd;
                pix = (img * p.oH + i * p.o_step + p.o_h0) * p.oW + j * p.o_step + p.o_w0;
            }
            ok = mbar_wait(smem_u32(&ctl->acc_full[b]), aph, abort_flag, p.status, 3);
            if (!ok) break;
            if (quarter == 0) GTRACE(6, tc);
            tc_fence_after();
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * p.BN);
            if (!APART && p.tma_store) {
                // Each warp stages its 32 rows x 64 channels (4 KB, 128-byte swizzle) and stores it with one TMA store,
                // which drops the channels past the true count and the rows past the last pixel. Two slabs alternate.
                const int n_chunks = (p.BN + 63) / 64;
                for (int ch = 0; ch < n_chunks; ++ch, sl ^= 1) {
                    const uint32_t slab = slab0 + (uint32_t)sl * 4096u;
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the slab's previous store has read it
                    __syncwarp();
                    const int groups = min(4, (p.BN - ch * 64) / 16);
                    uint32_t v[4][16];
                    // all of the chunk's TMEM loads are issued before the single wait
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (g < groups) tmem_ld16(lane_addr + (uint32_t)(ch * 64 + g * 16), v[g]);
                    tmem_ld_wait();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g >= groups) break;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            __nv_bfloat162 b0 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 0]), __uint_as_float(v[g][8 * h + 1]));
                            __nv_bfloat162 b1 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 2]), __uint_as_float(v[g][8 * h + 3]));
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 4]), __uint_as_float(v[g][8 * h + 5]));
                            __nv_bfloat162 b3 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 6]), __uint_as_float(v[g][8 * h + 7]));
                            const uint32_t j = (uint32_t)(g * 2 + h);
                            const uint32_t addr = slab + (uint32_t)lane * 128u + ((j ^ ((uint32_t)lane & 7u)) << 4);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(*reinterpret_cast<uint32_t *>(&b0)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b1)), "r"(*reinterpret_cast<uint32_t *>(&b2)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b3))
                                         : "memory");
                        }
                    }
                    if (ch + 1 >= n_chunks) {
                        // every TMEM read of this tile by this warp is done: hand the buffer back to the MMA issuer
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        if (m0 + quarter * 32 < p.M_total) tma_store_2d(&tmC, slab, n0 + ch * 64, m0 + quarter * 32);
                        tma_store_commit();
                    }
                    if (STATS && p.stats) {
                        const int left = p.M_total - (m0 + quarter * 32);
                        const uint32_t rows = left >= 32 ? 0xffffffffu : (left > 0 ? (1u << left) - 1u : 0u);
                        chunk_stats(slab, 0, rows, lane, st_acc + (uint32_t)ch * 512u);
                    }
                }
                if (quarter == 0) GTRACE(7, tc);
                continue;
            }
            if (APART) {
                // ---- strided stride-2 data-gradient outputs: through the warp's staging
                const uint32_t rows = __ballot_sync(0xffffffffu, row_ok);
                for (int c0 = 0; c0 < p.BN; c0 += 64) {
                    const int groups = min(4, (p.BN - c0) / 16);
                    uint32_t v[4][16];
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (g < groups) tmem_ld16(lane_addr + (uint32_t)(c0 + g * 16), v[g]);
                    tmem_ld_wait();
                    if (c0 + 64 >= p.BN) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                    }
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g >= groups) break;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            __nv_bfloat162 b0 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 0]), __uint_as_float(v[g][8 * h + 1]));
                            __nv_bfloat162 b1 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 2]), __uint_as_float(v[g][8 * h + 3]));
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 4]), __uint_as_float(v[g][8 * h + 5]));
                            __nv_bfloat162 b3 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 6]), __uint_as_float(v[g][8 * h + 7]));
                            const uint32_t j = (uint32_t)(g * 2 + h);
                            const uint32_t addr = slab0 + (uint32_t)lane * 128u + ((j ^ ((uint32_t)lane & 7u)) << 4);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(*reinterpret_cast<uint32_t *>(&b0)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b1)), "r"(*reinterpret_cast<uint32_t *>(&b2)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b3))
                                         : "memory");
                        }
                    }
                    __syncwarp();
                    store_rows_apart((__nv_bfloat16 *)p.out, p.ld_out, slab0, n0 + c0, min(groups * 2, (p.vec_cols - n0 - c0) >> 3), rows, pix, lane);
                    __syncwarp();
                }
                continue;
            }
            // ---- direct stores (fp32 outputs)
            for (int c0 = 0; c0 < p.BN; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(lane_addr + (uint32_t)c0, v);
                tmem_ld_wait();
                if (c0 + 16 >= p.BN) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                }
                const int col = n0 + c0;
                if (!row_ok || col >= p.n_cols) continue;
                const int nvalid = min(16, p.n_cols - col);
                float *o = (float *)p.out + (size_t)pix * (size_t)p.ld_out + col;
                if (nvalid == 16) {
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        reinterpret_cast<float4 *>(o)[g] = make_float4(__uint_as_float(v[4 * g]), __uint_as_float(v[4 * g + 1]),
                                                                      __uint_as_float(v[4 * g + 2]), __uint_as_float(v[4 * g + 3]));
                } else {
                    for (int e = 0; e < nvalid; ++e) o[e] = __uint_as_float(v[e]);
                }
            }
        }
        if (STATS && p.stats) {
            named_barrier(1, 128 * G);
            const int nt = (int)blockIdx.x % p.n_tiles;
            stats_store_cta(smem_base + (uint32_t)p.stats_off, (uint32_t)p.stats_warp, 4 * G, (int)threadIdx.x - 64, 128 * G,
                            p.stats + (size_t)(blockIdx.x / p.n_tiles) * (1 + p.stats_lo) * 2 * p.ld_out, p.ld_out, p.stats_lo, p.n_cols, nt * p.BN,
                            nt + 1 < p.n_tiles ? (nt + 1) * p.BN : p.ld_out);
        }
        if (p.tma_store && lane == 0) tma_store_wait_read();     // the staging slabs must outlive the stores' reads
        if (warp == 2) CTRACE(6);
        tc_fence_before();
    } else if (B_MN && p.zero_mask && warp < 14) {
        // ---------------- stride-2 data gradient: the pixels of each 2x2 cell that no tap reaches are zeros. They depend on no
        // accumulator: the warps past the epilogue groups (four or eight) write them, each for 32 of a tile's raster pixels and the
        // tile's columns, a row's whole 16-byte vectors on consecutive lanes. (Clearing dx in a pass of its own cost 25 of 70 us for
        // 77 <- 154 channels at 56x56, batch 256; one column tile writing the zeros of all 20 of 38 us for 418 <- 931 at 28x28.)
        const int z = warp - 2 - 4 * p.epi_groups, quarter = z & 3, nz = 3 - p.epi_groups;
        const size_t off1 = (size_t)p.ld_out, off2 = (size_t)p.oW * p.ld_out;
        for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
            const int n_tile = tile % p.n_tiles, m = tile / p.n_tiles * kBM + quarter * 32 + lane;
            const int n0 = n_tile * p.BN;
            int cell = 0, mask = 0;                 // the cell's first pixel, the parities to clear
            if (m < p.M_total) {
                const int j = m % p.Qd, t = m / p.Qd, i = t % p.Pd;
                cell = ((t / p.Pd) * p.oH + 2 * i) * p.oW + 2 * j;
                mask = p.zero_mask & (2 * i + 1 < p.oH ? 0xf : 0x3) & (2 * j + 1 < p.oW ? 0xf : 0x5);
            }
            const int np = p.out_f32 ? min(p.BN, p.n_cols - n0) : min(p.BN, p.vec_cols - n0) >> 3;      // floats or vectors per pixel
            const float inv_np = 1.0f / (float)np;
            for (int k = z >> 2; k < np; k += nz) {
                const int idx = k * 32 + lane, r = fast_div(idx, np, inv_np), e = idx - r * np;
                const size_t off = (size_t)__shfl_sync(0xffffffffu, cell, r) * (size_t)p.ld_out + (size_t)(n0 + (p.out_f32 ? e : e * 8));
                const int mk = __shfl_sync(0xffffffffu, mask, r);
                if (!APART) {
                    float *o = (float *)p.out + off;
                    if (mk & 1) o[0] = 0.f;
                    if (mk & 2) o[off1] = 0.f;
                    if (mk & 4) o[off2] = 0.f;
                    if (mk & 8) o[off2 + off1] = 0.f;
                } else {
                    __nv_bfloat16 *o = (__nv_bfloat16 *)p.out + off;
                    const uint4 zero = make_uint4(0, 0, 0, 0);
                    if (mk & 1) *reinterpret_cast<uint4 *>(o) = zero;
                    if (mk & 2) *reinterpret_cast<uint4 *>(o + off1) = zero;
                    if (mk & 4) *reinterpret_cast<uint4 *>(o + off2) = zero;
                    if (mk & 8) *reinterpret_cast<uint4 *>(o + off2 + off1) = zero;
                }
            }
        }
    }
    __syncthreads();
    if (warp == 0) CTRACE(7);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------ halo kernel (RxS, stride 1)
// For a stride-1 RxS filter the per-tap im2col loads fetch every input pixel R*S times. Here each input pixel row is
// fetched ONCE per 64-channel chunk: a tile is `nr` output rows of one image, laid out as a raster of pitch
// Wp = Q + S - 1 (the S - 1 extra columns per row are garbage outputs that are never stored). One tiled 4-D TMA load
// brings the (nr + R - 1) x Wp input positions of the tile, halo included, zero-filled outside the image. In that
// raster the input position of output position m for tap (r, s) is m + r*Wp + s, a constant row shift, and the
// 128-byte swizzle is a function of the absolute shared-memory address, so tap (r, s) is simply the same A tile read
// through a descriptor whose start address is (r*Wp + s) rows further on. Weights: if all taps x chunks of the CTA's
// channel tile fit in shared memory they are loaded once and stay resident; otherwise they stream through a ring.
struct HaloP {
    int N, P, Q, Wp, nr, row_tiles;      // images, output rows/cols, raster pitch, output rows per tile, tiles per image
    int n_cols, BN, n_tiles;
    int c_red, k_chunks, taps;
    int lo_h, lo_w;                      // source coordinate of raster position (0, 0) for tap offset (0, 0)
    int a_box_bytes, a_alloc;            // bytes one A load brings / bytes reserved per A stage
    int stages_a, stages_b, resident;    // ring depths; resident: weights loaded once
    int n_issuers, acc_per;              // MMA issuer warps (each with its own A ring of stages_a / n_issuers stages); accumulators per issuer (1 or 2)
    int shared_b;                        // two pipelines fed by ONE weight stream: a stage is read by both issuers (their tiles of a round)
    int lanes;                           // channel lanes per staged pixel: 64, 32 or 16 (128-, 64- or 32-byte rows and swizzle)
    int direct;                          // 1: at most 32 output channels, stored from registers (no staging)
    int b_slot, b_rows, staging, slabs;  // bytes reserved per weight tile, rows a K-major weight box brings, bytes and number of an epilogue group's staging slabs
    int direct_cols;                     // channels the direct stores cover (whole 16-byte vectors)
    int tmem_cols, tma_store, out_f32, ld_out;
    int oH, oW, o_step, o_h0, o_w0;      // direct stores: raster (n, i, j) -> out[((n*oH + i*o_step + o_h0)*oW + j*o_step + o_w0)*ld_out]
    int stats_off;                       // byte offset in shared memory of the epilogue warps' statistics accumulators
    int stats_warp;                      // bytes of one warp's accumulators: 512 per 64-channel chunk of the tile
    int stats_lo;                        // 1: two rows of sums per row of CTAs
    int test_skip;                       // test hook (pt_test_skip_next_arrive): the activation producers leave out their first box
    float *stats;                        // optional: rows [2][ld_out], one per n_tiles CTAs: sums and sums of squares of the stored bf16
    void *out;
    unsigned int *status;
    unsigned char tap_oh[kMaxTaps], tap_ow[kMaxTaps];
    unsigned short tap_wt[kMaxTaps];
};

constexpr int kHaloMaxIssuers = 4;
constexpr int kHaloMaxA = 8;             // activation stages: two per issuer (three measured the same or 2 us slower)

// Coordinates of the tiles t0, t0 + D, t0 + 2D, ... of a halo launch, advanced without integer divisions (a division costs
// a single issuing thread ~150 cycles, and the smallest tiles are only a few hundred cycles of work).
struct TileWalk {
    int n_tile, rt, img;          // channel tile, row tile within the image, image
    int dn, d_rt, d_img, n_tiles, row_tiles;
    __device__ __forceinline__ void init(int tile, int D, int n_tiles_, int row_tiles_)
    {
        n_tiles = n_tiles_; row_tiles = row_tiles_;
        n_tile = tile % n_tiles;
        const int m_tile = tile / n_tiles;
        img = m_tile / row_tiles; rt = m_tile - img * row_tiles;
        dn = D % n_tiles;
        const int dm = D / n_tiles;
        d_img = dm / row_tiles; d_rt = dm - d_img * row_tiles;
    }
    __device__ __forceinline__ void next()
    {
        n_tile += dn;
        rt += d_rt; img += d_img;
        if (n_tile >= n_tiles) { n_tile -= n_tiles; ++rt; }
        while (rt >= row_tiles) { rt -= row_tiles; ++img; }
    }
};
// Device-side timeline for tuning: a build with -DPT_DEVICE_TRACE makes CTA 0 stamp %globaltimer at the hand-over points of
// each role (producer issue, accumulator free, operands landed, MMAs committed, epilogue start, store issued) and exports
// pt_debug_halo_trace / pt_debug_wgrad_trace / pt_debug_gemm_trace to read the stamps back. The normal build compiles the macros away.
#ifdef PT_DEVICE_TRACE
__device__ unsigned long long g_halo_trace[8][64];
#define HTRACE(role, idx) do { if (blockIdx.x == 0 && (idx) < 64 && (threadIdx.x & 31) == 0) g_halo_trace[role][idx] = globaltimer_ns(); } while (0)
#else
#define HTRACE(role, idx) do { } while (0)
#endif

struct __align__(8) HCtl {
    uint64_t full_a[kHaloMaxA], empty_a[kHaloMaxA];
    uint64_t full_b[kMaxStages], empty_b[kMaxStages];
    uint64_t w_full;
    uint64_t acc_full[2 * kHaloMaxIssuers], acc_empty[2 * kHaloMaxIssuers];
    uint32_t tap_aoff[kMaxTaps];         // row shift of each tap in descriptor units (16 bytes)
    uint32_t tmem_base;
    int abort_flag;
};

// warp 0 (and 13): TMA producers (weights; with resident weights warp 0 also brings the activations); warps 14, 15: activation
// producers of the streamed-weight pipelines; warp 1 and warps 10..12: MMA issuers; warps 2..9: two groups of four epilogue warps
constexpr int kHaloThreads = 512;

// Issuing one tcgen05.mma costs the issuing warp 50 to 100 cycles of instruction time, more than a narrow MMA (N <= 64)
// takes to execute, so with a single issuer the tensor pipe of a small-channel layer idles most of the time. The
// kernel therefore runs up to four issuer warps, each on its own scheduler: issuer i owns accumulator buffer i and
// an A ring of its own (a waiter may lag an mbarrier by at most one phase, so issuers cannot share a ring), and takes
// the tiles i, i + I, i + 2I, ... of the CTA. Weights that stream through a ring keep a single issuer.
//   PL = 4: the forward pass at stride 2. The source pixels of either row and column parity are a plane (every other pixel: a tensor map of its
// own) in which the taps that read it are shifts of one pixel as at stride 1, so that every chunk of 64 channels is four boxes, each with its
// own taps, all into one accumulator. The im2col form loads a tile's 128 pixels once per tap (2304 rows a tile of 106 channels and nine taps
// against 1160). At PL = 1 the loops' bounds are read from the parameters as they stand: held in variables they cost the streamed layers 1 %
// (28x28, 106 -> 103, batch 64 19.1 and 19.35 us).
template <int PL> struct HaloMaps {
    CUtensorMap m[PL];
    int tap[PL + 1];           // the taps of plane i are tap[i] .. tap[i + 1] - 1
    int lo_h[PL], lo_w[PL];    // source coordinate of raster position (0, 0) in it
};
template <> struct HaloMaps<1> { CUtensorMap m[1]; };

template <bool B_MN, bool STATS, int PL>
__global__ void __launch_bounds__(kHaloThreads, 1) conv_halo_kernel(const __grid_constant__ HaloMaps<PL> tmA,
                                                                     const __grid_constant__ CUtensorMap tmB,
                                                                     const __grid_constant__ CUtensorMap tmC, const HaloP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    HCtl *ctl = reinterpret_cast<HCtl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t staging_base = (smem_base + (uint32_t)sizeof(HCtl) + 1023u) & ~1023u;
    const uint32_t b_base = staging_base + 2u * (uint32_t)(p.slabs * p.staging);
    // bytes one weight tile brings: a K-major tile only holds the rows (output channels) that exist
    const uint32_t row_bytes = (uint32_t)p.lanes * 2u, b_block = (uint32_t)p.lanes * 128u;   // (an MN-major block: 64 columns x `lanes` rows)
    const uint32_t b_bytes = B_MN ? (uint32_t)((p.BN + 63) / 64) * b_block : (uint32_t)p.b_rows * row_bytes;
    const uint32_t b_slot = (uint32_t)p.b_slot;
    const uint32_t n_bslots = p.resident ? (uint32_t)(p.taps * p.k_chunks) : (uint32_t)p.stages_b;
    const uint32_t a_base = b_base + n_bslots * b_slot;
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m_tiles = p.N * p.row_tiles;
    const int total_tiles = m_tiles * p.n_tiles;
    const int NI = p.n_issuers, SR = p.stages_a / NI;        // issuers, A stages per issuer ring
    const int boxes = p.k_chunks * PL;                       // activation boxes of a tile: chunk by chunk, every plane of it

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages_a; ++s) { mbar_init(smem_u32(&ctl->full_a[s]), 1); mbar_init(smem_u32(&ctl->empty_a[s]), 1); }
        for (int s = 0; s < p.stages_b; ++s) { mbar_init(smem_u32(&ctl->full_b[s]), 1); mbar_init(smem_u32(&ctl->empty_b[s]), p.shared_b ? 2 : 1); }
        mbar_init(smem_u32(&ctl->w_full), 1);
        for (int b = 0; b < 2 * kHaloMaxIssuers; ++b) { mbar_init(smem_u32(&ctl->acc_full[b]), 1); mbar_init(smem_u32(&ctl->acc_empty[b]), 4); }
        ctl->abort_flag = 0;
        fence_mbar_init();
#pragma unroll
        for (int i = 0; i < PL; ++i) prefetch_tmap(&tmA.m[i]);
        prefetch_tmap(&tmB);
        if (p.tma_store) prefetch_tmap(&tmC);
    }
    if (threadIdx.x < p.taps) ctl->tap_aoff[threadIdx.x] = (uint32_t)(p.tap_oh[threadIdx.x] * p.Wp + p.tap_ow[threadIdx.x]) * (row_bytes >> 4);
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int issuer = warp == 1 ? 0 : warp - 9;             // warps 10, 11, 12 -> issuers 1, 2, 3
    // the weight producers do not read the previous kernel's output: resident weights are issued first and the wait follows
    // them (below); the producers of streamed weights never need it
    // Warps that load activations wait just before their first activation load, after their set-up (tile walk, ring positions).
    if (!(warp == 0 || warp >= 13)) grid_dependency_wait();
    grid_launch_dependents();

    // Streamed weights with two issuers: two complete pipelines (producer warp, A ring, B ring, issuer warp, accumulators),
    // one per tile parity. Resident weights: every issuer's A ring has a producer warp of its own (a thread issues a box only every
    // 0.5 us, whatever it holds: one producer for four issuers made that the time of a tile), and they share the weights' loads.
    // With `shared_b` the two pipelines read the same weight stages: the tiles of a round (blockIdx.x + 2r*grid and + (2r+1)*grid)
    // use the same weights, so one stream through the whole ring feeds both issuers, half the bytes and twice the depth.
    const int n_prod = NI;
    const int SB = p.shared_b ? p.stages_b : p.stages_b / n_prod;     // weight stages per weight stream
    // Streamed weights: the activation boxes have a producer warp of their own per pipeline (14, 15), so that the next tile's
    // boxes go out as soon as their stage is free instead of behind the weight loads of the current tile, which wait for the
    // MMAs (the next tile's activations used to be issued only when the current tile was nearly done: ~4 us per tile exposed).
    const bool a_warp = !p.resident && (warp == 14 || (warp == 15 && n_prod == 2));
    if (warp == 0 || (p.resident ? warp >= 13 && warp - 12 < NI : (warp == 13 && n_prod == 2 && !p.shared_b) || a_warp)) {
        if (lane == 0) {
            // ---------------- TMA producer(s)
            const int pid = p.resident ? (warp == 0 ? 0 : warp - 12) : (warp == 0 || warp == 14) ? 0 : 1;
            const bool a_role = a_warp || p.resident, b_role = !a_warp && !p.resident;
            if (p.resident) {
                // n_tiles == 1 here: the whole weight tensor of the layer, tap by tap and chunk by chunk, once
                const uint32_t bar = smem_u32(&ctl->w_full);
                if (pid == 0) mbar_arrive_expect_tx(bar, (uint32_t)(p.taps * p.k_chunks) * b_bytes);
                for (int tap = pid; tap < p.taps; tap += n_prod)
                    for (int kc = 0; kc < p.k_chunks; ++kc) {
                        const uint32_t dst = b_base + (uint32_t)(tap * p.k_chunks + kc) * b_slot;
                        const int wtap = p.tap_wt[tap];
                        if (!B_MN) tma_load_3d(dst, &tmB, bar, kc * kKC, wtap, 0);
                        else for (int nb = 0; nb < (p.BN + 63) / 64; ++nb) tma_load_3d(dst + (uint32_t)nb * b_block, &tmB, bar, nb * 64, wtap, kc * kKC);
                    }
            }
            bool dep_waited = false;             // the activations are the previous kernel's output
            int tc = pid;
            TileWalk tw;
            tw.init((int)blockIdx.x + pid * (int)gridDim.x, n_prod * (int)gridDim.x, p.n_tiles, p.row_tiles);
            // ring = tc % NI; every ring has carried (tc / NI) * boxes boxes before its tile of this round: position and
            // phase of that count in a ring of SR stages, advanced per round
            int ring = pid % NI, base_pos = 0, base_ph = 0;
            const int kdiv = boxes / SR, kmod = boxes - kdiv * SR;
            int sb_pos = 0, sb_ph = 0;                         // position in this pipeline's weight ring
            const int skip_a = p.test_skip;
            int issued_a = 0, issued_b = 0;                    // stages filled (a producer of activations feeds one ring)
            for (int tile = blockIdx.x + pid * (int)gridDim.x; tile < total_tiles && !*abort_flag; tile += n_prod * (int)gridDim.x, tc += n_prod) {
                const int img = tw.img, p0 = tw.rt * p.nr;
                const int n0 = tw.n_tile * p.BN;
                bool ok = true;
                int pos = base_pos, pha = base_ph;
                for (int bx = 0; bx < p.k_chunks * PL && ok; ++bx) {
                    const int kc = bx / PL, pl = bx % PL;
                    [[maybe_unused]] int tap0 = 0, tap1 = 0, lo_h = p.lo_h, lo_w = p.lo_w;
                    if constexpr (PL > 1) { tap0 = tmA.tap[pl]; tap1 = tmA.tap[pl + 1]; lo_h = tmA.lo_h[pl]; lo_w = tmA.lo_w[pl]; }
                    const int sa = ring * SR + pos, ph_use = pha;
                    if (++pos == SR) { pos = 0; pha ^= 1; }
                    if (a_role) {
                        ok = mbar_wait(smem_u32(&ctl->empty_a[sa]), ph_use ^ 1, abort_flag, p.status, 11);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&ctl->full_a[sa]);
                        HTRACE(0, tc);
                        mbar_arrive_expect_tx(bar, (uint32_t)p.a_box_bytes);
                        if (!dep_waited) { grid_dependency_wait(); dep_waited = true; }
                        if (issued_a >= skip_a)                // (test hook: the first stage never becomes full)
                            tma_load_4d(a_base + (uint32_t)sa * (uint32_t)p.a_alloc, &tmA.m[pl], bar, kc * kKC, lo_w, p0 + lo_h, img);
                        ++issued_a;
                    }
                    if (!b_role) continue;
                    for (int tap = PL > 1 ? tap0 : 0; tap < (PL > 1 ? tap1 : p.taps); ++tap) {
                        const int sb = (p.shared_b ? 0 : pid * SB) + sb_pos, phb = sb_ph;
                        if (++sb_pos == SB) { sb_pos = 0; sb_ph ^= 1; }
                        ok = mbar_wait(smem_u32(&ctl->empty_b[sb]), phb ^ 1, abort_flag, p.status, 12);
                        if (!ok) break;
                        const uint32_t bbar = smem_u32(&ctl->full_b[sb]);
                        const uint32_t dst = b_base + (uint32_t)sb * b_slot;
                        const int wtap = p.tap_wt[tap];
                        mbar_arrive_expect_tx(bbar, b_bytes);
                        ++issued_b;
                        if (!B_MN) tma_load_3d(dst, &tmB, bbar, kc * kKC, wtap, n0);
                        else for (int nb = 0; nb < (p.BN + 63) / 64; ++nb) tma_load_3d(dst + (uint32_t)nb * b_block, &tmB, bbar, n0 + nb * 64, wtap, kc * kKC);
                    }
                }
                if (!ok) break;
                tw.next();
                ring += n_prod;
                while (ring >= NI) {                           // next round: every ring has carried `boxes` more
                    ring -= NI;
                    base_pos += kmod;
                    int wraps = kdiv;
                    if (base_pos >= SR) { base_pos -= SR; ++wraps; }
                    base_ph ^= wraps & 1;
                }
            }
            if (*abort_flag) {       // the copies this thread issued
                if (p.resident) drain_ring(smem_u32(&ctl->w_full), 1, 1);
                drain_ring(smem_u32(&ctl->full_a[pid * SR]), SR, issued_a);
                drain_ring(smem_u32(&ctl->full_b[p.shared_b ? 0 : pid * SB]), SB, issued_b);
            }
        }
    } else if (warp == 1 || (warp >= 10 && issuer < NI)) {
        // ---------------- MMA issuer `issuer`: the whole warp walks the loops in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(kBM, p.BN, 0, B_MN ? 1 : 0);
        const uint64_t a_desc0 = make_desc_rows(0u, row_bytes), b_desc0 = B_MN ? make_desc(0u, b_block, 1024u) : make_desc_rows(0u, row_bytes);
        const uint64_t bstep = B_MN ? 128ull : 2ull;
        int sb_pos = 0, sb_ph = 0;                            // position in this issuer's weight ring
        int s_loc = 0, pha = 0;                               // position in this issuer's A ring
        bool ok = true;
        if (p.resident) ok = mbar_wait(smem_u32(&ctl->w_full), 0, abort_flag, p.status, 13);
        int nt = 0;                                           // tiles this issuer has started
        for (int tc = issuer; ok; tc += NI, ++nt) {
            const int tile = blockIdx.x + tc * (int)gridDim.x;
            if (tile >= total_tiles) {
                // shared weight stream: the other issuer may still have a tile in this round; its stages need this issuer's
                // release too, given in step with the stream
                if (p.shared_b && issuer == 1 && tile - (int)gridDim.x < total_tiles) {
                    for (int i = 0; i < p.k_chunks * p.taps && ok; ++i) {
                        const int sb = sb_pos, phb = sb_ph;
                        if (++sb_pos == SB) { sb_pos = 0; sb_ph ^= 1; }
                        ok = mbar_wait(smem_u32(&ctl->full_b[sb]), phb, abort_flag, p.status, 16);
                        if (ok && lane == 0) mbar_arrive(smem_u32(&ctl->empty_b[sb]));
                    }
                }
                break;
            }
            // accumulator buffers issuer*acc_per .. +acc_per-1, used in turn
            const int b = p.acc_per == 2 ? issuer * 2 + (nt & 1) : issuer, aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1;
            ok = mbar_wait(smem_u32(&ctl->acc_empty[b]), aph ^ 1, abort_flag, p.status, 14);
            if (!ok) break;
            HTRACE(1, tc);
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(b * p.BN);
            uint32_t accumulate = 0u;
            for (int bx = 0; bx < p.k_chunks * PL && ok; ++bx) {
                const int kc = bx / PL;
                [[maybe_unused]] int t0 = 0, t1 = 0;
                if constexpr (PL > 1) { t0 = tmA.tap[bx % PL]; t1 = tmA.tap[bx % PL + 1]; }
                const int sa = issuer * SR + s_loc;
                ok = mbar_wait(smem_u32(&ctl->full_a[sa]), pha, abort_flag, p.status, 15);
                if (!ok) break;
                HTRACE(2, tc);
                tc_fence_after();
                const int rem = p.c_red - kc * kKC;
                const int ksteps = rem >= kKC ? 4 : (rem + 15) / 16;
                const uint64_t abase = a_desc0 | desc_addr(a_base + (uint32_t)sa * (uint32_t)p.a_alloc);
                if (p.resident) {
                    // every tap is the same A tile read through a descriptor that starts (r*Wp + s) rows further on
                    uint64_t bd0 = b_desc0 | desc_addr(b_base + (uint32_t)(t0 * p.k_chunks + kc) * b_slot);
                    const uint64_t b_tap_step = (uint64_t)(((uint32_t)p.k_chunks * b_slot) >> 4);
                    if (ksteps == 1) {
                        for (int tap = PL > 1 ? t0 : 0; tap < (PL > 1 ? t1 : p.taps); ++tap, bd0 += b_tap_step) {
                            umma_bf16_lead(d_tmem, abase + ctl->tap_aoff[tap], bd0, idesc, accumulate, leader);
                            accumulate = 1u;
                        }
                    } else if (ksteps == 4) {
                        for (int tap = PL > 1 ? t0 : 0; tap < (PL > 1 ? t1 : p.taps); ++tap, bd0 += b_tap_step) {
                            const uint64_t ad0 = abase + ctl->tap_aoff[tap];
#pragma unroll
                            for (int k = 0; k < 4; ++k) { umma_bf16_lead(d_tmem, ad0 + 2ull * k, bd0 + bstep * k, idesc, accumulate, leader); accumulate = 1u; }
                        }
                    } else {
                        for (int tap = PL > 1 ? t0 : 0; tap < (PL > 1 ? t1 : p.taps); ++tap, bd0 += b_tap_step) {
                            const uint64_t ad0 = abase + ctl->tap_aoff[tap];
                            for (int k = 0; k < ksteps; ++k) { umma_bf16_lead(d_tmem, ad0 + 2ull * k, bd0 + bstep * k, idesc, accumulate, leader); accumulate = 1u; }
                        }
                    }
                } else {
                    for (int tap = PL > 1 ? t0 : 0; tap < (PL > 1 ? t1 : p.taps); ++tap) {
                        const int sb = (p.shared_b ? 0 : issuer * SB) + sb_pos, phb = sb_ph;
                        if (++sb_pos == SB) { sb_pos = 0; sb_ph ^= 1; }
                        ok = mbar_wait(smem_u32(&ctl->full_b[sb]), phb, abort_flag, p.status, 16);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t ad0 = abase + ctl->tap_aoff[tap];
                        const uint64_t bd0 = b_desc0 | desc_addr(b_base + (uint32_t)sb * b_slot);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (k < ksteps) { umma_bf16_lead(d_tmem, ad0 + 2ull * k, bd0 + bstep * k, idesc, accumulate, leader); accumulate = 1u; }
                        umma_commit_lead(smem_u32(&ctl->empty_b[sb]), leader);
                    }
                }
                if (ok) umma_commit_lead(smem_u32(&ctl->empty_a[sa]), leader);
                if (++s_loc == SR) { s_loc = 0; pha ^= 1; }
            }
            if (ok) umma_commit_lead(smem_u32(&ctl->acc_full[b]), leader);
            HTRACE(3, tc);
        }
    } else if (warp >= 2 && warp < 10) {
        // ---------------- epilogue: group g (four warps) drains the accumulator buffers of its parity
        const int quarter = warp & 3, group = (warp - 2) >> 2;
        const int gtid = (warp - 2 - group * 4) * 32 + lane;         // 0..127 within the group
        // this thread's raster position: its output row within the tile and its column
        const int m = quarter * 32 + lane, ri = m / p.Wp, rj = m - ri * p.Wp;
        const bool on_raster = m < p.nr * p.Wp && rj < p.Q;
        uint32_t slab = staging_base + (uint32_t)(group * p.slabs) * (uint32_t)p.staging;
        int sl = 0;
        // statistics: accumulated over the warp's tiles in shared memory, combined at the end
        const uint32_t st_acc = smem_base + (uint32_t)p.stats_off + (uint32_t)(warp - 2) * (uint32_t)p.stats_warp;
        if (STATS && p.stats) {
            stats_clear(st_acc, lane, (p.BN + 63) / 64);
            __syncwarp();
        }
        bool ok = true;
        const int ni_shift = NI == 4 ? 2 : NI == 2 ? 1 : 0;   // NI is 1, 2 or 4
        TileWalk tw;
        tw.init((int)blockIdx.x + group * (int)gridDim.x, 2 * (int)gridDim.x, p.n_tiles, p.row_tiles);
        for (int tc = group; ok; tc += 2, tw.next()) {
            const int tile = blockIdx.x + tc * (int)gridDim.x;
            if (tile >= total_tiles) break;
            // tile tc is the nt-th tile of issuer tc % NI (NI is 1 or even, so a group always serves the same issuers)
            const int iss = tc & (NI - 1), nt = tc >> ni_shift;
            const int b = p.acc_per == 2 ? iss * 2 + (nt & 1) : iss, aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1;
            const int img = tw.img, p0 = tw.rt * p.nr;
            const int n0 = tw.n_tile * p.BN;
            ok = mbar_wait(smem_u32(&ctl->acc_full[b]), aph, abort_flag, p.status, 17);
            if (!ok) break;
            if (gtid == 0) HTRACE(4, tc);
            tc_fence_after();
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * p.BN);
            if (p.tma_store) {
                const int n_chunks = (p.BN + 63) / 64;
                for (int ch = 0; ch < n_chunks; ++ch) {
                    if (gtid == 0) {                                 // the slab's previous store has read it
                        if (p.slabs == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        else tma_store_wait_read();
                    }
                    if (gtid == 0) HTRACE(5, tc);
                    named_barrier(1 + group, 128);
                    const int groups = min(4, (p.BN - ch * 64) / 16);
                    uint32_t v[4][16];
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (g < groups) tmem_ld16(lane_addr + (uint32_t)(ch * 64 + g * 16), v[g]);
                    tmem_ld_wait();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g >= groups || m >= p.nr * p.Wp) break;   // the slab only holds the tile's raster rows
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            __nv_bfloat162 b0 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 0]), __uint_as_float(v[g][8 * h + 1]));
                            __nv_bfloat162 b1 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 2]), __uint_as_float(v[g][8 * h + 3]));
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 4]), __uint_as_float(v[g][8 * h + 5]));
                            __nv_bfloat162 b3 = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 6]), __uint_as_float(v[g][8 * h + 7]));
                            const uint32_t j = (uint32_t)(g * 2 + h);
                            const uint32_t addr = slab + (uint32_t)m * 128u + ((j ^ ((uint32_t)m & 7u)) << 4);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(*reinterpret_cast<uint32_t *>(&b0)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b1)), "r"(*reinterpret_cast<uint32_t *>(&b2)),
                                         "r"(*reinterpret_cast<uint32_t *>(&b3))
                                         : "memory");
                        }
                    }
                    if (ch + 1 >= n_chunks) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                    }
                    fence_proxy_async();
                    named_barrier(1 + group, 128);
                    // one store per tile and chunk: box = nr rows x Wp columns x 64 channels; the columns past Q, the rows
                    // past P and the channels past the true count fall outside the tensor and are dropped
                    if (gtid == 0) {
                        HTRACE(6, tc);
                        tma_store_4d(&tmC, slab, n0 + ch * 64, 0, p0, img);
                        tma_store_commit();
                        HTRACE(7, tc);
                    }
                    if (STATS && p.stats) {
                        // this thread's raster position is a real output pixel iff it lies inside the row and the image
                        const uint32_t rows = __ballot_sync(0xffffffffu, on_raster && p0 + ri < p.P);
                        chunk_stats(slab, quarter * 32, rows, lane, st_acc + (uint32_t)ch * 512u);
                    }
                    if (p.slabs == 2) { slab = sl ? slab - (uint32_t)p.staging : slab + (uint32_t)p.staging; sl ^= 1; }
                }
                continue;
            }
            // ---- direct stores (fp32 outputs, narrow bf16 outputs)
            const bool row_ok = on_raster && p0 + ri < p.P;
            const int pix = (img * p.oH + (p0 + ri) * p.o_step + p.o_h0) * p.oW + rj * p.o_step + p.o_w0;
            const size_t row_off = (size_t)pix * (size_t)p.ld_out;
            if (p.direct) {
                // a pixel's channels are 32 or 64 consecutive bytes: whole sectors from one thread, with no barrier among the warps and
                // no store to wait for before the next tile (whose staging made a tile cost 0.5 us however little it held)
                uint32_t v[2][16];
                tmem_ld16(lane_addr, v[0]);
                if (p.BN > 16) tmem_ld16(lane_addr + 16u, v[1]);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                if (!row_ok) continue;
                __nv_bfloat16 *o = (__nv_bfloat16 *)p.out + row_off;
#pragma unroll
                for (int q8 = 0; q8 < 4; ++q8) {
                    const uint32_t (&e)[16] = v[q8 >> 1];
                    const int h8 = (q8 & 1) * 8;
                    if (q8 * 8 >= p.direct_cols) continue;
                    __nv_bfloat162 b0 = __floats2bfloat162_rn(__uint_as_float(e[h8 + 0]), __uint_as_float(e[h8 + 1]));
                    __nv_bfloat162 b1 = __floats2bfloat162_rn(__uint_as_float(e[h8 + 2]), __uint_as_float(e[h8 + 3]));
                    __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(e[h8 + 4]), __uint_as_float(e[h8 + 5]));
                    __nv_bfloat162 b3 = __floats2bfloat162_rn(__uint_as_float(e[h8 + 6]), __uint_as_float(e[h8 + 7]));
                    *reinterpret_cast<uint4 *>(o + q8 * 8) = make_uint4(*reinterpret_cast<uint32_t *>(&b0), *reinterpret_cast<uint32_t *>(&b1),
                                                                        *reinterpret_cast<uint32_t *>(&b2), *reinterpret_cast<uint32_t *>(&b3));
                }
                continue;
            }
            for (int c0 = 0; c0 < p.BN; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(lane_addr + (uint32_t)c0, v);
                tmem_ld_wait();
                if (c0 + 16 >= p.BN) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                }
                const int col = n0 + c0;
                if (!row_ok || col >= p.n_cols) continue;
                const int nvalid = min(16, p.n_cols - col);
                float *o = (float *)p.out + row_off + col;
                for (int e = 0; e < nvalid; ++e) o[e] = __uint_as_float(v[e]);
            }
        }
        if (STATS && p.stats) {
            named_barrier(3, 256);
            const int nt = (int)blockIdx.x % p.n_tiles;
            stats_store_cta(smem_base + (uint32_t)p.stats_off, (uint32_t)p.stats_warp, 8, (int)threadIdx.x - 64, 256,
                            p.stats + (size_t)(blockIdx.x / p.n_tiles) * (1 + p.stats_lo) * 2 * p.ld_out, p.ld_out, p.stats_lo, p.n_cols, nt * p.BN,
                            nt + 1 < p.n_tiles ? (nt + 1) * p.BN : p.ld_out);
        }
        if (p.tma_store && gtid == 0) tma_store_wait_read();
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------ wgrad
// dw[k][tap][c] = sum over output pixels of dy[pixel][k] * x[pixel shifted by the tap][c]   (Eq. 4)
//   GEMM per tap: M = 128 output channels k, N = BN input channels c, reduction = output pixels, 64 per stage.
//   A operand: dy[pixel][k], k contiguous -> MN-major tiles (two 64-channel boxes of a 2-D tiled map).
//   B operand: x through the im2col map (same pixel raster as the forward pass, tap offset added by the TMA unit),
//              c contiguous -> MN-major tiles (one 64-channel box per 64 columns).
//   The pixel range is split across CTAs (blockIdx.y), at most one CTA per SM in total so that all of them are resident.
//   With more than one split every CTA stores its fp32 partial sums to the workspace from its registers, announces them on a
//   counter, waits (bounded) until all splits of its tile have arrived, and then sums its share of them over the splits in a
//   fixed order (wgrad_sum): deterministic, and no second kernel. Up to eight splits can meet in shared memory instead (wgrad_cluster_sum).
constexpr int kMaxRow = 8;  // filter rows and columns of the filter-row form
// The layer itself, for the sums that the raster forms cannot take from their accumulators (wgrad_pure).
struct WgradRaw {
    const __nv_bfloat16 *x, *dy;
    int N, H, W, C, K, P, Q, R, S, stride, pad, ldx, ldy;
};
struct WgradP {
    int K, C, taps;         // true channel counts, number of taps (R*S)
    int BN, n_tiles;        // input-channel tile
    int m_tiles;            // ceil(K / 128)
    int tpc, tap_groups;    // taps per CTA (they share the dy tile; one accumulator of BN columns each) and groups of taps
    int npix;               // N*P*Q
    int pix_per_split;      // multiple of 64
    int splits;
    int Pd, Qd, stride, lo_h, lo_w, S;
    int x_tiled;            // 1: 1x1 stride-1 filter without padding: x is a plain 2-D (channels, pixels) tiled map
    int stages, tmem_cols;
    // row-block form (stride-1 filters with several taps): a stage is `nr` output rows of one image
    int nr, Wp, RB;         // rows per unit, row pitch of both staged tiles in pixels (Q + S - 1), units per image
    int units, units_per_split;
    int ksteps;             // 16-pixel MMA steps per unit: ceil(nr * Wp / 16)
    int nb_a;               // 64-channel dy boxes per stage (1 when K <= 64)
    int lo_span;            // R - 1: extra rows of the x halo box
    int pair;               // row-block form: the M side of an MMA is two taps x 64 or four taps x 32 channel lanes of the x tile (a
                            // tap is another one shifted: the operand's block stride is that shift) and the N side is the output
                            // channels; accumulator lanes = (tap, c), columns = k
    int lanes, dy_lanes;    // row-block form: channel lanes per staged pixel of x and of dy (rows of 128 or 64 bytes)
    int lane_shift;         // log2 of `lanes`
    int row_lanes;          // packed form: channel lanes from one pixel of dy to the next (16 or 32)
    int acc_row;            // 32 lanes: accumulators per filter row, ceil(S / 4): each holds four neighbouring taps
    struct { int C, R, S, off; } stem;      // the space-to-depth stem: channels of the image (0: not the stem) and the real filter, for dw
    int G;                  // packed form: pixels side by side in a staged row of x (64 / lanes)
    // filter-row form: the taps of one filter row share a unit; a tap is plane tap_plane[s] of the unit's x rows (stride 2: the columns of
    // either parity are a plane each), tap_shift[s] pixels on
    int planes;
    int plane_lo[2];                                    // first column of a unit's rows in either plane
    unsigned char tap_plane[kMaxRow], tap_shift[kMaxRow];
    unsigned char row_par[kMaxRow];                     // filter row -> parity of the x rows it reads
    signed char row_off[kMaxRow];                       //               and their offset from the output row
    int cluster;            // 1: the splits of a tile are one thread-block cluster and meet in shared memory (no workspace)
    int apc;                // accumulators per CTA (= tpc in the generic form)
    int acc_cols;           // columns of one accumulator (= BN, or the padded K in the paired form)
    unsigned a_box, b_box;  // bytes reserved per dy box and per x box (multiples of 1024)
    unsigned data_bytes;    // shared memory behind the control block: the stages, and what the exchange of the splits may use
    float *out;             // dw
    int test_skip;          // test hook (pt_test_skip_next_arrive): split 0 does not announce its partial tile
    WgradRaw raw;           // raster forms (row-block, filter-row, packed)
    float *partial;         // splits > 1: workspace [blockIdx.x][split], room for the accumulators of 128 x acc_cols floats (WgradShare)
    unsigned int *sync;     // splits > 1: two zeroed counters per blockIdx.x (arrived, seen by); left zero again at exit
    unsigned int *status;
};

#ifdef PT_DEVICE_TRACE
__device__ unsigned long long g_wg_trace[8][64];
#define WTRACE(i) do { if (blockIdx.x == 0 && blockIdx.y < 64 && (threadIdx.x & 31) == 0) g_wg_trace[i][blockIdx.y] = globaltimer_ns(); } while (0)
#else
#define WTRACE(i) do { } while (0)
#endif
__device__ __forceinline__ int pt_ceil_div_dev(int a, int b) { return (a + b - 1) / b; }

// Row-block form: the tap that the `g`-th group of lanes of accumulator `acc` (of all of the layer's) holds; `taps` where there is none.
__device__ __forceinline__ int wgrad_tap(const WgradP &p, int acc, int g)
{
    if (p.lanes == 64) return min(2 * acc + g, p.taps);
    const int r = p.acc_row == 1 ? acc : acc / p.acc_row, s = (acc - r * p.acc_row) * 4 + g;
    return s < p.S ? r * p.S + s : p.taps;
}

// The raster forms stage whole rows of pixels. Where a row of dy ends (or its last unit, or a column group) its staged zeros meet pixels of x
// that no tap pairs them with: 0 x Inf, a NaN in a sum that the pixel is no part of. A NaN among the sums that a thread has stored, the four at
// (k + e dk, tap, c + e dc), is therefore taken again from the layer itself: one product per output pixel, with zeros outside the image, as
// the pixel form multiplies. Whole warps: eight `bad` lanes or more take their own sums, fewer are done one after the other by the warp, a lane
// to an output row (a NaN in the last image, each lane its own sums or rows dealt out: 106 -> 103 3x3 at 28x28, batch 64, all lanes bad 6 and
// 36 ms; 19 -> 19 at 56x56, batch 256, packed, a lane or two of a warp 106 and 20). A sum that is a NaN in its own right takes the rows up to
// the first that makes it one (all of x NaN: 0.06 and 0.09 ms, against 0.035 and 0.04 of finite x). (Inline, and behind the store: a call costs the kernels hundreds of bytes of spilled registers.)
__device__ __forceinline__ bool wgrad_nan(const float4 &v, int nv)
{
    return v.x != v.x || (nv > 1 && v.y != v.y) || (nv > 2 && v.z != v.z) || (nv > 3 && v.w != v.w);
}
__device__ __forceinline__ void wgrad_pure(const WgradRaw &q, float *out, bool bad, int k_, int dk, int tap_, int c_, int dc)
{
    unsigned left = __ballot_sync(0xffffffffu, bad);
    const int lane = threadIdx.x & 31, rows = q.N * q.P;
    const bool own = __popc(left) >= 8;
    while (left) {
        const int src = own ? lane : __ffs((int)left) - 1;
        const int k = __shfl_sync(0xffffffffu, k_, src), tap = __shfl_sync(0xffffffffu, tap_, src), c = __shfl_sync(0xffffffffu, c_, src);
        const int r = tap / q.S, s = tap - r * q.S;
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int row0 = 0; row0 < rows; row0 += own ? 1 : 32) {
            const int row = row0 + (own ? 0 : lane), n = row / q.P, h = (row - n * q.P) * q.stride - q.pad + r;
            const bool in_h = h >= 0 && h < q.H;
            const __nv_bfloat16 *const xr = q.x + ((size_t)n * q.H + (in_h ? h : 0)) * q.W * q.ldx, *const yr = q.dy + (size_t)row * q.Q * q.ldy;
            float part[4] = {0.f, 0.f, 0.f, 0.f};          // (a row's sum by itself: shorter chains)
            if (own ? bad : row < rows) {
#pragma unroll 4
                for (int j = 0; j < q.Q; ++j) {
                    const int w = j * q.stride - q.pad + s;
                    const bool in = in_h && w >= 0 && w < q.W;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        part[e] = fmaf(__bfloat162float(yr[(size_t)j * q.ldy + min(k + e * dk, q.K - 1)]),
                                       in ? __bfloat162float(xr[(size_t)w * q.ldx + min(c + e * dc, q.C - 1)]) : 0.f, part[e]);
                }
            }
            bool numbers = false;
#pragma unroll
            for (int e = 0; e < 4; ++e) { sum[e] += part[e]; numbers |= sum[e] == sum[e]; }
            if (own ? __all_sync(0xffffffffu, !bad || !numbers) : __any_sync(0xffffffffu, !numbers)) break;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (!own)
#pragma unroll
                for (int o = 16; o; o >>= 1) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
            if (!bad || lane != src || k + e * dk >= q.K || c + e * dc >= q.C) continue;
            float *const at = out + ((size_t)(k + e * dk) * q.R * q.S + tap) * q.C + c + e * dc;
            if (*at != *at) *at = sum[e];
        }
        left = own ? 0u : left & (left - 1u);
    }
}

// Row-block form: where the sums of (tap, lane c) are in dw; false: nowhere. In the stem a tap is a pair of filter rows and a lane one of four
// neighbouring positions' (a, b, channel): filter row 2 tap + a - off, column 2 (c / 16) + b - off, where the filter has them. (A launch of
// its own for this took 2 us and its start.)
__device__ __forceinline__ bool wgrad_pair_place(const WgradP &p, int &tap, int &c)
{
    if (!p.stem.C) return tap < p.taps && c < p.C;
    const int e = c & 15, ab = (e >= p.stem.C ? 1 : 0) + (e >= 2 * p.stem.C ? 1 : 0) + (e >= 3 * p.stem.C ? 1 : 0);
    const int r = 2 * tap + (ab >> 1) - p.stem.off, s = 2 * (c >> 4) + (ab & 1) - p.stem.off;
    c = e - ab * p.stem.C;
    tap = r * p.stem.S + s;
    return c < p.stem.C && r >= 0 && r < p.stem.R && s >= 0 && s < p.stem.S;
}
// The sums of the output channels k .. k + 3 at (tap, c) of dw (wgrad_pair_place).
__device__ __forceinline__ void wgrad_pair_store(const WgradP &p, int k, int tap, int c, const float4 &v)
{
    const int C = p.raw.C, pitch = p.raw.R * p.raw.S * C;
    float *const dst = p.out + (size_t)k * pitch + (size_t)tap * C + c;
    const float v4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (k + e < p.K) dst[(size_t)e * pitch] = v4[e];
}

// 32 columns (16 where the accumulator ends) of a warp's 32 TMEM lanes; zeros for a CTA that had no work.
__device__ __forceinline__ void wgrad_load32(uint32_t taddr, bool second, bool any, uint32_t (&v)[32])
{
    uint32_t lo[16], hi[16];
    if (any) {
        tmem_ld16(taddr, lo);
        if (second) tmem_ld16(taddr + 16u, hi);
        tmem_ld_wait();
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) { v[e] = any ? lo[e] : 0u; v[16 + e] = any && second ? hi[e] : 0u; }
}

// Four consecutive floats of dw, nv of which exist (a dw row starts on a 16-byte boundary only if C allows it).
__device__ __forceinline__ void wgrad_store4(float *dst, const float4 &v, int nv)
{
    if (nv == 4 && ((uintptr_t)dst & 15) == 0) { *reinterpret_cast<float4 *>(dst) = v; return; }
    if (nv == 4 && ((uintptr_t)dst & 7) == 0) {
        reinterpret_cast<float2 *>(dst)[0] = make_float2(v.x, v.y);
        reinterpret_cast<float2 *>(dst)[1] = make_float2(v.z, v.w);
        return;
    }
    dst[0] = v.x;
    if (nv > 1) dst[1] = v.y;
    if (nv > 2) dst[2] = v.z;
    if (nv > 3) dst[3] = v.w;
}

// The splits of a tile as one cluster: the accumulators, cut into slots of 32 lanes x 32 columns, are dealt out to the CTAs; every
// CTA writes each of its slots straight from its registers into the shared memory of the slot's owner (in that CTA's then idle
// stage memory, the sources side by side), and the owner adds the sources in ascending order and stores dw. Through the workspace the
// same exchange costs three round trips to L2 (store the partial tile, wait for its arrival counter, load: 7 us whatever the size);
// here it is two cluster barriers and the bytes (about 2.5 us). At most eight splits: what a portable cluster can be.
// Every thread of every CTA of the cluster calls this, with the same trip counts, and aborting CTAs too (they hand on zeros; dw is
// then undefined and the time-out already recorded): the barriers always complete.
template <bool RASTER, bool PAIR>
__device__ __forceinline__ void wgrad_cluster_sum(const WgradP &p, Ctl *ctl, uint32_t data_base, uint32_t tmem_base, int tap0, int k0, int c0,
                                                  int split, int iters, uint32_t ring_bytes, int n_acc, int acc_cols)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = p.splits, nch = pt_ceil_div_dev(acc_cols, 32);
    // quarters of the 128 lanes that hold something: output channels below K; in the row-block form the taps that exist
    const int nq = !p.pair ? min(4, pt_ceil_div_dev(p.K - k0, 32)) : p.lanes == 32 ? min(4, p.S) : 4;
    const int slots = n_acc * nch * nq, mine = pt_ceil_div_dev(slots, S);              // slot u: owner u % S, its (u / S)-th
    const int cap = (int)(ring_bytes / ((uint32_t)S * 4096u));                         // slots an owner can receive at a time
    const bool any = iters > 0 && !*(volatile int *)&ctl->abort_flag;
    for (int base = 0; base < mine; base += cap) {
        cluster_barrier();                     // every ring is idle (first round), every sum has been read (later rounds)
        const int n = min(cap, mine - base);
        if (warp >= 1) {
            const int quarter = warp & 3, wset = (warp >= 2 && warp < 6) ? 0 : 1;
            if (quarter < nq) {
                const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
                for (int ci = wset; ci < n_acc * nch; ci += 2) {
                    const int u = ci * nq + quarter, pos = u / S - base;
                    if (pos < 0 || pos >= n) continue;
                    const int tt = ci / nch, cc = (ci - tt * nch) * 32;
                    uint32_t v[32];
                    wgrad_load32(lane_addr + (uint32_t)(tt * acc_cols + cc), cc + 16 < acc_cols, any, v);
                    const uint32_t slab = map_to_rank(data_base + ((uint32_t)pos * (uint32_t)S + (uint32_t)split) * 4096u, (uint32_t)(u % S));
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        st_cluster_v4(slab + (uint32_t)lane * 128u + (((uint32_t)j ^ ((uint32_t)lane & 7u)) << 4), v[4 * j], v[4 * j + 1],
                                      v[4 * j + 2], v[4 * j + 3]);
                }
            }
        }
        cluster_barrier();                     // everything this CTA owns has arrived
        // a slot has 32 rows x 8 float4: in the paired form the row (input channel) varies fastest, so that lanes write consecutive
        // floats of dw; else the column
        for (int i = threadIdx.x; i < n * 256; i += kThreads) {
            const int pos = i >> 8, u = (base + pos) * S + split;
            if (u >= slots) break;
            const int ci = u / nq, quarter = u - ci * nq, tt = ci / nch, cc = (ci - tt * nch) * 32;
            const int r = p.pair ? i & 31 : (i >> 3) & 31, j = p.pair ? (i >> 5) & 7 : i & 7;
            const int row = quarter * 32 + r, col = cc + j * 4;
            const uint32_t a = data_base + (uint32_t)pos * (uint32_t)S * 4096u + (uint32_t)r * 128u + ((uint32_t)(j ^ (r & 7)) << 4);
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int z = 0; z < S; ++z) {
                float4 t;
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(a + (uint32_t)z * 4096u) : "memory");
                sum.x += t.x; sum.y += t.y; sum.z += t.z; sum.w += t.w;
            }
            if (PAIR) {
                int tap = wgrad_tap(p, tap0 + tt, row >> p.lane_shift), c = row & (p.lanes - 1);
                const bool here = wgrad_pair_place(p, tap, c) && col < p.K;
                if (here) wgrad_pair_store(p, col, tap, c, sum);
                wgrad_pure(p.raw, p.out, here && wgrad_nan(sum, p.K - col), col, 1, tap, c, 0);
            } else {
                const int nv = k0 + row < p.K && col < acc_cols ? min(4, p.C - (c0 + col)) : 0;
                if (nv > 0) wgrad_store4(p.out + ((size_t)(k0 + row) * p.taps + tap0 + tt) * p.C + c0 + col, sum, nv);
                if (RASTER) wgrad_pure(p.raw, p.out, nv > 0 && wgrad_nan(sum, nv), k0 + row, 0, tap0 + tt, c0 + col, 1);
            }
        }
    }
}

// A split's partial sums of a tile in the workspace: 16-byte pieces [accumulator][four columns][row], the rows and columns that are part of
// dw only (not the output channels past K; in the paired form not the channel lanes past C), so that a warp, whose lanes hold a row each
// when they read the tensor memory, stores 512 consecutive bytes at a time, and a CTA's share of the sum is one run of every
// split's pieces. (As 32 x 32 boxes through staging and TMA stores the 172 KB of three accumulators of 112 columns took 4.1 us to store,
// and 4.4 us to read back and sum; 2.2 and 2.9 this way. 418 -> 111 1x1 at 28x28, batch 64 21.8 -> 20.5 us a launch, 69 -> 418 19.8 -> 16.9,
// 8 -> 14 3x3 at 32x32, batch 128 16.6 -> 14.1; at a limit of 49 CTAs 112 -> 111 3x3/2 at 56x56 54.4 -> 50.8.)
struct WgradShare {
    int lanes_used, rows, quads;
    __device__ __forceinline__ WgradShare(const WgradP &p, int k0, int c0, int acc_cols)
    {
        const int groups = !p.pair ? 1 : p.lanes == 32 ? min(4, p.S) : 2;       // taps of an accumulator
        rows = !p.pair ? min(128, p.K - k0) : groups * p.C;
        lanes_used = !p.pair ? rows : groups << p.lane_shift;
        quads = pt_ceil_div_dev(p.pair ? p.K : min(acc_cols, p.C - c0), 4);
    }
    // the row of a TMEM lane; -1: none
    __device__ __forceinline__ int row(const WgradP &p, int l) const
    {
        if (!p.pair) return l < rows ? l : -1;
        const int g = l >> p.lane_shift, c = l & (p.lanes - 1);
        return l < lanes_used && c < p.C ? g * p.C + c : -1;
    }
    // where a split's pieces start, in floats (room for whole accumulators)
    __device__ __forceinline__ size_t split_off(const WgradP &p, int split, int acc_cols) const
    {
        return ((size_t)blockIdx.x * p.splits + split) * (size_t)p.apc * 128 * acc_cols;
    }
};

// One thread, behind a barrier of the threads that stored this split's partial sums: announces them, waits (bounded) for the tile's other
// splits, and the last CTA to see that all have arrived clears the counters (nobody looks at them again). Every split CTA of a tile is
// resident (the grid is at most one CTA per SM).
__device__ __forceinline__ void wgrad_arrive(const WgradP &p, int split, volatile int *abort_flag)
{
    unsigned int *arrived = p.sync + 2 * blockIdx.x;
    __threadfence();                                             // the CTA's stores (ordered before this by the barrier), then its arrival
    // (test hook: split 0 stays silent, so that every split of the tile runs into the bounded wait below)
    if (!(p.test_skip && split == 0)) atomicAdd(arrived, 1u);
    const uint64_t t0 = globaltimer_ns();
    unsigned int seen, polls = 0;
    for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(arrived) : "memory");
        if (seen >= (unsigned)p.splits || *abort_flag) break;
        if ((++polls & 63u) == 0u && globaltimer_ns() - t0 > *(volatile unsigned long long *)&g_wait_limit_ns) {
            record_timeout(p.status, 8);
            *abort_flag = 1;
            break;
        }
    }
    if (seen >= (unsigned)p.splits && atomicAdd(arrived + 1, 1u) == (unsigned)p.splits - 1u) {
        arrived[0] = 0u;
        arrived[1] = 0u;
    }
}

// Pieces of a chunk that `bytes` of shared memory hold from each of Z sources: an odd number (see wgrad_bring), at least one.
__device__ __forceinline__ int wgrad_chunk(uint32_t bytes, int Z)
{
    const int cap = (int)(bytes / ((uint32_t)Z * 16u));
    return cap - 1 + (cap & 1);
}
// All threads: the run of `n` 16-byte pieces at `src` of each of Z sources, `stride` pieces apart, into shared memory: piece i of source z
// at z * (n | 1) + i (an odd pitch: lanes on neighbouring sources do not share a bank; with a source's pieces apart instead, the copies'
// writes do: 418 -> 111 1x1 at 28x28, batch 64 20.4 -> 22.9 us).
__device__ __forceinline__ void wgrad_bring(uint32_t dst, const float4 *src, size_t stride, int Z, int n)
{
    // copies are dealt out evenly, i fastest
    const int pitch = n | 1;
    int z = threadIdx.x / n, i = threadIdx.x - z * n;
    const int dz = kThreads / n, di = kThreads - dz * n;
    while (z < Z) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(z * pitch + i) * 16u), "l"(src + (size_t)z * stride + i) : "memory");
        z += dz; i += di;
        if (i >= n) { i -= n; ++z; }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// log2 of the lanes that share the sum of a piece: a share of few pieces of many sources is one thread's long chain of adds otherwise
// (8 -> 8 3x3 at 32x32, batch 128 in the packed form: two pieces of 512 sources, 14.9 us against 10.7).
__device__ __forceinline__ int wgrad_sum_lanes(int n, int Z)
{
    int ls = 0;
    while (ls < 5 && (n << (ls + 1)) <= kThreads && (Z >> (ls + 1)) >= 4) ++ls;
    return ls;
}
// Piece k of what wgrad_bring brought (k >= n: none), summed over the sources: each of L = 2^ls neighbouring lanes every L-th of them in
// ascending order, then the lanes' sums pairwise: always the same way. Whole warps; the sum is in the first of the lanes.
__device__ __forceinline__ float4 wgrad_sum(uint32_t base, int k, int n, int Z, int ls)
{
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    const int step = 1 << ls, z0 = (int)(threadIdx.x & (unsigned)(step - 1)), z1 = k < n ? Z : 0;
    uint32_t a = base + (uint32_t)(z0 * (n | 1) + k) * 16u;
#pragma unroll 4
    for (int y = z0; y < z1; y += step, a += (uint32_t)(step * (n | 1)) * 16u) {
        float4 t;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(a) : "memory");
        sum.x += t.x; sum.y += t.y; sum.z += t.z; sum.w += t.w;
    }
    for (int o = 1; o < step; o <<= 1) {
        sum.x += __shfl_down_sync(0xffffffffu, sum.x, o); sum.y += __shfl_down_sync(0xffffffffu, sum.y, o);
        sum.z += __shfl_down_sync(0xffffffffu, sum.z, o); sum.w += __shfl_down_sync(0xffffffffu, sum.w, o);
    }
    return sum;
}

// Everything after the main loop of a weight-gradient kernel: the accumulators leave TMEM (directly to dw, or as this
// split's partial tile), the splits of a tile meet, and every CTA sums its share of the tile over the splits.
// `ring_bytes` of shared memory at `data_base` are free by then and serve as staging. `tap0` is the CTA's first tap (generic form) or
// accumulator (row-block form). RASTER: a form that pairs staged zeros of dy with pixels of x (wgrad_pure); PAIR: the row-block form.
template <bool RASTER, bool PAIR>
__device__ __forceinline__ void wgrad_finish(const WgradP &p, Ctl *ctl, uint32_t data_base, uint32_t tmem_base,
                                             int tap0, int k0, int c0, int split, int iters, uint32_t ring_bytes, int n_acc, int acc_cols)
{
    volatile int *abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= 1) {
        // ---------------- epilogue: the four epilogue warps and, once they are done issuing, the four issuer warps; a warp
        // may read the TMEM lanes of quarter warp % 4, so each quarter has two warps, which take alternate 32-column chunks
        const int quarter = warp & 3, wset = (warp >= 2 && warp < 6) ? 0 : 1;
        bool ok = true;
        if (iters > 0) ok = mbar_wait(smem_u32(&ctl->accum), 0, abort_flag, p.status, 6);
        ok = __all_sync(0xffffffffu, ok);                    // (the warp stays together below)
        if (warp == 2) WTRACE(3);
        tc_fence_after();
        if (ok) {
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
            if (p.cluster) {
                // the exchange is below: every thread of the cluster takes part in its barriers
            } else if (p.splits > 1) {
                // ---- (1) this CTA's partial sums go to the workspace straight from the registers (WgradShare: a lane's 16 bytes lie beside
                // its neighbour's, 512 bytes a store)
                const WgradShare sh(p, k0, c0, acc_cols);
                const int gtid = (warp - 1) * 32 + lane;
                const int row = sh.row(p, quarter * 32 + lane);
                float *const dst = p.partial + sh.split_off(p, split, acc_cols);
                int ci = 0;
                for (int tt = 0; tt < n_acc && quarter * 32 < sh.lanes_used; ++tt)
                for (int cc = 0; cc < acc_cols; cc += 32, ++ci) {
                    if ((ci & 1) != wset) continue;
                    uint32_t v[32];
                    wgrad_load32(lane_addr + (uint32_t)(tt * acc_cols + cc), cc + 16 < acc_cols, iters > 0, v);
                    float4 *const d4 = reinterpret_cast<float4 *>(dst) + (size_t)(tt * sh.quads + cc / 4) * sh.rows + row;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (row >= 0 && cc / 4 + j < sh.quads)
                            __stcg(d4 + (size_t)j * sh.rows, make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                                         __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])));
                }
                if (warp == 2) WTRACE(4);
                named_barrier(1, 256);
                // ---- (2) every split CTA of this tile is resident (the grid is at most one CTA per SM): wait for all of them
                if (gtid == 0) wgrad_arrive(p, split, abort_flag);
                named_barrier(1, 256);
                if (warp == 2) WTRACE(5);
            } else if (PAIR) {
                // lanes are (tap of the accumulator, input channel), columns are output channels: for one column a warp's lanes
                // write consecutive floats of dw
                // (addresses once per accumulator and a pitch per column: with the place in dw found anew for each float, two accumulators of 176
                // columns took 11 us, 6 before that)
                const int l = quarter * 32 + lane, C = p.raw.C;
                const size_t pitch = (size_t)p.raw.R * p.raw.S * C;
                int ci = 0;
                for (int tt = 0; tt < n_acc; ++tt) {
                    int tap = wgrad_tap(p, tap0 + tt, l >> p.lane_shift), c = l & (p.lanes - 1);
                    const bool here = wgrad_pair_place(p, tap, c);
                    float *const dst = p.out + (here ? (size_t)tap * C + c : 0);
                    for (int cc = 0; cc < acc_cols; cc += 16, ++ci) {
                        if ((ci & 1) != wset) continue;
                        uint32_t v[16];
                        if (iters > 0) {
                            tmem_ld16(lane_addr + (uint32_t)(tt * acc_cols + cc), v);
                            tmem_ld_wait();
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) v[e] = 0u;
                        }
                        const int n = here ? min(16, p.K - cc) : 0;
                        float *d = dst + (size_t)cc * pitch;
                        unsigned bad = 0u;                   // a bit per four sums
#pragma unroll
                        for (int e = 0; e < 16; ++e, d += pitch) {
                            const float f = __uint_as_float(v[e]);
                            if (e < n) *d = f;
                            if (e < n && f != f) bad |= 1u << (e >> 2);
                        }
                        if (__any_sync(0xffffffffu, bad != 0u))
#pragma unroll 1
                            for (int e = 0; e < 4; ++e) wgrad_pure(p.raw, p.out, (bad >> e) & 1u, cc + 4 * e, 1, tap, c, 0);
                    }
                }
            } else {
            float *obase = p.out;
            // The stages are free once the accumulator is complete: each warp transposes its 32 x 32 blocks through
            // a padded shared-memory square so that a warp writes 32 consecutive floats of one dw row at a time.
            const uint32_t sq = data_base + (uint32_t)(wset * 4 + quarter) * (32u * 33u * 4u);
            int ci = 0;
            for (int tt = 0; tt < n_acc; ++tt)
            for (int cc = 0; cc < acc_cols; cc += 32, ++ci) {
                if ((ci & 1) != wset) continue;
                const int tap = tap0 + tt;
                uint32_t v[32];
                if (iters > 0) {
                    uint32_t lo[16], hi[16];
                    tmem_ld16(lane_addr + (uint32_t)(tt * acc_cols + cc), lo);
                    if (cc + 16 < acc_cols) tmem_ld16(lane_addr + (uint32_t)(tt * acc_cols + cc) + 16u, hi);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) { v[e] = lo[e]; v[16 + e] = (cc + 16 < acc_cols) ? hi[e] : 0u; }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0u;
                }
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(sq + (uint32_t)(lane * 33 + e) * 4u), "r"(v[e]) : "memory");
                __syncwarp();
                const int col = c0 + cc + lane;
                [[maybe_unused]] unsigned bad = 0u;          // a bit per row
                for (int rr = 0; rr < 32; ++rr) {
                    const int kk = k0 + quarter * 32 + rr;
                    if (kk >= p.K) break;
                    uint32_t t;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(t) : "r"(sq + (uint32_t)(rr * 33 + lane) * 4u) : "memory");
                    if (col < p.C && cc + lane < p.BN) {
                        const float f = __uint_as_float(t);
                        obase[((size_t)kk * p.taps + tap) * p.C + col] = f;
                        if (RASTER && f != f) bad |= 1u << rr;
                    }
                }
                if (RASTER && __any_sync(0xffffffffu, bad != 0u))
#pragma unroll 1
                    for (int rr = 0; rr < 32; ++rr) wgrad_pure(p.raw, p.out, (bad >> rr) & 1u, k0 + quarter * 32 + rr, 0, tap, col, 0);
            }
            }
        }
        tc_fence_before();
    }
    if (p.cluster) {
        wgrad_cluster_sum<RASTER, PAIR>(p, ctl, data_base, tmem_base, tap0, k0, c0, split, iters, ring_bytes, n_acc, acc_cols);
        return;
    }
    __syncthreads();
    if (p.splits > 1 && !*abort_flag) {
        // ---- (3) all threads: this CTA sums its share of the tile's 16-byte pieces over the splits. The partial sums sit in L2 and what costs
        // time is a chain of dependent loads, so the asynchronous copies of the whole share, a run of every split's pieces, go out first, into
        // the (now idle) stage memory; the copies are then summed from there in a fixed order (wgrad_sum): deterministic, whichever CTA
        // does the work.
        const WgradShare sh(p, k0, c0, acc_cols);
        const int total = n_acc * sh.quads * sh.rows, per_cta = (total + p.splits - 1) / p.splits;
        const int it_beg = split * per_cta, it_end = min(total, it_beg + per_cta);
        const float4 *const pbase = reinterpret_cast<const float4 *>(p.partial + sh.split_off(p, 0, acc_cols));
        const size_t zstride = (size_t)p.apc * acc_cols * 32;                    // in pieces
        const int cap = wgrad_chunk(ring_bytes, p.splits);         // pieces the stage memory holds
        const float inv_rows = 1.0f / (float)sh.rows, inv_quads = 1.0f / (float)sh.quads;
        for (int c_beg = it_beg; c_beg < it_end; c_beg += cap) {
            const int n_chunk = min(cap, it_end - c_beg);
            wgrad_bring(data_base, pbase + c_beg, zstride, p.splits, n_chunk);
            const int ls = wgrad_sum_lanes(n_chunk, p.splits);
            for (int i = threadIdx.x; i < (((n_chunk << ls) + 31) & ~31); i += kThreads) {
                const int k = i >> ls;
                const float4 sum = wgrad_sum(data_base, k, n_chunk, p.splits, ls);
                const bool mine = k < n_chunk && !(i & ((1 << ls) - 1));
                const int piece = c_beg + k, tq = fast_div(piece, sh.rows, inv_rows), row = piece - tq * sh.rows;
                const int tt = fast_div(tq, sh.quads, inv_quads), col = (tq - tt * sh.quads) * 4;
                if (PAIR) {
                    // row = (tap of the accumulator, input channel), columns = output channels: consecutive threads, consecutive floats
                    const int g = (row >= p.C ? 1 : 0) + (row >= 2 * p.C ? 1 : 0) + (row >= 3 * p.C ? 1 : 0);
                    int tap = wgrad_tap(p, tap0 + tt, g), c = row - g * p.C;
                    const bool here = wgrad_pair_place(p, tap, c) && mine;
                    if (here) wgrad_pair_store(p, col, tap, c, sum);
                    wgrad_pure(p.raw, p.out, here && wgrad_nan(sum, p.K - col), col, 1, tap, c, 0);
                } else {
                    const int nv = min(4, p.C - (c0 + col));
                    if (mine) wgrad_store4(p.out + ((size_t)(k0 + row) * p.taps + tap0 + tt) * p.C + c0 + col, sum, nv);
                    if (RASTER) wgrad_pure(p.raw, p.out, mine && wgrad_nan(sum, nv), k0 + row, 0, tap0 + tt, c0 + col, 1);
                }
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) WTRACE(6);
    }
}

__global__ void __launch_bounds__(kThreads, 1) conv_wgrad_kernel(const __grid_constant__ CUtensorMap tmDy,
                                                              const __grid_constant__ CUtensorMap tmX, const __grid_constant__ WgradP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Ctl *ctl = reinterpret_cast<Ctl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t data_base = (smem_base + (uint32_t)sizeof(Ctl) + 1023u) & ~1023u;
    const uint32_t a_bytes = 2u * 8192u;
    const uint32_t nb_b = (uint32_t)((p.BN + 63) / 64);
    const uint32_t b_bytes = nb_b * 8192u;                            // one tap's x tile
    const uint32_t stage_bytes = a_bytes + (uint32_t)p.tpc * b_bytes;
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int bx = blockIdx.x;
    const int n_tile = bx % p.n_tiles; bx /= p.n_tiles;
    const int m_tile = bx % p.m_tiles; bx /= p.m_tiles;
    const int tap0 = bx * p.tpc;                                      // this CTA's taps: tap0 .. tap0 + ntap - 1
    const int ntap = min(p.tpc, p.taps - tap0);
    const int split = blockIdx.y;
    const int k0 = m_tile * 128, c0 = n_tile * p.BN;
    const int pix_beg = split * p.pix_per_split;
    const int pix_end = min(p.npix, pix_beg + p.pix_per_split);
    const int iters = pix_end > pix_beg ? (pix_end - pix_beg + 63) / 64 : 0;

    // Issuing is what a single thread does slowly (about 200 cycles per TMA instruction, 50 to 100 per MMA), so both
    // sides of the pipeline are spread over warps: warp 0 loads the dy tile, the four epilogue warps (idle until the
    // accumulators are complete) load the x tiles, and up to four issuer warps each own the accumulators of the taps
    // tt = i, i + NI, ... Every participant arrives on a stage's barriers itself.
    const int n_x = ntap * (int)nb_b;                                 // x boxes per stage
    const int NXP = n_x < 4 ? n_x : 4;                                // x producer warps in use
    const int NI = ntap < 4 ? ntap : 4;                               // MMA issuer warps in use
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1u + (uint32_t)NXP);
            mbar_init(smem_u32(&ctl->empty[s]), (uint32_t)NI);
        }
        mbar_init(smem_u32(&ctl->accum), (uint32_t)NI);
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmDy);
        prefetch_tmap(&tmX);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int issuer = warp == 1 ? 0 : warp - 5;                      // warps 6, 7, 8 -> issuers 1, 2, 3
    // Nothing above touches global memory. The producer threads wait for the previous kernel after their set-up (pixel
    // coordinates of the first stage: several divisions) instead of before it.
    if (!((warp == 0 || (warp >= 2 && warp < 2 + NXP)) && lane == 0)) grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x == 0) WTRACE(0);

    if (warp == 0 || (warp >= 2 && warp < 2 + NXP)) {
        if (lane == 0) {
            // ---------------- producers: warp 0 brings dy, warp 2 + j the x boxes j, j + 4, ... of every stage
            const bool is_dy = warp == 0;
            const int xp = warp - 2;
            // output channels k0+64.. of this tile do not exist when K - k0 <= 64: their accumulator rows are never
            // stored, so that half of the A tile is not loaded at all (the MMA reads stale shared memory there)
            const bool second = p.K - k0 > 64;
            uint32_t my_bytes;
            if (is_dy) my_bytes = second ? a_bytes : 8192u;
            else my_bytes = (uint32_t)((n_x - xp + 3) / 4) * 8192u;
            int q = pix_beg % p.Qd, t = pix_beg / p.Qd, pp = t % p.Pd, n = t / p.Pd;   // first pixel of the stage
            // a stage advances 64 pixels = dn images + dp rows + dq columns: carried without divisions in the loop
            const int dn = 64 / (p.Pd * p.Qd), rem64 = 64 - dn * p.Pd * p.Qd, dp = rem64 / p.Qd, dq = rem64 - dp * p.Qd;
            // this warp's x boxes (at most two per stage: tpc * BN/64 <= 8 boxes over four warps): tap and channel block of each
            int n_mine = 0, box_dst[2] = {0, 0}, box_c[2] = {0, 0};
            uint16_t box_sw[2] = {0, 0}, box_sh[2] = {0, 0};
            if (!is_dy)
                for (int j = xp; j < n_x && n_mine < 2; j += 4, ++n_mine) {
                    const int tt = j / (int)nb_b, nb = j - tt * (int)nb_b;
                    const int r = (tap0 + tt) / p.S;
                    box_dst[n_mine] = j * 8192; box_c[n_mine] = c0 + nb * 64;
                    box_sh[n_mine] = (uint16_t)r; box_sw[n_mine] = (uint16_t)((tap0 + tt) - r * p.S);
                }
            int s = 0, ph = 0, issued = 0;
            grid_dependency_wait();
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, p.status, 4)) break;
                const uint32_t bar = smem_u32(&ctl->full[s]);
                const uint32_t a_dst = data_base + (uint32_t)s * stage_bytes, b_dst = a_dst + a_bytes;
                mbar_arrive_expect_tx(bar, my_bytes);
                if (is_dy) {
                    const int pix = pix_beg + it * 64;
                    tma_load_2d(a_dst, &tmDy, bar, k0, pix);
                    if (second) tma_load_2d(a_dst + 8192u, &tmDy, bar, k0 + 64, pix);
                } else {
                    const int w = q * p.stride + p.lo_w, h = pp * p.stride + p.lo_h;
                    if (p.x_tiled) {
                        const int pix = pix_beg + it * 64;
                        tma_load_2d(b_dst + (uint32_t)box_dst[0], &tmX, bar, box_c[0], pix);
                        if (n_mine > 1) tma_load_2d(b_dst + (uint32_t)box_dst[1], &tmX, bar, box_c[1], pix);
                    } else {
                        tma_load_im2col_4d(b_dst + (uint32_t)box_dst[0], &tmX, bar, box_c[0], w, h, n, box_sw[0], box_sh[0]);
                        if (n_mine > 1) tma_load_im2col_4d(b_dst + (uint32_t)box_dst[1], &tmX, bar, box_c[1], w, h, n, box_sw[1], box_sh[1]);
                    }
                    q += dq; pp += dp; n += dn;                       // the next stage starts 64 pixels further on
                    if (q >= p.Qd) { q -= p.Qd; ++pp; }
                    if (pp >= p.Pd) { pp -= p.Pd; ++n; }
                }
                issued = it + 1;
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) drain_ring(smem_u32(&ctl->full[0]), p.stages, issued);
        }
        __syncwarp();
    }
    if (warp == 1 || (warp >= 6 && issuer < NI)) {
        // ---------------- MMA issuer `issuer`: the warp walks the loop in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, p.BN, 1, 1);
        bool ok = true;
        int s = 0, ph = 0;
        for (int it = 0; it < iters && ok; ++it) {
            ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status, 5);
            if (!ok) break;
            if (it == 0 && warp == 1) WTRACE(1);
            tc_fence_after();
            const int rem = pix_end - (pix_beg + it * 64);
            const int ksteps = rem >= 64 ? 4 : (rem + 15) / 16;
            const uint32_t a_src = data_base + (uint32_t)s * stage_bytes, b_src = a_src + a_bytes;
            const uint64_t ad0 = make_desc(a_src, 8192u, 1024u);
            const uint32_t acc = it != 0 ? 1u : 0u;
            for (int tt = issuer; tt < ntap; tt += NI) {
                const uint64_t bd0 = make_desc(b_src + (uint32_t)tt * b_bytes, 8192u, 1024u);
                const uint32_t d_tmem = tmem_base + (uint32_t)(tt * p.BN);
                if (ksteps == 4) {
                    umma_bf16_lead(d_tmem, ad0, bd0, idesc, acc, leader);
#pragma unroll
                    for (int k = 1; k < 4; ++k) umma_bf16_lead(d_tmem, ad0 + 128ull * k, bd0 + 128ull * k, idesc, 1u, leader);
                } else {
                    for (int k = 0; k < ksteps; ++k) umma_bf16_lead(d_tmem, ad0 + 128ull * k, bd0 + 128ull * k, idesc, k ? 1u : acc, leader);
                }
            }
            umma_commit_lead(smem_u32(&ctl->empty[s]), leader);
            if (++s == p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit_lead(smem_u32(&ctl->accum), leader);
        if (warp == 1) WTRACE(2);
    }
    wgrad_finish<false, false>(p, ctl, data_base, tmem_base, tap0, k0, c0, split, iters, p.data_bytes, ntap, p.BN);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// Row-block form of the weight gradient for stride-1 filters with several taps and at most 64 input channels. A stage is
// one unit = `nr` output rows of one image: dy as a box of nr rows x Wp columns (the columns past Q and the rows past P
// are zero-filled by the TMA unit) and x as the halo box of nr + R - 1 rows x Wp columns starting at (-pad, -pad) of the
// unit, both with one swizzle row per pixel. Pixel m = i * Wp + j of the dy box pairs with pixel
// m + r * Wp + s of the x box for tap (r, s), so every tap reads the SAME staged x tile through an operand descriptor
// whose start is shifted by r * Wp + s rows: x crosses the memory system once per unit instead of once per tap. Where
// j + s runs past the row the dy factor is a zero column. Rows past the boxes (up to the 16-pixel step) are zeroed once
// and never written again.
//   The x tile is the M side of the MMA and carries several taps. With 33 to 64 channels a pixel is a 128-byte row and M rows 0..63 are
// its 64 lanes at the first tap's shift, rows 64..127 the same lanes at the second tap's (the descriptor's block stride is the difference
// of the shifts). With at most 32 channels it is a 64-byte row and the four 32-lane blocks are the four neighbouring taps s, s + 1, ..
// of a filter row (block stride one pixel; past S they are not stored). The N side is dy's output channels. An accumulator therefore
// holds dw^T of two or four taps: lanes = (tap, c), columns = k -- a half or a third of the MMAs of the one-tap-per-accumulator form
// for a 3x3 filter. The MMAs (29 ns each however narrow) and the TMA unit's time per row bound the narrow layers, and a 64-byte
// row that ends inside a sector takes it 3.1 ns instead of 4.5.
__global__ void __launch_bounds__(kThreads, 1) conv_wgrad_rows_kernel(const __grid_constant__ CUtensorMap tmDy,
                                                                   const __grid_constant__ CUtensorMap tmX, const __grid_constant__ WgradP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Ctl *ctl = reinterpret_cast<Ctl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t data_base = (smem_base + (uint32_t)sizeof(Ctl) + 1023u) & ~1023u;
    const uint32_t nb_b = (uint32_t)((p.BN + 63) / 64);
    const uint32_t a_bytes = (uint32_t)p.nb_a * p.a_box;
    const uint32_t stage_bytes = a_bytes + nb_b * p.b_box;
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int bx = blockIdx.x;
    const int n_tile = bx % p.n_tiles; bx /= p.n_tiles;
    const int m_tile = bx % p.m_tiles; bx /= p.m_tiles;
    const int acc0 = bx * p.apc;                                      // this CTA's accumulators: acc0 .. acc0 + n_acc - 1
    const int split = blockIdx.y;
    const int k0 = m_tile * 128, c0 = n_tile * p.BN;
    const int u_beg = split * p.units_per_split;
    const int u_end = min(p.units, u_beg + p.units_per_split);
    const int iters = u_end > u_beg ? u_end - u_beg : 0;
    const int n_acc = min(p.apc, (p.lanes == 64 ? (p.taps + 1) / 2 : p.taps / p.S * p.acc_row) - acc0);
    const int NI = n_acc < 4 ? n_acc : 4;                             // MMA issuer warps in use: accumulators i, i + NI, ...
    const uint32_t x_row = (uint32_t)p.lanes * 2u, dy_row = (uint32_t)p.dy_lanes * 2u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2u);                   // the dy producer and the x producer
            mbar_init(smem_u32(&ctl->empty[s]), (uint32_t)NI);
        }
        mbar_init(smem_u32(&ctl->accum), (uint32_t)NI);
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmDy);
        prefetch_tmap(&tmX);
    }
    // the rows between the end of a box and the end of the last 16-pixel step are read by the MMAs (times zero) and must be finite
    {
        const uint32_t a_used = (uint32_t)(p.nr * p.Wp) * dy_row, b_used = (uint32_t)((p.nr + p.lo_span) * p.Wp) * x_row;
        const uint32_t a_rest = (p.a_box - a_used) / 16u, b_rest = (p.b_box - b_used) / 16u;
        const uint32_t per_stage = (uint32_t)p.nb_a * a_rest + nb_b * b_rest;
        for (uint32_t i = threadIdx.x; i < (uint32_t)p.stages * per_stage; i += kThreads) {
            const uint32_t st = i / per_stage, o = i - st * per_stage;
            const uint32_t at = o < (uint32_t)p.nb_a * a_rest ? (o / a_rest) * p.a_box + a_used + (o % a_rest) * 16u
                                                              : a_bytes + ((o - (uint32_t)p.nb_a * a_rest) / b_rest) * p.b_box + b_used +
                                                                    ((o - (uint32_t)p.nb_a * a_rest) % b_rest) * 16u;
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(data_base + st * stage_bytes + at), "r"(0u) : "memory");
        }
    }
    fence_proxy_async();
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int issuer = warp == 1 ? 0 : warp - 5;                      // warps 6, 7, 8 -> issuers 1, 2, 3
    // nothing above touches global memory; the producer threads wait after their set-up
    if (!((warp == 0 || warp == 2) && lane == 0)) grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x == 0) WTRACE(0);

    if (warp == 0 || warp == 2) {
        if (lane == 0) {
            // ---------------- producers: warp 0 brings the dy boxes of every unit, warp 2 the x halo boxes
            const bool is_dy = warp == 0;
            const int n_dy = p.nb_a;
            const uint32_t my_bytes = is_dy ? (uint32_t)(n_dy * p.nr * p.Wp) * dy_row
                                            : nb_b * (uint32_t)((p.nr + p.lo_span) * p.Wp) * x_row;
            int n = u_beg / p.RB, rb = u_beg - n * p.RB;
            int s = 0, ph = 0, issued = 0;
            grid_dependency_wait();
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, p.status, 4)) break;
                const uint32_t bar = smem_u32(&ctl->full[s]);
                const uint32_t a_dst = data_base + (uint32_t)s * stage_bytes, b_dst = a_dst + a_bytes;
                mbar_arrive_expect_tx(bar, my_bytes);
                const int p0 = rb * p.nr;
                if (is_dy) {
                    for (int b = 0; b < n_dy; ++b) tma_load_4d(a_dst + (uint32_t)b * p.a_box, &tmDy, bar, b * 64, 0, p0, n);
                } else {
                    for (uint32_t b = 0; b < nb_b; ++b)
                        tma_load_4d(b_dst + b * p.b_box, &tmX, bar, c0 + (int)b * 64, p.lo_w, p0 + p.lo_h, n);
                }
                if (++rb == p.RB) { rb = 0; ++n; }
                issued = it + 1;
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) drain_ring(smem_u32(&ctl->full[0]), p.stages, issued);
        }
        __syncwarp();
    }
    if (warp == 1 || (warp >= 6 && issuer < NI)) {
        // ---------------- MMA issuer `issuer`: the warp walks the loop in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, p.acc_cols, 1, 1);
        // this issuer's accumulators (at most four: 16 of 32 columns fill the tensor memory): byte offset of the first tap's rows in
        // the x tile and the distance to the next tap's rows
        uint32_t tap_shift[4] = {0u, 0u, 0u, 0u}, tap_lbo[4] = {x_row, x_row, x_row, x_row};
        int n_mine = 0;
        for (int a = issuer; a < n_acc && n_mine < 4; a += NI, ++n_mine) {
            const int t0 = wgrad_tap(p, acc0 + a, 0), r0 = t0 / p.S, sh0 = r0 * p.Wp + (t0 - r0 * p.S);
            tap_shift[n_mine] = (uint32_t)sh0 * x_row;
            if (p.lanes == 64 && t0 + 1 < p.taps) {                   // (an odd last tap: the upper 64 lanes are not stored)
                const int r1 = (t0 + 1) / p.S;
                tap_lbo[n_mine] = (uint32_t)(r1 * p.Wp + (t0 + 1 - r1 * p.S) - sh0) * x_row;
            }
        }
        const uint64_t x_step = x_row, dy_step = dy_row;              // 16 pixels further on, in units of 16 bytes
        bool ok = true;
        int s = 0, ph = 0;
        for (int it = 0; it < iters && ok; ++it) {
            ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status, 5);
            if (!ok) break;
            if (it == 0 && warp == 1) WTRACE(1);
            tc_fence_after();
            const uint32_t a_src = data_base + (uint32_t)s * stage_bytes, b_src = a_src + a_bytes;
            const uint64_t dyd = make_desc_mn(a_src, p.a_box, dy_row);
            const uint32_t acc = it != 0 ? 1u : 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= n_mine) break;
                const uint64_t xd = make_desc_mn(b_src + tap_shift[j], tap_lbo[j], x_row);
                const uint32_t d_tmem = tmem_base + (uint32_t)((issuer + j * NI) * p.acc_cols);
                umma_bf16_lead(d_tmem, xd, dyd, idesc, acc, leader);
                for (int k = 1; k < p.ksteps; ++k) umma_bf16_lead(d_tmem, xd + x_step * k, dyd + dy_step * k, idesc, 1u, leader);
            }
            umma_commit_lead(smem_u32(&ctl->empty[s]), leader);
            if (++s == p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit_lead(smem_u32(&ctl->accum), leader);
        if (warp == 1) WTRACE(2);
    }
    wgrad_finish<true, true>(p, ctl, data_base, tmem_base, acc0, k0, c0, split, iters, p.data_bytes, n_acc, p.acc_cols);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// Filter-row form of the weight gradient: filters of several columns at stride 1 (where the row-block form does not apply: more than 64
// input channels) or 2. A CTA has one filter row: a unit is `nr` output rows of one image, dy as a box of nr x Wp pixels (columns past Q
// and rows past P zero-filled) and the x rows that filter row reads, as a box of the same size; at stride 2 the columns of either parity
// are a box each (every other pixel: a tensor map of its own). The taps of the row are the same staged pixels one pixel apart, read
// through descriptors that start that many 128-byte rows further on, and have an accumulator each. Against the generic kernel, which loads a
// 64-pixel x tile per tap and reloads dy for every two taps or so: 33 KB instead of 72 KB per 64 pixels and three taps at stride 1
// (106 -> 103 channels, 48 against 72 at stride 2). What an SM can pull from L2, 130 to 140 GB/s, bounded that kernel; this one's matrix
// instructions (N = 112: 60 cycles) take as long as its loads.
struct TapMaps { CUtensorMap m[4]; };        // x: [row parity * 2 + column parity]; at stride 1 the first only

__global__ void __launch_bounds__(kThreads, 1) conv_wgrad_taps_kernel(const __grid_constant__ CUtensorMap tmDy, const __grid_constant__ TapMaps tmX, const __grid_constant__ WgradP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Ctl *ctl = reinterpret_cast<Ctl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t data_base = (smem_base + (uint32_t)sizeof(Ctl) + 1023u) & ~1023u;
    const uint32_t nb_b = (uint32_t)((p.BN + 63) / 64), x_boxes = (uint32_t)p.planes * nb_b;
    const uint32_t a_bytes = (uint32_t)p.nb_a * p.a_box, stage_bytes = a_bytes + x_boxes * p.b_box;
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int bx = blockIdx.x;
    const int n_tile = bx % p.n_tiles; bx /= p.n_tiles;
    const int m_tile = bx % p.m_tiles; bx /= p.m_tiles;
    const int r = bx;                                                 // this CTA's filter row
    const int split = blockIdx.y;
    const int k0 = m_tile * 128, c0 = n_tile * p.BN;
    const int u_beg = split * p.units_per_split;
    const int u_end = min(p.units, u_beg + p.units_per_split);
    const int iters = u_end > u_beg ? u_end - u_beg : 0;
    const uint32_t box_bytes = (uint32_t)(p.nr * p.Wp) * 128u;
    // blocks of 64 channels that exist: what an accumulator's other rows and columns hold is not stored, so they are not loaded
    const int n_dy = min(p.nb_a, pt_ceil_div_dev(p.K - k0, 64)), n_xb = min((int)nb_b, pt_ceil_div_dev(p.C - c0, 64)), n_x = p.planes * n_xb;
    const int NXP = n_x < 4 ? n_x : 4;                                // x producer warps in use
    const int NI = p.S < 4 ? p.S : 4;                                 // MMA issuer warps in use: taps i, i + NI, ... of the row

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1u + (uint32_t)NXP);
            mbar_init(smem_u32(&ctl->empty[s]), (uint32_t)NI);
        }
        mbar_init(smem_u32(&ctl->accum), (uint32_t)NI);
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmDy);
        prefetch_tmap(&tmX.m[p.row_par[r] * 2]);
        if (p.planes > 1) prefetch_tmap(&tmX.m[p.row_par[r] * 2 + 1]);
    }
    // rows past the end of a box, up to the last 16-pixel step and the largest shift: dy zeros, x times zero and must be finite
    {
        const uint32_t a_rest = (p.a_box - box_bytes) / 16u, b_rest = (p.b_box - box_bytes) / 16u;
        const uint32_t a_all = (uint32_t)p.nb_a * a_rest, per_stage = a_all + x_boxes * b_rest;
        for (uint32_t i = threadIdx.x; i < (uint32_t)p.stages * per_stage; i += kThreads) {
            const uint32_t st = i / per_stage, o = i - st * per_stage;
            const uint32_t at = o < a_all ? o / a_rest * p.a_box + o % a_rest * 16u : a_bytes + (o - a_all) / b_rest * p.b_box + (o - a_all) % b_rest * 16u;
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(data_base + st * stage_bytes + at + box_bytes), "r"(0u) : "memory");
        }
    }
    fence_proxy_async();
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int issuer = warp == 1 ? 0 : warp - 5;                      // warps 6, 7, 8 -> issuers 1, 2, 3
    // nothing above touches global memory; the producer threads wait after their set-up
    if (!((warp == 0 || (warp >= 2 && warp < 2 + NXP)) && lane == 0)) grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x == 0) WTRACE(0);

    if (warp == 0 || (warp >= 2 && warp < 2 + NXP)) {
        if (lane == 0) {
            // ---------------- producers: warp 0 brings the dy boxes of every unit, warp 2 + j the x boxes j, j + 4, ...
            const bool is_dy = warp == 0;
            const int xp = warp - 2;
            const uint32_t my_bytes = (uint32_t)(is_dy ? n_dy : (n_x - xp + 3) / 4) * box_bytes;
            const int row0 = p.row_off[r];
            int n = u_beg / p.RB, rb = u_beg - n * p.RB;
            int s = 0, ph = 0, issued = 0;
            grid_dependency_wait();
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, p.status, 4)) break;
                const uint32_t bar = smem_u32(&ctl->full[s]);
                const uint32_t a_dst = data_base + (uint32_t)s * stage_bytes, b_dst = a_dst + a_bytes;
                mbar_arrive_expect_tx(bar, my_bytes);
                const int p0 = rb * p.nr;
                if (is_dy) {
                    for (int b = 0; b < n_dy; ++b) tma_load_4d(a_dst + (uint32_t)b * p.a_box, &tmDy, bar, k0 + b * 64, 0, p0, n);
                } else {
                    for (int j = xp; j < n_x; j += 4) {
                        const int pl = j >= n_xb ? 1 : 0, b = j - pl * n_xb;
                        tma_load_4d(b_dst + ((uint32_t)pl * nb_b + (uint32_t)b) * p.b_box, &tmX.m[p.row_par[r] * 2 + pl], bar, c0 + b * 64, p.plane_lo[pl],
                                    p0 + row0, n);
                    }
                }
                if (++rb == p.RB) { rb = 0; ++n; }
                issued = it + 1;
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) drain_ring(smem_u32(&ctl->full[0]), p.stages, issued);
        }
        __syncwarp();
    }
    if (warp == 1 || (warp >= 6 && issuer < NI)) {
        // ---------------- MMA issuer `issuer`: the warp walks the loop in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, p.BN, 1, 1);
        bool ok = true;
        int s = 0, ph = 0;
        for (int it = 0; it < iters && ok; ++it) {
            ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status, 5);
            if (!ok) break;
            if (it == 0 && warp == 1) WTRACE(1);
            tc_fence_after();
            const uint32_t a_src = data_base + (uint32_t)s * stage_bytes, b_src = a_src + a_bytes;
            const uint64_t ad = make_desc(a_src, p.a_box, 1024u);
            const uint32_t acc = it != 0 ? 1u : 0u;
            for (int t = issuer; t < p.S; t += NI) {
                const uint64_t bd = make_desc(b_src + (uint32_t)p.tap_plane[t] * nb_b * p.b_box + (uint32_t)p.tap_shift[t] * 128u, p.b_box, 1024u);
                const uint32_t d_tmem = tmem_base + (uint32_t)(t * p.BN);
                umma_bf16_lead(d_tmem, ad, bd, idesc, acc, leader);
                for (int k = 1; k < p.ksteps; ++k) umma_bf16_lead(d_tmem, ad + 128ull * k, bd + 128ull * k, idesc, 1u, leader);
            }
            umma_commit_lead(smem_u32(&ctl->empty[s]), leader);
            if (++s == p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit_lead(smem_u32(&ctl->accum), leader);
        if (warp == 1) WTRACE(2);
    }
    wgrad_finish<true, false>(p, ctl, data_base, tmem_base, r * p.S, k0, c0, split, iters, p.data_bytes, p.S, p.BN);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// Packed form of the weight gradient: stride-1 filters of several columns whose pixels are 16 or 32 channels apart on both sides. G = 4 (or
// 2) neighbouring pixels make one 128-byte row, pad lanes and all (they only reach sums that are not stored), so that the reduction runs
// over rows of G pixels and a matrix instruction does 16 G pixels: with x rows of pixels G j .. and the row of the next G pixels on its M
// side (2 G x 64 / G lanes) and G pixels of dy on its N side, the sums of the tap s are the blocks (pixel a + s of x, pixel a of dy),
// a = 0 .. G - 1; the other blocks are dropped and these added when the splits are. A unit is `nr` such columns of an image, each a box of
// 64 elements x all rows of the image (and the R - 1 that the filter reaches over, zeros on the dy side), column behind column, so that the
// filter rows are row shifts with an accumulator each and the next G pixels are one column (`Wp` rows) on. Against the row-block form at
// 32x32, 8 -> 14 channels: 17 x 3 instructions per image instead of 68 x 3, and half as many
// staged rows: with 48 CTAs 22.3 -> 13.2 us at batch 128, alone 16.6 -> 11.3; 19 -> 19 at 56x56, batch 256 80.8 -> 53.1 and 37.2 -> 29.9. What is
// left there is the exchange (the dropped blocks are not stored, but the G pixels are G sources each) and a box per column, 0.2 us a thread.
__global__ void __launch_bounds__(kThreads, 1) conv_wgrad_packed_kernel(const __grid_constant__ CUtensorMap tmDy,
                                                                     const __grid_constant__ CUtensorMap tmX, const __grid_constant__ WgradP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Ctl *ctl = reinterpret_cast<Ctl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t data_base = (smem_base + (uint32_t)sizeof(Ctl) + 1023u) & ~1023u;
    const uint32_t a_bytes = (uint32_t)p.nb_a * p.a_box, stage_bytes = a_bytes + p.b_box;
    volatile int *abort_flag = &ctl->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.y, G = p.G, R = p.taps / p.S;
    const int u_beg = split * p.units_per_split, u_end = min(p.units, u_beg + p.units_per_split);
    const int iters = u_end > u_beg ? u_end - u_beg : 0;
    const uint32_t dy_row = (uint32_t)p.dy_lanes * 2u;                // bytes of a staged row of dy: 128, or 64 (two pixels of 16 channels)
    const uint32_t x_col = (uint32_t)p.Wp * 128u, dy_col = (uint32_t)p.Wp * dy_row;
    const int boxes = p.nr + 1 + p.nr * p.nb_a, NP = boxes < 5 ? boxes : 5;          // of a unit; producer warps 0, 2, 3, 4, 5
    const int NI = R < 4 ? R : 4;                                     // MMA issuer warps in use: filter rows i, i + NI, ...

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), (uint32_t)NP);
            mbar_init(smem_u32(&ctl->empty[s]), (uint32_t)NI);
        }
        mbar_init(smem_u32(&ctl->accum), (uint32_t)NI);
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmDy);
        prefetch_tmap(&tmX);
    }
    // rows past the last column, up to the last 16-row step and the largest shift: dy zeros, x times zero and must be finite
    {
        const uint32_t a_used = (uint32_t)p.nr * dy_col, b_used = (uint32_t)(p.nr + 1) * x_col;
        const uint32_t a_rest = (p.a_box - a_used) / 16u, b_rest = (p.b_box - b_used) / 16u, a_all = (uint32_t)p.nb_a * a_rest, per_stage = a_all + b_rest;
        for (uint32_t i = threadIdx.x; i < (uint32_t)p.stages * per_stage; i += kThreads) {
            const uint32_t st = i / per_stage, o = i - st * per_stage;
            const uint32_t at = o < a_all ? o / a_rest * p.a_box + a_used + o % a_rest * 16u : a_bytes + b_used + (o - a_all) * 16u;
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(data_base + st * stage_bytes + at), "r"(0u) : "memory");
        }
    }
    fence_proxy_async();
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int issuer = warp == 1 ? 0 : warp - 5;                      // warps 6, 7, 8 -> issuers 1, 2, 3
    const int pid = warp == 0 ? 0 : warp >= 2 && warp <= 5 ? warp - 1 : 5;
    // nothing above touches global memory; the producer threads wait after their set-up
    if (!(pid < NP && lane == 0)) grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x == 0) WTRACE(0);

    if (pid < NP) {
        if (lane == 0) {
            // ---------------- producers: the boxes pid, pid + NP, ... of every unit: nr + 1 columns of x, then nr of each dy block
            uint32_t my_bytes = 0;
            for (int b = pid; b < boxes; b += NP) my_bytes += b <= p.nr ? x_col : dy_col;
            const int x_step = G * p.lanes, dy_px = G * p.row_lanes;       // elements from one column to the next
            int n = u_beg / p.RB, rb = u_beg - n * p.RB;
            int s = 0, ph = 0, issued = 0;
            grid_dependency_wait();
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1, abort_flag, p.status, 4)) break;
                const uint32_t bar = smem_u32(&ctl->full[s]);
                const uint32_t a_dst = data_base + (uint32_t)s * stage_bytes, b_dst = a_dst + a_bytes;
                mbar_arrive_expect_tx(bar, my_bytes);
                const int j0 = rb * p.nr;
                for (int b = pid; b < boxes; b += NP) {
                    if (b <= p.nr) {
                        tma_load_3d(b_dst + (uint32_t)b * x_col, &tmX, bar, (j0 + b) * x_step + p.lo_w * p.lanes, p.lo_h, n);
                    } else {
                        int j = b - p.nr - 1, blk = 0;
                        if (j >= p.nr) { j -= p.nr; blk = 1; }
                        tma_load_3d(a_dst + (uint32_t)blk * p.a_box + (uint32_t)j * dy_col, &tmDy, bar, (j0 + j) * dy_px + blk * 64, 0, n);
                    }
                }
                if (++rb == p.RB) { rb = 0; ++n; }
                issued = it + 1;
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (*abort_flag) drain_ring(smem_u32(&ctl->full[0]), p.stages, issued);
        }
        __syncwarp();
    }
    if (warp == 1 || (warp >= 6 && issuer < NI)) {
        // ---------------- MMA issuer `issuer`: the warp walks the loop in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, p.acc_cols, 1, 1);
        const uint64_t dy_step = dy_row;                              // 16 rows further on, in units of 16 bytes
        bool ok = true;
        int s = 0, ph = 0;
        for (int it = 0; it < iters && ok; ++it) {
            ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status, 5);
            if (!ok) break;
            if (it == 0 && warp == 1) WTRACE(1);
            tc_fence_after();
            const uint32_t a_src = data_base + (uint32_t)s * stage_bytes, b_src = a_src + a_bytes;
            const uint64_t dyd = make_desc_mn(a_src, p.a_box, dy_row);
            const uint32_t acc = it != 0 ? 1u : 0u;
            for (int r = issuer; r < R; r += NI) {
                const uint64_t xd = make_desc_mn(b_src + (uint32_t)r * 128u, x_col, 128u);
                const uint32_t d_tmem = tmem_base + (uint32_t)(r * p.acc_cols);
                umma_bf16_lead(d_tmem, xd, dyd, idesc, acc, leader);
                for (int k = 1; k < p.ksteps; ++k) umma_bf16_lead(d_tmem, xd + 128ull * k, dyd + dy_step * k, idesc, 1u, leader);
            }
            umma_commit_lead(smem_u32(&ctl->empty[s]), leader);
            if (++s == p.stages) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit_lead(smem_u32(&ctl->accum), leader);
        if (warp == 1) WTRACE(2);
    }

    // ---------------- the sums: every split leaves G sources, one per pixel of dy in a row, of 16-byte pieces [filter row][four output
    // channels][tap column, input channel]; then each sums its share over the sources of all splits (as wgrad_finish does)
    const int KQ = pt_ceil_div_dev(p.K, 4), SC = p.S * p.C, total = R * KQ * SC;
    float4 *const part = reinterpret_cast<float4 *>(p.partial);
    if (warp >= 1) {
        const int quarter = warp & 3, wset = (warp >= 2 && warp < 6) ? 0 : 1;
        bool ok = true;
        if (iters > 0) ok = mbar_wait(smem_u32(&ctl->accum), 0, abort_flag, p.status, 6);
        if (warp == 2) WTRACE(3);
        tc_fence_after();
        if (ok) {
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
            const int l = quarter * 32 + lane, px = l >> p.lane_shift, c = l & (p.lanes - 1);
            // (all of a row's loads before the one wait: a load and its wait take 0.2 us, and there are up to 24)
            const bool here = c < p.C;
            int ci = 0;
            for (int r = 0; r < R; ++r)
                for (int h = 0; h < p.K; h += 16, ++ci) {
                    if ((ci & 1) != wset) continue;
                    uint32_t v[4][16];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
                        if (a < G && iters > 0) tmem_ld16(lane_addr + (uint32_t)(r * p.acc_cols + a * p.row_lanes + h), v[a]);
                    tmem_ld_wait();
                    float4 *const d4 = part + (size_t)(split * G) * total + (size_t)(r * KQ + (h >> 2)) * SC + c;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const int t = px - a;
                        if (a >= G || t < 0 || t >= p.S || !here) continue;
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if ((h >> 2) + j < KQ)
                                __stcg(d4 + (size_t)a * total + (size_t)j * SC + t * p.C,
                                       iters > 0 ? make_float4(__uint_as_float(v[a][4 * j]), __uint_as_float(v[a][4 * j + 1]), __uint_as_float(v[a][4 * j + 2]),
                                                               __uint_as_float(v[a][4 * j + 3]))
                                                 : make_float4(0.f, 0.f, 0.f, 0.f));
                    }
                }
        }
        if (warp == 2) WTRACE(4);
        named_barrier(1, 256);
        if (warp == 1 && lane == 0) wgrad_arrive(p, split, abort_flag);
        named_barrier(1, 256);
        if (warp == 2) WTRACE(5);
        tc_fence_before();
    }
    __syncthreads();
    if (!*abort_flag) {
        const int Z = p.splits * G, per_cta = (total + p.splits - 1) / p.splits;
        const int it_beg = split * per_cta, it_end = min(total, it_beg + per_cta);
        const int cap = wgrad_chunk(p.data_bytes, Z);
        const float inv_sc = 1.0f / (float)SC, inv_kq = 1.0f / (float)KQ;
        for (int c_beg = it_beg; c_beg < it_end; c_beg += cap) {
            const int n_chunk = min(cap, it_end - c_beg);
            wgrad_bring(data_base, part + c_beg, (size_t)total, Z, n_chunk);
            const int ls = wgrad_sum_lanes(n_chunk, Z);
            for (int i = threadIdx.x; i < (((n_chunk << ls) + 31) & ~31); i += kThreads) {
                const int k = i >> ls;
                const float4 sum = wgrad_sum(data_base, k, n_chunk, Z, ls);
                const bool mine = k < n_chunk && !(i & ((1 << ls) - 1));
                const int piece = c_beg + k, rq = fast_div(piece, SC, inv_sc), sc = piece - rq * SC, r = fast_div(rq, KQ, inv_kq), kk = (rq - r * KQ) * 4;
                const float v4[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (mine && kk + e < p.K) p.out[((size_t)(kk + e) * p.taps + r * p.S) * p.C + sc] = v4[e];      // (taps of a row side by side)
                if (__any_sync(0xffffffffu, mine && wgrad_nan(sum, p.K - kk)))
                    wgrad_pure(p.raw, p.out, mine && wgrad_nan(sum, p.K - kk), kk, 1, r * p.S + sc / p.C, sc % p.C, 0);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) WTRACE(6);
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------ few-channel stride-2 stem
// A stride-2 convolution over very few input channels (the 7x7 / 3-channel network stem) is rewritten as a stride-1
// convolution over a space-to-depth copy of the input: xs[n][i][j + pl][(a,b,c)] = x[n][2i+a][2j+b][c], 16 bf16 per pixel,
// with pl zero columns on the left and V-1-pl on the right. Consecutive pixels of a row are contiguous, so the V
// horizontal taps x 16 lanes of one output position are ONE run of 64 elements: the tensor map below gives every output
// column its own 128-byte row (overlapping windows, 32-byte stride), and the conv becomes U vertical taps of 64
// "channels" each -- full swizzle rows for TMA and UMMA instead of 49 taps of 3 channels.
//   h = 2p - pad + r = 2(p - pl) + t,  t = r + off,  off = 2*pl - pad,  u = t / 2, a = t % 2   (same for columns)
struct StemPlan {
    int ok;
    int pl, off, U, V, Hs, Ws, Wp, P, Q;
    size_t xs_bytes, w2_elems;     // padded space-to-depth input; weights / weight gradient as [K][U][64]
};

StemPlan stem_plan(const pt_conv_desc *d)
{
    StemPlan s;
    memset(&s, 0, sizeof(s));
    if (d->stride != 2 || d->C > 4 || (d->H & 1) || (d->W & 1) || d->R != d->S || d->ldx != 8) return s;
    s.pl = (d->pad + 1) / 2;
    s.off = 2 * s.pl - d->pad;
    s.U = (d->R - 1 + s.off) / 2 + 1;
    s.V = s.U;
    if (s.V > 4) return s;
    s.Hs = d->H / 2; s.Ws = d->W / 2;
    s.Wp = s.Ws + 3;                        // every window is 4 pixels wide whatever V is: pl zero columns left, 3 - pl right
    s.P = pt_out_dim(d->H, d->R, 2, d->pad);
    s.Q = pt_out_dim(d->W, d->S, 2, d->pad);
    if (s.Q > s.Ws || s.P > s.Hs + s.pl) return s;
    s.xs_bytes = pt_align_up((size_t)d->N * s.Hs * s.Wp * 32, 1024);
    s.w2_elems = (size_t)d->K * s.U * 64;
    s.ok = 1;
    return s;
}

// Forward pass of a few-channel stride-2 stem straight from the image (U >= 2; 64 to 125 output columns, at most 128 channels, bf16 out).
// A CTA has a run of consecutive output rows. Two teams of four warps turn each pair of image rows into one space-to-depth row in shared
// memory (every one of them once: the next output row needs one new one of its U), in a ring of rows of 32-byte positions with the
// swizzle of that width; an output row is then U x V matrix instructions on those rows (tap (u, v) starts at row u, v positions on) with the
// weights, laid out once per CTA, resident. Four issuers take output rows in turn (one needs 1.6 us for the 16 instructions, waits and
// commits of a row; two issuers 54.7 us for the launch), a group of epilogue warps every other one.
// Through a space-to-depth copy in memory it was two launches more (11 and 2 us at batch 64) and four staged rows per output row: 3 -> 55
// 7x7/2 at 224x224, batch 64 53.7 -> 37.5 us, 3 -> 19 at batch 256 153 -> 110. Bound by the matrix instructions' reads of shared memory
// (6 KB each, 16 a row: 0.4 us of the 0.6 to 0.7 a row takes) and by the stores.
constexpr int kStemAhead = 3;                                     // rows a converting thread has on their way (2 and 3: 38.8 and 37.5 us)
constexpr int kStemRing = 16, kStemSlot = 4352;                     // rows in the ring (a power of two); bytes of one: up to 131 positions of 32
constexpr int kStemIssuers = 4, kStemThreads = (kStemIssuers + 16) * 32;        // issuers, eight epilogue warps, two teams of four converting warps

struct StemP {
    int N, H, W, C, K, R, S, ldw;
    int P, Q, Hs, Ws, Wp, pl, off, U, V;
    int BN, rows, rows_per_cta;         // output rows in all (N * P) and of a CTA
    int tmem_cols, acc_per;
    int stats_off, stats_warp, stats_lo, ld_out;
    float *stats;
    const __nv_bfloat16 *x, *w;
    unsigned int *status;
    int test_skip;                      // test hook (pt_test_skip_next_arrive)
};

struct __align__(8) StemCtl {
    uint64_t full[kStemRing], empty[kStemRing];
    uint64_t acc_full[2 * kStemIssuers], acc_empty[2 * kStemIssuers];
    uint32_t tmem_base;
    int abort_flag;
};

// The output rows of a CTA image by image: first row, number of rows, position of the first space-to-depth row in the CTA's sequence.
struct StemWalk {
    int n, p0, len, q0, left;
    __device__ __forceinline__ void init(const StemP &p)
    {
        const int g0 = (int)blockIdx.x * p.rows_per_cta;
        left = min(p.rows_per_cta, p.rows - g0);
        n = g0 / p.P; p0 = g0 - n * p.P;
        len = min(left, p.P - p0); q0 = 0;
    }
    __device__ __forceinline__ void next(const StemP &p)
    {
        left -= len; q0 += len + p.U - 1;
        ++n; p0 = 0; len = min(left, p.P);
    }
};

// One position of a space-to-depth row: the four channels of four pixels of the image, zeros outside (i: the row, jp: the position), and
// the 16 lanes they make, pixel by pixel. (Plain loads: the kernel is on the SM before its predecessor, which may be writing the image, has
// ended; the read-only path is for what nothing writes while the kernel runs.)
__device__ __forceinline__ void stem_load(const StemP &p, int n, int i, int jp, uint2 (&px)[4])
{
    const int j = jp - p.pl;
    const bool in = i >= 0 && i < p.Hs && j >= 0 && j < p.Ws;
#pragma unroll
    for (int ab = 0; ab < 4; ++ab)
        px[ab] = in ? *reinterpret_cast<const uint2 *>(p.x + ((size_t)(n * p.H + 2 * i + (ab >> 1)) * p.W + 2 * j + (ab & 1)) * 8) : make_uint2(0, 0);
}
__device__ __forceinline__ void stem_pack(int C, const uint2 (&px)[4], uint4 &lo, uint4 &hi)
{
    hi = make_uint4(0, 0, 0, 0);
    if (C == 3) {
        lo = make_uint4(px[0].x, (px[0].y & 0xffffu) | (px[1].x << 16), (px[1].x >> 16) | (px[1].y << 16), px[2].x);
        hi.x = (px[2].y & 0xffffu) | (px[3].x << 16);
        hi.y = (px[3].x >> 16) | (px[3].y << 16);
    } else if (C == 4) {
        lo = make_uint4(px[0].x, px[0].y, px[1].x, px[1].y);
        hi = make_uint4(px[2].x, px[2].y, px[3].x, px[3].y);
    } else if (C == 2) {
        lo = make_uint4(px[0].x, px[1].x, px[2].x, px[3].x);
    } else {
        lo = make_uint4((px[0].x & 0xffffu) | (px[1].x << 16), (px[2].x & 0xffffu) | (px[3].x << 16), 0u, 0u);
    }
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

template <bool STATS>
__global__ void __launch_bounds__(kStemThreads, 1) conv_stem_kernel(const __grid_constant__ CUtensorMap tmC, const StemP p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    StemCtl *ctl = reinterpret_cast<StemCtl *>(smem_raw);
    const uint32_t smem_base = smem_u32(smem_raw);
    const uint32_t staging_base = (smem_base + (uint32_t)sizeof(StemCtl) + 1023u) & ~1023u;
    const uint32_t ring_base = staging_base + 8u * kSlabs * 4096u, w_base = ring_base + (uint32_t)(kStemRing * kStemSlot);
    const uint32_t w_tile = (uint32_t)p.BN * 32u;
    volatile int *abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStemRing; ++s) { mbar_init(smem_u32(&ctl->full[s]), 4); mbar_init(smem_u32(&ctl->empty[s]), kStemIssuers); }
        for (int b = 0; b < 2 * kStemIssuers; ++b) { mbar_init(smem_u32(&ctl->acc_full[b]), 1); mbar_init(smem_u32(&ctl->acc_empty[b]), 4); }
        ctl->abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmC);
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&ctl->tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (warp < kStemIssuers + 8) {
        // The weights as [tap (u, v)][output channel][16 lanes], K-major rows of 32 bytes, laid out like the positions: lane (a*2+b)*C + c
        // is filter position (2u + a - off, 2v + b - off), zeros outside the filter and past K. The converting warps are at work on the
        // image meanwhile. (Weights are not written by a kernel that releases its dependents early.)
        const unsigned short *w = reinterpret_cast<const unsigned short *>(p.w);
        for (int i = threadIdx.x; i < p.U * p.V * p.BN; i += (kStemIssuers + 8) * 32) {
            const int t = i / p.BN, k = i - t * p.BN, u = t / p.V, v = t - u * p.V;
            uint2 px[4];
#pragma unroll
            for (int ab = 0; ab < 4; ++ab) {
                const int r = 2 * u + (ab >> 1) - p.off, s = 2 * v + (ab & 1) - p.off;
                px[ab] = k < p.K && r >= 0 && r < p.R && s >= 0 && s < p.S ? __ldg(reinterpret_cast<const uint2 *>(w + ((size_t)(k * p.R + r) * p.S + s) * p.ldw))
                                                                           : make_uint2(0, 0);
            }
            uint4 lo, hi;
            stem_pack(p.C, px, lo, hi);
            const uint32_t row = w_base + (uint32_t)t * w_tile + (uint32_t)k * 32u, x = (row >> 3) & 16u;
            st_shared_v4(row + x, lo);
            st_shared_v4(row + (16u ^ x), hi);
        }
        fence_proxy_async();
        named_barrier(2, (kStemIssuers + 8) * 32);
        grid_dependency_wait();                                       // (the converting warps wait before their first load)
    }
    grid_launch_dependents();
    StemWalk sw;
    sw.init(p);

    if (warp < kStemIssuers) {
        // ---------------- MMA issuers: output rows warp, warp + kStemIssuers, ... of the CTA; the warp walks the loop in lockstep, lane 0 issues
        const uint32_t leader = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, p.BN, 0, 0);
        const uint64_t desc0 = make_desc_rows(0u, 32u);
        bool ok = true;
        int nt = 0, row0 = 0;                                        // rows this issuer has started; the segment's first row in the CTA's count
        for (; sw.left > 0 && ok; row0 += sw.len, sw.next(p)) {
            int rel = sw.q0;                                         // ring rows of the segment that this issuer has released
            const int end = sw.q0 + sw.len + p.U - 1;
            for (int l = (warp - row0) & (kStemIssuers - 1); l < sw.len && ok; l += kStemIssuers, ++nt) {
                const int b = p.acc_per == 2 ? warp * 2 + (nt & 1) : warp, aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1;
                ok = mbar_wait(smem_u32(&ctl->acc_empty[b]), aph ^ 1, abort_flag, p.status, 60);
                // (either team of converting warps fills its ring rows in order: behind the last two all are there)
                for (int q = sw.q0 + l + p.U - 2; q < sw.q0 + l + p.U && ok; ++q)
                    ok = mbar_wait(smem_u32(&ctl->full[q & (kStemRing - 1)]), (q / kStemRing) & 1, abort_flag, p.status, 61);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(b * p.BN);
                uint64_t bd = desc0 | desc_addr(w_base);
                const uint64_t b_step = w_tile >> 4;
                for (int u = 0; u < p.U; ++u) {
                    const uint64_t ad = desc0 | desc_addr(ring_base + (uint32_t)((sw.q0 + l + u) & (kStemRing - 1)) * kStemSlot);
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        if (v < p.V) umma_bf16_lead(d_tmem, ad + 2ull * v, bd + b_step * v, idesc, v == 0 ? (u ? 1u : 0u) : 1u, leader);
                    bd += b_step * p.V;
                }
                umma_commit_lead(smem_u32(&ctl->acc_full[b]), leader);
                // ring rows that this issuer needs no more: up to its next output row's first one, behind its last one all (those that
                // it never reads once they are there: an arrival belongs to the row's own turn in the ring)
                const int upto = l + kStemIssuers < sw.len ? sw.q0 + l + kStemIssuers : end;
                for (; rel < upto && ok; ++rel) {
                    const uint32_t bar = smem_u32(&ctl->empty[rel & (kStemRing - 1)]);
                    if (rel < sw.q0 + l + p.U) umma_commit_lead(bar, leader);
                    else {
                        ok = mbar_wait(smem_u32(&ctl->full[rel & (kStemRing - 1)]), (rel / kStemRing) & 1, abort_flag, p.status, 62);
                        if (ok && lane == 0) mbar_arrive(bar);
                    }
                }
            }
            for (; rel < end && ok; ++rel) {                          // (a segment without a row of this issuer)
                ok = mbar_wait(smem_u32(&ctl->full[rel & (kStemRing - 1)]), (rel / kStemRing) & 1, abort_flag, p.status, 63);
                if (ok && lane == 0) mbar_arrive(smem_u32(&ctl->empty[rel & (kStemRing - 1)]));
            }
        }
    } else if (warp < kStemIssuers + 8) {
        // ---------------- epilogue: group g (four warps) has every other output row
        const int ew = warp - kStemIssuers, quarter = warp & 3, group = ew >> 2;
        const uint32_t slab0 = staging_base + (uint32_t)ew * (kSlabs * 4096u);
        const uint32_t st_acc = smem_base + (uint32_t)p.stats_off + (uint32_t)ew * (uint32_t)p.stats_warp;
        const int n_chunks = (p.BN + 63) / 64;
        if (STATS) {
            stats_clear(st_acc, lane, n_chunks);
            __syncwarp();
        }
        const int valid = p.Q - quarter * 32;                         // pixels of this warp's 32 that exist
        const uint32_t rows = valid >= 32 ? 0xffffffffu : valid > 0 ? (1u << valid) - 1u : 0u;
        bool ok = true;
        int row0 = 0, sl = 0;
        for (; sw.left > 0 && ok; row0 += sw.len, sw.next(p))
            for (int l = (group - row0) & 1; l < sw.len; l += 2) {
                // the nt-th row of issuer `iss`
                const int iss = (row0 + l) & (kStemIssuers - 1), nt = (row0 + l) / kStemIssuers;
                const int b = p.acc_per == 2 ? iss * 2 + (nt & 1) : iss, aph = p.acc_per == 2 ? (nt >> 1) & 1 : nt & 1;
                ok = mbar_wait(smem_u32(&ctl->acc_full[b]), aph, abort_flag, p.status, 64);
                if (!ok) break;
                tc_fence_after();
                const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * p.BN);
                for (int ch = 0; ch < n_chunks; ++ch, sl ^= 1) {
                    const uint32_t slab = slab0 + (uint32_t)sl * 4096u;
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the slab's previous store has read it
                    __syncwarp();
                    const int groups = min(4, (p.BN - ch * 64) / 16);
                    // (with statistics two groups of 16 columns at a time: four of them do not fit the registers of 640 threads beside the sums)
                    constexpr int G = STATS ? 2 : 4;
#pragma unroll
                    for (int g0 = 0; g0 < 4; g0 += G) {
                        if (g0 >= groups) break;
                        uint32_t v[G][16];
#pragma unroll
                        for (int g = 0; g < G; ++g)
                            if (g0 + g < groups) tmem_ld16(lane_addr + (uint32_t)(ch * 64 + (g0 + g) * 16), v[g]);
                        tmem_ld_wait();
                        if (ch + 1 >= n_chunks && g0 + G >= groups) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                        }
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            if (g0 + g >= groups) break;
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                __nv_bfloat162 e[4];
#pragma unroll
                                for (int k = 0; k < 4; ++k) e[k] = __floats2bfloat162_rn(__uint_as_float(v[g][8 * h + 2 * k]), __uint_as_float(v[g][8 * h + 2 * k + 1]));
                                const uint32_t j = (uint32_t)((g0 + g) * 2 + h);
                                st_shared_v4(slab + (uint32_t)lane * 128u + ((j ^ ((uint32_t)lane & 7u)) << 4), *reinterpret_cast<uint4 *>(e));
                            }
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        if (valid > 0) tma_store_4d(&tmC, slab, ch * 64, quarter * 32, sw.p0 + l, sw.n);
                        tma_store_commit();
                    }
                    if (STATS) chunk_stats(slab, 0, rows, lane, st_acc + (uint32_t)ch * 512u);
                }
            }
        if (STATS) {
            named_barrier(1, 256);
            stats_store_cta(smem_base + (uint32_t)p.stats_off, (uint32_t)p.stats_warp, 8, (int)threadIdx.x - kStemIssuers * 32, 256,
                            p.stats + (size_t)blockIdx.x * (1 + p.stats_lo) * 2 * p.ld_out, p.ld_out, p.stats_lo, p.K, 0, p.ld_out);
        }
        if (lane == 0) tma_store_wait_read();                          // the staging slabs must outlive the stores' reads
        tc_fence_before();
    } else {
        // ---------------- converting warps: a team has every other ring row, a thread a position of it; the pixels of the team's next
        // kStemAhead rows are on their way meanwhile
        const int team = (warp - kStemIssuers - 8) >> 2, jp = (int)threadIdx.x - (kStemIssuers + 8 + team * 4) * 32;
        const bool on = jp < p.Wp;
        const uint32_t at = ring_base + (uint32_t)jp * 32u;
        uint2 px[kStemAhead][4];
        int total = 0;
        StemWalk lw = sw;                                              // where the next load is: row li of image lw.n, lrest more of the segment
        int li = lw.p0 - p.pl, lrest = lw.len + p.U - 1;
        for (; sw.left > 0; sw.next(p)) total += sw.len + p.U - 1;
        const auto skip = [&]() {
            ++li;
            if (--lrest == 0) { lw.next(p); li = lw.p0 - p.pl; lrest = lw.len + p.U - 1; }
        };
        const auto load = [&](uint2 (&d)[4]) {
            if (lw.left <= 0) return;
            if (on) stem_load(p, lw.n, li, jp, d);
            skip();
            if (lw.left > 0) skip();
        };
        grid_dependency_wait();
        if (team == 1) skip();
#pragma unroll
        for (int k = 0; k < kStemAhead; ++k) load(px[k]);
        bool ok = true;
        for (int q0 = team; q0 < total && ok; q0 += 2 * kStemAhead) {
#pragma unroll
            for (int k = 0; k < kStemAhead; ++k) {
                const int q = q0 + 2 * k, s = q & (kStemRing - 1);
                if (q >= total || !ok) break;
                ok = mbar_wait(smem_u32(&ctl->empty[s]), ((q / kStemRing) & 1) ^ 1, abort_flag, p.status, 65);
                if (!ok) break;
                if (on) {
                    uint4 lo, hi;
                    stem_pack(p.C, px[k], lo, hi);
                    const uint32_t a = at + (uint32_t)s * kStemSlot, x = (a >> 3) & 16u;
                    st_shared_v4(a + x, lo);
                    st_shared_v4(a + (16u ^ x), hi);
                }
                fence_proxy_async();
                __syncwarp();
                // (test hook: the last ring row of the CTA's first output row never becomes full)
                if (lane == 0 && !(p.test_skip && q == p.U - 1)) mbar_arrive(smem_u32(&ctl->full[s]));
                load(px[k]);
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// CT = channel count as a compile-time constant (1..4): the 16 output lanes are then plain registers
template <int CT>
__global__ void __launch_bounds__(256) stem_s2d_x_kernel_t(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ xs, int N, int H,
                                                           int W, int Hs, int Ws, int Wp, int pl)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)N * Hs * Wp;
    if (idx >= total) return;
    const int jp = (int)(idx % Wp);
    const size_t t = idx / Wp;
    const int i = (int)(t % Hs), n = (int)(t / Hs);
    __align__(16) unsigned short o[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) o[e] = 0;
    const int j = jp - pl;
    if (j >= 0 && j < Ws) {
        uint4 px[4];
#pragma unroll
        for (int ab = 0; ab < 4; ++ab)          // the four loads go out together
            px[ab] = __ldg(reinterpret_cast<const uint4 *>(x + ((size_t)(n * H + 2 * i + (ab >> 1)) * W + 2 * j + (ab & 1)) * 8));
#pragma unroll
        for (int ab = 0; ab < 4; ++ab) {
            const unsigned short *pe = reinterpret_cast<const unsigned short *>(&px[ab]);
#pragma unroll
            for (int c = 0; c < CT; ++c) o[ab * CT + c] = pe[c];
        }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(xs + idx * 16);
    dst[0] = *reinterpret_cast<uint4 *>(&o[0]);
    dst[1] = *reinterpret_cast<uint4 *>(&o[8]);
}

// (Launched plainly: a dependency wait in each of the thousands of blocks costs more than an earlier start saves, 142 -> 159 us for the
// weight gradient of 3 -> 19 at batch 256.)
void stem_s2d_x_kernel_launch(unsigned blocks, cudaStream_t st, const __nv_bfloat16 *x, __nv_bfloat16 *xs, int N, int H, int W, int C,
                              int Hs, int Ws, int Wp, int pl)
{
    switch (C) {
    case 1: stem_s2d_x_kernel_t<1><<<blocks, 256, 0, st>>>(x, xs, N, H, W, Hs, Ws, Wp, pl); break;
    case 2: stem_s2d_x_kernel_t<2><<<blocks, 256, 0, st>>>(x, xs, N, H, W, Hs, Ws, Wp, pl); break;
    case 3: stem_s2d_x_kernel_t<3><<<blocks, 256, 0, st>>>(x, xs, N, H, W, Hs, Ws, Wp, pl); break;
    default: stem_s2d_x_kernel_t<4><<<blocks, 256, 0, st>>>(x, xs, N, H, W, Hs, Ws, Wp, pl); break;
    }
}

// w2[k][u][v*16 + (a*2+b)*C + c] = w[k][2u+a-off][2v+b-off][c]  (0 where the tap falls outside the filter)
__global__ void stem_s2d_w_kernel(const __nv_bfloat16 *__restrict__ w, __nv_bfloat16 *__restrict__ w2, int K, int R, int S, int C,
                                  int ldw, int U, int V, int off)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= K * U * 64) return;
    const int l = idx & 63, u = (idx >> 6) % U, k = (idx >> 6) / U;
    const int v = l >> 4, e = l & 15;
    float val = 0.f;
    if (v < V && e < 4 * C) {
        const int ab = e / C, c = e - ab * C, a = ab >> 1, b = ab & 1;
        const int r = 2 * u + a - off, s = 2 * v + b - off;
        if (r >= 0 && r < R && s >= 0 && s < S) val = __bfloat162float(w[((size_t)(k * R + r) * S + s) * ldw + c]);
    }
    w2[idx] = __float2bfloat16_rn(val);
}

// dw[k][r][s][c] = dw2[k][u][v*16 + (a*2+b)*C + c] with (u,a) from r + off and (v,b) from s + off
__global__ void stem_dw_back_kernel(const float *__restrict__ dw2, float *__restrict__ dw, int K, int R, int S, int C, int U, int off)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= K * R * S * C) return;
    const int c = idx % C;
    int t = idx / C;
    const int s = t % S; t /= S;
    const int r = t % R, k = t / R;
    const int tr = r + off, ts = s + off;
    dw[idx] = dw2[((size_t)k * U + (tr >> 1)) * 64 + (ts >> 1) * 16 + ((tr & 1) * 2 + (ts & 1)) * C + c];
}

// ------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                   const int *, const int *, cuuint32_t, cuuint32_t, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

CUtensorMapSwizzle lanes_swizzle(int lanes)
{
    return lanes == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : lanes == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}

// bf16 tensor (C, W, H, N) with channel pitch ld: im2col map loading `pixels` x `lanes` channels.
bool make_im2col_map(const pt_ctx *c, CUtensorMap *tm, const void *base, int C, int W, int H, int N, int ld, int lo_w, int lo_h,
                     int up_w, int up_h, int stride, int pixels, int row_pixels = 0, int lanes = kKC)
{
    if (!c->encode_im2col) return false;
    if (lo_w < -128 || lo_h < -128 || up_w < -128 || up_h < -128 || lo_w > 127 || lo_h > 127 || up_w > 127 || up_h > 127) return false;
    const int rowp = row_pixels ? row_pixels : W;        // pixels between two image rows in memory (>= W)
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)ld * 2, (cuuint64_t)rowp * ld * 2, (cuuint64_t)H * rowp * ld * 2};
    int lo[2] = {lo_w, lo_h}, up[2] = {up_w, up_h};
    cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
    CUresult r = ((EncodeIm2colFn)c->encode_im2col)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, lo,
                                                    up, (cuuint32_t)lanes, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                    lanes_swizzle(lanes), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// bf16 activations as a plain 2-D tensor (channels, pixels) with row pitch ld: box 64 channels x `pixels`.
bool make_act2d_map(const pt_ctx *c, CUtensorMap *tm, const void *base, int C, long long npix, int ld, int pixels, int lanes = kKC)
{
    if (!c->encode_tiled) return false;
    cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)npix};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)lanes, (cuuint32_t)pixels}, estr[2] = {1, 1};
    CUresult r = ((CUresult(*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                               const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill))c->encode_tiled)(
        tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
        lanes_swizzle(lanes), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// bf16 weight shadow as (C, R*S, K) with row pitch ldw: box (lanes, 1, box_k).
bool make_weight_map(const pt_ctx *c, CUtensorMap *tm, const void *base, int C, int RS, int K, int ldw, int box_k, int lanes = kKC)
{
    if (!c->encode_tiled) return false;
    cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)RS, (cuuint64_t)K};
    cuuint64_t strides[2] = {(cuuint64_t)ldw * 2, (cuuint64_t)RS * ldw * 2};
    cuuint32_t box[3] = {(cuuint32_t)lanes, 1, (cuuint32_t)box_k};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = ((EncodeTiledFn)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box,
                                                  estr, CU_TENSOR_MAP_INTERLEAVE_NONE, lanes_swizzle(lanes),
                                                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// Tile width along the output channels. One tile: the ragged count rounded up to 16. Several tiles: a multiple of
// 64 (the TMA-store chunk) chosen to waste the fewest padded columns.
int tile_n(int cols, int *n_tiles, int m_tiles = 1 << 30, int sms = 0)
{
    int best = 256;
    if (cols <= 256) {
        *n_tiles = 1;
        best = pt_ceil_div(cols, 16) * 16;
    } else {
        int best_pad = 1 << 30;
        for (int bn = 256; bn >= 128; bn -= 64) {
            int pad = pt_ceil_div(cols, bn) * bn;
            if (pad < best_pad) { best_pad = pad; best = bn; }
        }
        *n_tiles = pt_ceil_div(cols, best);
    }
    if (sms <= 0 || m_tiles >= sms) return best;
    // Few pixel tiles (the 7x7 maps): a CTA's time is what it streams per reduction stage -- the 16 KB activation tile plus
    // bn x 128 bytes of weights -- times the waves of tiles. Narrower channel tiles put more SMs to work and cut the weight
    // bytes per CTA; the activation tile is then read by more CTAs, from L2. Taken when the estimate drops by 10 % or more.
    long long cost0 = (long long)pt_ceil_div(m_tiles * *n_tiles, sms) * (16 * 1024 + (long long)pt_ceil_div(best, 64) * 8192);
    for (int bn = 192; bn >= 64; bn -= 64) {
        if (bn >= best) continue;
        const int nt = pt_ceil_div(cols, bn);
        const long long cost = (long long)pt_ceil_div(m_tiles * nt, sms) * (16 * 1024 + (long long)bn * 128);
        if (cost * 10 <= cost0 * 9) { cost0 = cost; best = bn; *n_tiles = nt; }
    }
    return best;
}

int pow2_cols(int bn)
{
    int c = 32;
    while (c < bn) c <<= 1;
    return c;
}

// Pipeline depth for a kernel that owns the SM: as many stages as fit beside `reserved` bytes, at most kMaxStages.
// The GEMM-form kernel may take all but 1 KB of the 227 KB a CTA can have (one more stage for the wide 1x1 layers).
constexpr size_t kGemmSmemCap = (size_t)226 * 1024;
int pick_stages(size_t stage_bytes, int iters, size_t reserved, size_t *smem, size_t cap = (size_t)220 * 1024)
{
    int st = (int)((cap - 2048 - reserved) / stage_bytes);
    if (st > kMaxStages) st = kMaxStages;
    if (st > iters && iters >= 2) st = iters;
    if (st < 2) st = 2;
    *smem = 2048 + reserved + (size_t)st * stage_bytes;
    return st;
}

// bf16 output viewed as (channels, pixels) with row pitch ld: box 64 channels x 32 pixels, 128-byte swizzle.
// Channel extent of an output tensor map: the channel count rounded up to a whole 32-byte sector where the pitch has room
// for it (the pad lanes there receive zeros). A row whose last sector is only partly written costs a read-modify-write in
// the memory system: measured 35 us against 20 us for 56x56x209..216 channels at pitch 224.
// The operands of a weight gradient are loaded with the same extent: their channels are rows and columns of the result, so that whatever
// a pad lane holds (a NaN too) stays in sums that are not stored, and the TMA unit's time for a row that ends inside a box depends on
// where (ns per row with several issuing threads, box of 64 lanes: 64 channels 0.73, 57 to 63 1.03, 48 to 56 1.4 to 1.5, 41 to 47 1.6,
// 33 to 40 3.4; of 32 lanes: 32 0.53, 25 to 31 1.0, 17 to 24 1.5). Weight gradients of 106 -> 103 3x3 at 28x28, batch 64 27.2 -> 24.1 us,
// at 56x56 and stride 2 28.3 -> 25.2; 30 -> 33 at 56x56 22.8 -> 20.8; the 7x7 stem 3 -> 19, batch 256 156.9 -> 145.3.
int store_cols(int cols, int ld)
{
    const int up = pt_ceil_div(cols, 16) * 16;
    return up <= ld ? up : cols;
}

bool make_out_map(const pt_ctx *c, CUtensorMap *tm, void *base, int cols, int rows, int ld)
{
    cuuint64_t dims[2] = {(cuuint64_t)store_cols(cols, ld), (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, 32}, estr[2] = {1, 1};
    CUresult r = ((EncodeTiledFn)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// Tensor maps of a GEMM-form launch: activation tiles (of 64 lanes, and of the last chunk's) and weight tiles.
struct GemmMaps { CUtensorMap a, tail, b; };

// Lanes the last chunk of `c` reduction channels is staged with: the TMA unit's time is per row, and longer where a box is wider than
// what the tensor has left (128 rows of 13 of 64 lanes 0.62 us, of 16 lanes 0.48; 19 of 64 0.81, of 32 0.62).
int gemm_tail_lanes(int c)
{
    const int rem = c - (pt_ceil_div(c, kKC) - 1) * kKC;
    return rem <= 16 ? 16 : rem <= 32 ? 32 : 64;
}

template <bool B_MN>
pt_status launch_gemm(pt_ctx *c, const GemmMaps &tm, GemmP &p, cudaStream_t st)
{
    CUtensorMap tmC;
    memset(&tmC, 0, sizeof(tmC));
    p.tma_store = (!p.out_f32 && p.o_step == 1 && p.zero_mask == 0) ? 1 : 0;
    const bool apart = !p.out_f32 && !p.tma_store;
    if (apart && !B_MN) return PT_ERR_UNSUPPORTED;
    if (p.tma_store && !make_out_map(c, &tmC, p.out, p.n_cols, p.M_total, p.ld_out)) return PT_ERR_CUDA;
    const size_t a_bytes = kBM * kKC * 2;
    const size_t b_bytes = B_MN ? (size_t)pt_ceil_div(p.BN, 64) * 8192 : pt_align_up((size_t)p.BN * 128, 1024);
    size_t smem = 0;
    p.m_tiles = pt_ceil_div(p.M_total, kBM);
    const int total_tiles = p.m_tiles * p.n_tiles;
    const int per_cta = pt_ceil_div(total_tiles, c->sm_count);
    // accumulator buffers = epilogue groups: three when 3 * BN fits the 512 TMEM columns, else two; narrow layers whose
    // CTAs get a single tile need no more than that
    p.epi_groups = 3 * p.BN <= 512 ? 3 : 2;
    if (p.zero_mask) p.epi_groups = 2;                            // (the warps of the third write the zeros)
    if (per_cta < p.epi_groups) p.epi_groups = per_cta;           // a single tile per CTA: one group, and its staging goes to the ring
    // Small weights (one channel tile, all taps x chunks within 64 KB) stay resident: the ring then carries A tiles only and
    // holds more of them, which is what an activation-bound layer needs to cover the memory latency.
    const size_t w_all = (size_t)p.taps * p.k_chunks * b_bytes;
    p.resident = (p.n_tiles == 1 && w_all <= 64 * 1024 && per_cta >= 2) ? 1 : 0;
    p.n_issuers = 1; p.acc_per = 1;
    if (p.resident && per_cta >= 4 && 2 * p.BN <= 512) {
        // narrow tiles are bound by what one thread can issue: two issuer warps, two epilogue groups
        p.n_issuers = 2;
        p.epi_groups = 2;
        p.acc_per = 4 * p.BN <= 512 ? 2 : 1;
    }
    // one tile per CTA and streamed weights: the output is staged in the ring (all of its stages have been consumed when the
    // accumulator is complete), which leaves room for one more stage
    p.alias_staging = (per_cta == 1 && !p.resident) ? 1 : 0;
    // statistics mode: the epilogue warps' accumulators sit at the end of the shared memory (taken from the ring's room)
    p.stats_warp = pt_ceil_div(p.BN, 64) * (int)kStatsChunkBytes;
    const size_t st_smem = c->stats_mode ? (size_t)4 * p.epi_groups * p.stats_warp : 0;     // (the group count can only shrink below)
    size_t staging2 = p.alias_staging ? 0 : (size_t)p.epi_groups * 4 * kSlabs * 4096;
    if (p.resident) p.stages = pick_stages(a_bytes, p.taps * p.k_chunks * per_cta, staging2 + w_all + st_smem, &smem, kGemmSmemCap);
    else {
        p.stages = pick_stages(a_bytes + b_bytes, p.taps * p.k_chunks * per_cta, staging2 + st_smem, &smem, kGemmSmemCap);
        if (p.stages < 4 && p.epi_groups == 3 && p.taps * p.k_chunks * per_cta >= 4) {
            // a third epilogue group costs 32 KB of staging: with wide weight tiles that is the fourth pipeline stage
            p.epi_groups = 2;
            staging2 = (size_t)p.epi_groups * 4 * kSlabs * 4096;
            p.stages = pick_stages(a_bytes + b_bytes, p.taps * p.k_chunks * per_cta, staging2 + st_smem, &smem, kGemmSmemCap);
        }
    }
    p.stats_off = (int)(smem - st_smem);
    if (p.n_issuers == 2) {
        p.stages = p.stages / 2 * 2;
        if (p.stages < 2) { p.n_issuers = 1; p.acc_per = 1; p.stages = 2; }
    }
    p.n_a = (p.n_issuers == 2 && p.taps * p.k_chunks >= 2) ? 2 : 1;
    p.n_b = (B_MN && !p.resident && p.BN > 64) ? 2 : 1;
    p.vec_cols = pt_ceil_div(p.n_cols, 16) * 16 <= p.ld_out ? pt_ceil_div(p.n_cols, 16) * 16 : pt_ceil_div(p.n_cols, 8) * 8;
    p.tail_lanes = gemm_tail_lanes(p.c_red);
    p.tmem_cols = pow2_cols((p.n_issuers == 2 ? 2 * p.acc_per : p.epi_groups) * p.BN);
    // the statistics variant exists for the forward kernel only
    void (*kernel)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, GemmP) =
        (!B_MN && c->stats_mode) ? conv_gemm_kernel<false, true, false> : apart ? conv_gemm_kernel<true, false, true> : conv_gemm_kernel<B_MN, false, false>;
    const int kid = (!B_MN && c->stats_mode) ? 2 : apart ? 3 : (B_MN ? 1 : 0);
    if (!(c->attr_done & (kAttrGemm << kid))) {
        PT_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        c->attr_done |= kAttrGemm << kid;
    }
    int grid = total_tiles < c->sm_count ? total_tiles : c->sm_count;
    if (c->stats_mode) {
        if (!p.tma_store) return PT_ERR_UNSUPPORTED;
        if (grid > p.n_tiles) grid = grid / p.n_tiles * p.n_tiles;     // every CTA keeps one channel tile
        p.stats_lo = grid / p.n_tiles < kStatsFewRows ? 1 : 0;
        c->stats_parts = grid / p.n_tiles * (1 + p.stats_lo);
        if ((size_t)c->stats_parts * 2 * p.ld_out * sizeof(float) > c->stats_cap) return PT_ERR_WORKSPACE;
        p.stats = c->stats_out;
    }
    if (c->test_skip == 2) { p.test_skip = 1; c->test_skip = 0; }
    PT_CUDA_OK(pt_launch_pdl(kernel, dim3((unsigned)grid), dim3(kGemmThreads), smem, st, tm.a, tm.tail, tm.b, tmC, p));
    c->launches += 1;
    c->last_form = PT_FORM_GEMM;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Source activations as a tiled 4-D tensor (C, W, H, N): box 64 channels x box_w x box_h x 1 (the halo tile).
// `lanes` = 64, 32 or 16 (128-, 64- or 32-byte rows and swizzle).
// `row_pixels` > 0: pixels between the starts of consecutive rows when that is not W (a padded row).
bool make_halo_in_map(const pt_ctx *c, CUtensorMap *tm, const void *base, int C, int W, int H, int N, int ld, int box_w, int box_h,
                      int lanes = kKC, int row_pixels = 0)
{
    if (!c->encode_tiled || box_w > 256 || box_h > 256) return false;
    const cuuint64_t rp = row_pixels > 0 ? (cuuint64_t)row_pixels : (cuuint64_t)W;
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)ld * 2, rp * ld * 2, (cuuint64_t)H * rp * ld * 2};
    cuuint32_t box[4] = {(cuuint32_t)lanes, (cuuint32_t)box_w, (cuuint32_t)box_h, 1}, estr[4] = {1, 1, 1, 1};
    CUresult r = ((EncodeTiledFn)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box,
                                                  estr, CU_TENSOR_MAP_INTERLEAVE_NONE, lanes_swizzle(lanes),
                                                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// The pixels (a + i * stride, b + j * stride) of bf16 activations as a tiled 4-D tensor (C, columns j, rows i, N): box 64 channels x box_w x
// box_h x 1.
bool make_plane_map(const pt_ctx *c, CUtensorMap *tm, const void *base, int C, int W, int H, int N, int ld, int stride, int a, int b, int box_w, int box_h,
                    int lanes = kKC)
{
    if (!c->encode_tiled || box_w > 256 || box_h > 256 || a >= H || b >= W) return false;
    const char *first = (const char *)base + ((size_t)a * W + b) * ld * 2;
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)pt_ceil_div(W - b, stride), (cuuint64_t)pt_ceil_div(H - a, stride), (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)stride * ld * 2, (cuuint64_t)stride * W * ld * 2, (cuuint64_t)H * W * ld * 2};
    cuuint32_t box[4] = {(cuuint32_t)lanes, (cuuint32_t)box_w, (cuuint32_t)box_h, 1}, estr[4] = {1, 1, 1, 1};
    CUresult r = ((EncodeTiledFn)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<char *>(first), dims, strides, box, estr,
                                                  CU_TENSOR_MAP_INTERLEAVE_NONE, lanes_swizzle(lanes), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return map_ok(r, __LINE__);
}

// One launch of the halo kernel: a stride-1 correlation of `src` with a list of taps, written to a (possibly strided)
// view of the output.
struct HaloSpec {
    const void *src; int Cs, Ws, Hs, lds;            // activations read: channels, width, height, pitch
    int P, Q;                                        // output raster per image (rows, columns)
    int n_taps, span_h, span_w;                      // taps and the extent of their offsets (max offset + 1)
    int lo_h, lo_w;                                  // source coordinate of raster (0,0) at tap offset (0,0)
    int tap_oh[kMaxTaps], tap_ow[kMaxTaps], tap_wt[kMaxTaps];
    int n_cols, ld_out;                              // output channels and pitch
    int oH, oW, o_step, o_h0, o_w0;                  // output view: raster (i, j) -> pixel (i*o_step + o_h0, j*o_step + o_w0) of oH x oW
    int row32, w_taps;                               // 16-lane pixels (32-byte rows); taps per output channel in the weight tensor
    int plane_tap[5], plane_lo_h[4], plane_lo_w[4];  // stride-2 forward: the taps in the order of their parity planes, and where those start
    int max_ctas;                                    // > 0: grid limit (launches meant to run side by side share the SMs)
};

// Whether the parity planes pay, given a launch's rings: against the im2col form they have four boxes a chunk to wait for, whole raster rows in
// tiles of 128, and weights that stream once per round of tiles where they are not resident. By the times of 480 random stride-2 layers (5 to
// 400 channels, 2x2 to 5x5 filters, forward alone and with statistics; planes and im2col):
//   a tap to a plane (2x2): rows of at most 32 lanes (17 -> 149 at 14x14, batch 478 16 and 25 us; 151 -> 94 at 17x17, batch 117 25 and 13);
//   resident weights: always, but not with single stages for two issuers and more than two chunks (315 -> 32 at 27x27, batch 102 96 and 65) or, two
//     chunks or more a stage, in tiles that hold few output pixels (170 -> 7 at 13x13, batch 445 45 and 31; 159 -> 19 at 27x27 22 and 30);
//   streamed weights: rounds of tiles of which 55 % is work (354 -> 51 at 28x28, batch 12 58 and 41; 365 -> 190 at 28x28, batch 65 73 and 86), fewer
//     with up to two chunks (94 -> 82 at 8x8 19 and 16; 52 -> 177 at 28x22 17 and 21); one issuer with many taps only (64 -> 209 at 27x27,
//     batch 64 22 and 17; 41 -> 192 5x5 123 and 155); several channel tiles with narrow rows of one chunk only (83 -> 305 at 16x16 84 and 62; 17 ->
//     352 at 28x16 21 and 28).
// The layers take 0.71 of the im2col form's time by this rule, 0.74 without it and 0.71 by the faster of the two each.
bool planes_pay(const pt_ctx *c, const HaloP &p, int taps)
{
    const double useful = (double)p.P * p.Q / (p.row_tiles * 128.0), slot = (double)p.N * p.row_tiles * p.n_tiles / c->sm_count / p.n_issuers;
    const bool busy = useful * slot >= 0.55 * ceil(slot);
    const int per = p.stages_a / p.n_issuers;
    if (taps <= 4) return p.lanes < 64 && p.resident && (p.n_issuers == 4 || busy);
    if (p.resident) {
        if (taps >= 16 || per >= 2) return true;
        if (p.n_issuers == 2 && p.k_chunks > 2) return false;
        return useful >= 0.72 || p.k_chunks * (p.n_issuers == 2 ? 2 : 1) <= 2;
    }
    if (p.n_tiles > 1) return p.k_chunks == 1 && p.lanes < 64 && busy;
    if (p.n_issuers == 1) return taps >= 16 && busy;
    return busy || (p.k_chunks <= 2 && (taps >= 16 || useful >= 0.6));
}

template <bool B_MN, int PL = 1>
pt_status launch_halo(pt_ctx *c, const pt_conv_desc *d, const HaloSpec &h, const void *w, void *out, cudaStream_t st)
{
    const int Wp = h.Q + h.span_w - 1;
    if (h.n_taps < 1 || h.n_taps > kMaxTaps || Wp > 128 || (PL == 1 && h.Ws > 250)) return PT_ERR_UNSUPPORTED;
    HaloP p;
    memset(&p, 0, sizeof(p));
    p.N = d->N; p.P = h.P; p.Q = h.Q; p.Wp = Wp;
    p.nr = 128 / Wp < h.P ? 128 / Wp : h.P;
    p.row_tiles = pt_ceil_div(h.P, p.nr);
    p.n_cols = h.n_cols;
    p.BN = tile_n(h.n_cols, &p.n_tiles);
    // The planes pay where a CTA has several tiles, so that the boxes of one are on their way while another's are multiplied; with one or two
    // the im2col form's many small loads are sooner there (3x3/2, planes against im2col: 106 -> 103 at 56x56, batch 64, 448 tiles 23.6 and 25.7 us,
    // 38 -> 38 at 56x56, batch 256 33.7 and 48.5, 8 -> 17 at 32x32, batch 128, 384 tiles 6.4 and 10.6; 64 -> 128 at 32x32, batch 64, 192
    // tiles 11.1 and 7.9; 200 -> 200 at 28x28, batch 64, 128 tiles 23.4 and 19.6).
    if (PL > 1 && c->test_form != PT_FORM_PLANES && (long long)p.N * p.row_tiles * p.n_tiles <= 2 * c->sm_count) return PT_ERR_UNSUPPORTED;
    p.c_red = h.Cs; p.k_chunks = pt_ceil_div(h.Cs, kKC); p.taps = h.n_taps;
    // Channel lanes per staged pixel: narrow layers take rows of 64 or 32 bytes. The TMA unit's time is per row, and a row whose tensor
    // ends in the middle of a sector costs it twice as much in a 128-byte box (4.5 ns for 19 channels) as a whole one (2.3 ns); in a
    // box of the next width 3.1 ns. The rows also take less shared memory.
    p.lanes = h.Cs <= 16 ? 16 : h.Cs <= 32 ? 32 : 64;
    const int row_bytes = p.lanes * 2;
    if (h.row32 && (B_MN || h.Cs != 16)) return PT_ERR_UNSUPPORTED;
    p.lo_h = h.lo_h; p.lo_w = h.lo_w;
    for (int t = 0; t < h.n_taps; ++t) {
        p.tap_oh[t] = (unsigned char)h.tap_oh[t]; p.tap_ow[t] = (unsigned char)h.tap_ow[t];
        p.tap_wt[t] = (unsigned short)h.tap_wt[t];
    }
    const int box_h = p.nr + h.span_h - 1;
    if (box_h > 256) return PT_ERR_UNSUPPORTED;
    p.a_box_bytes = box_h * Wp * row_bytes;
    // The M = 128 MMAs of the last tap read up to this many rows; the rows past the box only feed raster positions that
    // are never stored, so consecutive A stages may overlap there (and a tail pad follows the last stage).
    const int need_rows = 128 + (h.span_h - 1) * Wp + h.span_w - 1;
    p.a_alloc = (int)pt_align_up((size_t)p.a_box_bytes, 1024);
    const size_t a_tail = need_rows * row_bytes > p.a_alloc ? pt_align_up((size_t)need_rows * row_bytes - p.a_alloc, 1024) : 0;
    // a K-major weight box brings the output channels that exist rounded up to 16 (the rows past the count are zero-filled
    // by the TMA unit): exactly the columns the output map covers, so the pad lanes it writes are zeros; the MMA may still
    // read up to BN rows, the rest from whatever follows in shared memory: columns that are never stored
    p.b_rows = p.BN < h.n_cols ? p.BN : pt_ceil_div(h.n_cols, 16) * 16;
    if (p.b_rows > p.BN) p.b_rows = p.BN;
    const size_t b_bytes = B_MN ? (size_t)pt_ceil_div(p.BN, 64) * p.lanes * 128 : (size_t)p.b_rows * row_bytes;
    p.b_slot = (int)b_bytes;
    // narrow outputs are stored from registers (the 16-byte vectors of a pixel must be whole: room in the pitch)
    p.direct_cols = pt_ceil_div(h.n_cols, 16) * 16 <= h.ld_out ? pt_ceil_div(h.n_cols, 16) * 16 : pt_ceil_div(h.n_cols, 8) * 8;
    const size_t w_all = (size_t)h.n_taps * p.k_chunks * b_bytes;
    // The rings of a launch, for outputs in fp32 or bf16, with statistics or without; false where they do not fit.
    const auto rings = [&](HaloP &p, bool f32, bool stats) {
        p.direct = (!f32 && !stats && p.n_tiles == 1 && p.BN <= 32) ? 1 : 0;
        // epilogue staging: a slab of the tile's raster rows x 128 bytes per group, two where the launch's other needs leave room (direct-store
        // launches use none)
        p.tma_store = (f32 || p.direct) ? 0 : 1;
        p.staging = !p.tma_store ? 0 : (int)pt_align_up((size_t)(p.nr * Wp < 128 ? p.nr * Wp : 128) * 128, 1024);
        p.slabs = 1;
        p.stats_warp = pt_ceil_div(p.BN, 64) * (int)kStatsChunkBytes;
        const size_t st_smem = stats ? (size_t)8 * p.stats_warp : 0;             // statistics accumulators of the eight epilogue warps
        const size_t budget = 227 * 1024 - 2048 - 2 * (size_t)p.staging - a_tail - st_smem;
        p.resident = (p.n_tiles == 1 && w_all + 2 * (size_t)p.a_alloc <= budget) ? 1 : 0;
        size_t left = budget - (p.resident ? w_all : 0);
        bool two_pipes = false;
        if (!p.resident) {
            // ring: at least two A stages, the rest for weight stages (at least 3)
            p.stages_a = 2;
            if (left < 2 * (size_t)p.a_alloc + 3 * b_bytes) return false;
            size_t sb = (left - 2 * (size_t)p.a_alloc) / b_bytes;
            p.stages_b = sb > kMaxStages ? kMaxStages : (int)sb;
            // two pipelines (one per tile parity) when each can have three weight stages and the CTAs get several tiles
            // (a launch that shares the SMs with others has fewer CTAs, each with more tiles)
            const int ctas_avail = (h.max_ctas > 0 && h.max_ctas < c->sm_count) ? h.max_ctas : c->sm_count;
            two_pipes = p.stages_b >= 6 && pt_ceil_div(p.N * p.row_tiles * p.n_tiles, ctas_avail) >= 2;
            if (two_pipes) p.stages_b = p.stages_b / 2 * 2;
            // Two pipelines on one weight stream (a single channel tile): every chunk of both tiles should have an activation stage
            // of its own -- a chunk that waits for the previous chunk's MMAs to free its stage exposes a DRAM round trip per tile
            // (28x28, 69 -> 93 channels, MN-major weights: two stages against four, 30 -> 22 us) -- as long as four weight stages
            // remain for the shared stream.
            const int want_a = 2 * p.k_chunks * PL > 4 ? 4 : 2 * p.k_chunks * PL;
            if (two_pipes && p.n_tiles == 1 && left >= (size_t)want_a * p.a_alloc + 4 * b_bytes) {
                const size_t sb2 = (left - (size_t)want_a * p.a_alloc) / b_bytes;
                if ((size_t)p.stages_b > sb2) p.stages_b = (int)sb2;
            }
            left -= (size_t)p.stages_b * b_bytes;
            int sa = (int)(left / p.a_alloc);
            p.stages_a = sa > 4 ? 4 : sa;
        } else {
            // (one stage per issuer leaves its load latency exposed on every tile: 19 -> 19 at 56x56, batch 256, 46 us with 4 stages, 36 with 8)
            int sa = (int)(left / p.a_alloc);
            p.stages_a = sa > kHaloMaxA ? kHaloMaxA : sa;
            p.stages_b = 1;
        }
        if (p.stages_a < 2) return false;
        if (p.tma_store && p.resident && left >= kHaloMaxA * (size_t)p.a_alloc + 2 * (size_t)p.staging) p.slabs = 2;
        // issuer warps: several only with resident weights; each needs an A stage of its own and an accumulator buffer
        p.n_issuers = 1;
        p.acc_per = 2;
        if (p.resident) {
            p.n_issuers = (p.stages_a >= 4 && 4 * p.BN <= 512) ? 4 : 2;
            p.acc_per = p.n_issuers * 2 * p.BN <= 512 ? 2 : 1;
        } else if (two_pipes) {
            p.n_issuers = 2;
            p.acc_per = 4 * p.BN <= 512 ? 2 : 1;
            p.shared_b = p.n_tiles == 1 ? 1 : 0;          // the tiles of a round then use the same weight columns
        }
        p.stages_a = p.stages_a / p.n_issuers * p.n_issuers;
        return true;
    };
    // (planes or not by the rings of the plain bf16 output, so that the same sums leave in every form: with statistics, in fp32)
    if (PL > 1 && c->test_form != PT_FORM_PLANES) {
        HaloP q = p;
        if (!rings(q, false, false) || !planes_pay(c, q, h.n_taps)) return PT_ERR_UNSUPPORTED;
    }
    if (!rings(p, d->out_f32 != 0, c->stats_mode != 0)) return PT_ERR_UNSUPPORTED;
    p.tmem_cols = pow2_cols(p.n_issuers * p.acc_per * p.BN);
    p.out = out; p.ld_out = h.ld_out; p.out_f32 = d->out_f32;
    p.oH = h.oH; p.oW = h.oW; p.o_step = h.o_step; p.o_h0 = h.o_h0; p.o_w0 = h.o_w0;
    p.status = c->d_status;
    HaloMaps<PL> tmA;
    if constexpr (PL > 1) {
        memcpy(tmA.tap, h.plane_tap, sizeof(tmA.tap));
        memcpy(tmA.lo_h, h.plane_lo_h, sizeof(tmA.lo_h));
        memcpy(tmA.lo_w, h.plane_lo_w, sizeof(tmA.lo_w));
    }
    CUtensorMap tmB, tmC;
    memset(&tmC, 0, sizeof(tmC));
    if (h.row32) {
        if (!p.resident) return PT_ERR_UNSUPPORTED;
        if (!make_halo_in_map(c, &tmA.m[0], h.src, h.Cs, h.Ws, h.Hs, d->N, h.lds, Wp, box_h, 16)) return PT_ERR_CUDA;
        // weights [K][w_taps][16]: one 32-byte row per output channel and tap
        cuuint64_t dims[3] = {16, (cuuint64_t)h.w_taps, (cuuint64_t)h.n_cols};
        cuuint64_t strides[2] = {32, (cuuint64_t)h.w_taps * 32};
        cuuint32_t box[3] = {16, 1, (cuuint32_t)p.b_rows}, estr[3] = {1, 1, 1};
        CUresult r = ((EncodeTiledFn)c->encode_tiled)(&tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(w), dims, strides, box,
                                                      estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                                                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (!map_ok(r, __LINE__)) return PT_ERR_CUDA;
    } else {
        for (int i = 0; i < PL; ++i)
            if (PL == 1 ? !make_halo_in_map(c, &tmA.m[0], h.src, h.Cs, h.Ws, h.Hs, d->N, h.lds, Wp, box_h, p.lanes)
                        : !make_plane_map(c, &tmA.m[i], h.src, h.Cs, h.Ws, h.Hs, d->N, h.lds, 2, i >> 1, i & 1, Wp, box_h, p.lanes)) return PT_ERR_CUDA;
        if (!make_weight_map(c, &tmB, w, d->C, d->R * d->S, d->K, d->ldw, B_MN ? p.lanes : p.b_rows, B_MN ? kKC : p.lanes)) return PT_ERR_CUDA;
    }
    if (p.tma_store) {
        // the output view as a 4-D tensor (channels, raster columns, raster rows, images); strided when o_step > 1
        const size_t es = 2;
        char *base = (char *)out + ((size_t)h.o_h0 * h.oW + h.o_w0) * h.ld_out * es;
        cuuint64_t dims[4] = {(cuuint64_t)store_cols(h.n_cols, h.ld_out), (cuuint64_t)h.Q, (cuuint64_t)h.P, (cuuint64_t)d->N};
        cuuint64_t strides[3] = {(cuuint64_t)h.o_step * h.ld_out * es, (cuuint64_t)h.o_step * h.oW * h.ld_out * es,
                                 (cuuint64_t)h.oH * h.oW * h.ld_out * es};
        cuuint32_t box[4] = {64, (cuuint32_t)Wp, (cuuint32_t)p.nr, 1}, estr[4] = {1, 1, 1, 1};
        CUresult r = ((EncodeTiledFn)c->encode_tiled)(&tmC, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                      CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (!map_ok(r, __LINE__)) return PT_ERR_CUDA;
    }
    const size_t st_smem = c->stats_mode ? (size_t)8 * p.stats_warp : 0;
    const size_t smem = 2048 + 2 * (size_t)p.slabs * p.staging + (p.resident ? w_all : (size_t)p.stages_b * b_bytes) + (size_t)p.stages_a * p.a_alloc + a_tail +
                        st_smem;
    p.stats_off = (int)(smem - st_smem);
    void (*kernel)(HaloMaps<PL>, CUtensorMap, CUtensorMap, HaloP) =
        (!B_MN && c->stats_mode) ? conv_halo_kernel<false, true, PL> : conv_halo_kernel<B_MN, false, PL>;
    const unsigned attr = PL > 1 ? kAttrPlanes << (c->stats_mode ? 1 : 0) : kAttrHalo << ((!B_MN && c->stats_mode) ? 2 : (B_MN ? 1 : 0));
    if (!(c->attr_done & attr)) {
        PT_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        c->attr_done |= attr;
    }
    const int total_tiles = p.N * p.row_tiles * p.n_tiles;
    int grid = total_tiles < c->sm_count ? total_tiles : c->sm_count;
    if (p.resident && p.k_chunks == 1 && total_tiles > c->sm_count / 2 && total_tiles <= 4 * (c->sm_count * 2 / 3)) {
        // Few short tiles: two to four per CTA on half to two thirds of the SMs. The launch is mostly its start and its drain; on the SMs it
        // leaves free the next kernel's CTAs run their set-up meanwhile (one CTA fills an SM), and a kernel of another stream finds room.
        // 54 -> 35 at 8x8, batch 128: 5.6 -> 4.7 us a launch, data gradient 6.4 -> 5.0; 21 -> 24 at 16x16 6.45 -> 6.1; with five
        // to ten tiles per CTA instead of three to seven it would be 0.6 to 1 us longer.
        const int want = c->sm_count * 2 / 3, rounds = total_tiles <= 2 * want ? 2 : pt_ceil_div(total_tiles, want);
        grid = pt_ceil_div(total_tiles, rounds);
    }
    // (the parities of a stride-2 data gradient share the SMs among themselves)
    if (B_MN && h.o_step == 1 && c->dgrad_ctas > 0 && grid > c->dgrad_ctas) grid = c->dgrad_ctas;
    if (h.max_ctas > 0 && grid > h.max_ctas) grid = h.max_ctas;
    if (c->stats_mode) {
        if (!p.tma_store || B_MN) return PT_ERR_UNSUPPORTED;
        if (grid > p.n_tiles) grid = grid / p.n_tiles * p.n_tiles;     // every CTA keeps one channel tile
        p.stats_lo = grid / p.n_tiles < kStatsFewRows ? 1 : 0;
        c->stats_parts = grid / p.n_tiles * (1 + p.stats_lo);
        if ((size_t)c->stats_parts * 2 * p.ld_out * sizeof(float) > c->stats_cap) return PT_ERR_WORKSPACE;
        p.stats = c->stats_out;
    }
    if (c->test_skip == 5) { p.test_skip = 1; c->test_skip = 0; }
    PT_CUDA_OK(pt_launch_pdl(kernel, dim3((unsigned)grid), dim3(kHaloThreads), smem, st, tmA, tmB, tmC, p));
    c->launches += 1;
    c->last_form = PL > 1 ? PT_FORM_PLANES : PT_FORM_HALO;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Stride-1 RxS forward (flip = false, src = x) or data gradient (flip = true, src = dy, padding R-1-pad).
void halo_spec_stride1(const pt_conv_desc *d, HaloSpec *h, const void *src, int Cs, int Ws, int Hs, int lds, int n_cols, int P, int Q,
                       int ld_out, int pad_h, int pad_w, bool flip)
{
    memset(h, 0, sizeof(*h));
    h->src = src; h->Cs = Cs; h->Ws = Ws; h->Hs = Hs; h->lds = lds;
    h->P = P; h->Q = Q; h->n_taps = d->R * d->S; h->span_h = d->R; h->span_w = d->S;
    h->lo_h = -pad_h; h->lo_w = -pad_w;
    for (int t = 0; t < h->n_taps && t < kMaxTaps; ++t) {
        h->tap_oh[t] = t / d->S; h->tap_ow[t] = t % d->S;
        h->tap_wt[t] = flip ? h->n_taps - 1 - t : t;
    }
    h->n_cols = n_cols; h->ld_out = ld_out;
    h->oH = P; h->oW = Q; h->o_step = 1; h->o_h0 = 0; h->o_w0 = 0;
}

// A CTA of a split weight gradient holds its tensor memory while it waits for the other splits of its tile. Two such CTAs
// on one SM could block each other's tensor-memory allocation (the second allocation waits for columns the first one
// frees only after a CTA that cannot start has arrived), so a split launch asks for more than half of an SM's shared
// memory: at most one of them per SM, whatever else runs beside it (kernels that wait for nobody always finish).
constexpr size_t kSplitSmemFloor = 116 * 1024;
// The least that a weight gradient has behind its control block: the squares that its epilogue transposes (34 KB) and the sums of the splits reuse
// the stages.
constexpr size_t kWgradSmemMin = 2048 + 8 * 2 * 4096;

// Launches the stem's forward kernel; PT_ERR_UNSUPPORTED where the space-to-depth copy serves the layer.
pt_status run_stem(pt_ctx *c, const pt_conv_desc *d, const StemPlan &sp, const void *x, const void *w, void *y, cudaStream_t st)
{
    // (narrower images would leave most of a row's 128 matrix rows empty; more channels do not fit beside two accumulators an issuer)
    if (d->out_f32 || sp.U < 2 || sp.Q < 64 || sp.Q > 128 || sp.Wp > 128 || sp.Q + sp.V - 1 > 128 + 3 || d->K > 128 || !c->encode_tiled) return PT_ERR_UNSUPPORTED;
    StemP p;
    memset(&p, 0, sizeof(p));
    p.N = d->N; p.H = d->H; p.W = d->W; p.C = d->C; p.K = d->K; p.R = d->R; p.S = d->S; p.ldw = d->ldw;
    p.P = sp.P; p.Q = sp.Q; p.Hs = sp.Hs; p.Ws = sp.Ws; p.Wp = sp.Wp; p.pl = sp.pl; p.off = sp.off; p.U = sp.U; p.V = sp.V;
    p.BN = pt_ceil_div(d->K, 16) * 16;
    p.rows = d->N * sp.P;
    p.rows_per_cta = pt_ceil_div(p.rows, c->sm_count);
    p.acc_per = 2 * kStemIssuers * p.BN <= 512 ? 2 : 1;
    p.tmem_cols = pow2_cols(kStemIssuers * p.acc_per * p.BN);
    p.x = (const __nv_bfloat16 *)x; p.w = (const __nv_bfloat16 *)w;
    p.status = c->d_status;
    p.ld_out = d->ldy;
    const int grid = pt_ceil_div(p.rows, p.rows_per_cta);
    p.stats_warp = pt_ceil_div(p.BN, 64) * (int)kStatsChunkBytes;
    const size_t st_smem = c->stats_mode ? (size_t)8 * p.stats_warp : 0;
    const size_t smem = 2048 + 8 * kSlabs * 4096 + (size_t)kStemRing * kStemSlot + (size_t)sp.U * sp.V * p.BN * 32 + st_smem;
    p.stats_off = (int)(smem - st_smem);
    CUtensorMap tmC;
    cuuint64_t dims[4] = {(cuuint64_t)store_cols(d->K, d->ldy), (cuuint64_t)sp.Q, (cuuint64_t)sp.P, (cuuint64_t)d->N};
    cuuint64_t strides[3] = {(cuuint64_t)d->ldy * 2, (cuuint64_t)sp.Q * d->ldy * 2, (cuuint64_t)sp.P * sp.Q * d->ldy * 2};
    cuuint32_t box[4] = {64, 32, 1, 1}, estr[4] = {1, 1, 1, 1};
    CUresult r = ((EncodeTiledFn)c->encode_tiled)(&tmC, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, y, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (!map_ok(r, __LINE__)) return PT_ERR_CUDA;
    void (*kernel)(CUtensorMap, StemP) = c->stats_mode ? conv_stem_kernel<true> : conv_stem_kernel<false>;
    if (!(c->attr_done & kAttrStem)) {
        PT_CUDA_OK(cudaFuncSetAttribute(conv_stem_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        PT_CUDA_OK(cudaFuncSetAttribute(conv_stem_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        c->attr_done |= kAttrStem;
    }
    if (c->stats_mode) {
        p.stats_lo = grid < kStatsFewRows ? 1 : 0;
        c->stats_parts = grid * (1 + p.stats_lo);
        if ((size_t)c->stats_parts * 2 * p.ld_out * sizeof(float) > c->stats_cap) return PT_ERR_WORKSPACE;
        p.stats = c->stats_out;
    }
    if (c->test_skip == 6) { p.test_skip = 1; c->test_skip = 0; }
    PT_CUDA_OK(pt_launch_pdl(kernel, dim3((unsigned)grid), dim3(kStemThreads), smem, st, tmC, p));
    c->launches += 1;
    c->last_form = PT_FORM_STEM;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Stride-2 forward by parity planes; false where some plane has no tap or the image not both parities.
bool halo_spec_stride2(const pt_conv_desc *d, HaloSpec *h, const void *src, int P, int Q)
{
    memset(h, 0, sizeof(*h));
    if (d->stride != 2 || d->H < 2 || d->W < 2 || d->R * d->S > kMaxTaps) return false;
    h->src = src; h->Cs = d->C; h->Ws = d->W; h->Hs = d->H; h->lds = d->ldx;
    h->P = P; h->Q = Q; h->span_h = h->span_w = 1;
    // filter row r reads image row 2 i + r - pad of output row i: row i + floor((r - pad) / 2) of the plane of its parity
    for (int pl = 0; pl < 4; ++pl) {
        h->plane_tap[pl] = h->n_taps;
        h->plane_lo_h[pl] = h->plane_lo_w[pl] = 1 << 20;
        for (int r = 0; r < d->R; ++r)
            for (int s = 0; s < d->S; ++s) {
                if (((r - d->pad) & 1) != pl >> 1 || ((s - d->pad) & 1) != (pl & 1)) continue;
                const int oh = (r - d->pad) >> 1, ow = (s - d->pad) >> 1, t = h->n_taps++;
                h->tap_oh[t] = oh; h->tap_ow[t] = ow; h->tap_wt[t] = r * d->S + s;
                if (oh < h->plane_lo_h[pl]) h->plane_lo_h[pl] = oh;
                if (ow < h->plane_lo_w[pl]) h->plane_lo_w[pl] = ow;
            }
        if (h->n_taps == h->plane_tap[pl]) return false;
        for (int t = h->plane_tap[pl]; t < h->n_taps; ++t) {
            h->tap_oh[t] -= h->plane_lo_h[pl]; h->tap_ow[t] -= h->plane_lo_w[pl];
            if (h->tap_oh[t] + 1 > h->span_h) h->span_h = h->tap_oh[t] + 1;
            if (h->tap_ow[t] + 1 > h->span_w) h->span_w = h->tap_ow[t] + 1;
        }
    }
    h->plane_tap[4] = h->n_taps;
    h->n_cols = d->K; h->ld_out = d->ldy;
    h->oH = P; h->oW = Q; h->o_step = 1;
    return true;
}

// ---- launch shape of a weight gradient
// The kernels cut the work three ways: tiles of dw (channels), groups of taps, and the pixels of the reduction over `splits` CTAs
// that exchange partial sums at the end. The shape is chosen by a rough time of one CTA (microseconds; the constants are measured):
//   first load 1.4, then per stage the longer of its matrix instructions and its staged rows, and what waiting and issuing add; then the
//   exchange of the sums that are part of dw: none (one split) 1 + bytes at 17 KB/us (transposed 4 bytes at a time); through the workspace
//   4 + bytes at 33 KB/us (stores, arrival counter, sum: three round trips), slower by what all CTAs exchange over 35 MB; in a cluster (2..8 splits) 2.6 + bytes at 20 KB/us (25 for two).
//   (512 -> 128 1x1 at 7x7, batch 16, 131 KB: workspace 7.9, clusters of two and four 9.9 and 9.2; 64 -> 256 at 14x14, batch 8, 32 KB: 4.5
//   and 3.9; 13 -> 27 3x3 at 16x16, batch 8, 16 KB: 4.3 and 2.9.)
// A cluster needs its CTAs free at the same time in one GPC: used while the device can hold all of the launch's clusters at once.
constexpr double kWgSearch = 400.0;      // generic kernel: layers whose tile takes one CTA less than this (us) also choose tap groups,
constexpr double kWgNarrow = 40.0;       // less than this: tile widths

// One MMA of M = 128, K = 16: cycles by its columns, and what one issuing warp needs where no other issues beside it.
double wg_mma_us(int n, bool several) { const double c = n <= 32 ? 40.0 : n <= 128 ? 32.0 + n * 0.25 : n * 0.5; return (several || c > 75.0 ? c : 75.0) / 1920.0; }
double wg_exchange_us(int tiles, int splits, bool cluster, double bytes)
{
    if (splits <= 1) return 1.0 + bytes / 17e3;
    return cluster ? 2.6 + bytes / (splits == 2 ? 25e3 : 20e3) : 4.0 + bytes / 33e3 * (1.0 + bytes * splits * tiles / 35e6);
}
// Nanoseconds the TMA unit takes per staged row of `cols` channels in boxes of 64 or 32 (see store_cols), all boxes together.
double wg_row_ns(int cols, int lanes = 64)
{
    if (lanes == 32) return cols == 32 ? 0.55 : cols > 16 && cols <= 24 ? 1.5 : 1.05;
    const int rest = cols & 63;
    return (cols >> 6) * 0.95 + (rest == 0 ? 0.0 : rest <= 32 ? 1.05 : rest <= 40 ? 3.4 : rest <= 56 ? 1.45 : 1.05);
}

int wg_max_clusters(const pt_ctx *c, int size);

// Taps handled by one weight-gradient CTA: they share the dy tile and get one TMEM accumulator of BN columns each.
// Bounded by the 512 TMEM columns and by a stage of 16 KB (dy) + taps x BN/64 x 8 KB (x) staying at or below 48 KB, so
// that at least four pipeline stages fit (measured: with two stages the kernel is slower than with one tap per CTA);
// the taps are then dealt out in equal groups.
int wgrad_taps_per_cta(int taps, int bn)
{
    int t = 512 / bn;
    const int by_smem = 4 / pt_ceil_div(bn, 64);
    if (t > by_smem) t = by_smem;
    if (t < 1) t = 1;
    if (t > taps) t = taps;
    const int groups = pt_ceil_div(taps, t);
    return pt_ceil_div(taps, groups);
}

int wgrad_budget(const pt_ctx *c) { return (c->wgrad_ctas > 0 && c->wgrad_ctas < c->sm_count) ? c->wgrad_ctas : c->sm_count; }

// Splits of a launch with `tiles` CTAs per split, at most `max_s`: all the budget holds through the workspace, or up to eight as
// clusters, whichever is estimated faster; `main_us(s)` is the main loop with s splits.
template <typename F>
double wg_pick_splits(const pt_ctx *c, int tiles, int max_s, double bytes, F main_us, int *splits, int *cluster)
{
    int s = wgrad_budget(c) / tiles;                       // at most one CTA per SM, one wave
    if (s > max_s) s = max_s;
    if (s > 512) s = 512;
    if (s < 1) s = 1;
    double best = main_us(s) + wg_exchange_us(tiles, s, false, bytes);
    *splits = s; *cluster = 0;
    for (int k = s < 8 ? s : 8; k >= 2; --k) {
        if (tiles > wg_max_clusters(c, k)) continue;
        const double t = main_us(k) + wg_exchange_us(tiles, k, true, bytes);
        if (t < best) { best = t; *splits = k; *cluster = 1; }
    }
    return best;
}

// Tile widths of the generic kernel: tile_n's, and for small layers a half and a quarter of it (a narrow accumulator is sooner exchanged, and
// more CTAs share the work). False past the last.
bool wgrad_gen_bn(const pt_conv_desc *d, int option, int *bn, int *n_tiles)
{
    *bn = tile_n(d->C, n_tiles);
    if (option == 0) return true;
    if (option > 2 || *bn >> option < 48) return false;
    *n_tiles <<= option;
    *bn = pt_ceil_div(pt_ceil_div(d->C, *n_tiles), 16) * 16;
    return (*n_tiles - 1) * *bn < d->C;
}
long long wgrad_gen_splits(const pt_conv_desc *d, int P, int Q) { return ((long long)d->N * P * Q + 127) / 128; }     // two 64-pixel stages each

// The generic kernel: 64 pixels per stage. Returns the estimated time.
double wgrad_gen_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, pt_wgrad_plan *w)
{
    memset(w, 0, sizeof(*w));
    const int taps = d->R * d->S;
    w->m_tiles = pt_ceil_div(d->K, 128);
    const long long stages = ((long long)d->N * P * Q + 63) / 64;
    long long max_s = wgrad_gen_splits(d, P, Q);
    if (max_s > 512) max_s = 512;
    const double dy_ns = wg_row_ns(d->K > 128 ? 128 : store_cols(d->K, d->ldy)), rows = d->K > 128 ? 128 : d->K;
    double best = 1e30;
    int bn, n_tiles;
    for (int o = 0; wgrad_gen_bn(d, o, &bn, &n_tiles); ++o) {
        const int base = wgrad_taps_per_cta(taps, bn), groups0 = pt_ceil_div(taps, base);
        const double x_ns = wg_row_ns(n_tiles > 1 ? bn : store_cols(d->C, d->ldx)) * (d->stride > 1 ? 1.08 : 1.0);     // (im2col boxes two pixels apart)
        double stage = 0.0;
        for (int g = groups0; g <= taps; g += groups0) {
            const int tpc = pt_ceil_div(taps, g), tiles = w->m_tiles * n_tiles * pt_ceil_div(taps, tpc);
            if ((o > 0 || g > groups0) && (2 * tiles > wgrad_budget(c) || pt_ceil_div(taps, tpc) != g)) continue;
            const double load = 64e-3 * (dy_ns + tpc * x_ns), mma = tpc * 4 * wg_mma_us(bn, tpc > 1);
            stage = load > mma ? load : mma;
            int s, cl;
            const double t = wg_pick_splits(c, tiles, (int)max_s, tpc * bn * rows * 4.0, [&](int k) { return 1.4 + (double)((stages + k - 1) / k) * stage; }, &s, &cl);
            if (t < best) {
                best = t;
                w->bn = w->acc_cols = bn; w->n_tiles = n_tiles;
                w->tpc = w->apc = tpc; w->tap_groups = pt_ceil_div(taps, tpc);
                w->splits = s; w->cluster = cl;
            }
            if ((double)stages * stage > kWgSearch) break;              // large: the fewest groups read the least
        }
        if ((double)stages * stage > kWgNarrow) break;
    }
    return best;
}

// The row-block kernel (stride-1 filters with at most 64 input channels): the estimated time, 1e30 where it does not apply.
double wgrad_rows_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, pt_wgrad_plan *w)
{
    memset(w, 0, sizeof(*w));
    const int taps = d->R * d->S;
    if (d->stride != 1 || taps > kMaxTaps) return 1e30;
    // a 1x1 filter has no halo to save, but the orientation (x on the M side, all of dy's channels on the N side: one tile
    // where the generic kernel needs two for K > 128) and the plain tiled loads (no im2col boxes on 96-byte pixel pitches)
    // still pay on large maps (56x56, 59 -> 143: 53 -> 31 us at 49 CTAs); small maps have too few units to split
    if (taps < 2 && P * Q < 784) return 1e30;
    w->Wp = Q + d->S - 1;
    if (w->Wp > 256 || P < 1 || Q < 1) return 1e30;
    // paired form only: the x tile is the M side (two taps x 64 channel lanes), dy's output channels the N side
    w->acc_cols = pt_ceil_div(d->K, 16) * 16;
    if (d->C > 64 || w->acc_cols > 256) return 1e30;
    w->bn = tile_n(d->C, &w->n_tiles);
    w->m_tiles = 1;
    w->lanes = d->C <= 32 ? 32 : 64;
    w->dy_lanes = d->K <= 32 ? 32 : 64;
    const size_t x_row = w->lanes * 2, dy_row = w->dy_lanes * 2;
    const int span = w->lanes == 64 ? d->S : pt_ceil_div(d->S, 4) * 4;                       // columns of shifts the operands reach
    const int pairs = w->lanes == 64 ? pt_ceil_div(taps, 2) : d->R * pt_ceil_div(d->S, 4);   // accumulators: of two or four taps
    int t = 512 / w->acc_cols;
    if (t > 16) t = 16;                                   // four issuer warps x four accumulators
    if (t > pairs) t = pairs;
    const int groups0 = pt_ceil_div(pairs, t);
    w->nb_a = pt_ceil_div(w->acc_cols, 64);
    const double dy_ns = wg_row_ns(store_cols(d->K, d->ldy), w->dy_lanes), x_ns = wg_row_ns(store_cols(d->C, d->ldx), w->lanes);
    const double rows_used = (w->lanes == 64 ? 2 : d->S < 4 ? d->S : 4) * d->C;              // of an accumulator
    // Rows per unit, tap groups and splits, by the estimated time: a unit takes the longer of its matrix instructions and its staged rows.
    // (Large layers took the unit with the least traffic and MMA steps per useful pixel instead, and no account of the rows: units of a
    // single row, or so large that the splits came out uneven. 10 -> 22 1x1 at 32x32, batch 253: 23.8 -> 15.4 us; 9 -> 13 at 37x37, batch
    // 58: 16.8 -> 13.4; 60 -> 29 at 56x56, batch 53: 23.8 -> 22.6; others the same.)
    double best_us = 1e30;
    for (int nr = 1; nr <= P && nr + d->R - 1 <= 256; ++nr) {
        const int ks = pt_ceil_div(nr * w->Wp, 16);
        const size_t a_box = (size_t)ks * 16 * dy_row;
        const size_t b_box = pt_align_up(((size_t)(d->R - 1) * w->Wp + span + (size_t)ks * 16) * x_row, 1024);
        const size_t stage = w->nb_a * a_box + b_box;
        const int st = (int)((220 * 1024 - 2048) / stage);
        if (st < 2) break;
        const int rb = pt_ceil_div(P, nr), units = d->N * rb;
        const double load = (dy_ns * nr + x_ns * (nr + d->R - 1)) * w->Wp * 1e-3;         // the TMA unit, by the row
        for (int g = groups0; g <= pairs; g += groups0) {
            const int apc = pt_ceil_div(pairs, g), tiles = pt_ceil_div(pairs, apc);
            if (g > groups0 && (tiles > wgrad_budget(c) || tiles != g)) continue;
            const double mma = ks * apc * wg_mma_us(w->acc_cols, apc > 1), unit = (load > mma ? load : mma) + 0.15;
            int s, cl;
            const double us = wg_pick_splits(c, tiles, units > 3 ? units / 2 : 1, apc * rows_used * d->K * 4.0,
                                             [&](int k) { return 1.4 + pt_ceil_div(units, k) * unit; }, &s, &cl);
            if (us >= best_us) continue;
            best_us = us;
            w->nr = nr; w->ksteps = ks; w->a_box = (unsigned)a_box; w->b_box = (unsigned)b_box;
            w->stages = st > kMaxStages ? kMaxStages : st;
            w->stage_bytes = stage; w->RB = rb; w->units = units;
            w->apc = apc; w->tap_groups = tiles;
            w->splits = s; w->cluster = cl;
        }
    }
    if (w->nr == 0) return 1e30;
    w->units_per_split = pt_ceil_div(w->units, w->splits);
    w->splits = pt_ceil_div(w->units, w->units_per_split);
    if (w->splits < 2) w->cluster = 0;
    if (w->stages > w->units_per_split && w->units_per_split >= 2) w->stages = w->units_per_split;
    w->smem = 2048 + (size_t)w->stages * w->stage_bytes;
    if (w->smem < kWgradSmemMin) w->smem = kWgradSmemMin;
    w->rows = 1;
    return best_us;
}

// Columns of an accumulator, and tiles of them, of the filter-row form: S accumulators fit the tensor memory.
int wgrad_taps_bn(const pt_conv_desc *d, int *n_tiles)
{
    int top = 512 / d->S / 16 * 16;
    if (top > 256) top = 256;
    *n_tiles = pt_ceil_div(d->C, top);
    return pt_ceil_div(pt_ceil_div(d->C, *n_tiles), 16) * 16;
}

bool wgrad_taps_ok(const pt_conv_desc *d)
{
    return d->S >= 2 && d->S <= kMaxRow && d->R <= kMaxRow && (d->stride == 1 || d->stride == 2) && d->pad <= 64 && d->H >= d->stride && d->W >= d->stride;
}

// The filter-row kernel: the estimated time, 1e30 where it does not apply.
double wgrad_taps_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, pt_wgrad_plan *w)
{
    memset(w, 0, sizeof(*w));
    if (!wgrad_taps_ok(d) || P < 1 || Q < 1) return 1e30;
    w->planes = d->stride;
    const int shift = d->stride == 1 ? d->S - 1 : d->S / 2;             // the largest one (at stride 2 and an even S it may be one less)
    w->Wp = Q + shift;
    if (w->Wp > 256) return 1e30;
    w->bn = w->acc_cols = wgrad_taps_bn(d, &w->n_tiles);
    if (w->n_tiles > 1) return 1e30;          // (dy would be loaded again: no fewer bytes, 147 -> 186 to 213 -> 242 3x3 at 14x14 no faster per SM)
    w->m_tiles = pt_ceil_div(d->K, 128);
    w->nb_a = d->K > 64 ? 2 : 1;
    w->tpc = w->apc = d->S; w->tap_groups = d->R;
    const int nb = pt_ceil_div(w->bn, 64), tiles = w->n_tiles * w->m_tiles * d->R;
    const double cyc = wg_mma_us(w->bn, true);
    const double dy_ns = wg_row_ns(d->K > 128 ? 128 : store_cols(d->K, d->ldy)), x_ns = wg_row_ns(w->n_tiles > 1 ? w->bn : store_cols(d->C, d->ldx));
    double best = 1e30;
    for (int nr = 1; nr <= P && nr <= 256; ++nr) {
        const int ks = pt_ceil_div(nr * w->Wp, 16);
        const size_t a_box = (size_t)ks * 2048, b_box = pt_align_up((size_t)(ks * 16 + shift) * 128, 1024);
        const size_t stage = w->nb_a * a_box + (size_t)w->planes * nb * b_box;
        int st = (int)((220 * 1024 - 2048) / stage);
        if (st < 3) break;
        if (st > kMaxStages) st = kMaxStages;
        const int rb = pt_ceil_div(P, nr), units = d->N * rb;
        // a unit takes the longest of its matrix instructions, its staged rows and a load's latency over the stages in flight
        const double mma = ks * d->S * cyc, load = (dy_ns + w->planes * x_ns) * nr * w->Wp * 1e-3, lat = 1.4 / (st - 1);
        double unit = mma > load ? mma : load;
        unit = (unit > lat ? unit : lat) + 0.08;
        int s, cl;
        const double us = wg_pick_splits(c, tiles, units > 3 ? units / 2 : 1, w->apc * w->bn * (d->K > 128 ? 128 : d->K) * 4.0,
                                         [&](int k) { return 1.4 + pt_ceil_div(units, k) * unit; }, &s, &cl);
        if (us >= best) continue;
        best = us;
        w->nr = nr; w->ksteps = ks; w->a_box = (unsigned)a_box; w->b_box = (unsigned)b_box;
        w->stages = st; w->stage_bytes = stage; w->RB = rb; w->units = units;
        w->splits = s; w->cluster = cl;
    }
    if (w->nr == 0) return 1e30;
    w->units_per_split = pt_ceil_div(w->units, w->splits);
    w->splits = pt_ceil_div(w->units, w->units_per_split);
    if (w->splits < 2) w->cluster = 0;
    if (w->stages > w->units_per_split && w->units_per_split >= 2) w->stages = w->units_per_split;
    w->smem = 2048 + (size_t)w->stages * w->stage_bytes;
    if (w->smem < kWgradSmemMin) w->smem = kWgradSmemMin;
    w->filter_row = 1;
    return best;
}

// The packed kernel: pixels of x 16 or 32 channels apart, of dy too; a staged row of x (64 / ldx pixels, G) and the next one hold what the
// S taps of G pixels read.
bool wgrad_packed_ok(const pt_conv_desc *d, int P)
{
    if (d->stride != 1 || (d->ldx != 16 && d->ldx != 32) || (d->ldy != 16 && d->ldy != 32) || d->S < 2) return false;
    const int G = 64 / d->ldx, N = G * d->ldy;
    return d->S - 1 <= G && d->R * N <= 512 && P >= 1 && P + d->R <= 256;
}
// 16-byte pieces that a split leaves (one source per pixel of dy in a row).
long long wgrad_packed_pieces(const pt_conv_desc *d) { return (long long)(64 / d->ldx) * d->R * pt_ceil_div(d->K, 4) * d->S * d->C; }

double wgrad_packed_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, pt_wgrad_plan *w)
{
    memset(w, 0, sizeof(*w));
    if (!wgrad_packed_ok(d, P) || Q < 1) return 1e30;
    const int G = 64 / d->ldx, cols = pt_ceil_div(Q, G), shift = d->R - 1;
    w->acc_cols = w->bn = G * d->ldy;
    w->n_tiles = w->m_tiles = w->tap_groups = 1;
    w->apc = w->tpc = d->R;
    w->lanes = d->ldx;
    w->dy_lanes = w->acc_cols < 64 ? 32 : 64;
    w->nb_a = w->acc_cols / w->dy_lanes;
    w->Wp = P + shift;
    if (w->dy_lanes == 32) w->Wp += w->Wp & 1;             // (a column of 64-byte rows starts on 128 bytes)
    const double bytes = (double)wgrad_packed_pieces(d) * 16.0;
    double best = 1e30;
    for (int nc = 1; nc <= cols; ++nc) {
        const int ks = pt_ceil_div(nc * w->Wp, 16);
        const size_t a_box = pt_align_up((size_t)ks * 16 * w->dy_lanes * 2, 1024), b_box = pt_align_up(((size_t)w->Wp + shift + (size_t)ks * 16) * 128, 1024);
        const size_t stage = w->nb_a * a_box + b_box;
        int st = (int)((220 * 1024 - 2048) / stage);
        if (st < 2) break;
        if (st > kMaxStages) st = kMaxStages;
        const int rb = pt_ceil_div(cols, nc), units = d->N * rb, boxes = nc + 1 + nc * w->nb_a;
        const double mma = ks * d->R * wg_mma_us(w->acc_cols, d->R > 1), issue = pt_ceil_div(boxes, 5) * 0.2;
        const double load = w->Wp * ((nc + 1) * 0.95e-3 + nc * w->nb_a * (w->dy_lanes == 64 ? 0.95e-3 : 0.55e-3)), lat = 1.4 / (st - 1);
        double unit = mma > load ? mma : load;
        if (unit < issue) unit = issue;
        unit = (unit > lat ? unit : lat) + 0.1;
        // splits: as few as share the units in the same number of turns
        const int most = wgrad_budget(c) < units ? wgrad_budget(c) : units, turns = pt_ceil_div(units, most), s = pt_ceil_div(units, turns);
        const double us = 1.4 + turns * unit + (s > 1 ? wg_exchange_us(1, s, false, bytes) : 3.0 + bytes / 33e3);
        if (us >= best) continue;
        best = us;
        w->nr = nc; w->ksteps = ks; w->a_box = (unsigned)a_box; w->b_box = (unsigned)b_box;
        w->stages = st; w->stage_bytes = stage; w->RB = rb; w->units = units; w->units_per_split = turns;
        w->splits = s;
    }
    if (w->nr == 0) return 1e30;
    if (w->stages > w->units_per_split && w->units_per_split >= 2) w->stages = w->units_per_split;
    w->smem = 2048 + (size_t)w->stages * w->stage_bytes;
    if (w->smem < kWgradSmemMin) w->smem = kWgradSmemMin;
    w->packed = 1;
    return best;
}

size_t wgrad_workspace_bound(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &w);

double wgrad_form_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, int form, pt_wgrad_plan *w)
{
    return form == PT_FORM_WGRAD_ROWS ? wgrad_rows_plan(c, d, P, Q, w) : form == PT_FORM_WGRAD_TAPS ? wgrad_taps_plan(c, d, P, Q, w)
         : form == PT_FORM_WGRAD_PACKED ? wgrad_packed_plan(c, d, P, Q, w) : wgrad_gen_plan(c, d, P, Q, w);
}

// The plan of a descriptor at the context's CTA limit. rows_only: only a row-block plan is asked for (its `rows` is 0 if there is none).
pt_wgrad_plan wgrad_plan(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, bool rows_only = false)
{
    pt_ctx::WgradKey key{*d, wgrad_budget(c), P, Q};
    static_assert(sizeof(key) == sizeof(pt_conv_desc) + 12, "the key is compared and hashed as words");
    const int form = rows_only || c->test_form > PT_FORM_WGRAD_PACKED ? (int)PT_FORM_ANY : c->test_form;
    key.d.ldw = key.d.out_f32 = 0; key.d.algo = rows_only ? 1 : 2 * form;
    std::lock_guard<std::mutex> lock(c->wgrad_mutex);
    const auto known = c->wgrad_plans.find(key);
    if (known != c->wgrad_plans.end()) return known->second;
    pt_wgrad_plan w;
    if (!form || wgrad_form_plan(c, d, P, Q, form, &w) > 1e29) {
        const double rows_us = wgrad_rows_plan(c, d, P, Q, &w);
        if (!rows_only && wgrad_packed_ok(d, P)) {
            pt_wgrad_plan k;
            if (wgrad_packed_plan(c, d, P, Q, &k) < (w.rows ? rows_us : 1e29)) w = k;
        }
        if (!w.rows && !w.packed && !rows_only) {
            pt_wgrad_plan g;
            // (measured against estimated times at all SMs and at 49: within 10 % of each other, so that near a tie either may be the faster;
            // 106 -> 103 3x3 at 28x28, batch 64 22.9 us generic, 21.8 by filter rows, 49.5 and 34.6 at 49; 128 -> 128 at 32x32 25.7 and 28.2,
            // 54.1 and 46.5; 147 -> 186 at 14x14 19.7 and 22.1, 44.5 and 32.1)
            if (0.98 * wgrad_gen_plan(c, d, P, Q, &g) <= wgrad_taps_plan(c, d, P, Q, &w)) w = g;
        }
    }
    w.ws_bytes = wgrad_workspace_bound(c, d, P, Q, w);
    if (c->wgrad_plans.size() >= pt_ctx::kWgradPlans) c->wgrad_plans.clear();
    c->wgrad_plans.emplace(key, w);
    return w;
}

// Workspace of the split weight gradient: one padded 128 x columns fp32 tile per (tile, split). (A cluster needs none, but the test
// hook of the arrival wait turns one into an exchange through the workspace.)
size_t wgrad_partial_bytes(const pt_wgrad_plan &w, const pt_conv_desc *d)
{
    if (w.packed) return (size_t)wgrad_packed_pieces(d) * 16 * (size_t)w.splits;
    if (w.splits <= 1) return 0;
    return (size_t)w.n_tiles * w.m_tiles * w.tap_groups * w.apc * w.splits * 128 * w.acc_cols * sizeof(float);
}

// What a caller is asked for: the most that a launch shape of this descriptor needs at the context's CTA limit, so that a workspace sized
// at one limit serves every smaller one too, whatever shape is chosen there (a smaller limit may well choose more splits, through the
// workspace, where a larger one takes a few in a cluster).
size_t wgrad_workspace_bound(const pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &w)
{
    const int taps = d->R * d->S, budget = wgrad_budget(c);
    // `parts` (taps, or accumulators of two or four taps) dealt out in groups, as few as fit one CTA (`most`) at most, each with `tiles1` tiles of
    // `cols` columns, and the most splits: floats
    const auto floats = [&](int parts, int most, int g_step, int tiles1, int cols, long long max_s) {
        long long tiles128 = 0;                            // 128 x cols tiles
        for (int g = pt_ceil_div(parts, most < parts ? most : parts); g <= parts; g += g_step) {
            const int per = pt_ceil_div(parts, g), tiles = tiles1 * pt_ceil_div(parts, per);
            long long s = budget / tiles;
            if (s > max_s) s = max_s;
            if (s >= 2 && tiles * s * per > tiles128) tiles128 = tiles * s * per;
        }
        return tiles128 * 128 * cols;
    };
    const long long units = (long long)d->N * P, unit_s = units > 3 ? units / 2 : 1;
    const size_t packed = wgrad_packed_ok(d, P) ? (size_t)wgrad_packed_pieces(d) * 16 * (size_t)budget : 0;
    if (w.rows || w.packed) {
        pt_wgrad_plan r = w;                               // (either may be the choice of a smaller limit)
        if (w.packed && wgrad_rows_plan(c, d, P, Q, &r) > 1e29) return packed;
        const size_t rows = (size_t)floats(r.lanes == 64 ? pt_ceil_div(taps, 2) : d->R * pt_ceil_div(d->S, 4), 512 / r.acc_cols < 16 ? 512 / r.acc_cols : 16, 1,
                              r.n_tiles * r.m_tiles, r.acc_cols, unit_s) * sizeof(float);
        return rows > packed ? rows : packed;
    }
    int bn, n_tiles;
    const int m_tiles = pt_ceil_div(d->K, 128);
    long long most = 0;
    for (int o = 0; wgrad_gen_bn(d, o, &bn, &n_tiles); ++o) {
        const long long t = floats(taps, wgrad_taps_per_cta(taps, bn), 1, n_tiles * m_tiles, bn, wgrad_gen_splits(d, P, Q));
        if (t > most) most = t;
    }
    const int bt = wgrad_taps_bn(d, &n_tiles);
    if (wgrad_taps_ok(d) && n_tiles == 1) {                // (either form may be the choice of a smaller limit)
        const long long t = floats(taps, d->S, taps, n_tiles * m_tiles, bt, unit_s);
        if (t > most) most = t;
    }
    const size_t bytes = (size_t)most * sizeof(float);
    return bytes > packed ? bytes : packed;
}

// Launch of a weight-gradient kernel: with programmatic stream serialization and, where the splits of a tile meet in shared memory,
// as clusters of `cluster` CTAs along y.
template <typename XMaps>
cudaError_t launch_wgrad(void (*kernel)(CUtensorMap, XMaps, WgradP), dim3 grid, int cluster, size_t smem, cudaStream_t st,
                         const CUtensorMap &a, const XMaps &b, const WgradP &p)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = (unsigned)cluster; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, a, b, p);
}

pt_status wgrad_attr(const pt_ctx *c)
{
    if (!(c->attr_done & kAttrWgrad)) {
        PT_CUDA_OK(cudaFuncSetAttribute(conv_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        PT_CUDA_OK(cudaFuncSetAttribute(conv_wgrad_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        PT_CUDA_OK(cudaFuncSetAttribute(conv_wgrad_packed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        PT_CUDA_OK(cudaFuncSetAttribute(conv_wgrad_taps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        c->attr_done |= kAttrWgrad;
    }
    return PT_OK;
}

// Clusters of `size` weight-gradient CTAs the device holds at once (one CTA per SM; a GPC whose SM count is no multiple leaves some over).
int wg_max_clusters(const pt_ctx *c, int size)
{
    if (size < 2 || size > 8) return 0;
    if (c->max_clusters[size] == 0) {
        // (a workspace query may come while another device is the current one)
        int n = 0, cur = c->device;
        (void)cudaGetDevice(&cur);
        if (cur != c->device) (void)cudaSetDevice(c->device);
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(1, (unsigned)size); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = 220 * 1024;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = (unsigned)size; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (wgrad_attr(c) != PT_OK || cudaOccupancyMaxActiveClusters(&n, conv_wgrad_kernel, &cfg) != cudaSuccess || n < 1) {
            (void)cudaGetLastError();
            n = -1;
        }
        if (cur != c->device) (void)cudaSetDevice(cur);
        c->max_clusters[size] = n;
    }
    return c->max_clusters[size] < 0 ? 0 : c->max_clusters[size];
}

WgradRaw wgrad_raw(const pt_conv_desc *d, int P, int Q, const void *x, const void *dy)
{
    return WgradRaw{(const __nv_bfloat16 *)x, (const __nv_bfloat16 *)dy, d->N, d->H, d->W, d->C, d->K, P, Q, d->R, d->S, d->stride, d->pad, d->ldx, d->ldy};
}

// What all forms have in common: tiles, splits and where the partial tiles go.
pt_status wgrad_common(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &w, float *out, void *ws, size_t ws_bytes, WgradP *p)
{
    memset(p, 0, sizeof(*p));
    p->K = d->K; p->C = d->C; p->taps = d->R * d->S; p->S = d->S;
    p->BN = w.bn; p->n_tiles = w.n_tiles; p->m_tiles = w.m_tiles;
    p->tpc = w.tpc; p->tap_groups = w.tap_groups; p->apc = w.apc; p->acc_cols = w.acc_cols;
    p->npix = d->N * P * Q;
    p->splits = w.splits; p->cluster = w.cluster;
    p->Pd = P; p->Qd = Q;
    p->tmem_cols = pow2_cols(w.apc * w.acc_cols);
    p->status = c->d_status;
    p->out = out;
    if (c->test_skip == 1 && p->splits > 1) { p->test_skip = 1; p->cluster = 0; c->test_skip = 0; }
    if ((p->splits > 1 && !p->cluster) || w.packed) {
        const int gx = p->n_tiles * p->m_tiles * p->tap_groups;
        if (!ws || ws_bytes < wgrad_partial_bytes(w, d)) return PT_ERR_WORKSPACE;
        p->partial = (float *)ws;
        // two self-resetting counters per tile from the context's ring (kernels of one stream run in order, and the ring
        // is far larger than the tiles of the few launches that can be in flight)
        if (2 * gx > 8192) return PT_ERR_UNSUPPORTED;
        if (c->sync_next + 2 * gx > 16384) c->sync_next = 0;
        p->sync = c->d_sync + c->sync_next;
        c->sync_next += 2 * gx;
    }
    return wgrad_attr(c);
}

// Launches the weight-gradient kernel for a problem whose x operand is described by `tmX` (64 pixels x 64 channels boxes).
pt_status run_wgrad(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &w, int stride, int lo_h, int lo_w, const CUtensorMap &tmX,
                    const void *dy, float *out, void *ws, size_t ws_bytes, cudaStream_t st, bool x_tiled = false)
{
    WgradP p;
    const pt_status r0 = wgrad_common(c, d, P, Q, w, out, ws, ws_bytes, &p);
    if (r0 != PT_OK) return r0;
    p.x_tiled = x_tiled ? 1 : 0;
    p.pix_per_split = pt_ceil_div(pt_ceil_div(p.npix, p.splits), 64) * 64;
    p.stride = stride; p.lo_h = lo_h; p.lo_w = lo_w;
    const int gx = p.n_tiles * p.m_tiles * p.tap_groups;
    // A: dy as a 2-D tensor (K channels, N*P*Q pixels), box 64 channels x 64 pixels
    if (!c->encode_tiled) return PT_ERR_CUDA;
    CUtensorMap tmA;
    {
        cuuint64_t dims[2] = {(cuuint64_t)store_cols(d->K, d->ldy), (cuuint64_t)p.npix};
        cuuint64_t strides[1] = {(cuuint64_t)d->ldy * 2};
        cuuint32_t box[2] = {64, 64}, estr[2] = {1, 1};
        CUresult r = ((EncodeTiledFn)c->encode_tiled)(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(dy), dims, strides, box,
                                                      estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (!map_ok(r, __LINE__)) return PT_ERR_CUDA;
    }
    size_t smem = 0;
    const size_t stage = 2 * 8192 + (size_t)p.tpc * pt_ceil_div(p.BN, 64) * 8192;
    p.stages = pick_stages(stage, pt_ceil_div(p.pix_per_split, 64), 0, &smem);
    if (smem < kWgradSmemMin) smem = kWgradSmemMin;
    if (p.splits > 1 && smem < kSplitSmemFloor) smem = kSplitSmemFloor;
    dim3 grid((unsigned)gx, (unsigned)p.splits);
    p.data_bytes = (unsigned)(smem - 2048);
    PT_CUDA_OK(launch_wgrad(conv_wgrad_kernel, grid, p.cluster ? p.splits : 1, smem, st, tmA, tmX, p));
    c->launches += 1;
    c->last_form = PT_FORM_WGRAD_PIXELS;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Launches the row-block weight-gradient kernel.
// `x_row_pixels` > 0 and (lo_h, lo_w): x is a view whose rows are x_row_pixels apart and whose raster origin for tap (0, 0)
// is at (lo_h, lo_w) instead of (-pad, -pad) -- the space-to-depth stem, whose "pixels" are overlapping 4-pixel windows; `stem` is that
// layer, `image` its input and out its dw.
pt_status run_wgrad_rows(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &wr, const void *x, const void *dy, float *out, void *ws,
                         size_t ws_bytes, cudaStream_t st, int x_row_pixels = 0, int lo_h = 0, int lo_w = 0, const pt_conv_desc *stem = nullptr, const void *image = nullptr, int off = 0)
{
    if (!c->encode_tiled) return PT_ERR_CUDA;
    WgradP p;
    CUtensorMap tmA, tmX;
    const pt_status r0 = wgrad_common(c, d, P, Q, wr, out, ws, ws_bytes, &p);
    if (r0 != PT_OK) return r0;
    p.pair = 1;
    p.raw = wgrad_raw(stem ? stem : d, P, Q, stem ? image : x, dy);
    p.stride = 1; p.lo_h = -d->pad; p.lo_w = -d->pad;
    if (x_row_pixels > 0) { p.lo_h = lo_h; p.lo_w = lo_w; }
    if (stem) { p.stem.C = stem->C; p.stem.R = stem->R; p.stem.S = stem->S; p.stem.off = off; }
    p.nr = wr.nr; p.Wp = wr.Wp; p.RB = wr.RB; p.units = wr.units; p.units_per_split = wr.units_per_split;
    p.ksteps = wr.ksteps; p.nb_a = wr.nb_a; p.lo_span = d->R - 1; p.a_box = wr.a_box; p.b_box = wr.b_box;
    p.stages = wr.stages;
    p.lanes = wr.lanes; p.dy_lanes = wr.dy_lanes; p.acc_row = pt_ceil_div(d->S, 4); p.lane_shift = wr.lanes == 64 ? 6 : 5;
    const int gx = p.n_tiles * p.m_tiles * p.tap_groups;
    // dy: box of nr rows x Wp columns (Wp > Q: the extra columns are out of bounds and read as zeros); x: the halo box
    if (!make_halo_in_map(c, &tmA, dy, store_cols(d->K, d->ldy), Q, P, d->N, d->ldy, wr.Wp, wr.nr, wr.dy_lanes)) return PT_ERR_UNSUPPORTED;
    if (!make_halo_in_map(c, &tmX, x, x_row_pixels > 0 ? d->C : store_cols(d->C, d->ldx), d->W, d->H, d->N, d->ldx, wr.Wp, wr.nr + d->R - 1, wr.lanes, x_row_pixels))
        return PT_ERR_UNSUPPORTED;
    dim3 grid((unsigned)gx, (unsigned)p.splits);
    const size_t smem = (p.splits > 1 && wr.smem < kSplitSmemFloor) ? kSplitSmemFloor : wr.smem;
    p.data_bytes = (unsigned)(smem - 2048);
    PT_CUDA_OK(launch_wgrad(conv_wgrad_rows_kernel, grid, p.cluster ? p.splits : 1, smem, st, tmA, tmX, p));
    c->launches += 1;
    c->last_form = PT_FORM_WGRAD_ROWS;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Launches the packed weight-gradient kernel.
pt_status run_wgrad_packed(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &wk, const void *x, const void *dy, float *out, void *ws,
                           size_t ws_bytes, cudaStream_t st)
{
    WgradP p;
    CUtensorMap tmA, tmX;
    const pt_status r0 = wgrad_common(c, d, P, Q, wk, out, ws, ws_bytes, &p);
    if (r0 != PT_OK) return r0;
    p.G = 64 / d->ldx; p.lanes = d->ldx; p.lane_shift = d->ldx == 32 ? 5 : 4; p.dy_lanes = wk.dy_lanes; p.row_lanes = d->ldy;
    p.lo_h = p.lo_w = -d->pad;
    p.raw = wgrad_raw(d, P, Q, x, dy);
    p.nr = wk.nr; p.Wp = wk.Wp; p.RB = wk.RB; p.units = wk.units; p.units_per_split = wk.units_per_split;
    p.ksteps = wk.ksteps; p.nb_a = wk.nb_a; p.a_box = wk.a_box; p.b_box = wk.b_box; p.stages = wk.stages;
    // image rows as rows of W x ld elements: a box of 64 (32) of them is the next pixels side by side, zeros past either end of the row
    const auto map = [&](CUtensorMap *tm, const void *base, int W, int H, int ld, int lanes) {
        cuuint64_t dims[3] = {(cuuint64_t)W * ld, (cuuint64_t)H, (cuuint64_t)d->N};
        cuuint64_t strides[2] = {(cuuint64_t)W * ld * 2, (cuuint64_t)H * W * ld * 2};
        cuuint32_t box[3] = {(cuuint32_t)lanes, (cuuint32_t)wk.Wp, 1}, estr[3] = {1, 1, 1};
        return map_ok(((EncodeTiledFn)c->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                                                       CU_TENSOR_MAP_INTERLEAVE_NONE, lanes_swizzle(lanes), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE), __LINE__);
    };
    if (!c->encode_tiled || !map(&tmA, dy, Q, P, d->ldy, wk.dy_lanes) || !map(&tmX, x, d->W, d->H, d->ldx, 64)) return PT_ERR_CUDA;
    const size_t smem = (p.splits > 1 && wk.smem < kSplitSmemFloor) ? kSplitSmemFloor : wk.smem;
    p.data_bytes = (unsigned)(smem - 2048);
    PT_CUDA_OK(launch_wgrad(conv_wgrad_packed_kernel, dim3(1u, (unsigned)p.splits), 1, smem, st, tmA, tmX, p));
    c->launches += 1;
    c->last_form = PT_FORM_WGRAD_PACKED;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Launches the filter-row weight-gradient kernel.
pt_status run_wgrad_taps(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const pt_wgrad_plan &wt, const void *x, const void *dy, float *out, void *ws,
                         size_t ws_bytes, cudaStream_t st)
{
    if (!c->encode_tiled) return PT_ERR_CUDA;
    WgradP p;
    CUtensorMap tmA;
    TapMaps tmX;
    memset(&tmX, 0, sizeof(tmX));
    const pt_status r0 = wgrad_common(c, d, P, Q, wt, out, ws, ws_bytes, &p);
    if (r0 != PT_OK) return r0;
    p.raw = wgrad_raw(d, P, Q, x, dy);
    p.nr = wt.nr; p.Wp = wt.Wp; p.RB = wt.RB; p.units = wt.units; p.units_per_split = wt.units_per_split;
    p.ksteps = wt.ksteps; p.nb_a = wt.nb_a; p.a_box = wt.a_box; p.b_box = wt.b_box; p.stages = wt.stages; p.planes = wt.planes;
    // tap column s reads pixel stride * j + s - pad of output column j: plane (s - pad) mod stride, column j + floor((s - pad) / stride) of it
    const int sh = d->stride - 1;                                     // (stride 1 or 2: shifts and masks)
    p.plane_lo[0] = p.plane_lo[1] = 1 << 20;
    for (int s = 0; s < d->S; ++s) {
        const int pl = (s - d->pad) & sh, off = (s - d->pad) >> sh;
        p.tap_plane[s] = (unsigned char)pl;
        if (off < p.plane_lo[pl]) p.plane_lo[pl] = off;
    }
    for (int s = 0; s < d->S; ++s) p.tap_shift[s] = (unsigned char)(((s - d->pad) >> sh) - p.plane_lo[p.tap_plane[s]]);
    for (int r = 0; r < d->R; ++r) {
        p.row_par[r] = (unsigned char)((r - d->pad) & sh);
        p.row_off[r] = (signed char)((r - d->pad) >> sh);
    }
    if (!make_halo_in_map(c, &tmA, dy, store_cols(d->K, d->ldy), Q, P, d->N, d->ldy, wt.Wp, wt.nr)) return PT_ERR_UNSUPPORTED;
    for (int a = 0; a < d->stride; ++a)
        for (int b = 0; b < d->stride; ++b)
            if (!make_plane_map(c, &tmX.m[a * 2 + b], x, store_cols(d->C, d->ldx), d->W, d->H, d->N, d->ldx, d->stride, a, b, wt.Wp, wt.nr)) return PT_ERR_UNSUPPORTED;
    dim3 grid((unsigned)(p.n_tiles * p.m_tiles * p.tap_groups), (unsigned)p.splits);
    const size_t smem = (p.splits > 1 && wt.smem < kSplitSmemFloor) ? kSplitSmemFloor : wt.smem;
    p.data_bytes = (unsigned)(smem - 2048);
    PT_CUDA_OK(launch_wgrad(conv_wgrad_taps_kernel, grid, p.cluster ? p.splits : 1, smem, st, tmA, tmX, p));
    c->launches += 1;
    c->last_form = PT_FORM_WGRAD_TAPS;
    PT_CUDA_OK(cudaGetLastError());
    return PT_OK;
}

// Stride-2 data gradient of a bf16 dx with even H and W: the input pixels split by the parity (a, b) of (h, w) into four
// stride-1 correlations over dy (pixel h = 2i + a receives tap r iff a + pad - r is even, from dy row i + (a + pad - r)/2).
// Each parity with taps is one halo-kernel launch that TMA-stores into the strided view of dx holding that parity; if some
// parity has no tap, dx is cleared first (1x1 filters without padding go to the GEMM kernel, which writes those zeros itself). Returns PT_ERR_UNSUPPORTED for shapes the halo kernel declines
// (nothing has been launched then).
pt_status dgrad_stride2_halo(pt_ctx *c, const pt_conv_desc *d, int P, int Q, const void *dy, const void *w, void *dx, cudaStream_t st)
{
    HaloSpec hs[4];
    int n_launch = 0;
    bool any_empty = false;
    for (int ab = 0; ab < 4; ++ab) {
        const int pa = ab >> 1, pb = ab & 1;
        HaloSpec &h = hs[n_launch];
        memset(&h, 0, sizeof(h));
        int oh[kMaxTaps], ow[kMaxTaps], nt = 0;
        for (int r = 0; r < d->R; ++r) {
            if ((pa + d->pad - r) & 1) continue;
            for (int sft = 0; sft < d->S; ++sft) {
                if ((pb + d->pad - sft) & 1) continue;
                if (nt >= kMaxTaps) return PT_ERR_UNSUPPORTED;
                oh[nt] = (pa + d->pad - r) / 2; ow[nt] = (pb + d->pad - sft) / 2;
                h.tap_wt[nt] = r * d->S + sft;
                ++nt;
            }
        }
        if (nt == 0) { any_empty = true; continue; }
        int min_oh = oh[0], min_ow = ow[0], max_oh = oh[0], max_ow = ow[0];
        for (int t = 0; t < nt; ++t) {
            min_oh = oh[t] < min_oh ? oh[t] : min_oh; max_oh = oh[t] > max_oh ? oh[t] : max_oh;
            min_ow = ow[t] < min_ow ? ow[t] : min_ow; max_ow = ow[t] > max_ow ? ow[t] : max_ow;
        }
        for (int t = 0; t < nt; ++t) { h.tap_oh[t] = oh[t] - min_oh; h.tap_ow[t] = ow[t] - min_ow; }
        h.src = dy; h.Cs = d->K; h.Ws = Q; h.Hs = P; h.lds = d->ldy;
        h.P = d->H / 2; h.Q = d->W / 2;
        h.n_taps = nt; h.span_h = max_oh - min_oh + 1; h.span_w = max_ow - min_ow + 1;
        h.lo_h = min_oh; h.lo_w = min_ow;
        h.n_cols = d->C; h.ld_out = d->ldx;
        h.oH = d->H; h.oW = d->W; h.o_step = 2; h.o_h0 = pa; h.o_w0 = pb;
        if (h.Q + h.span_w - 1 > 128) return PT_ERR_UNSUPPORTED;      // (so a tile has a row)
        ++n_launch;
    }
    if (n_launch == 0) return PT_ERR_UNSUPPORTED;
    // a 1x1 filter reads every pixel of dy once and has no halo: the pixel-linear tiles of the GEMM kernel, which also writes the
    // zeros of the parities without a tap. It anchors them at parity (0, 0), which the tap of a filter with padding 1 does not reach:
    // that one stays here, unless the maps are so small that a tile is mostly padding
    if (d->R * d->S == 1 && ((d->pad & 1) == 0 || (d->H / 2) * (d->W / 2) < 64)) return PT_ERR_UNSUPPORTED;
    if (any_empty) PT_CUDA_OK(cudaMemsetAsync(dx, 0, (size_t)d->N * d->H * d->W * d->ldx * 2, st));
    // The parity classes write disjoint pixels of dx and read the same inputs: launches 1.. go to the context's helper
    // streams (forked from and joined back to the caller's stream by events) so that their fills and drains overlap.
    if (n_launch > 1 && !c->fork_ev) {
        bool ok = cudaEventCreateWithFlags(&c->fork_ev, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; i < 3 && ok; ++i)
            ok = cudaStreamCreateWithFlags(&c->fork_stream[i], cudaStreamNonBlocking) == cudaSuccess &&
                 cudaEventCreateWithFlags(&c->join_ev[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) { (void)cudaGetLastError(); return PT_ERR_CUDA; }
    }
    if (n_launch > 1) {
        // Each parity launch would fill the device on its own and they would run one after the other, each paying its start and drain:
        // they get shares of the SMs on which they run side by side and end together. A tile takes its taps' matrix work (0.066 us per
        // 64 x 64 channels and tap) and 0.22 us; the shares are the smallest that finish all of their tiles, in whole rounds, within
        // the shortest time for which they fit. 103 -> 106 at 56x56, batch 64: 40.6 -> 23.3 us; 64 -> 64, batch 256 49 -> 30;
        // 11 -> 21 at 32x32, batch 128 15.6 -> 8.9; 200 -> 200 at 28x28, batch 64 40.7 -> 24.5.
        int n_tiles, tiles[4], share[4];
        const int bn = tile_n(d->C, &n_tiles);
        double cost[4], lo = 0.0, hi = 0.0;
        for (int i = 0; i < n_launch; ++i) {
            const int wp = hs[i].Q + hs[i].span_w - 1, nr = 128 / wp < hs[i].P ? 128 / wp : hs[i].P;
            tiles[i] = d->N * pt_ceil_div(hs[i].P, nr) * n_tiles;
            cost[i] = 0.066 * hs[i].n_taps * pt_ceil_div(d->K, kKC) * (bn > 64 ? bn / 64.0 : 1.0) + 0.22;
            if (tiles[i] * cost[i] > hi) hi = tiles[i] * cost[i];
        }
        const auto fits = [&](double t) {
            int sum = 0;
            for (int i = 0; i < n_launch; ++i) {
                const int rounds = (int)(t / cost[i] + 1e-6);
                share[i] = rounds < 1 ? tiles[i] + c->sm_count : pt_ceil_div(tiles[i], rounds);
                sum += share[i];
            }
            return sum <= c->sm_count;
        };
        while (!fits(hi)) hi *= 2.0;                  // (one CTA per launch fits)
        for (int it = 0; it < 24; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (fits(mid)) hi = mid; else lo = mid;
        }
        (void)fits(hi);
        for (int i = 0; i < n_launch; ++i) hs[i].max_ctas = share[i];
    }
    if (n_launch > 1) PT_CUDA_OK(cudaEventRecord(c->fork_ev, st));
    pt_status first = PT_OK;
    for (int i = 0; i < n_launch; ++i) {
        cudaStream_t si = i == 0 ? st : c->fork_stream[i - 1];
        if (i > 0) PT_CUDA_OK(cudaStreamWaitEvent(si, c->fork_ev, 0));
        pt_status r = launch_halo<true>(c, d, hs[i], w, dx, si);
        if (i > 0) {                                   // join even after a failure, so that a capture stays well formed
            PT_CUDA_OK(cudaEventRecord(c->join_ev[i - 1], si));
            PT_CUDA_OK(cudaStreamWaitEvent(st, c->join_ev[i - 1], 0));
        }
        if (r != PT_OK && first == PT_OK)
            first = (r == PT_ERR_UNSUPPORTED && i == 0 && !any_empty) ? r : (r == PT_ERR_UNSUPPORTED ? PT_ERR_CUDA : r);
        if (first != PT_OK && i == 0) return first;    // nothing forked yet
    }
    return first;
}

}  // namespace

bool pt_sm100_conv_supported(const pt_ctx *c, const pt_conv_desc *d, int which)
{
    if (!c->encode_tiled || !c->encode_im2col) return false;
    if (d->stride > 8 || d->pad > 100 || d->R * d->S > kMaxTaps) return false;
    if (which == PT_CONV_FWD) return true;
    if (which == PT_CONV_DGRAD) return (d->stride == 1 && d->pad <= d->R - 1 && d->pad <= d->S - 1) || d->stride == 2;
    return true;
}

// The stem's weight gradient as the generic kernel sees it: U taps of 64 "channels".
static pt_conv_desc stem_virtual_desc(const pt_conv_desc *d, const StemPlan &sp)
{
    pt_conv_desc v = *d;
    v.C = 64; v.R = sp.U; v.S = 1;
    return v;
}

// The same for the row-block kernel: a stride-1 U x 1 filter over Q x Hs "pixels" of 64 lanes whose rows are Wp real pixels
// (16 lanes each) apart; pixel j of a row is the window of real pixels j .. j+3.
static pt_conv_desc stem_rows_desc(const pt_conv_desc *d, const StemPlan &sp)
{
    pt_conv_desc v = stem_virtual_desc(d, sp);
    v.stride = 1; v.W = sp.Q; v.H = sp.Hs; v.ldx = 16;
    return v;
}

// CTAs the weight gradient of `d` launches at the context's current CTA limit: tiles x splits; *waits = 1 if they wait for
// one another (splits > 1).
int pt_sm100_wgrad_ctas(const pt_ctx *c, const pt_conv_desc *d, int *waits)
{
    const StemPlan sp = stem_plan(d);
    pt_conv_desc v = sp.ok ? stem_virtual_desc(d, sp) : *d;
    const int P = sp.ok ? sp.P : pt_out_dim(d->H, d->R, d->stride, d->pad), Q = sp.ok ? sp.Q : pt_out_dim(d->W, d->S, d->stride, d->pad);
    const pt_conv_desc vr = sp.ok ? stem_rows_desc(d, sp) : v;
    pt_wgrad_plan w = wgrad_plan(c, &vr, P, Q, sp.ok);
    if (sp.ok && !w.rows) w = wgrad_plan(c, &v, P, Q);
    if (waits) *waits = w.splits > 1 ? 1 : 0;
    return w.n_tiles * w.m_tiles * w.tap_groups * w.splits;
}

size_t pt_sm100_conv_workspace(const pt_ctx *c, const pt_conv_desc *d, int which)
{
    const StemPlan sp = stem_plan(d);
    if (sp.ok && which == PT_CONV_FWD) return sp.xs_bytes + pt_align_up(sp.w2_elems * 2, 1024);
    if (sp.ok && which == PT_CONV_WGRAD) {
        const pt_conv_desc v = stem_virtual_desc(d, sp), vr = stem_rows_desc(d, sp);
        const pt_wgrad_plan wa = wgrad_plan(c, &v, sp.P, sp.Q), wb = wgrad_plan(c, &vr, sp.P, sp.Q, true);
        const size_t pa = wa.ws_bytes, pb = wb.rows ? wb.ws_bytes : 0;
        return sp.xs_bytes + pt_align_up(sp.w2_elems * 4, 1024) + (pa > pb ? pa : pb);
    }
    if (which != PT_CONV_WGRAD) return 0;
    const int P = pt_out_dim(d->H, d->R, d->stride, d->pad), Q = pt_out_dim(d->W, d->S, d->stride, d->pad);
    return wgrad_plan(c, d, P, Q).ws_bytes;
}

pt_status pt_sm100_conv(pt_ctx *c, const pt_conv_desc *d, int which, const void *a, const void *b, void *out, void *ws,
                        size_t ws_bytes, cudaStream_t st)
{
    const int P = pt_out_dim(d->H, d->R, d->stride, d->pad), Q = pt_out_dim(d->W, d->S, d->stride, d->pad);
    GemmMaps tm;
    const StemPlan sp = stem_plan(d);
    if (which == PT_CONV_WGRAD) {
        if (sp.ok) {
            // stem: space-to-depth copy of x, generic wgrad over U taps x 64 lanes, then back to [K][R][S][C]
            char *wsb = (char *)ws;
            __nv_bfloat16 *xs = (__nv_bfloat16 *)wsb;
            float *dw2 = (float *)(wsb + sp.xs_bytes);
            char *part = wsb + sp.xs_bytes + pt_align_up(sp.w2_elems * 4, 1024);
            const pt_conv_desc v = stem_virtual_desc(d, sp);
            const size_t tot = (size_t)d->N * sp.Hs * sp.Wp;
            stem_s2d_x_kernel_launch((unsigned)((tot + 255) / 256), st, (const __nv_bfloat16 *)a, xs, d->N, d->H, d->W, d->C, sp.Hs, sp.Ws, sp.Wp, sp.pl);
            c->launches += 1;
            // the row-block kernel first: the windows of a unit of rows are staged once for all U vertical taps and two taps share
            // an MMA (M = 128 lanes where the generic kernel has 55 output channels on its M side)
            const pt_conv_desc vr = stem_rows_desc(d, sp);
            const pt_wgrad_plan wr = wgrad_plan(c, &vr, sp.P, sp.Q, true);
            pt_status r = PT_ERR_UNSUPPORTED;
            if (wr.rows) {
                r = run_wgrad_rows(c, &vr, sp.P, sp.Q, wr, xs, b, (float *)out, part, ws_bytes - (size_t)(part - wsb), st, sp.Wp, -sp.pl, 0, d, a, sp.off);
                if (r != PT_ERR_UNSUPPORTED) return r;
            }
            if (r == PT_ERR_UNSUPPORTED) {
                CUtensorMap tmX;
                const int up_h = (sp.P - 1) - sp.pl - (sp.Hs - 1);
                if (!make_im2col_map(c, &tmX, xs, 64, sp.Q, sp.Hs, d->N, 16, 0, -sp.pl, 0, up_h, 1, 64, sp.Wp)) return PT_ERR_CUDA;
                r = run_wgrad(c, &v, sp.P, sp.Q, wgrad_plan(c, &v, sp.P, sp.Q), 1, -sp.pl, 0, tmX, b, dw2, part, ws_bytes - (size_t)(part - wsb), st);
            }
            if (r != PT_OK) return r;
            const int n = d->K * d->R * d->S * d->C;
            stem_dw_back_kernel<<<(n + 255) / 256, 256, 0, st>>>(dw2, (float *)out, d->K, d->R, d->S, d->C, sp.U, sp.off);
            c->launches += 1;
            PT_CUDA_OK(cudaGetLastError());
            return PT_OK;
        }
        pt_wgrad_plan w = wgrad_plan(c, d, P, Q);
        if (w.packed) return run_wgrad_packed(c, d, P, Q, w, a, b, (float *)out, ws, ws_bytes, st);
        if (w.rows) {
            const pt_status r = run_wgrad_rows(c, d, P, Q, w, a, b, (float *)out, ws, ws_bytes, st);
            if (r != PT_ERR_UNSUPPORTED) return r;
            wgrad_gen_plan(c, d, P, Q, &w);
        }
        if (w.filter_row) {
            const pt_status r = run_wgrad_taps(c, d, P, Q, w, a, b, (float *)out, ws, ws_bytes, st);
            if (r != PT_ERR_UNSUPPORTED) return r;
            wgrad_gen_plan(c, d, P, Q, &w);
        }
        CUtensorMap tmX;
        const int up_w = (Q - 1) * d->stride - d->pad - (d->W - 1), up_h = (P - 1) * d->stride - d->pad - (d->H - 1);
        const bool plain = d->R == 1 && d->S == 1 && d->stride == 1 && d->pad == 0;     // pixels of x and dy coincide
        if (plain) {
            if (!make_act2d_map(c, &tmX, a, store_cols(d->C, d->ldx), (long long)d->N * d->H * d->W, d->ldx, 64)) return PT_ERR_CUDA;
        } else if (!make_im2col_map(c, &tmX, a, store_cols(d->C, d->ldx), d->W, d->H, d->N, d->ldx, -d->pad, -d->pad, up_w, up_h, d->stride, 64)) return PT_ERR_CUDA;
        return run_wgrad(c, d, P, Q, w, d->stride, -d->pad, -d->pad, tmX, b, (float *)out, ws, ws_bytes, st, plain);
    }

    GemmP p;
    memset(&p, 0, sizeof(p));
    p.status = c->d_status;
    p.out = out;
    p.out_f32 = d->out_f32;
    if (which == PT_CONV_FWD && sp.ok) {
        const pt_status direct = run_stem(c, d, sp, a, b, out, st);
        if (direct != PT_ERR_UNSUPPORTED) return direct;
        char *wsb = (char *)ws;
        __nv_bfloat16 *xs = (__nv_bfloat16 *)wsb, *w2 = (__nv_bfloat16 *)(wsb + sp.xs_bytes);
        const size_t tot = (size_t)d->N * sp.Hs * sp.Wp;
        stem_s2d_x_kernel_launch((unsigned)((tot + 255) / 256), st, (const __nv_bfloat16 *)a, xs, d->N, d->H, d->W, d->C, sp.Hs, sp.Ws, sp.Wp, sp.pl);
        stem_s2d_w_kernel<<<(unsigned)((sp.w2_elems + 255) / 256), 256, 0, st>>>((const __nv_bfloat16 *)b, w2, d->K, d->R, d->S, d->C, d->ldw,
                                                                              sp.U, sp.V, sp.off);
        c->launches += 2;
        // (plain launches: the convolution below loads w2 before its dependency wait, which is safe because stem_s2d_w_kernel
        // does not release its dependents before it has completed)
        if (!d->out_f32) {
            // row-block form on 32-byte pixels: the U x V taps are row shifts of one staged tile (each xs byte read once)
            HaloSpec h;
            memset(&h, 0, sizeof(h));
            h.src = xs; h.Cs = 16; h.Ws = sp.Wp; h.Hs = sp.Hs; h.lds = 16;
            h.P = sp.P; h.Q = sp.Q;
            h.n_taps = sp.U * sp.V; h.span_h = sp.U; h.span_w = sp.V;
            h.lo_h = -sp.pl; h.lo_w = 0;
            for (int t = 0; t < h.n_taps; ++t) { h.tap_oh[t] = t / sp.V; h.tap_ow[t] = t % sp.V; h.tap_wt[t] = (t / sp.V) * 4 + t % sp.V; }
            h.n_cols = d->K; h.ld_out = d->ldy;
            h.oH = sp.P; h.oW = sp.Q; h.o_step = 1; h.o_h0 = 0; h.o_w0 = 0;
            h.row32 = 1; h.w_taps = sp.U * 4;
            const pt_status r = launch_halo<false>(c, d, h, w2, out, st);
            if (r != PT_ERR_UNSUPPORTED) return r;
        }
        p.M_total = d->N * sp.P * sp.Q;
        p.n_cols = d->K;
        p.BN = tile_n(d->K, &p.n_tiles);
        p.c_red = 64;
        p.k_chunks = 1;
        p.taps = sp.U;
        for (int t = 0; t < p.taps; ++t) { p.tap_oh[t] = (unsigned char)t; p.tap_ow[t] = 0; p.tap_wt[t] = (unsigned short)t; }
        p.Pd = sp.P; p.Qd = sp.Q; p.stride = 1; p.lo_h = -sp.pl; p.lo_w = 0;
        p.oH = sp.P; p.oW = sp.Q; p.o_step = 1; p.o_h0 = 0; p.o_w0 = 0; p.ld_out = d->ldy; p.zero_mask = 0;
        p.tmem_cols = pow2_cols(p.BN);
        const int up_h = (sp.P - 1) - sp.pl - (sp.Hs - 1);
        if (!make_im2col_map(c, &tm.a, xs, 64, sp.Q, sp.Hs, d->N, 16, 0, -sp.pl, 0, up_h, 1, kBM, sp.Wp)) return PT_ERR_CUDA;
        tm.tail = tm.a;
        if (!make_weight_map(c, &tm.b, w2, 64, sp.U, d->K, 64, p.BN)) return PT_ERR_CUDA;
        return launch_gemm<false>(c, tm, p, st);
    }
    // A halo tile is whole raster rows of ONE image in at most 128 MMA rows: on small maps most of the tile is padding (7x7:
    // 49 useful rows of 128), and the pixel-linear tiles of the im2col kernel do better (7x7, 345 -> 374: 23 us against 30)
    const int raster_h = which == PT_CONV_FWD ? P : d->H, raster_w = which == PT_CONV_FWD ? Q : d->W;
    const int halo_wp = raster_w + d->S - 1;
    const int halo_nr = halo_wp <= 128 ? (128 / halo_wp < raster_h ? 128 / halo_wp : raster_h) : 1;
    const bool sparse_tiles = 2 * raster_h * raster_w < pt_ceil_div(raster_h, halo_nr) * 128;
    if (!sparse_tiles && which == PT_CONV_FWD && d->stride == 1 && d->R * d->S > 1 && d->R * d->S <= kMaxTaps) {
        HaloSpec h;
        halo_spec_stride1(d, &h, a, d->C, d->W, d->H, d->ldx, d->K, P, Q, d->ldy, d->pad, d->pad, false);
        pt_status r = launch_halo<false>(c, d, h, b, out, st);
        if (r != PT_ERR_UNSUPPORTED) return r;
    }
    if ((!sparse_tiles || c->test_form == PT_FORM_PLANES) && which == PT_CONV_FWD && d->stride == 2 && d->R * d->S > 1) {
        HaloSpec h;
        if (halo_spec_stride2(d, &h, a, P, Q)) {
            const pt_status r = launch_halo<false, 4>(c, d, h, b, out, st);
            if (r != PT_ERR_UNSUPPORTED) return r;
        }
    }
    if (!sparse_tiles && which == PT_CONV_DGRAD && d->stride == 1 && d->R * d->S > 1 && d->R * d->S <= kMaxTaps && d->pad <= d->R - 1 &&
        d->pad <= d->S - 1) {
        // dx = correlation of dy (padding R-1-pad) with the taps visited flipped
        HaloSpec h;
        halo_spec_stride1(d, &h, a, d->K, Q, P, d->ldy, d->C, d->H, d->W, d->ldx, d->R - 1 - d->pad, d->S - 1 - d->pad, true);
        pt_status r = launch_halo<true>(c, d, h, b, out, st);
        if (r != PT_ERR_UNSUPPORTED) return r;
    }
    if (which == PT_CONV_DGRAD && d->stride == 2 && !d->out_f32 && (d->H % 2 == 0) && (d->W % 2 == 0)) {
        pt_status r = dgrad_stride2_halo(c, d, P, Q, a, b, out, st);
        if (r != PT_ERR_UNSUPPORTED) return r;
    }
    const int tail = gemm_tail_lanes(which == PT_CONV_FWD ? d->C : d->K);
    if (which == PT_CONV_FWD) {
        // raster = output pixels (P x Q per image); source = x
        p.M_total = d->N * P * Q;
        p.n_cols = d->K;
        p.BN = tile_n(d->K, &p.n_tiles, pt_ceil_div(p.M_total, kBM), c->sm_count);
        p.c_red = d->C;
        p.k_chunks = pt_ceil_div(d->C, kKC);
        p.taps = d->R * d->S;
        for (int t = 0; t < p.taps; ++t) { p.tap_oh[t] = (unsigned char)(t / d->S); p.tap_ow[t] = (unsigned char)(t % d->S); p.tap_wt[t] = (unsigned short)t; }
        p.Pd = P; p.Qd = Q; p.stride = d->stride; p.lo_h = -d->pad; p.lo_w = -d->pad;
        p.oH = P; p.oW = Q; p.o_step = 1; p.o_h0 = 0; p.o_w0 = 0; p.ld_out = d->ldy; p.zero_mask = 0;
        p.tmem_cols = pow2_cols(p.BN);
        // the box of base positions must hold exactly P x Q positions at the traversal stride
        const int up_w = (Q - 1) * d->stride - d->pad - (d->W - 1), up_h = (P - 1) * d->stride - d->pad - (d->H - 1);
        if (d->R == 1 && d->S == 1 && d->stride == 1 && d->pad == 0) {
            p.a_tiled = 1;
            if (!make_act2d_map(c, &tm.a, a, d->C, (long long)d->N * d->H * d->W, d->ldx, kBM) ||
                !make_act2d_map(c, &tm.tail, a, d->C, (long long)d->N * d->H * d->W, d->ldx, kBM, tail)) return PT_ERR_CUDA;
        } else if (!make_im2col_map(c, &tm.a, a, d->C, d->W, d->H, d->N, d->ldx, -d->pad, -d->pad, up_w, up_h, d->stride, kBM) ||
                   !make_im2col_map(c, &tm.tail, a, d->C, d->W, d->H, d->N, d->ldx, -d->pad, -d->pad, up_w, up_h, d->stride, kBM, 0, tail)) return PT_ERR_CUDA;
        if (!make_weight_map(c, &tm.b, b, d->C, d->R * d->S, d->K, d->ldw, p.BN)) return PT_ERR_CUDA;
        return launch_gemm<false>(c, tm, p, st);
    }
    if (which != PT_CONV_DGRAD) return PT_ERR_UNSUPPORTED;
    p.n_cols = d->C;
    p.BN = tile_n(d->C, &p.n_tiles, pt_ceil_div(d->N * d->H * d->W / (d->stride * d->stride), kBM), c->sm_count);
    p.c_red = d->K;
    p.k_chunks = pt_ceil_div(d->K, kKC);
    p.tmem_cols = pow2_cols(p.BN);
    p.oH = d->H; p.oW = d->W; p.ld_out = d->ldx;
    if (!make_weight_map(c, &tm.b, b, d->C, d->R * d->S, d->K, d->ldw, kKC)) return PT_ERR_CUDA;
    if (d->stride == 1) {
        // raster = input pixels (H x W per image); source = dy with padding R-1-pad and the taps visited flipped:
        // dx[h,w] = sum_{r',s'} dy[h - (R-1-pad) + r', w - (S-1-pad) + s'] * w[R-1-r', S-1-s']
        const int ph = d->R - 1 - d->pad, pw = d->S - 1 - d->pad;
        if (ph < 0 || pw < 0) return PT_ERR_UNSUPPORTED;
        p.M_total = d->N * d->H * d->W;
        p.taps = d->R * d->S;
        for (int t = 0; t < p.taps; ++t) {
            p.tap_oh[t] = (unsigned char)(t / d->S); p.tap_ow[t] = (unsigned char)(t % d->S);
            p.tap_wt[t] = (unsigned short)(p.taps - 1 - t);
        }
        p.Pd = d->H; p.Qd = d->W; p.stride = 1; p.lo_h = -ph; p.lo_w = -pw;
        p.o_step = 1; p.o_h0 = 0; p.o_w0 = 0; p.zero_mask = 0;
        const int up_w = (d->W - 1) - pw - (Q - 1), up_h = (d->H - 1) - ph - (P - 1);
        if (d->R == 1 && d->S == 1 && d->pad == 0) {
            p.a_tiled = 1;
            if (!make_act2d_map(c, &tm.a, a, d->K, (long long)d->N * P * Q, d->ldy, kBM) ||
                !make_act2d_map(c, &tm.tail, a, d->K, (long long)d->N * P * Q, d->ldy, kBM, tail)) return PT_ERR_CUDA;
        } else if (!make_im2col_map(c, &tm.a, a, d->K, Q, P, d->N, d->ldy, -pw, -ph, up_w, up_h, 1, kBM) ||
                   !make_im2col_map(c, &tm.tail, a, d->K, Q, P, d->N, d->ldy, -pw, -ph, up_w, up_h, 1, kBM, 0, tail)) return PT_ERR_CUDA;
        return launch_gemm<true>(c, tm, p, st);
    }
    if (d->stride != 2) return PT_ERR_UNSUPPORTED;
    // Stride 2: the input pixels split by the parity (a, b) of (h, w) into four stride-1 problems over dy.
    // Pixel h = 2i + a receives tap r iff (a + pad - r) is even, from dy row p = i + (a + pad - r)/2.
    // Parities no tap reaches are zero-filled by the epilogue of the first launched parity.
    struct Par { int a, b, nt; int oh[kMaxTaps], ow[kMaxTaps], wt[kMaxTaps]; };
    Par par[4];
    int empty_mask = 0, first = -1;
    for (int ab = 0; ab < 4; ++ab) {
        Par &q = par[ab];
        q.a = ab >> 1; q.b = ab & 1; q.nt = 0;
        for (int r = 0; r < d->R; ++r) {
            if ((q.a + d->pad - r) & 1) continue;
            for (int s = 0; s < d->S; ++s) {
                if ((q.b + d->pad - s) & 1) continue;
                q.oh[q.nt] = (q.a + d->pad - r) / 2;      // exact: the difference is even (may be negative)
                q.ow[q.nt] = (q.b + d->pad - s) / 2;
                q.wt[q.nt] = r * d->S + s;
                ++q.nt;
            }
        }
        const int rows = (d->H - q.a + 1) / 2, cols = (d->W - q.b + 1) / 2;
        if (rows <= 0 || cols <= 0) { q.nt = -1; continue; }          // no pixel has this parity
        if (q.nt == 0) empty_mask |= 1 << ab; else if (first < 0) first = ab;
    }
    if (first < 0) return PT_ERR_UNSUPPORTED;
    if (empty_mask && (par[first].a != 0 || par[first].b != 0)) return PT_ERR_UNSUPPORTED;   // cells are anchored at parity (0,0)
    for (int ab = 0; ab < 4; ++ab) {
        Par &q = par[ab];
        if (q.nt <= 0) continue;
        int min_oh = q.oh[0], min_ow = q.ow[0];
        for (int t = 0; t < q.nt; ++t) { min_oh = q.oh[t] < min_oh ? q.oh[t] : min_oh; min_ow = q.ow[t] < min_ow ? q.ow[t] : min_ow; }
        const int rows = (d->H - q.a + 1) / 2, cols = (d->W - q.b + 1) / 2;
        p.M_total = d->N * rows * cols;
        p.taps = q.nt;
        for (int t = 0; t < q.nt; ++t) {
            p.tap_oh[t] = (unsigned char)(q.oh[t] - min_oh); p.tap_ow[t] = (unsigned char)(q.ow[t] - min_ow);
            p.tap_wt[t] = (unsigned short)q.wt[t];
        }
        p.Pd = rows; p.Qd = cols; p.stride = 1; p.lo_h = min_oh; p.lo_w = min_ow;
        p.o_step = 2; p.o_h0 = q.a; p.o_w0 = q.b;
        p.zero_mask = (ab == first) ? empty_mask : 0;
        const int up_w = (cols - 1) + min_ow - (Q - 1), up_h = (rows - 1) + min_oh - (P - 1);
        p.a_tiled = (q.nt == 1 && min_oh == 0 && min_ow == 0 && rows == P && cols == Q) ? 1 : 0;      // dy's pixels in order
        if (p.a_tiled) {
            if (!make_act2d_map(c, &tm.a, a, d->K, p.M_total, d->ldy, kBM) || !make_act2d_map(c, &tm.tail, a, d->K, p.M_total, d->ldy, kBM, tail))
                return PT_ERR_CUDA;
        } else if (!make_im2col_map(c, &tm.a, a, d->K, Q, P, d->N, d->ldy, min_ow, min_oh, up_w, up_h, 1, kBM) ||
                   !make_im2col_map(c, &tm.tail, a, d->K, Q, P, d->N, d->ldy, min_ow, min_oh, up_w, up_h, 1, kBM, 0, tail)) return PT_ERR_CUDA;
        pt_status s = launch_gemm<true>(c, tm, p, st);
        if (s != PT_OK) return s;
    }
    return PT_OK;
}

// Sets the limit of the bounded device-side waits of this file's kernels (the variable lives in this translation unit).
pt_status pt_sm100_set_wait_limit_ns(unsigned long long ns)
{
    PT_CUDA_OK(cudaMemcpyToSymbol(g_wait_limit_ns, &ns, sizeof(ns)));
    return PT_OK;
}

#ifdef PT_DEVICE_TRACE
extern "C" int pt_debug_wgrad_trace(unsigned long long *host_out)
{
    return (int)cudaMemcpyFromSymbol(host_out, g_wg_trace, sizeof(unsigned long long) * 8 * 64);
}
extern "C" int pt_debug_chain_trace(unsigned long long *host_out, int reset)
{
    cudaError_t e = cudaMemcpyFromSymbol(host_out, g_chain_trace, sizeof(unsigned long long) * 256 * 12);
    if (reset) {
        static const unsigned long long zeros[256 * 12] = {0};
        const unsigned int z = 0;
        (void)cudaMemcpyToSymbol(g_chain_trace, zeros, sizeof(zeros));
        (void)cudaMemcpyToSymbol(g_chain_seq, &z, sizeof(z));
    }
    return (int)e;
}
extern "C" int pt_debug_gemm_trace(unsigned long long *host_out)
{
    return (int)cudaMemcpyFromSymbol(host_out, g_gemm_trace, sizeof(unsigned long long) * 8 * 64);
}
extern "C" int pt_debug_halo_trace(unsigned long long *host_out)
{
    return (int)cudaMemcpyFromSymbol(host_out, g_halo_trace, sizeof(unsigned long long) * 8 * 64);
}
#endif
