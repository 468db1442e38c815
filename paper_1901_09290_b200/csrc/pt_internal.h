// Internal declarations shared by the translation units of the library (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <string.h>
#include <atomic>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "../../include/pt.h"

// The CUDA call that last failed on this thread: kept for pt_last_cuda_error.
void pt_note_cuda_error(cudaError_t e, const char *call, const char *file, int line);

#define PT_CUDA_OK(call)                                   \
    do {                                                   \
        cudaError_t e__ = (call);                          \
        if (e__ != cudaSuccess) {                          \
            pt_note_cuda_error(e__, #call, __FILE__, __LINE__); \
            (void)cudaGetLastError();                      \
            return PT_ERR_CUDA;                            \
        }                                                  \
    } while (0)

// Device status word layout: [0] = first error code recorded (0 = none), [1] = detail (where), [2] = ticket of the
// keep-set scan (self-resetting), [3] spare.
enum { PT_DEV_OK = 0, PT_DEV_TIMEOUT = 1, PT_DEV_BAD_INDEX = 2 };

struct pt_region {              // one cached table: a slot of the arena, or memory of its own for a larger one
    char *dev = nullptr, *host = nullptr;               // where it is on the device and its pinned staging
    size_t cap = 0;
    char *large_dev = nullptr, *large_host = nullptr;
    std::vector<char> key;      // host bytes the current device copy was built from
    bool valid = false;
};

// One cached table of the lasso step or the detection: the layers array it was built from, and what the launches need to know of it.
struct pt_group_slot {
    pt_region reg;
    std::vector<char> args;
    size_t chunks_off = 0, jobs_off = 0;
    unsigned n_chunks = 0, n_jobs = 0;
    bool small = false;
    std::vector<int> first_chunk;
    size_t ws[11];                  // offsets of the workspace's parts
};

// Kernels whose opt-in to more than 48 KB of dynamic shared memory a context has set (pt_ctx::attr_done). The attribute belongs to a
// device, so it is remembered per context and not per process; setting it twice does no harm.
enum : unsigned { kAttrGemm = 1u << 0 /* four variants */, kAttrHalo = 1u << 4 /* three */, kAttrWgrad = 1u << 7, kAttrBn = 1u << 8 /* four */,
                  kAttrGate = 1u << 12 /* three */, kAttrStem = 1u << 15, kAttrPlanes = 1u << 16 /* two */ };

// Launch shape of a weight gradient. rows = 1: the row-block kernel (stride-1 filters with at most 64 input channels).
struct pt_wgrad_plan {
    int rows;
    int bn, n_tiles, m_tiles, tpc, tap_groups, apc, acc_cols;
    int splits, cluster;            // CTAs that share a tile's pixels; 1: they are one thread-block cluster
    // row-block form
    int nr, Wp, RB, units, units_per_split, ksteps, nb_a, stages;
    int lanes, dy_lanes;            // channel lanes per staged pixel of x (64: two taps per accumulator, 32: four) and of dy
    unsigned a_box, b_box;
    size_t stage_bytes, smem;
    size_t ws_bytes;                // workspace that a caller is asked for
    int packed;                     // packed form (nr: columns per unit; Wp: rows of a column; RB, units, ... as above)
    int filter_row, planes;         // filter-row form (nr, Wp, RB, units, ksteps, nb_a, stages, boxes as above); x boxes per unit and block
};

struct pt_ctx {
    int device = 0;
    int sm_count = 0;
    mutable std::atomic<unsigned> attr_done{0};
    int cc_major = 0, cc_minor = 0;
    unsigned int *d_status = nullptr;   // 4 words, device
    unsigned int *h_status = nullptr;   // 4 words, pinned host
    char *d_arena = nullptr;            // table arena, device
    char *h_stage = nullptr;            // pinned staging copy of the arena
    size_t arena_bytes = 0;
    cudaEvent_t upload_done = nullptr;  // last staging->arena copy
    bool upload_pending = false;
    // Cached device tables. A captured CUDA graph embeds the device address of the table its kernels read, so tables of
    // different callers must not evict each other: the lasso step and the detection have their own slot sets.
    pt_group_slot lasso_tab[3], detect_tab[2];
    pt_region graph_tab;
    int lasso_next = 0, detect_next = 0;
    // pt_reconfigure: four cached gather tables, each with the argument bytes it was built from and its launch shape. A call
    // with the same arguments (every reconfiguration of a fixed pair of models, or of a fixed part of them) launches straight
    // from its table; a caller that gathers a model in two parts keeps both tables alive.
    struct GatherSlot {
        pt_region reg;
        std::vector<char> args;
        unsigned chunks = 0;
        size_t jobs_bytes = 0;
    } gather_slot[4];
    int gather_next = 0;
    int32_t *h_counts = nullptr;        // pinned, for pt_reconfigure_plan: [0] = flag the kernel raises, [16..] = counts
    unsigned int plan_seq = 0;          // sequence number of the last plan's flag
    int plan_spaces = 0;                // number of spaces of the last plan
    void *plan_stream = nullptr;        // the stream it was enqueued on
    unsigned int *d_sync = nullptr;     // zero-initialised, self-resetting arrival counters of the split weight gradient
    unsigned int sync_next = 0;         // ring position in d_sync
    uint64_t launches = 0;
    int wgrad_ctas = 0;                 // CTA limit of a weight-gradient launch (0 = all SMs)
    // pt_conv_fwd_stats: non-zero while that call runs: the forward kernels also leave per-warp channel sums in stats_out
    // (stats_cap bytes) and the launcher records how many rows of partial sums there are
    int stats_mode = 0;
    int stats_parts = 0;
    float *stats_out = nullptr;
    size_t stats_cap = 0;
    int test_skip = 0;                  // pt_test_skip_next_arrive: 1 = next split weight gradient, 2 = next fwd/dgrad GEMM-form launch,
                                        // 3 = next batch-norm pass, 4 = next staged gate, 5 = next halo-form launch, 6 = next direct stem
    int test_form = 0, last_form = 0;   // pt_test_form, pt_test_last_form
    int dgrad_ctas = 0;                 // pt_set_dgrad_cta_limit (0: none)
    // Plans of the weight-gradient descriptors met so far: choosing one walks a few hundred candidates (about 10 us), a call must not.
    // A network has about fifty, each at a few CTA limits; past kWgradPlans the table starts again.
    struct WgradKey {
        pt_conv_desc d;
        int limit, P, Q;
        bool operator==(const WgradKey &o) const { return memcmp(this, &o, sizeof(o)) == 0; }
    };
    struct WgradHash {
        size_t operator()(const WgradKey &k) const {
            uint64_t h = 1469598103934665603ull;
            for (size_t i = 0; i < sizeof(k) / 4; ++i) h = (h ^ reinterpret_cast<const uint32_t *>(&k)[i]) * 1099511628211ull;
            return (size_t)(h ^ (h >> 32));
        }
    };
    static constexpr size_t kWgradPlans = 2048;
    mutable std::unordered_map<WgradKey, pt_wgrad_plan, WgradHash> wgrad_plans;
    mutable std::mutex wgrad_mutex;
    mutable int max_clusters[9] = {0};  // co-resident weight-gradient clusters of 2..8 CTAs (0: not asked yet)
    // Helper streams for independent launches inside one call (the parity classes of a stride-2 data gradient): the caller's
    // stream forks to them and joins them back through events, which a stream capture records as graph edges.
    cudaStream_t fork_stream[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t fork_ev = nullptr, join_ev[3] = {nullptr, nullptr, nullptr};
    // tcgen05 conv path
    void *encode_tiled = nullptr;       // cuTensorMapEncodeTiled
    void *encode_im2col = nullptr;      // cuTensorMapEncodeIm2col
};

static inline int pt_ceil_div(int a, int b) { return (a + b - 1) / b; }
static inline size_t pt_align_up(size_t a, size_t b) { return (a + b - 1) / b * b; }
static inline int pt_out_dim(int H, int R, int stride, int pad) {
    int t = H + 2 * pad - R;
    return t < 0 ? 0 : t / stride + 1;
}

// Launch with programmatic stream serialization: the kernel may be scheduled while the previous kernel of the stream is still
// draining, so that its launch latency and prologue overlap that kernel's tail. In a kernel launched this way every thread executes
// griddepcontrol.wait before it touches anything a predecessor wrote, and all but the producers before they release its dependents. Those
// wait later, right before their first load, or not at all where what they load has been complete for longer: weights, which no kernel
// that releases its dependents early writes, and the inputs of a batch-norm apply pass, whose predecessor reads them too.
template <typename... KArgs, typename... Args>
cudaError_t pt_launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Copies `bytes` of host data into the region's slot of the arena if it differs from what is there.
// Returns the device address of the slot.
pt_status pt_upload_table(pt_ctx *ctx, pt_region *reg, const void *host, size_t bytes, cudaStream_t st, char **dev);
// Validation shared by the conv entry points. Fills P, Q.
pt_status pt_conv_validate(const pt_ctx *ctx, const pt_conv_desc *d, int *P, int *Q);

// SIMT (CUDA-core) convolution kernels: every legal shape.
pt_status pt_simt_conv(pt_ctx *ctx, const pt_conv_desc *d, int which, const void *a, const void *b, void *out,
                       void *ws, size_t ws_bytes, cudaStream_t st);
size_t pt_simt_conv_workspace(const pt_ctx *ctx, const pt_conv_desc *d, int which);

// tcgen05 / TMEM / TMA convolution kernels: returns PT_ERR_UNSUPPORTED for shapes they do not cover.
bool pt_sm100_conv_supported(const pt_ctx *ctx, const pt_conv_desc *d, int which);
pt_status pt_sm100_conv(pt_ctx *ctx, const pt_conv_desc *d, int which, const void *a, const void *b, void *out,
                        void *ws, size_t ws_bytes, cudaStream_t st);
size_t pt_sm100_conv_workspace(const pt_ctx *ctx, const pt_conv_desc *d, int which);
int pt_sm100_wgrad_ctas(const pt_ctx *ctx, const pt_conv_desc *d, int *waits);
pt_status pt_sm100_set_wait_limit_ns(unsigned long long ns);
pt_status pt_bn_set_wait_limit_ns(unsigned long long ns);
pt_status pt_gate_set_wait_limit_ns(unsigned long long ns);
