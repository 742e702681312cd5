// C ABI of the FFF inference library: handle management, argument checks,
// stage planning and kernel launches.  Declarations and the contract of every
// entry point are in include/fff.h.
#include "../../include/fff.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <new>
#include <set>
#include <vector>

#include "kernels/block_forward.cuh"
#include "kernels/block_tiles.cuh"
#include "kernels/bucket.cuh"
#include "kernels/common.cuh"
#include "kernels/descent_mma.cuh"
#include "kernels/descent_umma.cuh"
#include "kernels/descent_warp.cuh"
#include "kernels/gemm_umma.cuh"
#include "kernels/leaf_mma.cuh"
#include "kernels/leaf_mma_warp.cuh"
#include "kernels/leaf_umma.cuh"
#include "kernels/leaf_warp.cuh"
#include "kernels/stack.cuh"
#include "kernels/token_block.cuh"

namespace {

constexpr uint64_t kMagic = 0x4646465f42323030ull;   // "FFF_B200"

struct DeviceGuard {
    int prev = -1;
    bool switched = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) switched = (cudaSetDevice(dev) == cudaSuccess);
    }
    ~DeviceGuard() { if (switched) cudaSetDevice(prev); }
};

}  // namespace

struct fff_handle_s {
    uint64_t magic = kMagic;
    int device = 0;
    int sm_count = 148;
    int D = 0, O = 0, depth = 0, l = 0;
    int Dp = 0;                   // D rounded up to the K step of the tensor-core images, which are padded with zero columns
    bool padded() const { return D != Dp; }      // the leaf kernels then keep the hidden values' float32 precision (kSplit in leaf_umma.cuh)
    int act = 0, dtype = 0;
    size_t esize = 4;
    int64_t n_nodes = 0, n_leaves = 1;
    bool vec_ok = false;          // rows of x / W start on 16-byte boundaries and D % kVec == 0

    // library-owned copies of the parameters, caller layout
    void *node_w = nullptr, *node_b = nullptr, *w1 = nullptr, *b1 = nullptr, *w2 = nullptr, *b2 = nullptr;

    // tensor-core leaf path: padded hidden width (0 = shapes not eligible) and pre-swizzled stage images
    int LP = 0;
    __nv_bfloat16* w1img = nullptr;
    float* b1img = nullptr;
    unsigned char* w2img = nullptr;
    unsigned char* w2uimg = nullptr;   // W2 pieces (+ biases) of the tcgen05 leaf kernel (nullptr = kernel not available)
    int* ws_sched = nullptr;           // its tile counter and finished-CTA counter (zero between launches); 8-bit weights: [2] has NaN codes
    // 8-bit leaf weights (fff_create_w8): code images of the tcgen05 leaf kernel and the per-leaf scales
    bool w8 = false;
    unsigned char *w1codes = nullptr, *w2codes = nullptr;
    float *scale1 = nullptr, *scale2 = nullptr;
    // grouped tiles of the tcgen05 leaf kernel (8 leaves per tile, bins = the nodes three levels above the leaves):
    // weight images (nullptr = shapes not eligible) and the first stage that ends at those nodes
    __nv_bfloat16* g_w1 = nullptr;
    float* g_b1 = nullptr;
    unsigned char* g_w2 = nullptr;
    bool slots_no_pos2 = false;        // the stage that files the tokens does not end at the leaves: no second copy of its positions
    // direct lists between the first and the second descent stage (two-stage trees): per node of the first stage's last
    // level a list of the tokens that reached it, filled by the first stage and read by the grouped second stage
    int32_t* ws_nslots = nullptr;      // [2^k0][nslot_cap]
    int32_t* ws_ncursor = nullptr;     // [kUGMaxBins] counts (zero between forwards) + [1] finished-CTA counter
    int64_t nslot_cap = 0;
    bool ncursor_dirty = false;
    bool nslots_here = false;          // the stage being launched files its tokens under the nodes it reaches
    fff::Tile* ws_tiles = nullptr;

    // workspace
    int64_t cap_B = 0;
    uint64_t epoch = 0;           // counts its allocations: a recorded graph holds the addresses of one
    int32_t *ws_leaf = nullptr, *ws_perm = nullptr, *ws_offsets = nullptr;
    int32_t* ws_rank = nullptr;   // per-token rank scratch of the bucketing kernel (large batches only)
    uint8_t* ws_rank8 = nullptr;  // rank of every token inside its 128-token tile, left by the first descent stage
    uint8_t* ws_counts8 = nullptr;   // and that stage's per-tile counts, [ceil(B/128)][<= 256]
    int32_t* ws_blocksum = nullptr;  // [4] CTA counter of k_bucket_ranked, then the counts summed over blocks of 16 tiles
    size_t blocksum_bytes = 0;
    bool blocksum_dirty = false;     // a descent has added to the table and no ranked bucketing has cleared it since
    bool blocksum_wanted = false;    // k_bucket_ranked follows the first descent stage of the call in progress
    // direct lists (slot_tokens in descent_umma.cuh): when one tcgen05 stage is the whole descent and the tcgen05
    // leaf kernel follows, the descent files every token under its leaf itself and no bucketing kernel runs
    int32_t* ws_slots = nullptr;     // [n_leaves][slot_cap] token numbers
    int32_t* ws_cursor = nullptr;    // [n_leaves] entries used, [1] finished CTAs, [1] CTAs at k_block_forward's barrier; zero between calls
    int64_t slot_cap = 0;
    bool cursor_dirty = false;       // a descent has filled the lists and no leaf kernel has cleared the counts since
    bool slots_now = false;          // the call in progress uses the direct lists
    bool slots_here = false;         // ... and the descent stage being launched is the one that fills them (the last)
    int max_bucket_clusters = 8;
    int32_t* last_perm = nullptr; // where the most recent forward left its leaf permutation
    bool bucketing_pending = false;   // the last forward skipped the leaf bucketing; ws_leaf holds its leaf indices
    bool pending_in_staging = false;  // ... or, after a host-buffer forward in chunks, st_leaf
    int* ws_matrix = nullptr;     // per-CTA bin totals of the grid-wide bucketing kernel
    int coop_ctas = 0;            // CTAs of that kernel that are resident at once (0 = cooperative launch unavailable)
    int32_t* ws_perm2 = nullptr;  // second permutation buffer: successive bucketings alternate between the two
    int32_t* ws_offsets2[2] = {nullptr, nullptr};   // offsets of the intermediate (node) bucketings

    // one-launch forward on CUDA cores (block_forward.cuh): its CTAs per SM (0: shapes not eligible), and whether the layer
    // may be pinned to it (FFF_PATH_FUSED)
    int bf_per_sm = 0;
    bool bf_pinnable = false;
    float* w2t = nullptr;         // float32: output weights as [leaf][l][O] for k_block_tiles (nullptr: shapes not eligible)
    int64_t bt_B = -1;            // its plan for the batch size last used
    bool bt_fits = false;
    fff::BlockTilesLayout bt_lay = {};

    // FORWARD_T (fff_forward_train): transposed output weights with the output biases appended along K, and the
    // workspace of the three GEMMs (allocated on first use)
    __nv_bfloat16* tr_w2t = nullptr;     // [O][tr_Kp]
    __nv_bfloat16* tr_w1t = nullptr;     // hidden weights in the order of the GEMM's columns, and their biases
    float* tr_b1t = nullptr;
    __nv_bfloat16* tr_wn = nullptr;      // node weights in the order of k_train_nodes' columns (1 <= depth <= 8), and their biases
    float* tr_bn = nullptr;
    bool tr_packed = false;              // the images below exist
    int tr_Kp = 0;                       // 2^d l + 2^d rounded up to 64 (0 = shapes not eligible)
    int64_t tr_cap_B = 0;
    float *tr_c = nullptr, *tr_mix = nullptr, *tr_entpart = nullptr;
    __nv_bfloat16* tr_hp = nullptr;

    // staged descent on tensor cores: consecutive groups of levels, each with its weight image
    struct DenseStage {
        int L0 = 0, k = 0, NP = 0;
        bool umma = false;            // first stage on the tcgen05 kernel (up to 8 levels)
        __nv_bfloat16* wimg = nullptr;
        float* bimg = nullptr;
    };
    std::vector<DenseStage> stages;
    std::vector<DenseStage> gstages;   // grouped tiles: one stage of depth - 3 levels
    // the same with a first stage of up to 8 levels on the tcgen05 kernel (empty = not available)
    std::vector<DenseStage> ustages;
    DenseStage halves;                 // the levels of ustages[0] below the root as two images (k_descent_umma<NP, true>); NP = 0: none
    int32_t* ws_pos[2] = {nullptr, nullptr};
    int *d_status = nullptr;

    // staging for the host-buffer entry point
    int64_t cap_host_B = 0;
    void *st_x = nullptr, *st_y = nullptr;
    int32_t *st_leaf = nullptr;
    // copy streams and events of the chunked host-buffer pipeline (created on first use)
    static constexpr int kMaxHostChunks = 16;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t ev_in[kMaxHostChunks] = {}, ev_done[kMaxHostChunks] = {}, ev_start = nullptr, ev_end = nullptr;

    int path = FFF_PATH_AUTO;
    bool tune[FFF_TUNE_COUNT] = {true, true, true, true, true, true, true, true};      // fff_set_tuning; every switch defaults to on
    bool pdl = true;              // launch every kernel of a forward but the first as a programmatic dependent
    int launches = 0;
    int64_t last_B = -1;
    int64_t plan_B = 0;           // chunk of a larger batch: kernels that round differently are chosen as for that many tokens (0: the call's own)

    // optional per-launch timing of forwards (fff_profile_*)
    static constexpr int kMaxProfLaunches = 16;
    int prof_max_steps = 0, prof_steps = 0;
    bool prof_active = false;                     // this forward is being recorded
    int prof_nlaunch = 0;                         // launches per forward of the recorded steps
    const char* prof_names[kMaxProfLaunches] = {};
    std::vector<cudaEvent_t> prof_events;         // [prof_max_steps][kMaxProfLaunches + 1]
};

// Several layers behind one handle (fff_stack_*): the layers stay the caller's; the stack owns the buffers
// between them, the normalisation parameters and, when asked to, one instantiated CUDA graph of its forward.
struct fff_stack_s {
    uint64_t magic = 0;
    int device = 0, sm_count = 148;
    std::vector<fff_handle_s*> layers;
    std::vector<void*> gamma, beta;       // per layer, library-owned copies (nullptr = 1 / 0)
    bool layer_norm = false, residual = false;
    float eps = 1e-5f;
    int D = 0, dtype = 0;
    size_t esize = 4;
    int64_t cap_B = 0;
    void *buf_z = nullptr, *buf_y = nullptr, *buf_x[2] = {nullptr, nullptr};
    // graph replay: the key of the forward that the instantiated graph holds, and of the last eager forward
    bool want_graph = false, graph_failed = false;
    cudaGraphExec_t exec = nullptr;
    const void *key_x = nullptr, *key_y = nullptr, *key_leaf = nullptr, *seen_x = nullptr, *seen_y = nullptr, *seen_leaf = nullptr;
    int64_t key_B = -1, seen_B = -1;
    uint64_t key_epoch = 0;               // sum of the layers' epochs at the recording
    cudaStream_t key_stream = nullptr, seen_stream = nullptr;
    int launches = 0;
    bool replayed = false;
};

namespace {

constexpr uint64_t kStackMagic = 0x4646465f53544b31ull;   // "FFF_STK1"

std::mutex g_mu;
std::set<fff_handle_s*> g_live;
std::set<fff_stack_s*> g_live_stacks;

bool live_stack(fff_stack_s* s) {
    if (!s) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_live_stacks.count(s) != 0 && s->magic == kStackMagic;
}

bool live(fff_handle_t h) {
    if (!h) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_live.count(h) != 0 && h->magic == kMagic;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

fff_status_t dmalloc(void** p, size_t bytes) {
    *p = nullptr;
    bytes = std::max<size_t>((bytes + 15) & ~(size_t)15, 16);      // (whole 16-byte vectors: bulk copies read the last one)
    return cudaMalloc(p, bytes) == cudaSuccess ? FFF_OK : (cudaGetLastError(), FFF_ERR_ALLOC);
}

void dfree(void* p) { if (p) cudaFree(p); }

// A copy of `src`, or zeroes, made on the default stream: the call returns before they are in place (default_stream_done).
fff_status_t clone(void** dst, const void* src, size_t bytes) {
    fff_status_t s = dmalloc(dst, bytes);
    if (s != FFF_OK) return s;
    cudaError_t e = src ? cudaMemcpy(*dst, src, bytes, cudaMemcpyDeviceToDevice) : cudaMemset(*dst, 0, bytes ? bytes : 16);
    return e == cudaSuccess ? FFF_OK : (cudaGetLastError(), FFF_ERR_CUDA);
}

// Waits for copies and memsets of device memory on the default stream, which return before they are done: a caller's
// non-blocking stream does not wait for that stream, so whoever allocates on behalf of a call in progress does it here.
fff_status_t default_stream_done(cudaError_t e) {
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    return e == cudaSuccess ? FFF_OK : (cudaGetLastError(), FFF_ERR_CUDA);
}

// Launch a kernel of the forward chain.  Every launch after the first of a call carries the
// programmatic-stream-serialization attribute: the kernel may be scheduled while its predecessor is
// still draining, runs its prologue, and waits in griddepcontrol.wait (cudaGridDependencySynchronize)
// until the predecessor has completed and flushed its results.  Every kernel launched through here
// calls that wait before its first global read.
template <typename... KArgs, typename... Args>
cudaError_t launch_chain(fff_handle_s* h, void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                         int cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    // (also the first kernel of a call: it may then start its prologue while the last kernel of the
    // previous call on this stream drains; with any other predecessor the attribute changes nothing)
    if (h->pdl && !h->prof_active) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)n;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

void prof_free(fff_handle_s* h) {
    for (cudaEvent_t e : h->prof_events) cudaEventDestroy(e);
    h->prof_events.clear();
    h->prof_max_steps = h->prof_steps = h->prof_nlaunch = 0;
    h->prof_active = false;
}

void release(fff_handle_s* h) {
    dfree(h->w2t);
    dfree(h->node_w); dfree(h->node_b); dfree(h->w1); dfree(h->b1); dfree(h->w2); dfree(h->b2);
    dfree(h->ws_leaf); dfree(h->ws_perm); dfree(h->ws_perm2); dfree(h->ws_offsets); dfree(h->ws_offsets2[0]); dfree(h->ws_offsets2[1]);
    dfree(h->d_status); dfree(h->st_x); dfree(h->st_y); dfree(h->st_leaf);
    for (auto& sg : h->stages) { dfree(sg.wimg); dfree(sg.bimg); }
    for (auto& sg : h->ustages) { dfree(sg.wimg); dfree(sg.bimg); }
    dfree(h->halves.wimg); dfree(h->halves.bimg);
    for (auto& sg : h->gstages) { dfree(sg.wimg); dfree(sg.bimg); }
    dfree(h->g_w1); dfree(h->g_b1); dfree(h->g_w2);
    dfree(h->ws_pos[0]); dfree(h->ws_pos[1]);
    dfree(h->w1codes); dfree(h->w2codes); dfree(h->scale1); dfree(h->scale2);
    dfree(h->tr_w2t); dfree(h->tr_w1t); dfree(h->tr_b1t); dfree(h->tr_wn); dfree(h->tr_bn); dfree(h->tr_c); dfree(h->tr_mix); dfree(h->tr_entpart); dfree(h->tr_hp);
    dfree(h->w1img); dfree(h->b1img); dfree(h->w2img); dfree(h->w2uimg); dfree(h->ws_sched); dfree(h->ws_tiles); dfree(h->ws_rank); dfree(h->ws_rank8); dfree(h->ws_counts8); dfree(h->ws_blocksum); dfree(h->ws_matrix); dfree(h->ws_slots); dfree(h->ws_cursor); dfree(h->ws_nslots); dfree(h->ws_ncursor);
    if (h->copy_in) cudaStreamDestroy(h->copy_in);
    if (h->copy_out) cudaStreamDestroy(h->copy_out);
    for (int i = 0; i < fff_handle_s::kMaxHostChunks; ++i) {
        if (h->ev_in[i]) cudaEventDestroy(h->ev_in[i]);
        if (h->ev_done[i]) cudaEventDestroy(h->ev_done[i]);
    }
    if (h->ev_start) cudaEventDestroy(h->ev_start);
    if (h->ev_end) cudaEventDestroy(h->ev_end);
    prof_free(h);
    h->magic = 0;
    delete h;
}

constexpr int kMinTileRows = 32;

constexpr int kMaxDevices = 64;          // device ordinals the per-device tables below cover (fff_create checks)
std::mutex g_attr_mu;

// Raises a kernel's dynamic shared-memory limit on the handle's device, once per device and kernel
// (`done` is that kernel's table).  Handles on different host threads may get here at the same time.
template <typename K>
bool raise_smem_limit(K kern, int device, int bytes, bool (&done)[kMaxDevices]) {
    std::lock_guard<std::mutex> lk(g_attr_mu);
    if (done[device]) return true;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
        return cudaGetLastError(), false;
    done[device] = true;
    return true;
}

// Length of a tile list: floor(B / tile_rows) + nbins entries, some of them empty (see k_bucket_cluster).
int tile_list_len(int64_t B, int tile_rows, int nbins) { return (int)(B / tile_rows) + nbins; }

// Leaves whose tiles the mma.sync leaf kernel derives from the lists' counts (more would cost it its second CTA per SM),
// and the batches for which their number fits 16 bits.
constexpr int kMaxListedLeaves = 2048;
constexpr int64_t kMaxListedTokens = 1 << 20;
constexpr size_t kMaxSlotBytes = (size_t)1 << 30;      // largest table of direct lists a handle allocates

// Capacity of the tile buffer: the longest list any stage can ask for.
size_t max_tiles(const fff_handle_s* h, int64_t B) { return (size_t)(B / kMinTileRows + h->n_leaves + 1); }

// Which tensor-core leaf kernel runs, and on tiles of how many token rows.
struct LeafPlan {
    int tile_rows = 0;
    bool umma = false;
    bool resident = false;         // the tiles of all leaves run at once
};

// Tiles of tile_rows rows that B tokens spread over the leaves fill, on average (a leaf's count is about Poisson): the sum over k
// of the chance that a leaf has more than k tiles' worth of tokens.  Once counts spread over whole tiles (standard deviation of
// tile_rows) the last tile of a leaf is half full on average and the sum is its mean plus a half.
double expected_tiles(const fff_handle_s* h, int64_t B, int tile_rows) {
    const double mean = (double)B / (double)h->n_leaves, sd2 = std::sqrt(2.0 * mean);
    if (mean >= (double)tile_rows * tile_rows) return (mean / tile_rows + 0.5) * (double)h->n_leaves;
    double per_leaf = 1.0 - std::exp(-mean);
    for (int k = 1; (k * tile_rows - mean) / sd2 < 4.5; ++k) per_leaf += 0.5 * std::erfc((k * tile_rows + 0.5 - mean) / sd2);
    return per_leaf * (double)h->n_leaves;
}

template <int LP, int TM, int S> int leaf_mma_slots(const fff_handle_s* h) {
    using L = fff::LeafMmaLayout<LP, TM, S>;
    const int smem = L::kSmemBytes + L::list_bytes((int)std::min<int64_t>(h->n_leaves, kMaxListedLeaves));
    return h->sm_count * std::max(1, std::min(2, (227 * 1024) / (smem + 1024)));
}
// CTAs of the mma.sync leaf kernel that are resident at once (ring depths as in run_leaf_mma).
int leaf_mma_slots(const fff_handle_s* h, int tile_rows) {
    switch (h->LP) {
        case 16: return tile_rows == 32 ? leaf_mma_slots<16, 32, 6>(h) : leaf_mma_slots<16, 64, 4>(h);
        case 32: return tile_rows == 32 ? leaf_mma_slots<32, 32, 5>(h) : leaf_mma_slots<32, 64, 3>(h);
        default: return tile_rows == 32 ? leaf_mma_slots<64, 32, 4>(h) : leaf_mma_slots<64, 64, 4>(h);
    }
}

LeafPlan leaf_plan(const fff_handle_s* h, int64_t B) {
    if (h->w8) return LeafPlan{fff::kLUM, true};
    // While the tiles of all leaves are resident at once, the mma.sync kernel (two CTAs per SM for leaves of up to 32 neurons,
    // no tensor memory to set up) is ahead: 768 -> 768, 256 leaves of 12, with the descent: 19.3 against 24.1 us at 4096 tokens
    // and 19.6 against 24.6 at 6144 (32-row tiles), 22.7 against 25.8 at 8192 and 25.0 against 30.1 at 12 608 (64-row tiles);
    // a second round of tiles costs more than it saves: 38.3 against 34.0 at 16 384.
    for (int rows : {32, 64})
        if (expected_tiles(h, B, rows) <= 0.98 * leaf_mma_slots(h, rows)) return LeafPlan{rows, false, true};
    // The tcgen05 kernel works on 128-row tiles.  Measured against the mma.sync kernel it is far ahead when
    // some buckets are large (skewed routing), about level with uniformly thin buckets of 32 tokens, and is
    // left out only when buckets are thinner still (tiles of at most 64 rows are stacked in the MMA rows, so the
    // epilogue's cost follows the rows; the rest of a tile's cost is fixed).
    if (h->w2uimg && h->tune[FFF_TUNE_TCGEN05_LEAF] && B >= 16 * h->n_leaves) {
        return LeafPlan{fff::kLUM, true};
    }
    return LeafPlan{B / h->n_leaves <= 40 ? 32 : 64, false};
}

// Whether a forward whose descent files the tokens runs a warp per tile of up to 16 tokens (k_leaf_mma_warp) instead: thin
// buckets, more of them than CTAs at once.  Forwards, us, with the other kernels and with it: 768 -> 768, 2048 leaves of 12:
// 2500 tokens 53.0 and 40.0, 8192 68.1 and 55.2, 16 384 75.6 and 69.1; 1024 leaves of 16: 2500 43.9 and 32.3, 12 000 48.8 and
// 41.5; 512 leaves of 16: 8192 42.5 and 33.9, 16 384 47.2 and 42.6; 256 -> 256, 2048 leaves of 10: 8192 42.5 and 26.4, 24 000
// 48.4 and 36.6.  It fetches a row in pieces of 64 bytes, which tells once the rows outweigh the weights: 1024 -> 1024, 2048
// leaves of 16: 16 384 tokens (32 MB) 91.1 and 90.2, 20 000 94.8 and 100.9; 768 -> 768, 1024 leaves of 16: 32 768 73.2 and 85.5.
// With tokens of 16 clusters, which fill a few leaves (their weights then come from L2): 768 -> 768, 2048 leaves of 12: 16 384 tokens
// 58.2 and 41.0; 1024 of 16: 16 384 47.4 and 37.3; 512 of 16: 8192 37.4 and 31.1, 19 968 55.5 and 48.0; 256 -> 256, 2048 of 10: 16 384
// 44.9 and 27.6.
bool warp_tiles(const fff_handle_s* h, const LeafPlan& plan, int64_t B) {
    return h->LP == 16 && !plan.resident && h->n_leaves <= kMaxListedLeaves && B < 40 * h->n_leaves &&
           B * h->D * h->esize <= ((int64_t)32 << 20);
}

bool use_tensor_leaf(const fff_handle_s* h) {
    if (h->w8) return true;            // 8-bit leaf weights exist for the tcgen05 leaf kernel only
    if (h->LP == 0 || h->path == FFF_PATH_WARP) return false;
    return h->path == FFF_PATH_TENSOR || h->l >= 8;
}

// Tokens for which the leaves' lists stay within kMaxSlotBytes, and the fewest that k_block_forward is given at a time.
int64_t listed_tokens(const fff_handle_s* h) { return (int64_t)(kMaxSlotBytes / sizeof(int32_t)) / h->n_leaves; }
constexpr int64_t kMinListedTokens = 1024;
size_t cursor_bytes(const fff_handle_s* h) { return sizeof(int32_t) * (size_t)(h->n_leaves + 2); }

// Whether forwards of this handle, as it is pinned now, run as the one-launch kernel on CUDA cores: the layers without a
// tensor-core leaf path, and those pinned to it.  Shapes and the path alone decide, not what the handle has served before.
bool runs_block_forward(const fff_handle_s* h) {
    return h->bf_per_sm > 0 && (h->path == FFF_PATH_FUSED || (h->path == FFF_PATH_AUTO && h->LP == 0));
}

fff_status_t grow_workspace(fff_handle_s* h, int64_t B) {
    if (B <= h->cap_B) return FFF_OK;
    if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    // the last forward's permutation and leaf indices go with the buffers (a bucketing still to be made from the staging buffers stays)
    if (!(h->pending_in_staging && h->bucketing_pending)) h->last_B = -1;
    ++h->epoch;
    dfree(h->ws_leaf); dfree(h->ws_perm); dfree(h->ws_perm2); dfree(h->ws_tiles); dfree(h->ws_rank); dfree(h->ws_pos[0]);
    dfree(h->ws_rank8); dfree(h->ws_counts8); dfree(h->ws_blocksum); dfree(h->ws_slots); dfree(h->ws_cursor); dfree(h->ws_nslots);
    dfree(h->ws_ncursor);
    h->ws_slots = h->ws_cursor = h->ws_nslots = h->ws_ncursor = nullptr;
    h->slot_cap = 0;
    h->ws_rank8 = h->ws_counts8 = nullptr;
    h->ws_blocksum = nullptr;
    dfree(h->ws_pos[1]);
    h->ws_leaf = h->ws_perm = h->ws_perm2 = h->ws_rank = h->ws_pos[0] = h->ws_pos[1] = nullptr;
    h->ws_tiles = nullptr;
    h->cap_B = 0;
    fff_status_t s;
    if ((s = dmalloc((void**)&h->ws_leaf, sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->ws_perm, sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->ws_perm2, sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->ws_rank, sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
    if (!h->ustages.empty()) {
        if ((s = dmalloc((void**)&h->ws_rank8, (size_t)B)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->ws_counts8, (size_t)((B + 127) / 128) * 256)) != FFF_OK) return s;
        h->blocksum_bytes = sizeof(int32_t) * (4 + (size_t)(((B + 127) / 128 + fff::kRankBlock - 1) / fff::kRankBlock) * 256);
        if ((s = clone((void**)&h->ws_blocksum, nullptr, h->blocksum_bytes)) != FFF_OK) return s;      // zeroed
        h->blocksum_dirty = false;
    }
    if (h->stages.size() > 1 || h->ustages.size() > 1 || h->g_w1) {
        if ((s = dmalloc((void**)&h->ws_pos[0], sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->ws_pos[1], sizeof(int32_t) * (size_t)B)) != FFF_OK) return s;
    }
    if ((s = dmalloc((void**)&h->ws_tiles, sizeof(fff::Tile) * max_tiles(h, B))) != FFF_OK) return s;
    // direct lists: every leaf's list can take the whole batch, so their size grows with n_leaves * B; beyond
    // kMaxSlotBytes the forward keeps the bucketing kernel instead.  k_block_forward has no other way: for the layers that
    // run it the table stops growing there, and larger batches go through it in parts.
    const bool filed_by_descent = !h->ustages.empty() && h->ustages.back().umma &&
                                  h->ustages.back().L0 + h->ustages.back().k == h->depth && (h->w2uimg || h->w2codes);
    const int64_t most = listed_tokens(h);
    if (runs_block_forward(h) || ((filed_by_descent || (h->bf_per_sm > 0 && h->bf_pinnable)) && B <= most)) {
        int64_t cap = std::min(B, most);
        s = dmalloc((void**)&h->ws_slots, sizeof(int32_t) * (size_t)h->n_leaves * (size_t)cap);
        // (short of memory: smaller parts)
        while (s != FFF_OK && runs_block_forward(h) && cap > kMinListedTokens) {
            cap = std::max(cap / 4 & ~int64_t(15), kMinListedTokens);
            s = dmalloc((void**)&h->ws_slots, sizeof(int32_t) * (size_t)h->n_leaves * (size_t)cap);
        }
        if (s != FFF_OK) return s;
        if ((s = clone((void**)&h->ws_cursor, nullptr, cursor_bytes(h))) != FFF_OK) return s;
        h->slot_cap = cap;
        h->cursor_dirty = false;
    }
    // node lists for trees whose descent runs as two tcgen05 stages (a forward decides: the stages it runs depend on B):
    // [nodes of the first stage][B]
    if (h->ustages.size() >= 2 && h->ustages[0].umma && h->ustages[1].umma && (1 << h->ustages[0].k) <= fff::kUGMaxBins &&
        ((size_t)B << h->ustages[0].k) * sizeof(int32_t) <= kMaxSlotBytes) {
        if ((s = dmalloc((void**)&h->ws_nslots, sizeof(int32_t) * ((size_t)B << h->ustages[0].k))) != FFF_OK) return s;
        if ((s = clone((void**)&h->ws_ncursor, nullptr, sizeof(int32_t) * (fff::kUGMaxBins + 1))) != FFF_OK) return s;
        h->nslot_cap = B;
        h->ncursor_dirty = false;
    }
    if ((s = default_stream_done(cudaSuccess)) != FFF_OK) return s;       // the counters are zero on every stream
    h->cap_B = B;
    return FFF_OK;
}

// Called after every kernel launch: counts it, records its profiling event, reports launch errors.
fff_status_t launched(fff_handle_s* h, cudaStream_t st, const char* name) {
    const int i = h->launches++;
    if (h->prof_active && i < fff_handle_s::kMaxProfLaunches) {
        h->prof_names[i] = name;
        cudaEventRecord(h->prof_events[(size_t)h->prof_steps * (fff_handle_s::kMaxProfLaunches + 1) + i + 1], st);
    }
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}


// ---- stage launchers -------------------------------------------------------

// Whether k_bucket_ranked can follow a first descent stage over B tokens (few enough 128-token tiles per CTA).
bool ranked_bucketing_fits(const fff_handle_s* h, int64_t B) {
    const int64_t n_src = (B + fff::kRankTile - 1) / fff::kRankTile;
    const int64_t ctas = std::min<int64_t>(h->sm_count, n_src);
    return B > 0 && h->ws_rank8 && h->ws_counts8 && h->ws_blocksum &&
           (n_src + ctas - 1) / ctas <= fff::kRankedMaxTilesPerCta;
}

// The block-sum table the first descent stage adds to, ready for use: null when no ranked bucketing can follow,
// cleared first if an earlier descent was not followed by one.
fff_status_t blocksum_for_descent(fff_handle_s* h, int64_t B, bool ranked, cudaStream_t st, int32_t** table) {
    *table = nullptr;
    if (!ranked || !h->blocksum_wanted || !ranked_bucketing_fits(h, B)) return FFF_OK;
    if (h->blocksum_dirty && cudaMemsetAsync(h->ws_blocksum, 0, h->blocksum_bytes, st) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    h->blocksum_dirty = true;
    *table = h->ws_blocksum + 4;
    return FFF_OK;
}

// What a bucketing refines: nothing (all tokens in natural order), or the previous bucketing.
struct Coarse {
    const int32_t* perm = nullptr;      // previous permutation
    const int32_t* offsets = nullptr;   // its offsets, one segment per coarse bin
    int bins = 0;                       // number of coarse bins
    bool ranked = false;                // no previous bucketing, but the keys come with the first descent stage's
                                        // per-tile ranks and counts (ws_rank8, ws_counts8)
};

template <int NW>
cudaError_t launch_bucket(fff_handle_s* h, int clusters, size_t smem, cudaStream_t st, const int32_t* keys,
                          const int32_t* perm_in, const int32_t* seg_offsets, int32_t* offsets, int32_t* perm, int B, int nbins,
                          int nb, int bin_bits, int tile_rows, fff::Tile* tiles, int n_tiles_total, int32_t* rank_tmp) {
    return launch_chain(h, fff::k_bucket_cluster<NW>, (unsigned)(clusters * fff::kBucketClusterSize), NW * 32, smem, st,
                        fff::kBucketClusterSize, keys, perm_in, seg_offsets, offsets, perm, B, nbins, nb, bin_bits, tile_rows,
                        tiles, n_tiles_total, rank_tmp);
}

// Stable bucketing of B keys in [0, nbins) into (offsets, perm).  If `coarse` describes a bucketing by
// key >> log2(nbins / coarse.bins), only the inside of each coarse bucket is re-ordered (one cluster per
// coarse bucket); otherwise clusters split the bin range and each scans all keys.
// tile_rows > 0 also writes the tile list (tile_list_len(B, tile_rows, nbins) entries) into ws_tiles.
fff_status_t run_bucket(fff_handle_s* h, const int32_t* keys, int nbins, const Coarse& coarse, int32_t* offsets,
                        int32_t* perm, int64_t B, cudaStream_t st, int tile_rows, const char* name) {
    const int n_tiles_total = tile_rows > 0 ? tile_list_len(B, tile_rows, nbins) : 0;
    cudaError_t e;
    const int64_t n_src = (B + fff::kRankTile - 1) / fff::kRankTile;
    const int64_t ranked_ctas = std::min<int64_t>(h->sm_count, n_src);
    if (coarse.ranked && !coarse.perm && nbins >= 16 && nbins <= 256 && ranked_bucketing_fits(h, B)) {
        // the descent kernel has done the ranking: sum its per-tile counts and scatter
        if (launch_chain(h, fff::k_bucket_ranked, (unsigned)ranked_ctas, fff::kRankedThreads,
                         sizeof(int) * (size_t)(3 + fff::kRankedMaxTilesPerCta) * nbins, st, 1, keys, (const uint8_t*)h->ws_rank8,
                         (const uint8_t*)h->ws_counts8, h->ws_blocksum + 4, (int*)h->ws_blocksum, offsets, perm, (int)B, nbins,
                         tile_rows, h->ws_tiles, n_tiles_total) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        h->blocksum_dirty = false;          // the kernel clears the table when all its CTAs have read it
        return launched(h, st, name);
    }
    // Refining pays while the coarse buckets are few and large; thousands of tiny buckets would mean
    // thousands of tiny clusters, and scanning all keys from a few clusters is cheaper then.
    if (coarse.perm && nbins / coarse.bins <= fff::kBucketMaxBinsPerCta && coarse.bins <= 256) {
        const int nb = nbins / coarse.bins;
        int bin_bits = 0;
        while ((1 << bin_bits) < nb) ++bin_bits;
        if (nb <= 256)
            e = launch_bucket<8>(h, coarse.bins, sizeof(int) * (size_t)(8 + 1) * nb, st, keys, coarse.perm, coarse.offsets, offsets,
                                 perm, (int)B, nbins, nb, bin_bits, tile_rows, h->ws_tiles, n_tiles_total, h->ws_rank);
        else
            e = launch_bucket<32>(h, coarse.bins, sizeof(int) * (size_t)(32 + 1) * nb, st, keys, coarse.perm, coarse.offsets,
                                  offsets, perm, (int)B, nbins, nb, bin_bits, tile_rows, h->ws_tiles, n_tiles_total, h->ws_rank);
    } else if (h->coop_ctas > 0 && nbins <= fff::kBucketMaxBinsPerCta && B >= 4096) {
        // few bins, no previous bucketing: one token slice per SM and one grid-wide barrier
        const int ctas = (int)std::min<int64_t>(h->coop_ctas, (B + 255) / 256);
        int bin_bits = 0;
        while ((1 << bin_bits) < nbins) ++bin_bits;
        int Bi = (int)B, tr = tile_rows, nbi = nbins, ntt = n_tiles_total;
        const int32_t* k = keys;
        fff::Tile* tiles = h->ws_tiles;
        int32_t* rank = h->ws_rank;
        int* matrix = h->ws_matrix;
        void* args[] = {&k, &offsets, &perm, &Bi, &nbi, &bin_bits, &tr, &tiles, &ntt, &rank, &matrix};
        e = cudaLaunchCooperativeKernel((const void*)fff::k_bucket_coop, dim3((unsigned)ctas), dim3(fff::kCoopThreads), args,
                                        sizeof(int) * (size_t)(fff::kCoopWarps + 2) * nbins, st);
    } else {
        // Every cluster reads all keys, so more clusters do not shorten the kernel; they only shrink the
        // bin range (and the number of ballots per step).
        int clusters = std::max(1, std::min(std::min(nbins / 32, 8), h->max_bucket_clusters));
        int nb = (nbins + clusters - 1) / clusters;
        if (nb > fff::kBucketMaxBinsPerCta) nb = fff::kBucketMaxBinsPerCta;
        clusters = (nbins + nb - 1) / nb;
        int bin_bits = 0;
        while ((1 << bin_bits) < nb) ++bin_bits;
        e = launch_bucket<32>(h, clusters, sizeof(int) * (size_t)(32 + 1) * nb, st, keys, nullptr, nullptr, offsets, perm, (int)B,
                              nbins, nb, bin_bits, tile_rows, h->ws_tiles, n_tiles_total, h->ws_rank);
    }
    if (e != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, name);
}

constexpr int kSmemBudget = 227 * 1024 - 1024;      // usable shared memory of an SM, less the per-CTA reservation

template <int NP>
fff_status_t launch_descent_mma(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, const int32_t* perm,
                                bool grouped, int32_t* pos_out, int64_t B, cudaStream_t st) {
    using L = fff::DescentMmaLayout<NP>;
    // A single-group stage keeps its weight image resident if at least 3 ring stages still fit.
    const int res_bytes = NP * h->Dp * 2;
    const bool resident = !grouped && L::smem_bytes(3, res_bytes) <= kSmemBudget;
    // two CTAs per SM when that leaves at least 3 stages each, else one CTA with as many as fit
    auto stages_for = [&](int budget) {
        const int per = resident ? L::kXStageBytes : L::kStageStride;
        return std::min((int)fff::kMaxStages, (budget - L::kFixedBytes - (resident ? res_bytes : 0)) / per);
    };
    int per_sm = 2, stages = stages_for(kSmemBudget / 2 - 1024);
    if (stages < 3) { per_sm = 1; stages = stages_for(kSmemBudget); }
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    const int smem = L::smem_bytes(stages, resident ? res_bytes : 0);
    const int n_tiles = grouped ? tile_list_len(B, fff::kDTM, 1 << sg.L0) : (int)((B + fff::kDTM - 1) / fff::kDTM);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sm_count * per_sm, n_tiles));
    if (launch_chain(h, fff::k_descent_mma<NP>, (unsigned)grid, fff::kDescentThreads, (size_t)smem, st, 1,
                     (const __nv_bfloat16*)x, grouped ? perm : nullptr, grouped ? h->ws_tiles : nullptr, n_tiles, sg.wimg,
                     sg.bimg, pos_out, h->D, h->Dp, (int)B, sg.k, stages, resident ? 1 : 0, h->d_status) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "tree_descent_mma");
}

fff_status_t run_descent_mma(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, const int32_t* perm,
                             bool grouped, int32_t* pos_out, int64_t B, cudaStream_t st) {
    switch (sg.NP) {
        case 16: return launch_descent_mma<16>(h, sg, x, perm, grouped, pos_out, B, st);
        case 32: return launch_descent_mma<32>(h, sg, x, perm, grouped, pos_out, B, st);
        case 64: return launch_descent_mma<64>(h, sg, x, perm, grouped, pos_out, B, st);
    }
    return FFF_ERR_UNSUPPORTED;
}

// cuTensorMapEncodeTiled, looked up once through the runtime (the library does not link the driver).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// Tensor map of the bf16 token matrix x[B, D] for boxes of box_rows x 64 columns, 128-byte swizzled;
// rows past B read as zeros.
bool make_x_tensor_map(CUtensorMap* tm, const void* x, int64_t B, int D, int box_rows, bool swizzle = true) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)D, (cuuint64_t)B};
    const cuuint64_t gstride[1] = {(cuuint64_t)D * 2};
    const cuuint32_t box[2] = {(cuuint32_t)fff::kUKB, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), gdim, gstride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Arguments of the first descent stage for the direct lists (all null unless the call in progress uses them);
// the positions are also kept in the workspace, from which a bucketing can be made on demand afterwards.
struct SlotArgs {
    int32_t *pos2 = nullptr, *cursor = nullptr, *slots = nullptr;
    int cap = 0;
};
SlotArgs slot_args(const fff_handle_s* h, const int32_t* pos_out) {
    SlotArgs a;
    if (h->nslots_here) {              // the lists between the first and the second stage
        a.cursor = h->ws_ncursor;
        a.slots = h->ws_nslots;
        a.cap = (int)h->nslot_cap;
        return a;
    }
    if (!h->slots_here) return a;
    a.pos2 = pos_out == h->ws_leaf || h->slots_no_pos2 ? nullptr : h->ws_leaf;
    a.cursor = h->ws_cursor;
    a.slots = h->ws_slots;
    a.cap = (int)h->slot_cap;
    return a;
}

// CTAs for `units` equal work units walked with a static stride on at most `max_ctas` CTAs: the fewest CTAs that
// still need no more rounds, so that all of them finish together (512 tiles on 148 SMs: 128 CTAs with 4 tiles
// each instead of 68 with 4 and 80 with 3; the memory system is shared, so the idle SMs cost nothing).
int64_t balanced_grid(int64_t max_ctas, int64_t units) {
    max_ctas = std::max<int64_t>(1, max_ctas);
    if (units <= max_ctas) return std::max<int64_t>(1, units);
    const int64_t rounds = (units + max_ctas - 1) / max_ctas;
    return (units + rounds - 1) / rounds;
}

template <int NP, bool kHalves = false>
fff_status_t launch_descent_umma(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, int32_t* pos_out,
                                 int64_t B, cudaStream_t st) {
    using L = fff::DescentUmmaLayout<NP>;
    const int stages = std::min((int)fff::kUmmaMaxStages, (kSmemBudget - L::smem_bytes(0)) / L::kStageBytes);
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    CUtensorMap tm;
    if (!make_x_tensor_map(&tm, x, B, h->D, fff::kUM)) return FFF_ERR_CUDA;
    const int64_t n_tiles = (B + fff::kUM - 1) / fff::kUM;
    const int64_t grid = kHalves ? 2 * n_tiles : balanced_grid(h->sm_count, n_tiles);
    const bool ranked = !kHalves && !h->nslots_here && sg.k >= 4 && h->ws_rank8 && h->ws_counts8;      // also rank the tokens for the bucketing that follows
    int32_t* sums = nullptr;
    if (blocksum_for_descent(h, B, ranked, st, &sums) != FFF_OK) return FFF_ERR_CUDA;
    const SlotArgs sl = slot_args(h, pos_out);
    if (launch_chain(h, fff::k_descent_umma<NP, kHalves>, (unsigned)grid, fff::kUmmaThreads, (size_t)L::smem_bytes(stages), st, 1, tm,
                     (const __nv_bfloat16*)sg.wimg, (const float*)sg.bimg, pos_out, ranked ? h->ws_rank8 : (uint8_t*)nullptr,
                     ranked ? h->ws_counts8 : (uint8_t*)nullptr, sums, sl.pos2, sl.cursor, sl.slots, sl.cap, h->Dp, (int)B, sg.k + (kHalves ? 1 : 0),
                     stages, h->d_status) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "tree_descent_umma");
}

// The same on CTA pairs that share the weight K-blocks (NP >= 128, where re-streaming them binds the kernel).
template <int NP>
fff_status_t launch_descent_umma_pair(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, int32_t* pos_out,
                                      int64_t B, cudaStream_t st) {
    using L = fff::DescentUmmaPairLayout<NP>;
    const int stages = std::min((int)fff::kUmmaMaxStages, (kSmemBudget - L::smem_bytes(0)) / L::kStageBytes);
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_descent_umma_pair<NP>, h->device, kSmemBudget, limit_raised)) return FFF_ERR_CUDA;
    CUtensorMap tm, tw;
    if (!make_x_tensor_map(&tm, x, B, h->D, fff::kUM)) return FFF_ERR_CUDA;
    // the weight image as (D/64) * NP rows of 64 columns, stored pre-swizzled: copied as it is
    if (!make_x_tensor_map(&tw, sg.wimg, (int64_t)(h->Dp / fff::kUKB) * NP, fff::kUKB, NP / 2, false)) return FFF_ERR_CUDA;
    const int64_t n_pairs = ((B + fff::kUM - 1) / fff::kUM + 1) / 2;
    const int64_t grid = 2 * balanced_grid(h->sm_count / 2, n_pairs);
    const bool ranked = !h->nslots_here && sg.k >= 4 && h->ws_rank8 && h->ws_counts8;
    int32_t* sums = nullptr;
    if (blocksum_for_descent(h, B, ranked, st, &sums) != FFF_OK) return FFF_ERR_CUDA;
    const SlotArgs sl = slot_args(h, pos_out);
    if (launch_chain(h, fff::k_descent_umma_pair<NP>, (unsigned)grid, fff::kUmmaThreads, (size_t)L::smem_bytes(stages), st, 2, tm,
                     tw, (const float*)sg.bimg, pos_out, ranked ? h->ws_rank8 : (uint8_t*)nullptr,
                     ranked ? h->ws_counts8 : (uint8_t*)nullptr, sums, sl.pos2, sl.cursor, sl.slots, sl.cap, h->Dp, (int)B, sg.k,
                     stages, h->d_status) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "tree_descent_umma");
}

fff_status_t run_descent_umma(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, int32_t* pos_out, int64_t B,
                              cudaStream_t st) {
    const bool no_pair = !h->tune[FFF_TUNE_CTA_PAIRS];
    // pairs pay once there is more than one round of tiles (measured: 29.1 vs 31.2 us at 394 tiles, 18.7 vs 17.0 at 128)
    if (!no_pair && (B + fff::kUM - 1) / fff::kUM > h->sm_count && h->sm_count >= 2) {
        if (sg.NP == 128) return launch_descent_umma_pair<128>(h, sg, x, pos_out, B, st);
        if (sg.NP == 256) return launch_descent_umma_pair<256>(h, sg, x, pos_out, B, st);
    }
    // Two CTAs per tile while they are all resident at once (where the tokens are filed, not ranked: a rank needs the whole
    // tile).  Forwards of the 768 -> 768 layer with 256 leaves of 12, one CTA and two: 600 tokens 18.8 and 17.4 us, 3152 19.2
    // and 18.4, 6304 20.6 and 19.9, 9472 23.9 and 23.2; 256 -> 256: 3152 tokens 13.8 and 12.5; 1024 -> 1024, leaves of 24: 9472
    // tokens 32.5 and 31.3; 7 levels: 17.2 and 17.0 at 1024.  A second round of tiles would cost more than half an image saves.
    if (h->halves.NP != 0 && &sg == &h->ustages[0] && (h->slots_here || h->nslots_here) &&
        2 * ((B + fff::kUM - 1) / fff::kUM) <= h->sm_count)
        return h->halves.NP == 64 ? launch_descent_umma<64, true>(h, h->halves, x, pos_out, B, st)
                                  : launch_descent_umma<128, true>(h, h->halves, x, pos_out, B, st);
    switch (sg.NP) {
        case 32: return launch_descent_umma<32>(h, sg, x, pos_out, B, st);
        case 64: return launch_descent_umma<64>(h, sg, x, pos_out, B, st);
        case 128: return launch_descent_umma<128>(h, sg, x, pos_out, B, st);
        case 256: return launch_descent_umma<256>(h, sg, x, pos_out, B, st);
    }
    return FFF_ERR_UNSUPPORTED;
}

template <int NP>
fff_status_t launch_descent_umma_grouped(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, const int32_t* perm,
                                         int32_t* pos_out, int64_t B, cudaStream_t st) {
    const bool node_lists = perm == h->ws_nslots && h->ws_nslots != nullptr;      // tiles from the node counts, not from ws_tiles
    using L = fff::DescentUmmaGroupedLayout<NP>;
    const int stages = std::min((int)fff::kUmmaMaxStages, (kSmemBudget - L::smem_bytes(0)) / L::kStageBytes);
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_descent_umma_grouped<NP>, h->device, kSmemBudget, limit_raised)) return FFF_ERR_CUDA;
    CUtensorMap tm;
    if (!make_x_tensor_map(&tm, x, B, h->D, 1)) return FFF_ERR_CUDA;       // one-row boxes: rows are gathered four at a time
    const int n_tiles = tile_list_len(B, fff::kUM, 1 << sg.L0);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(h->sm_count, n_tiles));
    const SlotArgs sl = slot_args(h, pos_out);
    if (launch_chain(h, fff::k_descent_umma_grouped<NP>, (unsigned)grid, fff::kUGThreads, (size_t)L::smem_bytes(stages), st, 1, tm,
                     perm, (const fff::Tile*)h->ws_tiles, n_tiles, (const __nv_bfloat16*)sg.wimg, (const float*)sg.bimg, pos_out,
                     sl.pos2, sl.cursor, sl.slots, sl.cap, h->Dp, sg.k, stages, h->d_status, node_lists ? h->ws_ncursor : (int32_t*)nullptr,
                     1 << sg.L0, (int)h->nslot_cap) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "tree_descent_umma_grouped");
}

fff_status_t run_descent_umma_grouped(fff_handle_s* h, const fff_handle_s::DenseStage& sg, const void* x, const int32_t* perm,
                                      int32_t* pos_out, int64_t B, cudaStream_t st) {
    switch (sg.NP) {
        case 16: return launch_descent_umma_grouped<16>(h, sg, x, perm, pos_out, B, st);
        case 32: return launch_descent_umma_grouped<32>(h, sg, x, perm, pos_out, B, st);
        case 64: return launch_descent_umma_grouped<64>(h, sg, x, perm, pos_out, B, st);
    }
    return FFF_ERR_UNSUPPORTED;
}

template <typename T>
fff_status_t run_descent_warp(fff_handle_s* h, const void* x, int level0, int levels, const int32_t* pos_in,
                              int32_t* pos_out, int64_t B, cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((B + fff::kDescentWarps - 1) / fff::kDescentWarps, (int64_t)h->sm_count * 8);
    if (launch_chain(h, fff::k_descent_warp<T>, (unsigned)blocks, fff::kDescentWarps * 32, 0, st, 1, (const T*)x,
                     (const T*)h->node_w, (const T*)h->node_b, h->D, level0, levels, pos_in, pos_out, B,
                     h->vec_ok && aligned16(x)) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "tree_descent_warp");
}

// Number of leading tensor-core stages to run for a batch of B tokens: a stage pays off while the
// groups it works on (tokens that share the node at the stage's first level) hold enough tokens to
// reuse the subtree's weights.
const std::vector<fff_handle_s::DenseStage>& stage_plan(const fff_handle_s* h) {
    return h->ustages.empty() || !h->tune[FFF_TUNE_TCGEN05_DESCENT] ? h->stages : h->ustages;
}

// Tokens that a call of B is planned for: those of the whole batch when it is one chunk of several.  Everything that chooses
// between kernels which round differently goes by this number; only capacities go by the chunk's own.
int64_t planned_tokens(const fff_handle_s* h, int64_t B) { return std::max(B, h->plan_B); }

// Whether a later descent stage's groups fill 128-row tiles well enough.
bool fills_grouped_tiles(const fff_handle_s* h, int64_t B, int L0) { return (planned_tokens(h, B) >> L0) >= 64; }

// Whether the lists between the first and the second descent stage hold this call's tokens (and would hold the whole batch's).
bool node_lists_fit(const fff_handle_s* h, int64_t B) {
    const int k = h->ustages[0].k;
    return h->ws_nslots && B <= h->nslot_cap && (h->nslot_cap << k) <= INT32_MAX &&      // (a tile's start is an int)
           ((size_t)planned_tokens(h, B) << k) * sizeof(int32_t) <= kMaxSlotBytes;
}

// Likewise the leaves' lists.
bool leaf_lists_fit(const fff_handle_s* h, int64_t B) {
    return h->ws_slots && B <= h->slot_cap && h->n_leaves * h->slot_cap <= INT32_MAX && planned_tokens(h, B) <= listed_tokens(h);
}

// Thin leaves that are evaluated token by token anyway, with fewer than four tokens each: whether the leaf kernel's own walk through
// all levels beats the stages, their bucketing and the walk through the rest.  The line lies where the walk's row loads end: its
// loop takes 256 columns at a time, and widths that fill the steps (or end in the third) are cheap.  us, walk and stages:
//   256, 512, 768, 1024 columns and 513 to 768: 768 columns, 14 levels, 3000 tokens 20.7 and 22.8, 5409 27.6 and 35.1, 6900 33.0 and
//   36.2, 8192 39.8 and 40.8; 12 levels, 5409 24.8 and 29.2, 8192 35.1 and 33.0;
//   other widths below 512: 328 columns, 14 levels, 4096 tokens 22.7 and 26.8, 4800 26.8 and 26.9, 6144 31.0 and 26.9;
//   other widths above 768: 896 columns, 12 levels, 4096 tokens 31.1 and 33.1, 5409 39.0 and 34.7, 8192 53.4 and 39.2; against a single
//   stage (fewer than 16 tokens per group of the second) 824 columns, 14 levels, 3000 tokens 28.9 and 28.9, 3600 34.9 and 31.0; against
//   two, 4096 35.0 and 38.8, 4800 42.9 and 39.2.
bool walks_alone(const fff_handle_s* h, const std::vector<fff_handle_s::DenseStage>& plan, int64_t B) {
    if (use_tensor_leaf(h) || B >= 4 * h->n_leaves) return false;
    if (h->D % 256 == 0 || (h->D > 512 && h->D <= 768)) return B <= 7000;
    if (h->D < 512) return B <= 5000;
    const bool one_stage = plan.size() < 2 || (B >> plan[1].L0) < 16;
    return B <= (one_stage ? 3072 : 4608);
}

// leaf_walks: a leaf kernel follows that can walk the levels left over itself.
int dense_stage_count(const fff_handle_s* h, int64_t call_B, bool leaf_walks) {
    const int64_t B = planned_tokens(h, call_B);
    const auto& plan = stage_plan(h);
    if (plan.empty() || h->path == FFF_PATH_WARP) return 0;
    if (h->path == FFF_PATH_TENSOR) return (int)plan.size();
    if (leaf_walks && walks_alone(h, plan, B)) return 0;
    int n = 0;
    for (const auto& sg : plan) {
        if ((B >> sg.L0) < 16) break;
        ++n;
    }
    return n;
}

// The whole descent: tensor-core stages (with a bucketing by current node between them), then the
// remaining levels, if any, one warp per token.  leaf_out receives the leaf index.  *coarse describes
// the last node bucketing made on the way (the leaf bucketing can refine it instead of starting over).
// Levels of the descent that the caller's leaf kernel will walk itself (k_leaf_warp), instead of a launch of
// k_descent_warp: the walk starts at level `level0` from the positions `pos` (NULL = the root).
struct DescentTail {
    int level0 = 0, levels = 0;
    const int32_t* pos = nullptr;
};

// leaf_bucketing_follows: the caller buckets by leaf right after (run_bucket with *coarse).
fff_status_t run_descent(fff_handle_s* h, const void* x, int32_t* leaf_out, Coarse* coarse, int64_t B, cudaStream_t st,
                         DescentTail* defer_tail = nullptr, bool leaf_bucketing_follows = false) {
    fff_status_t s = FFF_OK;
    const int n_dense = dense_stage_count(h, B, defer_tail != nullptr);
    // the first stage's counts are summed per block of tiles only if the bucketing kernel that reads (and clears)
    // the sums comes next: a node bucketing before the second stage, or the caller's leaf bucketing
    h->blocksum_wanted = n_dense > 1 || (n_dense == 1 && leaf_bucketing_follows && coarse != nullptr &&
                                         stage_plan(h)[0].k == h->depth);
    int level = 0;
    const int32_t* pos = nullptr;
    Coarse prev;
    const auto& plan = stage_plan(h);
    // Two tcgen05 stages and nobody downstream who would refine the node bucketing: the first stage files the tokens
    // under the nodes it reaches and the second derives its tiles from the counts; no bucketing launch in between.
    const bool node_lists = n_dense == 2 && &plan == &h->ustages && plan[0].umma && plan[1].umma && node_lists_fit(h, B) &&
                            h->tune[FFF_TUNE_DIRECT_LISTS] && h->tune[FFF_TUNE_TCGEN05_GROUPED] &&
                            (coarse == nullptr || defer_tail != nullptr);
    if (node_lists) {
        if (h->ncursor_dirty &&
            cudaMemsetAsync(h->ws_ncursor, 0, sizeof(int32_t) * (fff::kUGMaxBins + 1), st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        h->ncursor_dirty = true;
        h->blocksum_wanted = false;
    }
    for (int i = 0; i < n_dense; ++i) {
        const auto& sg = plan[i];
        // later stages: the tcgen05 kernel on 128-row tiles when the groups fill them reasonably, else mma.sync on 64-row tiles
        // (with node lists there is no bucketing launch that the thinner tiles would have to pay for)
        const bool grouped_umma = i > 0 && sg.umma && h->tune[FFF_TUNE_TCGEN05_GROUPED] && (node_lists || fills_grouped_tiles(h, B, sg.L0));
        if (i > 0 && !node_lists) {
            // bucket by the node reached so far; buffers alternate so that the previous level stays readable
            int32_t* perm_out = (i & 1) ? h->ws_perm2 : h->ws_perm;
            int32_t* off_out = h->ws_offsets2[i & 1];
            prev.ranked = i == 1 && plan[0].umma && plan[0].k >= 4 && h->ws_rank8 != nullptr;
            s = run_bucket(h, pos, 1 << level, prev, off_out, perm_out, B, st, grouped_umma ? fff::kUM : fff::kDTM, "node_bucketing");
            prev.ranked = false;
            if (s != FFF_OK) return s;
            prev.perm = perm_out;
            prev.offsets = off_out;
            prev.bins = 1 << level;
        }
        const bool last = level + sg.k == h->depth;
        int32_t* out = last ? leaf_out : h->ws_pos[i & 1];
        h->slots_here = h->slots_now && last;
        h->nslots_here = node_lists && i == 0;
        s = i == 0 && sg.umma ? run_descent_umma(h, sg, x, out, B, st)
            : grouped_umma    ? run_descent_umma_grouped(h, sg, x, node_lists ? h->ws_nslots : prev.perm, out, B, st)
                              : run_descent_mma(h, sg, x, prev.perm, i > 0, out, B, st);
        h->slots_here = false;
        h->nslots_here = false;
        if (s != FFF_OK) return s;
        if (node_lists && i == 1) h->ncursor_dirty = false;       // its last CTA clears the counts
        level += sg.k;
        pos = out;
    }
    if (level < h->depth && defer_tail) {
        defer_tail->level0 = level;
        defer_tail->levels = h->depth - level;
        defer_tail->pos = pos;
    } else if (level < h->depth || h->depth == 0) {
        s = h->dtype == FFF_DTYPE_F32 ? run_descent_warp<float>(h, x, level, h->depth - level, pos, leaf_out, B, st)
                                      : run_descent_warp<__nv_bfloat16>(h, x, level, h->depth - level, pos, leaf_out, B, st);
    }
    // one tcgen05 stage was the whole descent: the leaf indices come with its ranks and counts
    prev.ranked = n_dense == 1 && level == h->depth && plan[0].umma && plan[0].k >= 4 && h->ws_rank8 != nullptr;
    if (coarse) *coarse = prev;
    return s;
}

// Packs the weight image of one stage (levels L0 .. L0 + k - 1) and appends it to `plan`.
template <typename T>
fff_status_t pack_stage(fff_handle_s* h, std::vector<fff_handle_s::DenseStage>& plan, int L0, int k, int NP, bool umma) {
    fff_handle_s::DenseStage sg;
    sg.L0 = L0;
    sg.k = k;
    sg.NP = NP;
    sg.umma = umma;
    const size_t groups = (size_t)1 << L0;
    fff_status_t s;
    if ((s = dmalloc((void**)&sg.wimg, groups * sg.NP * h->Dp * 2)) != FFF_OK) return s;
    plan.push_back(sg);                            // owned by the handle from here on
    if ((s = dmalloc((void**)&plan.back().bimg, groups * sg.NP * 4)) != FFF_OK) return s;
    fff::k_pack_nodes<T><<<h->sm_count * 8, 256>>>((const T*)h->node_w, (const T*)h->node_b, plan.back().wimg, plan.back().bimg,
                                                  sg.L0, sg.k, sg.NP, h->D, h->Dp, false);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// Levels per stage when `levels` levels are cut into stages of at most 6, larger stages first.
std::vector<int> cut_levels(int levels) {
    std::vector<int> ks;
    const int n_st = (levels + 5) / 6;
    for (int i = 0; i < n_st; ++i) ks.push_back(levels / n_st + (i < levels % n_st ? 1 : 0));
    return ks;
}

template <typename T>
fff_status_t pack_node_images(fff_handle_s* h) {
    const int d = h->depth;
    fff_status_t s;
    // plan for the mma.sync kernels alone: stages of at most 6 levels
    int L0 = 0;
    for (int k : cut_levels(d)) {
        if ((s = pack_stage<T>(h, h->stages, L0, k, std::max(16, 1 << k), false)) != FFF_OK) return s;
        L0 += k;
    }
    // plan with a first stage of up to 8 levels on the tcgen05 kernel, the rest as above
    if (encode_tiled_fn()) {
        std::vector<int> ks;
        // Measured: up to 8 levels in one stage when that is the whole tree (no node bucketing at all); two
        // balanced stages up to depth 12 ([6,5] beats [8,3]: 64 bins instead of 256 and fatter groups);
        // deeper trees as few stages as possible, 8 levels first and then 6 at a time ([8,6,1] beats [5,5,5]:
        // one pass over x and one bucketing less, the last thin levels go to the warp kernel anyway).
        if (d <= 8) ks = {d};
        else if (d <= 12) ks = cut_levels(d);
        else {
            ks.push_back(8);
            for (int rest = d - 8; rest > 0; rest -= 6) ks.push_back(std::min(rest, 6));
        }
        L0 = 0;
        for (size_t i = 0; i < ks.size(); ++i) {
            const int np = i == 0 ? std::max(32, 1 << ks[i]) : std::max(16, 1 << ks[i]);
            if ((s = pack_stage<T>(h, h->ustages, L0, ks[i], np, true)) != FFF_OK) return s;
            L0 += ks[i];
        }
        if (ks[0] >= 7) {
            auto& hv = h->halves;
            hv.L0 = 1;
            hv.k = ks[0] - 1;
            hv.umma = true;
            const int np = 1 << hv.k;
            if ((s = dmalloc((void**)&hv.wimg, (size_t)2 * np * h->Dp * 2)) != FFF_OK) return s;
            if ((s = dmalloc((void**)&hv.bimg, (size_t)2 * np * 4)) != FFF_OK) return s;
            fff::k_pack_nodes<T><<<h->sm_count * 8, 256>>>((const T*)h->node_w, (const T*)h->node_b, hv.wimg, hv.bimg, hv.L0, hv.k, np,
                                                          h->D, h->Dp, true);
            hv.NP = np;
        }
        cudaFuncSetAttribute(fff::k_descent_umma<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        cudaFuncSetAttribute(fff::k_descent_umma<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        cudaFuncSetAttribute(fff::k_descent_umma<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        cudaFuncSetAttribute(fff::k_descent_umma<256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        cudaFuncSetAttribute(fff::k_descent_umma<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        cudaFuncSetAttribute(fff::k_descent_umma<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
    }
    cudaFuncSetAttribute(fff::k_descent_mma<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
    cudaFuncSetAttribute(fff::k_descent_mma<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
    cudaFuncSetAttribute(fff::k_descent_mma<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// Which form of k_leaf_warp: while the warps of all tokens are resident at once with the registers that the general form wants
// (three CTAs per SM, four where the kernel walks the last levels too), that one; beyond, the loads of six CTAs per SM outweigh the
// few that each has in flight, as long as the leaves are narrow and rows come in vectors (769 columns, 4096 leaves of 16, 12 000 tokens
// 460 and 508).  us, general and six CTAs: float32, 768 -> 768, 1024 leaves of 3 behind a bucketing, 3000 tokens 27.2 and 29.0, 12 000
// 130.6 and 116.7; 512 leaves of 32, 3000 tokens 387 and 621; walking 4096 leaves of 6, 3000 tokens 60.0 and 65.1, 12 000 161 and 140; of 16, 6000 tokens 272 and 237.  Leaves of two and four neurons in vectors
// gain at any size (768 -> 768, 4096 leaves of 2, 3000 tokens 31.3 and 28.3), leaves of one where the kernel walks (15 levels, 16 384
// tokens 35.5 and 31.9; 12 levels behind a bucketing 35.6 and 37.2 per forward).
template <typename T>
fff_status_t run_leaf(fff_handle_s* h, const void* x, const int32_t* leaf_idx, const int32_t* perm, void* y,
                      int64_t B, cudaStream_t st, const DescentTail& tail = DescentTail(), int32_t* leaf_out = nullptr) {
    const int64_t blocks = std::min<int64_t>((B + fff::kLeafWarps - 1) / fff::kLeafWarps, (int64_t)h->sm_count * 8);
    const size_t smem = sizeof(float) * (size_t)fff::kLeafWarps * h->l;
    auto launch = [&](auto kern) {
        return launch_chain(h, kern, (unsigned)blocks, fff::kLeafWarps * 32, smem, st, 1, (const T*)x, leaf_idx, perm,
                            (const T*)h->w1, (const T*)h->b1, (const T*)h->w2, (const T*)h->b2, (T*)y, h->D, h->O, h->l, h->act, B,
                            h->vec_ok && aligned16(x), (const T*)h->node_w, (const T*)h->node_b, tail.level0, tail.levels, tail.pos,
                            leaf_out);
    };
    const bool walk = tail.levels > 0, vec = h->vec_ok && aligned16(x);
    const bool crowded = B > (int64_t)h->sm_count * fff::kLeafWarps * (walk ? 4 : 3);
    const bool thin = vec && h->O % fff::Elem<T>::kVec == 0 && (h->l == 2 || h->l == 4 || (h->l == 1 && walk && crowded));
    const bool dense = vec && crowded && h->l <= (walk ? 16 : 8) && (walk || h->l > 1);
    auto kernel = [&](auto tail_form) {
        constexpr bool kTail = decltype(tail_form)::value;
        return thin    ? fff::k_leaf_warp<T, kTail, fff::kLeafThin>
               : dense ? fff::k_leaf_warp<T, kTail, fff::kLeafDense>
                       : fff::k_leaf_warp<T, kTail, fff::kLeafWide>;
    };
    if (launch(walk ? kernel(std::true_type{}) : kernel(std::false_type{})) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, tail.levels > 0 ? "descent_tail+leaf_ff_warp" : "grouped_leaf_ff_warp");
}

template <int LP, int TM, int S, bool kSplit>
fff_status_t launch_leaf_mma(fff_handle_s* h, const void* x, const int32_t* perm, void* y, int64_t B, cudaStream_t st) {
    const int n_tiles = tile_list_len(B, TM, (int)h->n_leaves);
    using L = fff::LeafMmaLayout<LP, TM, S>;
    // direct lists: perm is the table of lists, the tiles come from its counts
    int32_t* counts = h->slots_now && perm == h->ws_slots ? h->ws_cursor : nullptr;
    const int smem = L::kSmemBytes + (counts ? L::list_bytes((int)h->n_leaves) : 0);
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_leaf_mma<LP, TM, S, kSplit>, h->device, L::kSmemBytes + L::list_bytes(kMaxListedLeaves), limit_raised)) return FFF_ERR_CUDA;
    const int per_sm = std::max(1, std::min(2, (int)((227 * 1024) / (smem + 1024))));
    const int64_t grid = std::min<int64_t>((int64_t)h->sm_count * per_sm, n_tiles);
    if (launch_chain(h, fff::k_leaf_mma<LP, TM, S, kSplit>, (unsigned)grid, L::kThreads, (size_t)smem, st, 1,
                     (const __nv_bfloat16*)x, perm, h->ws_tiles, n_tiles, h->w1img, h->b1img, h->w2img, (__nv_bfloat16*)y, h->D, h->Dp,
                     h->O, h->act, h->d_status, counts, (int)h->n_leaves, (int)h->slot_cap) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "grouped_leaf_ff_mma");
}

template <int LP, int TM, int S>
fff_status_t launch_leaf_mma(fff_handle_s* h, const void* x, const int32_t* perm, void* y, int64_t B, cudaStream_t st) {
    return h->padded() ? launch_leaf_mma<LP, TM, S, true>(h, x, perm, y, B, st) : launch_leaf_mma<LP, TM, S, false>(h, x, perm, y, B, st);
}

fff_status_t launch_leaf_mma_warp(fff_handle_s* h, const void* x, const int32_t* slots, void* y, int64_t B, cudaStream_t st) {
    const int64_t n_tiles = tile_list_len(B, fff::kLWRows, (int)h->n_leaves);
    const int64_t grid = std::min<int64_t>((int64_t)h->sm_count * 2, n_tiles);
    if (launch_chain(h, h->padded() ? fff::k_leaf_mma_warp<true> : fff::k_leaf_mma_warp<false>, (unsigned)grid, fff::kLWThreads, sizeof(int) * (size_t)(h->n_leaves + 1), st, 1,
                     (const __nv_bfloat16*)x, slots, (const __nv_bfloat16*)h->w1img, (const float*)h->b1img, (const unsigned char*)h->w2img,
                     (__nv_bfloat16*)y, h->D, h->Dp, h->O, h->act, h->ws_cursor, (int)h->n_leaves, (int)h->slot_cap) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "grouped_leaf_ff_mma_warp");
}

template <int LP, bool kFold, bool kW8, bool kSplit>
fff_status_t launch_leaf_umma_tiles(fff_handle_s* h, const void* x, const int32_t* perm, void* y, int64_t B, int tile_rows,
                                    cudaStream_t st) {
    using L = fff::LeafUmmaLayout<LP, kW8, 1, kSplit>;
    constexpr auto kernel = fff::k_leaf_umma<LP, kFold, kW8, 1, kSplit>;
    const int n_tiles = tile_list_len(B, tile_rows, (int)h->n_leaves);
    const int stages = std::min((int)fff::kLUMaxStages, (kSmemBudget - L::smem_bytes(0)) / L::kStageBytes);
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(kernel, h->device, kSmemBudget, limit_raised)) return FFF_ERR_CUDA;
    CUtensorMap tm;
    if (!make_x_tensor_map(&tm, x, B, h->D, 1)) return FFF_ERR_CUDA;       // one-row boxes: rows are gathered four at a time
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(h->sm_count, n_tiles));
    const int wide = (reinterpret_cast<uintptr_t>(y) & 31u) == 0 ? 1 : 0;
    const int passes = 1;      // two passes (full tiles first) measured slightly slower
    // direct lists: perm is the table of lists, the tiles come from its counts
    int32_t* counts = h->slots_now && perm == h->ws_slots ? h->ws_cursor : nullptr;
    if (launch_chain(h, kernel, (unsigned)grid, fff::LeafUmmaWarps<kW8>::kThreads, (size_t)L::smem_bytes(stages), st, 1, tm, perm,
                     (const fff::Tile*)h->ws_tiles, n_tiles, (const __nv_bfloat16*)h->w1img, (const float*)h->b1img,
                     (const unsigned char*)(kW8 ? h->w2codes : h->w2uimg), (__nv_bfloat16*)y, h->Dp, h->O, h->l, h->act, stages, wide, passes, h->ws_sched,
                     counts, (int)h->n_leaves, (int)h->slot_cap, h->d_status, (const unsigned char*)h->w1codes, (const float*)h->scale1,
                     (const float*)h->scale2, (const float*)nullptr, (int32_t*)nullptr, (int32_t*)nullptr) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, kW8 ? "grouped_leaf_ff_umma_w8" : "grouped_leaf_ff_umma");
}

template <int LP, bool kFold, bool kW8 = false>
fff_status_t launch_leaf_umma(fff_handle_s* h, const void* x, const int32_t* perm, void* y, int64_t B, int tile_rows,
                              cudaStream_t st) {
    if constexpr (!kW8)
        if (h->padded()) return launch_leaf_umma_tiles<LP, kFold, false, true>(h, x, perm, y, B, tile_rows, st);
    return launch_leaf_umma_tiles<LP, kFold, kW8, false>(h, x, perm, y, B, tile_rows, st);
}

// Ring depth per (LP, TM): what fits twice into an SM's shared memory (once for LP = 64).
fff_status_t run_leaf_mma(fff_handle_s* h, const void* x, const int32_t* perm, void* y, int64_t B, const LeafPlan& plan,
                          cudaStream_t st) {
    const int tile_rows = plan.tile_rows;
    if (h->w8) {
        switch (h->LP) {
            case 16: return launch_leaf_umma<16, false, true>(h, x, perm, y, B, tile_rows, st);
            case 32: return launch_leaf_umma<32, false, true>(h, x, perm, y, B, tile_rows, st);
            case 64: return launch_leaf_umma<64, false, true>(h, x, perm, y, B, tile_rows, st);
        }
        return FFF_ERR_UNSUPPORTED;
    }
    if (plan.umma && h->w2uimg) {
        switch (h->LP) {
            case 16: return h->l < 16 ? launch_leaf_umma<16, true>(h, x, perm, y, B, tile_rows, st)
                                      : launch_leaf_umma<16, false>(h, x, perm, y, B, tile_rows, st);
            case 32: return h->l < 32 ? launch_leaf_umma<32, true>(h, x, perm, y, B, tile_rows, st)
                                      : launch_leaf_umma<32, false>(h, x, perm, y, B, tile_rows, st);
            case 64: return h->l < 64 ? launch_leaf_umma<64, true>(h, x, perm, y, B, tile_rows, st)
                                      : launch_leaf_umma<64, false>(h, x, perm, y, B, tile_rows, st);
        }
    }
    if (tile_rows == fff::kLWRows) return launch_leaf_mma_warp(h, x, perm, y, B, st);
    if (tile_rows == 32) {
        switch (h->LP) {
            case 16: return launch_leaf_mma<16, 32, 6>(h, x, perm, y, B, st);
            case 32: return launch_leaf_mma<32, 32, 5>(h, x, perm, y, B, st);
            case 64: return launch_leaf_mma<64, 32, 4>(h, x, perm, y, B, st);
        }
    } else {
        switch (h->LP) {
            case 16: return launch_leaf_mma<16, 64, 4>(h, x, perm, y, B, st);
            case 32: return launch_leaf_mma<32, 64, 3>(h, x, perm, y, B, st);
            case 64: return launch_leaf_mma<64, 64, 4>(h, x, perm, y, B, st);
        }
    }
    return FFF_ERR_UNSUPPORTED;
}

// Build the pre-swizzled stage images of the tensor-core leaf kernel (once, at creation).
template <typename T>
fff_status_t pack_leaf_images(fff_handle_s* h) {
    const int LP = h->LP, U2 = (h->O + fff::kNC - 1) / fff::kNC;
    const size_t nl = (size_t)h->n_leaves;
    const size_t stage2 = (size_t)fff::kNC * LP * 2 + fff::kNC * 4;
    fff_status_t s;
    if ((s = dmalloc((void**)&h->w1img, nl * LP * h->Dp * 2)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->b1img, nl * LP * 4)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->w2img, nl * U2 * stage2)) != FFF_OK) return s;
    const int blocks = h->sm_count * 8;
    fff::k_pack_w1<T><<<blocks, 256>>>((const T*)h->w1, h->w1img, (int)nl, h->l, LP, h->D, h->Dp);
    fff::k_pack_b1<T><<<blocks, 256>>>((const T*)h->b1, h->b1img, (int)nl, h->l, LP);
    fff::k_pack_w2<T><<<blocks, 256>>>((const T*)h->w2, (const T*)h->b2, h->w2img, (int)nl, h->l, LP, h->O);
    if (cudaGetLastError() != cudaSuccess) return FFF_ERR_CUDA;
    // the tcgen05 kernel: W2 in pieces of 128 output features, and its scheduler words
    if (encode_tiled_fn() && h->O % 16 == 0) {
        const size_t P = (size_t)(h->O + fff::kLUPiece - 1) / fff::kLUPiece;
        if ((s = dmalloc((void**)&h->w2uimg, nl * P * ((size_t)fff::kLUPiece * LP * 2 + fff::kLUPiece * 4))) != FFF_OK) return s;
        if ((s = clone((void**)&h->ws_sched, nullptr, 4 * sizeof(int))) != FFF_OK) return s;
        fff::k_pack_w2_umma<T><<<blocks, 256>>>((const T*)h->w2, (const T*)h->b2, h->w2uimg, (int)nl, h->l, LP, h->O);
        if (cudaGetLastError() != cudaSuccess) return FFF_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// Grouped tiles (8 leaves per tile of the tcgen05 leaf kernel): for leaves whose padded width 16 leaves a spare hidden
// column for the output bias, and trees whose levels above the last three fit one tcgen05 descent stage.
template <typename T>
fff_status_t pack_group_images(fff_handle_s* h) {
    const int d = h->depth, kd = d - 3;
    if (h->LP != 16 || h->l >= 16 || kd < 1 || kd > 8 || h->ustages.size() < 2 || !encode_tiled_fn()) return FFF_OK;
    const size_t bins = (size_t)1 << kd, N1 = (size_t)fff::kLUGroup * h->LP + 16;
    const size_t P = (size_t)(h->O + fff::kLUPiece - 1) / fff::kLUPiece;
    const size_t w2_bytes = bins * P * ((size_t)fff::kLUPiece * fff::kLUGroup * h->LP * 2 + fff::kLUPiece * 4);
    fff_status_t s;
    if ((s = pack_stage<T>(h, h->gstages, 0, kd, std::max(32, 1 << kd), true)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->g_b1, bins * N1 * 4)) != FFF_OK) return s;
    if ((s = clone((void**)&h->g_w2, nullptr, w2_bytes)) != FFF_OK) return s;                    // zeroed
    if ((s = dmalloc((void**)&h->g_w1, bins * N1 * h->Dp * 2)) != FFF_OK) return s;                 // (last: it marks the images as usable)
    fff::k_pack_leaf_groups<T><<<h->sm_count * 8, 256>>>((const T*)h->w1, (const T*)h->b1, (const T*)h->w2, (const T*)h->b2,
                                                        (const T*)h->node_w, (const T*)h->node_b, h->g_w1, h->g_b1, h->g_w2, (int)bins, d,
                                                        h->l, h->LP, h->D, h->Dp, h->O);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// Whether a forward of B tokens runs on grouped tiles.  Measured (D = O = 768, l = 12, 50 432 tokens; D = O = 1024 and
// 65 536 tokens at depth 11): depth 9: 70.8 against 82.1 us, depth 10: 81.4 against 88.3, depth 11: 138.7 against
// 155.5, but depth 8: 69.2 against 65.5.  A grouped tile streams the weights of 8 leaves (3 x the bytes into the SM
// per tile), which costs more than it saves unless it also replaces a second descent stage and its node bucketing:
// so only trees that the staged descent would cut in two.  The nodes three levels above the leaves must receive
// whole tiles on average, and the lists must fit.
bool use_group_tiles(const fff_handle_s* h, int64_t B) {
    if (!h->g_w1 || h->path == FFF_PATH_WARP || h->path == FFF_PATH_FUSED) return false;
    if (h->ustages.size() < 2) return false;
    if (!h->tune[FFF_TUNE_GROUP_TILES] || !h->tune[FFF_TUNE_TCGEN05_DESCENT] || !h->tune[FFF_TUNE_TCGEN05_LEAF] ||
        !h->tune[FFF_TUNE_DIRECT_LISTS])
        return false;
    const int64_t bins = h->n_leaves / fff::kLUGroup;
    return leaf_lists_fit(h, B) && planned_tokens(h, B) >= fff::kLUM * bins;
}

// First stage (depth - 3 levels, files the tokens under the nodes it reaches), then the leaf kernel on grouped tiles,
// which finishes the descent itself and reports the leaves.
template <bool kSplit>
fff_status_t run_forward_grouped_tiles(fff_handle_s* h, const void* x, void* y, int32_t* leaf, int64_t B, cudaStream_t st) {
    using L = fff::LeafUmmaLayout<16, false, fff::kLUGroup, kSplit>;
    constexpr auto kernel = fff::k_leaf_umma<16, true, false, fff::kLUGroup, kSplit>;
    const int bins = (int)(h->n_leaves / fff::kLUGroup);
    if (h->cursor_dirty && cudaMemsetAsync(h->ws_cursor, 0, cursor_bytes(h), st) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    h->cursor_dirty = true;
    h->blocksum_wanted = false;
    h->slots_here = true;
    h->slots_no_pos2 = true;
    fff_status_t s = run_descent_umma(h, h->gstages[0], x, h->ws_pos[0], B, st);
    h->slots_here = false;
    h->slots_no_pos2 = false;
    if (s != FFF_OK) return s;
    const int stages = std::min((int)fff::kLUMaxStages, (kSmemBudget - L::smem_bytes(0)) / L::kStageBytes);
    if (stages < 2) return FFF_ERR_UNSUPPORTED;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(kernel, h->device, kSmemBudget, limit_raised)) return FFF_ERR_CUDA;
    CUtensorMap tm;
    if (!make_x_tensor_map(&tm, x, B, h->D, 1)) return FFF_ERR_CUDA;
    const int n_tiles = tile_list_len(B, fff::kLUM, bins);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(h->sm_count, n_tiles));
    const int wide = (reinterpret_cast<uintptr_t>(y) & 31u) == 0 ? 1 : 0;
    if (launch_chain(h, kernel, (unsigned)grid, fff::kLUThreads, (size_t)L::smem_bytes(stages), st,
                     1, tm, (const int32_t*)h->ws_slots, (const fff::Tile*)h->ws_tiles, n_tiles, (const __nv_bfloat16*)h->g_w1,
                     (const float*)h->b1img, (const unsigned char*)h->g_w2, (__nv_bfloat16*)y, h->Dp, h->O, h->l, h->act, stages, wide, 1,
                     h->ws_sched, h->ws_cursor, bins, (int)h->slot_cap, h->d_status, (const unsigned char*)nullptr,
                     (const float*)nullptr, (const float*)nullptr, (const float*)h->g_b1, leaf,
                     leaf == h->ws_leaf ? (int32_t*)nullptr : h->ws_leaf) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    s = launched(h, st, "grouped_leaf_ff_umma_8");
    if (s == FFF_OK) h->cursor_dirty = false;
    return s;
}

fff_status_t run_forward_grouped(fff_handle_s* h, const void* x, void* y, int32_t* leaf, int64_t B, cudaStream_t st) {
    return h->padded() ? run_forward_grouped_tiles<true>(h, x, y, leaf, B, st) : run_forward_grouped_tiles<false>(h, x, y, leaf, B, st);
}

// The one-launch kernel on CUDA cores: eligibility (at creation).
size_t block_forward_smem(const fff_handle_s* h) {
    return sizeof(int) * (size_t)((h->n_leaves + 1 + 3) & ~(int64_t)3) + sizeof(float) * (size_t)h->l * fff::kBFTile;
}

template <typename T>
fff_status_t plan_block_forward(fff_handle_s* h) {
    const size_t smem = block_forward_smem(h);
    if (h->coop_ctas <= 0 || h->n_leaves > fff::kBFMaxLeaves || smem > 96 * 1024) return FFF_OK;
    static bool raised[2][kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_block_forward<T, 1>, h->device, 96 * 1024, raised[0]) ||
        !raise_smem_limit(fff::k_block_forward<T, 4>, h->device, 96 * 1024, raised[1]))
        return FFF_ERR_CUDA;
    int n1 = 0, n4 = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n1, fff::k_block_forward<T, 1>, fff::kBFThreads, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n4, fff::k_block_forward<T, 4>, fff::kBFThreads, smem) != cudaSuccess)
        return cudaGetLastError(), FFF_OK;
    h->bf_per_sm = std::min(2, std::min(n1, n4));
    // The layers that may be pinned to it (FFF_PATH_FUSED, FFF_CAP_FUSED_SMALL): a promise of the interface, small trees with thin
    // leaves and rows that are not too wide, and narrower than what the kernel takes (above).
    int lp = 1;
    while (lp < h->l) lp <<= 1;
    const int64_t Dr = (h->D + 3) & ~3, rows = std::max<int64_t>(Dr, 512);
    h->bf_pinnable = h->bf_per_sm > 0 && h->l <= 32 && (h->n_leaves * lp + 31) / 32 <= h->sm_count &&
                     128 * Dr + 256 * (int64_t)h->O + 32 * rows + 5432 <= kSmemBudget;
    return FFF_OK;
}

// How k_block_forward runs B tokens: one token per warp in the descent or four (one: 2048 tokens of 768 columns keep 14 warps per SM
// busy instead of 3.5; four: a quarter of the node rows' traffic), and rows per tile (thinner ones while full ones would leave CTAs
// without work, unless the leaves are thin themselves).
bool block_forward_single(const fff_handle_s* h, int64_t B) { return B <= (int64_t)h->sm_count * 2 * fff::kBFWarps * 2; }
int block_forward_rows(const fff_handle_s* h, int64_t B) {
    return B <= 8 * (int64_t)h->sm_count * h->bf_per_sm && B >= 32 * h->n_leaves ? 8 : fff::kBFTile;
}

// float32 layers whose operands fit shared memory in pieces have k_block_tiles too (block_tiles_plan says for which batches), which reads a
// transposed copy of W2.  Rows of fewer than 128 columns and leaves of fewer than 48 neurons, or rows of more than 1500 and leaves of one, have
// nothing for its copies to hide: of 369 random sizes of them it was faster on 19, and 1.25 times as long on average.
fff_status_t plan_block_tiles(fff_handle_s* h) {
    fff::BlockTilesLayout lay;
    if (h->bf_per_sm <= 0 || h->dtype != FFF_DTYPE_F32 || h->O > fff::kBTMaxOut || (h->D < 128 && h->l < 48) || (h->l == 1 && h->D > 1500) ||
        !lay.plan(h->D, h->O, h->l, (int)h->n_leaves, 8, 1, kSmemBudget))
        return FFF_OK;
    static bool raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_block_tiles, h->device, kSmemBudget, raised)) return FFF_ERR_CUDA;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fff::k_block_tiles, fff::kBTThreads, kSmemBudget) != cudaSuccess || n < 1)
        return cudaGetLastError(), FFF_OK;
    if (dmalloc((void**)&h->w2t, sizeof(float) * (size_t)h->n_leaves * h->l * h->O) != FFF_OK) return FFF_OK;      // (without it: k_block_forward)
    fff::k_pack_w2_columns<<<h->sm_count * 8, 256>>>((const float*)h->w2, h->w2t, h->n_leaves, h->l, h->O);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// Estimates, in us, of what k_block_forward and k_block_tiles take for B tokens, less what both have in common (the launch, the barrier,
// the rows of x and y): the passes of the descent (k steps of 128 columns for each chain of levels) and the rounds of tiles, a round being a
// tile on every CTA.  The factors are a least-squares fit to 802 random sizes (128 to 2400 columns, 1 to 1024 outputs, 1 to
// 4096 leaves of 2 to 80 neurons, 515 to 80 000 tokens); the whole estimates are 9 and 8 % off on average.
double block_forward_us(const fff_handle_s* h, int64_t B) {
    const int slots = h->sm_count * h->bf_per_sm, tile_rows = block_forward_rows(h, B);
    const bool single = block_forward_single(h, B);
    const double tiles = std::max(1.0, expected_tiles(h, B, tile_rows)), rounds = std::ceil(tiles / slots);
    const double passes = std::ceil((double)B / (slots * fff::kBFWarps * (single ? 1 : 4)));
    const int k = (h->D + 127) / 128, low = std::max(h->depth - 3, 0), chains = single ? (low + 2) / 3 : low;      // below the first three levels
    // blocks of 4 x 8 products per warp, 2.3 times as long where rows are read value by value
    const double blocks = std::ceil(std::ceil(std::min<double>(tile_rows, B / tiles) / 4) * ((h->l + 7) / 8) / fff::kBFWarps) * (h->vec_ok ? 1.0 : 2.3);
    return passes * (3.7 + 0.48 * k * chains) +
           rounds * (2.3 + 0.42 * blocks * k + 0.074 * h->l * ((h->O + 255) / 256) + 1.35e-4 * h->l * (h->D + h->O));
}
double block_tiles_us(const fff_handle_s* h, int64_t B, const fff::BlockTilesLayout& lay, double tiles) {
    const double rounds = std::ceil(tiles / h->sm_count), rows = std::min<double>(lay.tile_rows, B / tiles);
    const double passes = std::ceil((double)B / (h->sm_count * fff::kBTWarps * lay.tok));
    const int k = (h->D + 127) / 128, low = std::max(h->depth - 3, 0), chains = lay.tok == 1 ? (low + 2) / 3 : low;
    const int sent = (h->l + lay.w1_units - 1) / lay.w1_units + (h->l + lay.w2_units - 1) / lay.w2_units;      // ring slots per tile
    const double blocks = std::ceil(rows / 4) * ((h->l + 7) / 8) / fff::kBTWarps;
    return 3.4 + passes * (2.7 + chains * (0.41 + 0.085 * k * lay.tok)) + 0.012 * h->n_leaves +
           rounds * (1.6 + 0.52 * sent + 0.39 * blocks * k + 0.047 * h->l * ((h->O + 255) / 256) * rows / 16 + 0.66e-4 * h->l * (h->D + h->O));
}

// How k_block_tiles runs B tokens; false: not at all, k_block_forward is expected to be faster.  The more rows and weights a tile has, the
// more there is for the copies to hide; thin tiles cost their hand-overs, and one CTA per SM has no other to run meanwhile, so that a batch
// can need two rounds of tiles where two CTAs of the other kernel need one.  Measured, us, k_block_forward and it: 768 -> 768, 256
// leaves of 12, 6304 tokens 49.0 and 44.0, 50 432 tokens 285 and 251; 512 -> 512, 32 leaves of 16, 700 tokens 18.5 and 16.5; 1523 -> 745, 32 leaves of
// 37, 640 tokens 76 and 33; not taken: 768 -> 768, 256 leaves of 12, 1576 tokens 26.7 and 29.9; 516 -> 780, 32 leaves of 19, 9080 tokens 51.3
// and 67.7; 256 -> 256, 4096 leaves of 8, 16 384 tokens 135 and 175.  Over 1598 random sizes, times against the better of the two:
// this rule 1.007 on average, always k_block_forward 1.087, it wherever it fits 1.089; more than 3 % slower than k_block_forward are 3 % of
// the sizes with the rule and 37 % without.
// The line is drawn 6 % past equal estimates: sizes in between are ahead as often as behind.
// Tokens per warp in the descent: so many that the batch is one pass.  Rows per tile: a tile costs about as much as 20 rows before its
// first (its weights' way through the ring, the two barriers), and the launch lasts as long as the CTA with the most tiles.
bool block_tiles_plan(fff_handle_s* h, const void* x, int64_t B, fff::BlockTilesLayout* lay) {
    if (!h->w2t || !aligned16(x)) return false;
    if (h->bt_B == B) return *lay = h->bt_lay, h->bt_fits;
    const int64_t per_sm = (B + h->sm_count - 1) / h->sm_count;
    const int tok = (int)std::min<int64_t>(fff::kBTMaxTok, (per_sm + fff::kBTWarps - 1) / fff::kBTWarps);
    double best_cost = 0.0, best_us = 0.0;
    for (int rows : {8, 16, 32}) {
        fff::BlockTilesLayout l;
        if (!l.plan(h->D, h->O, h->l, (int)h->n_leaves, rows, tok, kSmemBudget)) continue;
        const double tiles = std::max(1.0, expected_tiles(h, B, rows));
        const double cost = std::ceil(tiles / h->sm_count) * (20.0 + std::min<double>(rows, B / tiles));
        if (best_cost == 0.0 || cost < best_cost) {
            h->bt_lay = l;
            best_cost = cost;
            best_us = block_tiles_us(h, B, l, tiles);
        }
    }
    h->bt_B = B;
    h->bt_fits = best_cost > 0.0 && best_us < 1.06 * block_forward_us(h, B);
    return *lay = h->bt_lay, h->bt_fits;
}

// Whether a forward of B tokens runs as the one-launch kernel: when pinned to it, or by default for layers that have no
// tensor-core leaf path, where it is faster than one warp per token (three launches): float32, 768 -> 768, 256 leaves of 12, 6304 tokens
// 44 against 95 us, 50 432 tokens 251 against 646; 1024 -> 1024, 512 leaves of 32, 8192 tokens 141 against 1151; 512 -> 512, 32 leaves of 16,
// 8192 tokens 35 against 174; 784 -> 10, 8 leaves of 32, 2048 tokens 21 against 44; 256 -> 64, one leaf of 16, 65 536 tokens 128 against
// 286.  CTAs of k_block_forward per SM: two (three leave 85 registers to the 32 sums of a block: 26 against 18 us).
// A tile fetches its leaf's weights once for its tokens; a leaf of a few neurons with a few tokens has little to share, while the
// warp per token (which with fewer than four of them needs neither bucketing nor barrier) has all of its loads to itself.  One
// launch (k_block_forward, which block_tiles_plan leaves only for less) and a warp per token, us, 768 columns, r tokens per leaf (over
// 1200 sizes the rule costs 1 % against the better of the two each time, always taking the one launch 29 %):
//   r < 4, float32: 512 leaves of 8, r = 2 30.0 and 31.0; 2048 leaves of 16, r = 1 106.9 and 117.9; 4096 leaves of 2, r = 1 108.5 and
//     35.1; bf16 -> 300 (whose descent runs on tensor cores then): 2048 leaves of 16, r = 2 81.1 and 59.7;
//   r >= 4, float32: 4096 leaves of 4, r = 4 223.9 and 146.3, r = 12 368.3 and 375.0; of 8, r = 6 314.6 and 375.9; bf16 -> 300: 4096
//     leaves of 8, r = 4 183.9 and 107.6; of 12, r = 12 321.8 and 332.7.
bool use_block_forward(const fff_handle_s* h, int64_t B) {
    if (!runs_block_forward(h) || !h->ws_slots || !h->tune[FFF_TUNE_FUSED_SMALL]) return false;
    if (h->path == FFF_PATH_FUSED) return true;
    const bool bf16 = h->dtype == FFF_DTYPE_BF16;
    if (B < 4 * h->n_leaves) return (int64_t)h->l * h->l * B >= h->n_leaves * (h->depth <= 9 ? 128 : 256) * (bf16 ? 2 : 1);
    if (h->depth <= 9 || h->l >= (bf16 ? 12 : 8)) return true;
    return !bf16 && B >= 10 * h->n_leaves && (h->l >= 4 || h->depth == 10);
}

template <typename T>
fff_status_t launch_block_forward(fff_handle_s* h, const void* x, void* y, int32_t* leaf_out, int32_t* leaf_out2, int64_t B,
                                  cudaStream_t st) {
    if (h->cursor_dirty && cudaMemsetAsync(h->ws_cursor, 0, cursor_bytes(h), st) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    h->cursor_dirty = true;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = h->pdl && !h->prof_active ? 2 : 1;
    cudaError_t e = cudaErrorUnknown;
    bool staged = false;
    if constexpr (sizeof(T) == 4) {
        fff::BlockTilesLayout lay;
        if (block_tiles_plan(h, x, B, &lay)) {
            staged = true;
            cfg.gridDim = dim3((unsigned)std::min<int64_t>(h->sm_count, B));
            cfg.blockDim = dim3(fff::kBTThreads);
            cfg.dynamicSmemBytes = lay.total_bytes;
            e = cudaLaunchKernelEx(&cfg, fff::k_block_tiles, (const float*)x, (const float*)h->node_w, (const float*)h->node_b, (const float*)h->w1,
                                   (const float*)h->b1, (const float*)h->w2t, (const float*)h->b2, (float*)y, leaf_out, leaf_out2, h->ws_slots,
                                   h->ws_cursor, (int)h->slot_cap, h->D, h->O, h->depth, h->l, h->act, (int)B, (int)h->n_leaves, lay, h->d_status);
        }
    }
    if (!staged) {
        cfg.gridDim = dim3((unsigned)std::min((int64_t)h->sm_count * h->bf_per_sm, std::max<int64_t>(B, 1)));
        cfg.blockDim = dim3(fff::kBFThreads);
        cfg.dynamicSmemBytes = block_forward_smem(h);
        e = cudaLaunchKernelEx(&cfg, block_forward_single(h, B) ? fff::k_block_forward<T, 1> : fff::k_block_forward<T, 4>, (const T*)x, (const T*)h->node_w,
                               (const T*)h->node_b, (const T*)h->w1, (const T*)h->b1, (const T*)h->w2, (const T*)h->b2, (T*)y, leaf_out, leaf_out2,
                               h->ws_slots, h->ws_cursor, (int)h->slot_cap, h->D, h->O, h->depth, h->l, h->act, (int)B,
                               h->vec_ok && aligned16(x), (int)h->n_leaves, block_forward_rows(h, B), h->d_status);
    }
    if (e != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    const fff_status_t s = launched(h, st, "fused_forward_blocks");
    if (s == FFF_OK) h->cursor_dirty = false;
    return s;
}

// In parts of as many tokens as the lists hold (a part's rows start on 16-byte boundaries where the batch's do: slot_cap is a
// multiple of 16 whenever there is more than one).
template <typename T>
fff_status_t run_block_forward(fff_handle_s* h, const void* x, void* y, int32_t* leaf_out, int32_t* leaf_out2, int64_t B,
                               cudaStream_t st) {
    fff_status_t s = FFF_OK;
    for (int64_t b0 = 0; b0 < B && s == FFF_OK; b0 += h->slot_cap)
        s = launch_block_forward<T>(h, (const T*)x + b0 * h->D, (T*)y + b0 * h->O, leaf_out + b0, leaf_out2 ? leaf_out2 + b0 : nullptr,
                                    std::min(h->slot_cap, B - b0), st);
    return s;
}

// Whether a forward of B tokens runs as one CTA per token.  While the CTAs of all tokens are resident at once (four per SM
// with bf16) the launch takes one chain of latencies whatever B is, and the other paths take two to five such chains:
// 768 -> 768, 256 leaves of 12, bf16: 7.4 us at one token, 8.5 at 197, 11.2 at 512 (three launches: 17.6, 19.0, 19.1);
// float32 7.5 / 9.1 / 16.8 us (18 / 20 / 20).  Past that the weights fetched token by token cost more than the launches:
// 1024 tokens 19.5 against 19.4 us, 2048 34.6 against 20.6.  Trees that the staged descent cuts in two would run five
// launches on thin groups: 1024 -> 1024, 2048 leaves of 32: 43 against 68 us at 1024 tokens, 79 against 97 at 2048, 149
// against 94 at 4096.  With leaves of up to 16 neurons those launches end in a warp per tile, and two or two and a half rounds
// of CTAs (four per SM) are the line: 768 -> 768, 1024 leaves of 16: 23.1 against 29.9 us at 1024 tokens, 33.7 against 30.7 at
// 1500, 43.2 against 30.9 at 2048; 2048 leaves of 12: 24.9 against 34.6, 35.1 against 35.8, 45.0 against 37.6.
constexpr int64_t kTokenBlockMaxB = 512, kTokenBlockMaxBDeep = 2048, kTokenBlockMaxBytes = (int64_t)96 << 20;

bool use_token_block(const fff_handle_s* h, int64_t B) {
    if (h->w8 || h->path != FFF_PATH_AUTO || !h->tune[FFF_TUNE_TOKEN_BLOCKS]) return false;
    if (fff::TokenBlockLayout{h->D, h->l, (int)h->esize}.total() > 100 * 1024) return false;
    const bool two_stages = use_tensor_leaf(h) && h->ustages.size() >= 2;
    if (two_stages) {
        const bool thin = h->LP == 16 && h->n_leaves <= kMaxListedLeaves && h->w2uimg;
        const int64_t most = thin ? (int64_t)h->sm_count * (h->n_leaves > 1024 ? 10 : 8) : kTokenBlockMaxBDeep;
        return B <= std::max(kTokenBlockMaxB, std::min(most, 2 * h->n_leaves));
    }
    const int full = h->depth / fff::kTBLevels, rest = h->depth % fff::kTBLevels;
    const int64_t nodes = (int64_t)full * ((1 << fff::kTBLevels) - 1) + ((1 << rest) - 1);
    const int64_t per_token = (nodes * h->D + (int64_t)h->l * (h->D + h->O)) * (int64_t)h->esize;
    return B <= kTokenBlockMaxB && B * per_token <= kTokenBlockMaxBytes;
}

template <typename T>
fff_status_t run_token_block(fff_handle_s* h, const void* x, void* y, int32_t* leaf_out, int32_t* leaf_out2, int64_t B, cudaStream_t st) {
    const size_t smem = fff::TokenBlockLayout{h->D, h->l, (int)h->esize}.total();
    static bool limit_raised[kMaxDevices] = {};
    if (smem > 48 * 1024 && !raise_smem_limit(fff::k_token_block<T>, h->device, 100 * 1024, limit_raised)) return FFF_ERR_CUDA;
    if (launch_chain(h, fff::k_token_block<T>, (unsigned)B, fff::kTBThreads, smem, st, 1, (const T*)x, (const T*)h->node_w,
                     (const T*)h->node_b, (const T*)h->w1, (const T*)h->b1, (const T*)h->w2, (const T*)h->b2, (T*)y, leaf_out, leaf_out2, h->D,
                     h->O, h->depth, h->l, h->act, (int)B, h->vec_ok && aligned16(x)) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "forward_token_blocks");
}

// FORWARD_T: the weight images of the GEMMs.  Sizes at creation (tr_Kp; 0: shapes not eligible), the images with the first
// call, like its workspace: layers that only infer do not pay for them.
constexpr int kTrainMaxFusedDepth = 8;      // deepest tree whose node logits fit one tile of k_train_nodes

void plan_train(fff_handle_s* h) {
    if (h->dtype != FFF_DTYPE_BF16 || h->D % fff::kGKB != 0 || !encode_tiled_fn() || h->n_leaves * (h->l + 1) > (1 << 24)) return;
    const int hidden = fff::train_hidden_columns((int)h->n_leaves, h->l);
    h->tr_Kp = (int)((hidden + h->n_leaves + fff::kGKB - 1) / fff::kGKB * fff::kGKB);
}

fff_status_t pack_train_images(fff_handle_s* h) {
    const int hidden = fff::train_hidden_columns((int)h->n_leaves, h->l), Kp = h->tr_Kp;
    const int padded = (hidden + 255) / 256 * 256, NP = std::max<int>(32, (int)h->n_leaves);
    const int blocks = h->sm_count * 8;
    const __nv_bfloat16 *w1 = (const __nv_bfloat16*)h->w1, *b1 = (const __nv_bfloat16*)h->b1;
    fff_status_t s;
    if ((s = dmalloc((void**)&h->tr_w2t, sizeof(__nv_bfloat16) * (size_t)h->O * Kp)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->tr_w1t, sizeof(__nv_bfloat16) * (size_t)hidden * h->D)) != FFF_OK) return s;
    if ((s = dmalloc((void**)&h->tr_b1t, sizeof(float) * (size_t)padded)) != FFF_OK) return s;
    fff::k_pack_w2_transposed<__nv_bfloat16><<<blocks, 256>>>((const __nv_bfloat16*)h->w2, (const __nv_bfloat16*)h->b2, h->tr_w2t,
                                                             (int)h->n_leaves, h->l, h->O, Kp);
    fff::k_pack_train_hidden<__nv_bfloat16><<<blocks, 256>>>(w1, b1, h->tr_w1t, h->tr_b1t, (int)h->n_leaves, h->l, h->D, padded);
    if (h->depth >= 1 && h->depth <= kTrainMaxFusedDepth) {
        if ((s = dmalloc((void**)&h->tr_wn, sizeof(__nv_bfloat16) * (size_t)NP * h->D)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->tr_bn, sizeof(float) * (size_t)NP)) != FFF_OK) return s;
        fff::k_pack_train_nodes<__nv_bfloat16><<<blocks, 256>>>((const __nv_bfloat16*)h->node_w, (const __nv_bfloat16*)h->node_b, h->tr_wn,
                                                               h->tr_bn, h->depth, NP, h->D);
    }
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    h->tr_packed = true;
    return FFF_OK;
}

// Tensor map of a row-major matrix (element size 2 or 4, `pitch` elements between rows) for boxes of box_cols x box_rows,
// swizzled in the mode of the box's row width (32, 64 or 128 bytes).
bool make_matrix_map(CUtensorMap* tm, const void* p, int esize, int64_t rows, int64_t cols, int64_t pitch, int box_cols, int box_rows) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)pitch * esize};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    const int width = box_cols * esize;
    return enc(tm, esize == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(p), gdim, gstride,
               box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
               width == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : width == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// C [M, N] = epilogue(A [M, K] . B [N, K]^T) on CTA pairs; lda = row pitch of A; out / out_cols / ld_out: the bf16 matrix that
// the epilogue stores through a tensor map (nullptr: it stores by itself).
template <int MODE, int BN>
fff_status_t launch_gemm_tiles(fff_handle_s* h, const void* a, int64_t M, int lda, const void* b, int64_t N, int64_t K,
                               fff::GemmEpilogueArgs ep, void* out, cudaStream_t st, const char* name) {
    using L = fff::GemmLayout<MODE, BN>;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_gemm_pair<MODE, BN>, h->device, L::kSmemBytes, limit_raised)) return FFF_ERR_CUDA;
    CUtensorMap ta, tb, tc, tx;
    if (!make_matrix_map(&ta, a, 2, M, K, lda, fff::kGKB, fff::kGRows) || !make_matrix_map(&tb, b, 2, N, K, K, fff::kGKB, BN / 2))
        return FFF_ERR_CUDA;
    tc = tx = ta;                          // unused ones still have to be valid maps
    if (out && !make_matrix_map(&tc, out, 2, M, N, ep.ld_out, L::kColsPerWarp, 32)) return FFF_ERR_CUDA;
    if (MODE == fff::kGemmHidden && ep.n_leaves >= 32 && !make_matrix_map(&tx, ep.mix, 4, M, ep.n_leaves, ep.n_leaves, 32, fff::kGRows)) return FFF_ERR_CUDA;
    const int64_t tiles = ((M + fff::kGM - 1) / fff::kGM) * ((N + BN - 1) / BN);
    const int64_t grid = 2 * (MODE == fff::kGemmHidden ? std::min<int64_t>(h->sm_count / 2, tiles) : balanced_grid(h->sm_count / 2, tiles));
    if (launch_chain(h, fff::k_gemm_pair<MODE, BN>, (unsigned)grid, fff::kGPairThreads, (size_t)L::kSmemBytes, st, 2, ta, tb, tc, tx, (int)M, (int)N,
                     (int)K, ep, h->d_status) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, name);
}

template <int MODE>
fff_status_t launch_gemm(fff_handle_s* h, const void* a, int64_t M, int lda, const void* b, int64_t N, int64_t K,
                         const fff::GemmEpilogueArgs& ep, void* out, cudaStream_t st, const char* name) {
    // 256 columns per tile unless that leaves pairs of SMs without a tile
    const int64_t tiles = ((M + fff::kGM - 1) / fff::kGM) * ((N + 255) / 256);
    return tiles >= h->sm_count / 2 ? launch_gemm_tiles<MODE, 256>(h, a, M, lda, b, N, K, ep, out, st, name)
                                    : launch_gemm_tiles<MODE, 128>(h, a, M, lda, b, N, K, ep, out, st, name);
}

template <int DEPTH>
fff_status_t launch_train_nodes(fff_handle_s* h, const void* x, float* mix, float* ent_part, int64_t B, cudaStream_t st, int* ctas) {
    using L = fff::TrainNodesLayout<DEPTH>;
    static bool limit_raised[kMaxDevices] = {};
    if (!raise_smem_limit(fff::k_train_nodes<DEPTH>, h->device, L::kSmemBytes, limit_raised)) return FFF_ERR_CUDA;
    const int hidden = fff::train_hidden_columns((int)h->n_leaves, h->l);
    CUtensorMap tx, tw, tm, tt;
    if (!make_matrix_map(&tx, x, 2, B, h->D, h->D, fff::kGKB, fff::kGRows) || !make_matrix_map(&tw, h->tr_wn, 2, L::NP, h->D, h->D, fff::kGKB, L::NP / 2))
        return FFF_ERR_CUDA;
    tm = tt = tx;
    if (L::kStaged && (!make_matrix_map(&tm, mix, 4, B, h->n_leaves, h->n_leaves, L::kPart, 32) ||
                       !make_matrix_map(&tt, h->tr_hp + hidden, 2, B, h->n_leaves, h->tr_Kp, L::kPart, 32)))
        return FFF_ERR_CUDA;
    const int64_t grid = 2 * balanced_grid(h->sm_count / 2, (B + fff::kGM - 1) / fff::kGM);
    *ctas = (int)grid;
    if (launch_chain(h, fff::k_train_nodes<DEPTH>, (unsigned)grid, fff::kGThreads, (size_t)L::kSmemBytes, st, 2, tx, tw, tm, tt, (const float*)h->tr_bn, mix,
                     h->tr_hp, h->tr_Kp, hidden, ent_part, (int)B, h->D, h->d_status) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    return launched(h, st, "train_node_choices");
}

fff_status_t run_train_nodes(fff_handle_s* h, const void* x, float* mix, float* ent_part, int64_t B, cudaStream_t st, int* ctas) {
    switch (h->depth) {
        case 1: return launch_train_nodes<1>(h, x, mix, ent_part, B, st, ctas);
        case 2: return launch_train_nodes<2>(h, x, mix, ent_part, B, st, ctas);
        case 3: return launch_train_nodes<3>(h, x, mix, ent_part, B, st, ctas);
        case 4: return launch_train_nodes<4>(h, x, mix, ent_part, B, st, ctas);
        case 5: return launch_train_nodes<5>(h, x, mix, ent_part, B, st, ctas);
        case 6: return launch_train_nodes<6>(h, x, mix, ent_part, B, st, ctas);
        case 7: return launch_train_nodes<7>(h, x, mix, ent_part, B, st, ctas);
        case 8: return launch_train_nodes<8>(h, x, mix, ent_part, B, st, ctas);
    }
    return FFF_ERR_UNSUPPORTED;
}

fff_status_t run_forward_train(fff_handle_s* h, const void* x, void* y, float* mixture, float* node_entropy, int64_t B,
                               cudaStream_t st) {
    const int64_t nl = h->n_leaves, nn = h->n_nodes, hidden = fff::train_hidden_columns((int)nl, h->l);
    if (!h->tr_packed) {
        // (a packing that failed half-way starts over)
        dfree(h->tr_w2t); dfree(h->tr_w1t); dfree(h->tr_b1t); dfree(h->tr_wn); dfree(h->tr_bn);
        h->tr_w2t = h->tr_w1t = h->tr_wn = nullptr;
        h->tr_b1t = h->tr_bn = nullptr;
        const fff_status_t ps = pack_train_images(h);
        if (ps != FFF_OK) return ps;
    }
    const bool fused = h->tr_wn != nullptr;
    const int ldc = (int)std::max<int64_t>((nn + 3) & ~(int64_t)3, 4);      // rows of c start on 16-byte boundaries
    const int64_t n_mt = (B + fff::kGRows - 1) / fff::kGRows;
    if (B > h->tr_cap_B) {
        if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        dfree(h->tr_c); dfree(h->tr_mix); dfree(h->tr_entpart); dfree(h->tr_hp);
        h->tr_c = h->tr_mix = h->tr_entpart = nullptr;
        h->tr_hp = nullptr;
        h->tr_cap_B = 0;
        fff_status_t s;
        if (!fused && (s = dmalloc((void**)&h->tr_c, sizeof(float) * (size_t)B * ldc)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->tr_mix, sizeof(float) * (size_t)B * nl)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->tr_entpart, sizeof(float) * (fused ? (size_t)h->sm_count * nl : (size_t)n_mt * 4 * ldc))) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->tr_hp, sizeof(__nv_bfloat16) * (size_t)B * h->tr_Kp)) != FFF_OK) return s;
        // the columns of h' past the mixture weights stay zero
        const int pad = h->tr_Kp - (int)(hidden + nl);
        if (pad > 0 && (s = default_stream_done(cudaMemset2D(h->tr_hp + hidden + nl, (size_t)h->tr_Kp * 2, 0, (size_t)pad * 2, (size_t)B))) != FFF_OK)
            return s;
        h->tr_cap_B = B;
    }
    fff_status_t s = FFF_OK;
    fff::GemmEpilogueArgs ep = {};
    float* mix = h->tr_mix;
    int ent_ctas = 0;
    if (fused) {
        // the caller's matrix is the one that the hidden GEMM reads, where its tensor map can take it
        if (mixture && aligned16(mixture)) mix = mixture;
        if ((s = run_train_nodes(h, x, mix, node_entropy ? h->tr_entpart : nullptr, B, st, &ent_ctas)) != FFF_OK) return s;
        if (mixture && mix != mixture &&
            cudaMemcpyAsync(mixture, mix, sizeof(float) * (size_t)B * nl, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
    } else {
        if (nn > 0) {
            ep.bias_bf16 = (const __nv_bfloat16*)h->node_b;
            ep.out_f32 = h->tr_c;
            ep.ent_part = node_entropy ? h->tr_entpart : nullptr;
            ep.ld_out = ldc;
            if ((s = launch_gemm<fff::kGemmNodes>(h, x, B, h->D, h->node_w, nn, h->D, ep, nullptr, st, "train_node_choices")) != FFF_OK) return s;
            if (node_entropy) {
                fff::k_entropy_reduce<<<(unsigned)((nn + 7) / 8), 256, 0, st>>>(h->tr_entpart, (int)((B + 31) / 32), (int)nn, B, node_entropy);
                if ((s = launched(h, st, "train_node_entropy")) != FFF_OK) return s;
            }
        }
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((B + fff::kMixTokens - 1) / fff::kMixTokens, (int64_t)h->sm_count * 16));
        fff::k_mixture_weights<<<(unsigned)blocks, 256, 0, st>>>(h->tr_c, ldc, h->tr_mix, mixture, h->tr_hp, h->tr_Kp, (int)hidden,
                                                                 h->depth, B);
        if ((s = launched(h, st, "train_mixture_weights")) != FFF_OK) return s;
    }
    ep = {};
    ep.bias = h->tr_b1t;
    ep.mix = mix;
    ep.out_bf16 = h->tr_hp;
    ep.ld_out = h->tr_Kp;
    ep.n_leaves = (int)nl;
    ep.l = h->l;
    ep.act = h->act;
    if (fused && node_entropy) {
        ep.ent_part = h->tr_entpart;
        ep.ent_out = node_entropy;
        ep.ent_rows = ent_ctas;
        ep.ent_depth = h->depth;
    }
    if ((s = launch_gemm<fff::kGemmHidden>(h, x, B, h->D, h->tr_w1t, hidden, h->D, ep, h->tr_hp, st, "train_hidden_all_leaves")) != FFF_OK) return s;
    ep = {};
    ep.out_bf16 = (__nv_bfloat16*)y;
    ep.ld_out = h->O;
    ep.tma_out = h->O % 8 == 0 ? 1 : 0;
    return launch_gemm<fff::kGemmOutput>(h, h->tr_hp, B, h->tr_Kp, h->tr_w2t, h->O, h->tr_Kp, ep, ep.tma_out ? y : nullptr, st,
                                         "train_output_mixture");
}

#define FFF_DISPATCH(h, fn, ...) \
    ((h)->dtype == FFF_DTYPE_F32 ? fn<float>(__VA_ARGS__) : fn<__nv_bfloat16>(__VA_ARGS__))

fff_status_t check_forward_args(fff_handle_t h, int64_t B) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (B < 0) return FFF_ERR_INVALID_ARG;
    if (B > FFF_MAX_TOKENS) return FFF_ERR_UNSUPPORTED;
    return FFF_OK;
}

}  // namespace

// Self-test of the bounded waits: one CTA waits, through the same helpers as the tensor-core kernels, on a barrier
// that nothing ever arrives on.  The wait gives up after limit_cycles, the thread records kDevTimeout in the status
// word, as those kernels do, and the kernel ends; nothing faults and nothing waits longer than the limit.
namespace fff {
__global__ void k_selftest_bounded_wait(int* __restrict__ status, long long limit_cycles)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    bool timed_out = false;
    if (threadIdx.x == 0 && !ptx::mbar_wait(&bar, 0, limit_cycles)) timed_out = true;
    if (threadIdx.x == 32 && !ptx::mbar_wait_relaxed(&bar, 0, limit_cycles)) timed_out = true;
    if (timed_out) atomicExch(status, kDevTimeout);
}
}  // namespace fff

// ---- scratch of fff_leaf_bucketing_static ----------------------------------------------------
// Two histogram buffers of FFF_STATIC_MAX_BINS counters each, resident on every device that loads the
// library.  In host code this name only stands for the symbol; the device address comes from
// cudaGetSymbolAddress (static_scratch_for_current_device).
static __device__ __align__(256) int g_static_bucket_scratch[2 * FFF_STATIC_MAX_BINS];

namespace {

std::mutex g_static_mu;
int* g_static_ptr[kMaxDevices] = {};

// Device address of the static scratch on the current device; looked up once per device.
fff_status_t static_scratch_for_current_device(int** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return FFF_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_ptr[dev]) {
        int* p = nullptr;
        if (cudaGetSymbolAddress((void**)&p, g_static_bucket_scratch) != cudaSuccess || !p)
            return cudaGetLastError(), FFF_ERR_CUDA;
        if (cudaFuncSetAttribute(fff::k_bucket, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(int) * fff::kBucketWarps * fff::kBucketMaxBinsPerCta)) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        g_static_ptr[dev] = p;
    }
    *out = g_static_ptr[dev];
    return FFF_OK;
}

}  // namespace

extern "C" {

fff_status_t fff_leaf_bucketing_static(const int32_t* leaf_idx, int32_t* offsets, int32_t* perm, int64_t B,
                                       int depth, void* cuda_stream) {
    if (B < 0 || depth < 0) return FFF_ERR_INVALID_ARG;
    if (depth > FFF_STATIC_MAX_DEPTH || B > FFF_MAX_TOKENS) return FFF_ERR_TOO_LARGE;
    if (!offsets || (B > 0 && (!leaf_idx || !perm))) return FFF_ERR_INVALID_ARG;
    int* scratch = nullptr;
    fff_status_t s = static_scratch_for_current_device(&scratch);
    if (s != FFF_OK) return s;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int nbins = 1 << depth;
    int* hist = scratch;                          // must start at zero: holds the previous call's counts
    int* spare = scratch + FFF_STATIC_MAX_BINS;   // only written (zeroed) by the bucketing kernel
    if (cudaMemsetAsync(hist, 0, sizeof(int) * (size_t)nbins, st) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    if (B > 0) {
        int sms = 148;
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int64_t blocks = std::min<int64_t>((B + 255) / 256, (int64_t)sms * 4);
        fff::k_histogram<<<(unsigned)blocks, 256, 0, st>>>(leaf_idx, hist, B, nbins);
        if (cudaGetLastError() != cudaSuccess) return FFF_ERR_CUDA;
    }
    int ctas = std::min(nbins, 32);
    int per = (nbins + ctas - 1) / ctas;
    if (per > fff::kBucketMaxBinsPerCta) {
        per = fff::kBucketMaxBinsPerCta;
        ctas = (nbins + per - 1) / per;
    }
    fff::k_bucket<<<ctas, fff::kBucketThreads, sizeof(int) * (size_t)fff::kBucketWarps * per, st>>>(
        leaf_idx, hist, spare, offsets, perm, (int)B, nbins, per, 0, nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

const char* fff_status_string(fff_status_t s) {
    switch (s) {
        case FFF_OK: return "ok";
        case FFF_ERR_INVALID_ARG: return "invalid argument";
        case FFF_ERR_UNSUPPORTED: return "unsupported configuration";
        case FFF_ERR_ALLOC: return "allocation failed";
        case FFF_ERR_CUDA: return "CUDA runtime error";
        case FFF_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        case FFF_ERR_BAD_HANDLE: return "bad handle";
        case FFF_ERR_TOO_LARGE: return "size exceeds the capacity of the static scratch";
    }
    return "unknown status";
}

}  // extern "C"

namespace {

// fff_create and fff_create_w8: w1_scale != nullptr means leaf_w1 / leaf_w2 are e4m3 codes with per-leaf scales.
fff_status_t create_common(fff_handle_t* out, int D, int O, int depth, int leaf_width, fff_activation_t act,
                           fff_dtype_t dtype, const void* node_w, const void* node_b, const void* leaf_w1,
                           const void* leaf_b1, const void* leaf_w2, const void* leaf_b2, const float* w1_scale,
                           const float* w2_scale) {
    if (!out) return FFF_ERR_INVALID_ARG;
    *out = nullptr;
    if (D < 1 || O < 1 || leaf_width < 1 || depth < 0) return FFF_ERR_INVALID_ARG;
    if (act != FFF_ACT_RELU && act != FFF_ACT_GELU && act != FFF_ACT_GELU_TANH && act != FFF_ACT_SILU) return FFF_ERR_INVALID_ARG;
    if (dtype != FFF_DTYPE_F32 && dtype != FFF_DTYPE_BF16) return FFF_ERR_INVALID_ARG;
    if (depth > FFF_MAX_DEPTH) return FFF_ERR_UNSUPPORTED;
    if (!leaf_w1 || !leaf_w2 || (depth > 0 && !node_w)) return FFF_ERR_INVALID_ARG;
    for (const void* p : {node_w, node_b, leaf_w1, leaf_b1, leaf_w2, leaf_b2, (const void*)w1_scale, (const void*)w2_scale})
        if (p && !aligned16(p)) return FFF_ERR_INVALID_ARG;
    const bool w8 = w1_scale != nullptr;
    if (w8 && (!w2_scale || dtype != FFF_DTYPE_BF16)) return FFF_ERR_INVALID_ARG;
    // 8-bit leaf weights run on the tcgen05 leaf kernel only
    if (w8 && (D % fff::kKS != 0 || O % 16 != 0 || leaf_width > 64 || !encode_tiled_fn())) return FFF_ERR_UNSUPPORTED;

    fff_handle_s* h = new (std::nothrow) fff_handle_s();
    if (!h) return FFF_ERR_ALLOC;
    if (cudaGetDevice(&h->device) != cudaSuccess) { delete h; return cudaGetLastError(), FFF_ERR_CUDA; }
    if (h->device < 0 || h->device >= kMaxDevices) { delete h; return FFF_ERR_UNSUPPORTED; }
    cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device);
    {
        const int smem_max = (int)(sizeof(int) * (fff::kBucketWarps + 1) * fff::kBucketMaxBinsPerCta);
        cudaFuncSetAttribute(fff::k_bucket_cluster<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(fff::kBucketClusterSize);
        cfg.blockDim = dim3(fff::kBucketThreads);
        cfg.dynamicSmemBytes = 4096;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = fff::kBucketClusterSize;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fff::k_bucket_cluster<32>, &cfg) == cudaSuccess && n > 0)
            h->max_bucket_clusters = n;
        else
            cudaGetLastError();
    }
    h->D = D; h->O = O; h->depth = depth; h->Dp = (D + fff::kKS - 1) / fff::kKS * fff::kKS; h->l = leaf_width; h->act = act; h->dtype = dtype;
    h->esize = dtype == FFF_DTYPE_F32 ? 4 : 2;
    h->n_nodes = ((int64_t)1 << depth) - 1;
    h->n_leaves = (int64_t)1 << depth;
    h->vec_ok = (D % (int)(16 / h->esize)) == 0;

    const size_t e = h->esize, nn = (size_t)h->n_nodes, nl = (size_t)h->n_leaves;
    fff_status_t s = FFF_OK;
    if (s == FFF_OK) s = clone(&h->node_w, node_w, nn * D * e);
    if (s == FFF_OK) s = clone(&h->node_b, node_b, nn * e);
    h->w8 = w8;
    if (s == FFF_OK && !w8) s = clone(&h->w1, leaf_w1, nl * leaf_width * D * e);
    if (s == FFF_OK) s = clone(&h->b1, leaf_b1, nl * leaf_width * e);
    if (s == FFF_OK && !w8) s = clone(&h->w2, leaf_w2, nl * O * leaf_width * e);
    if (s == FFF_OK) s = clone(&h->b2, leaf_b2, nl * O * e);
    if (s == FFF_OK) s = clone((void**)&h->ws_offsets, nullptr, sizeof(int32_t) * (nl + 1));
    if (s == FFF_OK) s = clone((void**)&h->ws_offsets2[0], nullptr, sizeof(int32_t) * (nl + 1));
    if (s == FFF_OK) s = clone((void**)&h->ws_offsets2[1], nullptr, sizeof(int32_t) * (nl + 1));
    if (s == FFF_OK) s = clone((void**)&h->d_status, nullptr, sizeof(int));
    {
        int coop = 0, per_sm = 0;
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device);
        const int smem_max = (int)(sizeof(int) * (fff::kCoopWarps + 2) * fff::kBucketMaxBinsPerCta);
        cudaFuncSetAttribute(fff::k_bucket_coop, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        if (coop && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fff::k_bucket_coop, fff::kCoopThreads, smem_max) ==
                        cudaSuccess &&
            per_sm > 0) {
            h->coop_ctas = h->sm_count;          // one CTA per SM is always resident
            if (s == FFF_OK)
                s = clone((void**)&h->ws_matrix, nullptr, sizeof(int) * (size_t)h->coop_ctas * fff::kBucketMaxBinsPerCta);
        } else {
            cudaGetLastError();
        }
    }
    if (s == FFF_OK && dtype == FFF_DTYPE_BF16 && D % 8 == 0 && depth > 0) s = pack_node_images<__nv_bfloat16>(h);
    if (s == FFF_OK && w8) {
        h->LP = leaf_width <= 16 ? 16 : (leaf_width <= 32 ? 32 : 64);
        const int LP = h->LP;
        const size_t P = (size_t)(O + fff::kLUPiece - 1) / fff::kLUPiece;
        if (s == FFF_OK) s = dmalloc((void**)&h->w1codes, nl * LP * D);
        if (s == FFF_OK) s = dmalloc((void**)&h->w2codes, nl * P * ((size_t)fff::kLUPiece * LP + fff::kLUPiece * 4));
        if (s == FFF_OK) s = dmalloc((void**)&h->b1img, nl * LP * 4);
        if (s == FFF_OK) s = clone((void**)&h->scale1, w1_scale, nl * sizeof(float));
        if (s == FFF_OK) s = clone((void**)&h->scale2, w2_scale, nl * sizeof(float));
        if (s == FFF_OK) s = clone((void**)&h->ws_sched, nullptr, 4 * sizeof(int));
        if (s == FFF_OK) {
            // (the caller's code arrays are read directly: nothing else of the library needs a copy of them)
            fff::k_pack_leaf_codes<__nv_bfloat16><<<h->sm_count * 8, 256>>>((const unsigned char*)leaf_w1, (const unsigned char*)leaf_w2,
                                                                           (const __nv_bfloat16*)h->b2, h->w1codes, h->w2codes, (int)nl,
                                                                           leaf_width, LP, D, O, h->ws_sched + 2);
            fff::k_pack_b1<__nv_bfloat16><<<h->sm_count * 8, 256>>>((const __nv_bfloat16*)h->b1, h->b1img, (int)nl, leaf_width, LP);
            if (cudaGetLastError() != cudaSuccess) s = FFF_ERR_CUDA;
        }
    } else if (s == FFF_OK && dtype == FFF_DTYPE_BF16 && D % 8 == 0 && O % 8 == 0 && leaf_width <= 64) {
        h->LP = leaf_width <= 16 ? 16 : (leaf_width <= 32 ? 32 : 64);
        s = pack_leaf_images<__nv_bfloat16>(h);
    }
    if (s == FFF_OK && !w8 && h->w2uimg) s = pack_group_images<__nv_bfloat16>(h);
    if (s == FFF_OK && !w8) s = FFF_DISPATCH(h, plan_block_forward, h);
    if (s == FFF_OK) s = plan_block_tiles(h);
    if (s == FFF_OK && !w8) plan_train(h);
    if (s == FFF_OK && cudaDeviceSynchronize() != cudaSuccess) s = (cudaGetLastError(), FFF_ERR_CUDA);
    if (s != FFF_OK) { release(h); return s; }
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_live.insert(h);
    }
    *out = h;
    return FFF_OK;
}

}  // namespace

extern "C" {

fff_status_t fff_create(fff_handle_t* out, int D, int O, int depth, int leaf_width, fff_activation_t act,
                        fff_dtype_t dtype, const void* node_w, const void* node_b, const void* leaf_w1,
                        const void* leaf_b1, const void* leaf_w2, const void* leaf_b2) {
    return create_common(out, D, O, depth, leaf_width, act, dtype, node_w, node_b, leaf_w1, leaf_b1, leaf_w2, leaf_b2, nullptr,
                         nullptr);
}

fff_status_t fff_create_w8(fff_handle_t* out, int D, int O, int depth, int leaf_width, fff_activation_t act,
                           const void* node_w, const void* node_b, const uint8_t* leaf_w1_e4m3, const float* leaf_w1_scale,
                           const void* leaf_b1, const uint8_t* leaf_w2_e4m3, const float* leaf_w2_scale, const void* leaf_b2) {
    if (!leaf_w1_scale || !leaf_w2_scale) return out ? (*out = nullptr, FFF_ERR_INVALID_ARG) : FFF_ERR_INVALID_ARG;
    return create_common(out, D, O, depth, leaf_width, act, FFF_DTYPE_BF16, node_w, node_b, leaf_w1_e4m3, leaf_b1, leaf_w2_e4m3,
                         leaf_b2, leaf_w1_scale, leaf_w2_scale);
}

fff_status_t fff_destroy(fff_handle_t h) {
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!h || g_live.erase(h) == 0) return FFF_ERR_BAD_HANDLE;
    }
    DeviceGuard g(h->device);
    cudaDeviceSynchronize();
    release(h);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

fff_status_t fff_reserve(fff_handle_t h, int64_t max_B) {
    fff_status_t s = check_forward_args(h, max_B);
    if (s != FFF_OK) return s;
    DeviceGuard g(h->device);
    return grow_workspace(h, max_B);
}

fff_status_t fff_set_path(fff_handle_t h, fff_path_t path) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (path != FFF_PATH_AUTO && path != FFF_PATH_WARP && path != FFF_PATH_TENSOR && path != FFF_PATH_FUSED)
        return FFF_ERR_INVALID_ARG;
    // (pinning to the tensor-core kernels stays reserved to layers whose rows they take unpadded)
    if (path == FFF_PATH_TENSOR && ((h->LP == 0 && h->stages.empty()) || h->D != h->Dp)) return FFF_ERR_UNSUPPORTED;
    if (path == FFF_PATH_FUSED && !h->bf_pinnable) return FFF_ERR_UNSUPPORTED;
    if (h->w8 && path != FFF_PATH_AUTO && path != FFF_PATH_TENSOR) return FFF_ERR_UNSUPPORTED;
    h->path = path;
    if (runs_block_forward(h) && h->cap_B > 0 && !h->ws_slots) {      // a workspace sized without its lists
        DeviceGuard g(h->device);
        const int64_t B = h->cap_B;
        h->cap_B = 0;
        return grow_workspace(h, B);
    }
    return FFF_OK;
}

fff_status_t fff_set_tuning(fff_handle_t h, fff_tuning_t key, int value) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if ((int)key < 0 || (int)key >= FFF_TUNE_COUNT || (value != 0 && value != 1)) return FFF_ERR_INVALID_ARG;
    h->tune[key] = value != 0;
    return FFF_OK;
}

fff_status_t fff_tree_descent(fff_handle_t h, const void* x, int32_t* leaf_idx, int64_t B, void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (B == 0) { h->launches = 0; return FFF_OK; }
    if (!x || !leaf_idx || !aligned16(x)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if ((s = grow_workspace(h, B)) != FFF_OK) return s;
    h->launches = 0;
    return run_descent(h, x, leaf_idx, nullptr, B, (cudaStream_t)cuda_stream);
}

fff_status_t fff_leaf_bucketing(fff_handle_t h, const int32_t* leaf_idx, int32_t* offsets, int32_t* perm, int64_t B,
                                void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (!offsets || (B > 0 && (!leaf_idx || !perm))) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if ((s = grow_workspace(h, B)) != FFF_OK) return s;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    h->launches = 0;
    return run_bucket(h, leaf_idx, (int)h->n_leaves, Coarse(), offsets, perm, B, st, 0, "leaf_bucketing");
}

fff_status_t fff_grouped_leaf_ff(fff_handle_t h, const void* x, const int32_t* leaf_idx, const int32_t* offsets,
                                 const int32_t* perm, void* y, int64_t B, void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (B == 0) { h->launches = 0; return FFF_OK; }
    if (!x || !y || !leaf_idx || !offsets || !perm || !aligned16(x) || !aligned16(y)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    h->launches = 0;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (use_tensor_leaf(h)) {
        if ((s = grow_workspace(h, B)) != FFF_OK) return s;
        const LeafPlan plan = leaf_plan(h, B);
        const int tile_rows = plan.tile_rows;
        fff::k_tiles_from_offsets<<<1, fff::kBucketThreads, 0, st>>>(offsets, (int)h->n_leaves, tile_rows, h->ws_tiles,
                                                                     tile_list_len(B, tile_rows, (int)h->n_leaves));
        if ((s = launched(h, st, "tiles_from_offsets")) != FFF_OK) return s;
        return run_leaf_mma(h, x, perm, y, B, plan, st);
    }
    return FFF_DISPATCH(h, run_leaf, h, x, leaf_idx, perm, y, B, st);
}

fff_status_t fff_forward_infer(fff_handle_t h, const void* x, void* y, int32_t* leaf_idx, int64_t B, void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (B == 0) { h->launches = 0; h->last_B = 0; return FFF_OK; }
    if (!x || !y || !aligned16(x) || !aligned16(y)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if ((s = grow_workspace(h, B)) != FFF_OK) return s;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int32_t* leaf = leaf_idx ? leaf_idx : h->ws_leaf;
    h->launches = 0;
    h->last_B = B;
    h->pending_in_staging = false;
    h->prof_active = h->prof_steps < h->prof_max_steps;
    if (h->prof_active)
        cudaEventRecord(h->prof_events[(size_t)h->prof_steps * (fff_handle_s::kMaxProfLaunches + 1)], st);
    const int64_t plan_B = planned_tokens(h, B);
    const bool token_blocks = use_token_block(h, plan_B);
    if (token_blocks || use_block_forward(h, plan_B)) {
        // one launch: a CTA per token; or descent, grid barrier, leaves.  The stable bucketing is made on demand from the leaf
        // indices that are left in the workspace
        s = token_blocks ? FFF_DISPATCH(h, run_token_block, h, x, y, h->ws_leaf, leaf_idx, B, st)
                         : FFF_DISPATCH(h, run_block_forward, h, x, y, h->ws_leaf, leaf_idx, B, st);
        h->last_perm = h->ws_perm;
        h->bucketing_pending = true;
        if (h->prof_active) {
            h->prof_active = false;
            if (s == FFF_OK && (h->prof_steps == 0 || h->prof_nlaunch == h->launches)) {
                h->prof_nlaunch = std::min(h->launches, (int)fff_handle_s::kMaxProfLaunches);
                ++h->prof_steps;
            }
        }
        return s;
    }
    const bool tensor_leaf = use_tensor_leaf(h);
    // With fewer than about 4 tokens per leaf the warp leaf kernel gains nothing from bucket order (no
    // weights to share), so the bucketing is left out of the forward and made on demand
    // (fff_debug_get_bucketing) from the leaf indices, which then also live in the workspace.
    const bool lazy_bucketing = !tensor_leaf && plan_B < 4 * h->n_leaves;
    if (lazy_bucketing) leaf = h->ws_leaf;
    Coarse coarse;
    DescentTail tail;
    LeafPlan plan = tensor_leaf ? leaf_plan(h, plan_B) : LeafPlan{};
    const int tile_rows = plan.tile_rows;
    // The descent ends with a tcgen05 stage and a tensor-core leaf kernel follows: that stage files the tokens under their
    // leaves itself and the leaf kernel follows at once, on tiles it derives from the lists' counts.
    h->slots_now = h->tune[FFF_TUNE_DIRECT_LISTS] && h->tune[FFF_TUNE_TCGEN05_DESCENT] && tensor_leaf && !h->ustages.empty() &&
                   leaf_lists_fit(h, B) &&
                   (plan.umma ? tile_rows == fff::kLUM : h->n_leaves <= kMaxListedLeaves && plan_B <= kMaxListedTokens) && h->ustages.back().umma &&
                   h->ustages.back().L0 + h->ustages.back().k == h->depth &&
                   dense_stage_count(h, B, false) == (int)h->ustages.size() &&
                   (h->ustages.size() == 1 ||
                    (h->tune[FFF_TUNE_TCGEN05_GROUPED] && (fills_grouped_tiles(h, B, h->ustages.back().L0) ||
                                                           (h->ustages.size() == 2 && node_lists_fit(h, B)))));
    const bool group_tiles = tensor_leaf && plan.umma && use_group_tiles(h, B);
    if (h->slots_now && !group_tiles && !h->w8 && warp_tiles(h, plan, plan_B)) plan = LeafPlan{fff::kLWRows};
    if (group_tiles) {
        h->slots_now = false;
        s = run_forward_grouped(h, x, y, leaf, B, st);
        h->last_perm = h->ws_perm;
        h->bucketing_pending = true;          // the stable permutation is made on demand from ws_leaf
        if (h->prof_active) {
            h->prof_active = false;
            if (s == FFF_OK && (h->prof_steps == 0 || h->prof_nlaunch == h->launches)) {
                h->prof_nlaunch = std::min(h->launches, (int)fff_handle_s::kMaxProfLaunches);
                ++h->prof_steps;
            }
        }
        return s;
    }
    if (h->slots_now) {
        if (h->cursor_dirty && cudaMemsetAsync(h->ws_cursor, 0, cursor_bytes(h), st) != cudaSuccess)
            return h->slots_now = false, cudaGetLastError(), FFF_ERR_CUDA;
        h->cursor_dirty = true;
        s = run_descent(h, x, leaf, nullptr, B, st);
        h->last_perm = h->ws_perm;
        h->bucketing_pending = true;          // the stable permutation is made on demand from ws_leaf
        if (s == FFF_OK) s = run_leaf_mma(h, x, h->ws_slots, y, B, plan, st);
        if (s == FFF_OK) h->cursor_dirty = false;
        h->slots_now = false;
        if (h->prof_active) {
            h->prof_active = false;
            if (s == FFF_OK && (h->prof_steps == 0 || h->prof_nlaunch == h->launches)) {
                h->prof_nlaunch = std::min(h->launches, (int)fff_handle_s::kMaxProfLaunches);
                ++h->prof_steps;
            }
        }
        return s;
    }
    // without a bucketing in between, the warp leaf kernel also walks the levels the staged descent leaves over
    s = run_descent(h, x, leaf, &coarse, B, st, lazy_bucketing ? &tail : nullptr, !lazy_bucketing);
    // the final permutation goes to whichever buffer the last node bucketing did not use
    h->last_perm = coarse.perm == h->ws_perm ? h->ws_perm2 : h->ws_perm;
    h->bucketing_pending = lazy_bucketing;
    if (lazy_bucketing) {
        if (s == FFF_OK) s = FFF_DISPATCH(h, run_leaf, h, x, leaf, nullptr, y, B, st, tail, leaf);
        if (s == FFF_OK && leaf_idx &&
            cudaMemcpyAsync(leaf_idx, leaf, sizeof(int32_t) * (size_t)B, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            s = (cudaGetLastError(), FFF_ERR_CUDA);
    } else {
        if (s == FFF_OK)
            s = run_bucket(h, leaf, (int)h->n_leaves, coarse, h->ws_offsets, h->last_perm, B, st, tile_rows, "leaf_bucketing");
        if (s == FFF_OK)
            s = tensor_leaf ? run_leaf_mma(h, x, h->last_perm, y, B, plan, st)
                            : FFF_DISPATCH(h, run_leaf, h, x, leaf, h->last_perm, y, B, st);
    }
    if (h->prof_active) {
        h->prof_active = false;
        if (s == FFF_OK && (h->prof_steps == 0 || h->prof_nlaunch == h->launches)) {
            h->prof_nlaunch = std::min(h->launches, (int)fff_handle_s::kMaxProfLaunches);
            ++h->prof_steps;
        }
    }
    return s;
}

fff_status_t fff_forward_train(fff_handle_t h, const void* x, void* y, float* mixture, float* node_entropy, int64_t B,
                               void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (h->tr_Kp == 0) return FFF_ERR_UNSUPPORTED;
    if (B == 0) { h->launches = 0; return FFF_OK; }
    if (!x || !y || !aligned16(x) || !aligned16(y)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    h->launches = 0;
    return run_forward_train(h, x, y, mixture, node_entropy, B, (cudaStream_t)cuda_stream);
}

// Chunks of a host-buffer forward: of 8192 tokens, or two for a smaller batch of at least 4 MB of x and y (less, and the
// second chunk's submission and launches cost what the overlap saves), as long as the weights that a chunk fetches again cost
// less than a quarter of its copies (16 times its bytes: memory is about 120 times as fast as the link).  One chunk against
// two, us, 768 -> 768, bf16, 256 leaves of 12: 3 MB 104 and 104, 4 MB 128 and 115, 8 MB 193 and 174, 12 MB 272 and 242, 24 MB
// 484 and 412; three or four are level with two or behind.  A smaller first or last chunk gains nothing: a copy that runs
// while another one goes the other way costs about 7 us more than its bytes.
// Copies of pageable memory hold up the host and overlap nothing, so those batches stay whole up to 16 384 tokens (cut in two:
// 4 MB 405 against 334 us, 9 MB 607 against 547, 17 MB 1030 against 965).
static bool pinned(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) return cudaGetLastError(), false;
    return a.type == cudaMemoryTypeHost || a.type == cudaMemoryTypeManaged;
}

static int host_chunks(const fff_handle_s* h, const void* x_host, const void* y_host, int64_t B) {
    const int64_t per_token = (int64_t)(h->D + h->O) * (int64_t)h->esize, half = (B + 1) / 2;
    const bool profiled = h->prof_steps < h->prof_max_steps;      // a profiled step is a whole forward
    const bool halves = !profiled && B < 16384 && B * per_token >= 4000000 && std::min<int64_t>(h->n_leaves, half) * h->l <= 16 * half &&
                        pinned(x_host) && pinned(y_host);
    return (int)std::max<int64_t>(halves ? 2 : 1, std::min<int64_t>(fff_handle_s::kMaxHostChunks, B / 8192));
}

fff_status_t fff_forward_infer_host(fff_handle_t h, const void* x_host, void* y_host, int32_t* leaf_idx_host,
                                    int64_t B, void* cuda_stream) {
    fff_status_t s = check_forward_args(h, B);
    if (s != FFF_OK) return s;
    if (B == 0) { h->launches = 0; h->last_B = 0; return FFF_OK; }
    if (!x_host || !y_host) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (B > h->cap_host_B) {
        if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        h->last_B = -1;                     // (a bucketing made on demand would read the leaf indices that are freed here)
        h->pending_in_staging = false;
        dfree(h->st_x); dfree(h->st_y); dfree(h->st_leaf);
        h->st_x = h->st_y = nullptr; h->st_leaf = nullptr; h->cap_host_B = 0;
        if ((s = dmalloc(&h->st_x, (size_t)B * h->D * h->esize)) != FFF_OK) return s;
        if ((s = dmalloc(&h->st_y, (size_t)B * h->O * h->esize)) != FFF_OK) return s;
        if ((s = dmalloc((void**)&h->st_leaf, (size_t)B * sizeof(int32_t))) != FFF_OK) return s;
        h->cap_host_B = B;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // Batches go through in chunks so that the copy of chunk i+1 to the device, the kernels of chunk i
    // and the copy of chunk i-1 back overlap (tokens are independent, so chunking does not change any result).
    const int n_chunks = host_chunks(h, x_host, y_host, B);
    if (n_chunks == 1) {
        if (cudaMemcpyAsync(h->st_x, x_host, (size_t)B * h->D * h->esize, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        if ((s = fff_forward_infer(h, h->st_x, h->st_y, h->st_leaf, B, cuda_stream)) != FFF_OK) return s;
        if (cudaMemcpyAsync(y_host, h->st_y, (size_t)B * h->O * h->esize, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        if (leaf_idx_host &&
            cudaMemcpyAsync(leaf_idx_host, h->st_leaf, (size_t)B * sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        return FFF_OK;
    }
    if (!h->copy_in) {
        bool ok = cudaStreamCreateWithFlags(&h->copy_in, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&h->copy_out, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaEventCreateWithFlags(&h->ev_start, cudaEventDisableTiming) == cudaSuccess &&
                  cudaEventCreateWithFlags(&h->ev_end, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; ok && i < fff_handle_s::kMaxHostChunks; ++i)
            ok = cudaEventCreateWithFlags(&h->ev_in[i], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&h->ev_done[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) return cudaGetLastError(), FFF_ERR_CUDA;
    }
    const int64_t chunk = (((B + n_chunks - 1) / n_chunks) + 127) & ~int64_t(127);
    const int n_full = (int)((B + chunk - 1) / chunk);
    const size_t xrow = (size_t)h->D * h->esize, yrow = (size_t)h->O * h->esize;
    auto copy_leaves = [&](int64_t from, int64_t to) {
        return !leaf_idx_host || cudaMemcpyAsync(leaf_idx_host + from, h->st_leaf + from, (size_t)(to - from) * sizeof(int32_t),
                                                 cudaMemcpyDeviceToHost, h->copy_out) == cudaSuccess;
    };
    bool ok = cudaEventRecord(h->ev_start, st) == cudaSuccess &&              // the copies come after what the caller enqueued
              cudaStreamWaitEvent(h->copy_in, h->ev_start, 0) == cudaSuccess &&
              cudaStreamWaitEvent(h->copy_out, h->ev_start, 0) == cudaSuccess;
    for (int c = 0; ok && c < n_full; ++c) {
        const int64_t b0 = c * chunk, n = std::min(chunk, B - b0);
        ok = cudaMemcpyAsync((char*)h->st_x + b0 * xrow, (const char*)x_host + b0 * xrow, (size_t)n * xrow, cudaMemcpyHostToDevice,
                             h->copy_in) == cudaSuccess &&
             cudaEventRecord(h->ev_in[c], h->copy_in) == cudaSuccess;
    }
    for (int c = 0; ok && c < n_full; ++c) {
        const int64_t b0 = c * chunk, n = std::min(chunk, B - b0);
        ok = cudaStreamWaitEvent(st, h->ev_in[c], 0) == cudaSuccess;
        if (!ok) break;
        h->plan_B = B;           // results do not depend on the chunking
        s = fff_forward_infer(h, (char*)h->st_x + b0 * xrow, (char*)h->st_y + b0 * yrow, h->st_leaf + b0, n, cuda_stream);
        h->plan_B = 0;
        if (s != FFF_OK) return s;
        ok = cudaEventRecord(h->ev_done[c], st) == cudaSuccess && cudaStreamWaitEvent(h->copy_out, h->ev_done[c], 0) == cudaSuccess &&
             cudaMemcpyAsync((char*)y_host + b0 * yrow, (char*)h->st_y + b0 * yrow, (size_t)n * yrow, cudaMemcpyDeviceToHost,
                             h->copy_out) == cudaSuccess &&
             (c != n_full - 2 || copy_leaves(0, b0 + n)) &&            // the leaves of all chunks but the last in one copy
             (c != n_full - 1 || copy_leaves(n_full > 1 ? b0 : 0, b0 + n));
    }
    ok = ok && cudaEventRecord(h->ev_end, h->copy_out) == cudaSuccess && cudaStreamWaitEvent(st, h->ev_end, 0) == cudaSuccess &&
         cudaStreamSynchronize(st) == cudaSuccess;
    // the workspace holds the last chunk only: the bucketing of a small batch is made on demand from the staged leaf indices,
    // that of a large one is not reported
    h->last_B = ok && B < 16384 ? B : -1;
    h->bucketing_pending = h->pending_in_staging = true;
    return ok ? FFF_OK : (cudaGetLastError(), FFF_ERR_CUDA);
}

fff_status_t fff_debug_get_bucketing(fff_handle_t h, int32_t* perm, int32_t* offsets, void* cuda_stream) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (!offsets || h->last_B < 0 || (h->last_B > 0 && !perm)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (h->last_B > 0 && h->bucketing_pending) {
        if (h->pending_in_staging) {
            const fff_status_t gs = grow_workspace(h, h->last_B);      // (it was sized for a chunk)
            if (gs != FFF_OK) return gs;
            h->last_perm = h->ws_perm;
        }
        const int saved = h->launches;
        h->launches = 0;           // an ordinary launch: nothing of this call precedes it in the stream
        const fff_status_t bs = run_bucket(h, h->pending_in_staging ? h->st_leaf : h->ws_leaf, (int)h->n_leaves, Coarse(), h->ws_offsets, h->last_perm, h->last_B, st,
                                           0, "leaf_bucketing");
        h->launches = saved;
        if (bs != FFF_OK) return bs;
        h->bucketing_pending = false;
    }
    if (h->last_B > 0 &&
        cudaMemcpyAsync(perm, h->last_perm, sizeof(int32_t) * (size_t)h->last_B, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return cudaGetLastError(), FFF_ERR_CUDA;
    if (h->last_B > 0) {
        if (cudaMemcpyAsync(offsets, h->ws_offsets, sizeof(int32_t) * (size_t)(h->n_leaves + 1), cudaMemcpyDeviceToDevice,
                            st) != cudaSuccess)
            return cudaGetLastError(), FFF_ERR_CUDA;
    } else if (cudaMemsetAsync(offsets, 0, sizeof(int32_t) * (size_t)(h->n_leaves + 1), st) != cudaSuccess) {
        return cudaGetLastError(), FFF_ERR_CUDA;
    }
    return FFF_OK;
}

fff_status_t fff_get_last_status(fff_handle_t h) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    DeviceGuard g(h->device);
    if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    int word = 0;
    if (cudaMemcpy(&word, h->d_status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    if (word != fff::kDevOk) {
        const fff_status_t cs = default_stream_done(cudaMemset(h->d_status, 0, sizeof(int)));
        return cs != FFF_OK ? cs : FFF_ERR_DEVICE_TIMEOUT;
    }
    return FFF_OK;
}

fff_status_t fff_selftest_bounded_wait(fff_handle_t h, int64_t limit_cycles, void* cuda_stream) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (limit_cycles < 1 || limit_cycles > (int64_t)1 << 24) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    fff::k_selftest_bounded_wait<<<1, 64, 0, (cudaStream_t)cuda_stream>>>(h->d_status, (long long)limit_cycles);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

int fff_last_launch_count(fff_handle_t h) { return live(h) ? h->launches : -1; }

int fff_capabilities(fff_handle_t h) {
    if (!live(h)) return -1;
    int caps = 0;
    if (h->D == h->Dp) {
        if (!h->stages.empty() || !h->ustages.empty()) caps |= FFF_CAP_TENSOR_DESCENT;
        if (!h->ustages.empty()) caps |= FFF_CAP_TCGEN05_DESCENT;
        if (h->LP != 0) caps |= FFF_CAP_TENSOR_LEAF;
        if (h->w2uimg || h->w2codes) caps |= FFF_CAP_TCGEN05_LEAF;
    } else if (!h->ustages.empty() || h->LP != 0) {
        caps |= FFF_CAP_PADDED;
    }
    if (h->bf_pinnable) caps |= FFF_CAP_FUSED_SMALL;
    if (h->tr_Kp != 0) caps |= FFF_CAP_FORWARD_TRAIN;
    if (h->g_w1) caps |= FFF_CAP_GROUP_TILES;
    return caps;
}

fff_status_t fff_profile_begin(fff_handle_t h, int max_steps) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (max_steps < 0 || max_steps > (1 << 20)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    prof_free(h);
    const size_t n = (size_t)max_steps * (fff_handle_s::kMaxProfLaunches + 1);
    h->prof_events.reserve(n);
    for (size_t i = 0; i < n; ++i) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) { prof_free(h); return cudaGetLastError(), FFF_ERR_ALLOC; }
        h->prof_events.push_back(e);
    }
    h->prof_max_steps = max_steps;
    return FFF_OK;
}

int fff_profile_launches(fff_handle_t h) { return live(h) ? h->prof_nlaunch : -1; }

const char* fff_profile_launch_name(fff_handle_t h, int i) {
    if (!live(h) || i < 0 || i >= h->prof_nlaunch || !h->prof_names[i]) return "";
    return h->prof_names[i];
}

fff_status_t fff_profile_end(fff_handle_t h, double* mean_ms, int* steps) {
    if (!live(h)) return FFF_ERR_BAD_HANDLE;
    if (!mean_ms || !steps) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    *steps = h->prof_steps;
    const int stride = fff_handle_s::kMaxProfLaunches + 1;
    for (int i = 0; i < h->prof_nlaunch; ++i) {
        double sum = 0.0;
        for (int s = 0; s < h->prof_steps; ++s) {
            float ms = 0.0f;
            if (cudaEventElapsedTime(&ms, h->prof_events[(size_t)s * stride + i], h->prof_events[(size_t)s * stride + i + 1]) !=
                cudaSuccess)
                return cudaGetLastError(), FFF_ERR_CUDA;
            sum += ms;
        }
        mean_ms[i] = h->prof_steps ? sum / h->prof_steps : 0.0;
    }
    h->prof_max_steps = 0;      // stop recording; names and counts stay readable until the next begin
    return FFF_OK;
}


}  // extern "C"

// ---- stacks of layers --------------------------------------------------------------------------------------

namespace {

void stack_release(fff_stack_s* s) {
    if (s->exec) cudaGraphExecDestroy(s->exec);
    for (void* p : s->gamma) dfree(p);
    for (void* p : s->beta) dfree(p);
    dfree(s->buf_z); dfree(s->buf_y); dfree(s->buf_x[0]); dfree(s->buf_x[1]);
    s->magic = 0;
    delete s;
}

template <typename T>
fff_status_t stack_glue(fff_stack_s* s, const void* x_prev, const void* y_prev, void* x_out, void* z, int layer, int64_t B,
                        cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((B + fff::kStackWarps - 1) / fff::kStackWarps, (int64_t)s->sm_count * 8);
    const bool vec = s->D % (int)(16 / s->esize) == 0 && aligned16(x_prev) && aligned16(y_prev) && aligned16(x_out) && aligned16(z);
    const T *g = z ? (const T*)s->gamma[layer] : nullptr, *b = z ? (const T*)s->beta[layer] : nullptr;
    cudaError_t e;
    if (vec && s->D <= 32 * 32)          // (in registers: 32 values per lane)
        e = launch_chain(s->layers[0], fff::k_stack_glue_rows<T>, (unsigned)blocks, fff::kStackWarps * 32, 0, st, 1, (const T*)x_prev,
                         (const T*)y_prev, (T*)x_out, (T*)z, g, b, s->eps, s->D, B);
    else
        e = launch_chain(s->layers[0], fff::k_stack_glue<T>, (unsigned)blocks, fff::kStackWarps * 32, 0, st, 1, (const T*)x_prev,
                         (const T*)y_prev, (T*)x_out, (T*)z, g, b, s->eps, s->D, B, vec);
    if (e != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
    ++s->launches;
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

// The forward of the whole stack, enqueued kernel by kernel.
fff_status_t stack_enqueue(fff_stack_s* s, const void* x, void* y, int32_t* leaf_idx, int64_t B, cudaStream_t st) {
    const int K = (int)s->layers.size();
    const void* x_cur = x;           // x_k
    const void* y_prev = nullptr;    // y_{k-1}, not yet added to x_{k-1} (residual stacks)
    fff_status_t rc = FFF_OK;
    s->launches = 0;
    for (int k = 0; k < K && rc == FFF_OK; ++k) {
        const void* ffn_in = x_cur;
        if (s->residual && y_prev) {
            // x_k = x_{k-1} + y_{k-1}, and its normalisation in the same pass
            void* x_new = s->buf_x[k & 1];
            rc = s->dtype == FFF_DTYPE_F32 ? stack_glue<float>(s, x_cur, y_prev, x_new, s->layer_norm ? s->buf_z : nullptr, k, B, st)
                                           : stack_glue<__nv_bfloat16>(s, x_cur, y_prev, x_new, s->layer_norm ? s->buf_z : nullptr, k, B, st);
            x_cur = x_new;
            ffn_in = s->layer_norm ? s->buf_z : x_new;
        } else if (s->layer_norm) {
            rc = s->dtype == FFF_DTYPE_F32 ? stack_glue<float>(s, x_cur, nullptr, nullptr, s->buf_z, k, B, st)
                                           : stack_glue<__nv_bfloat16>(s, x_cur, nullptr, nullptr, s->buf_z, k, B, st);
            ffn_in = s->buf_z;
        }
        if (rc != FFF_OK) break;
        // without residual connections the last layer writes y itself, the others into the buffer the next one reads
        void* out = (!s->residual && k == K - 1) ? y : (s->residual ? s->buf_y : s->buf_x[k & 1]);
        rc = fff_forward_infer(s->layers[k], ffn_in, out, leaf_idx ? leaf_idx + (int64_t)k * B : nullptr, B, (void*)st);
        s->launches += s->layers[k]->launches;
        if (s->residual) y_prev = out;
        else x_cur = out;
    }
    if (rc == FFF_OK && s->residual)
        rc = s->dtype == FFF_DTYPE_F32 ? stack_glue<float>(s, x_cur, y_prev, y, nullptr, 0, B, st)
                                       : stack_glue<__nv_bfloat16>(s, x_cur, y_prev, y, nullptr, 0, B, st);
    return rc;
}

}  // namespace

extern "C" {

fff_status_t fff_stack_create(fff_stack_t* out, int n_layers, const fff_handle_t* layers, int layer_norm, const void* const* ln_gamma,
                              const void* const* ln_beta, float eps, int residual) {
    if (!out) return FFF_ERR_INVALID_ARG;
    *out = nullptr;
    if (n_layers < 1 || n_layers > 1024 || !layers || !(eps >= 0.0f)) return FFF_ERR_INVALID_ARG;
    for (int k = 0; k < n_layers; ++k)
        if (!live(layers[k])) return FFF_ERR_BAD_HANDLE;
    const fff_handle_s* first = layers[0];
    for (int k = 0; k < n_layers; ++k) {
        const fff_handle_s* h = layers[k];
        if (h->device != first->device || h->dtype != first->dtype) return FFF_ERR_INVALID_ARG;
        // a layer reads what the one before it wrote; residual connections and shared buffers need one width
        if (h->D != first->D || h->O != first->D) return FFF_ERR_INVALID_ARG;
        for (int j = 0; j < k; ++j)
            if (layers[j] == layers[k]) return FFF_ERR_INVALID_ARG;      // a handle serves one forward at a time
    }
    fff_stack_s* s = new (std::nothrow) fff_stack_s();
    if (!s) return FFF_ERR_ALLOC;
    s->device = first->device;
    s->sm_count = first->sm_count;
    s->D = first->D;
    s->dtype = first->dtype;
    s->esize = first->esize;
    s->layer_norm = layer_norm != 0;
    s->residual = residual != 0;
    s->eps = eps;
    s->layers.assign(layers, layers + n_layers);
    s->gamma.assign(n_layers, nullptr);
    s->beta.assign(n_layers, nullptr);
    DeviceGuard g(s->device);
    fff_status_t rc = FFF_OK;
    for (int k = 0; k < n_layers && rc == FFF_OK && s->layer_norm; ++k) {
        if (ln_gamma && ln_gamma[k]) rc = clone(&s->gamma[k], ln_gamma[k], (size_t)s->D * s->esize);
        if (rc == FFF_OK && ln_beta && ln_beta[k]) rc = clone(&s->beta[k], ln_beta[k], (size_t)s->D * s->esize);
    }
    if (rc == FFF_OK && cudaDeviceSynchronize() != cudaSuccess) rc = (cudaGetLastError(), FFF_ERR_CUDA);
    if (rc != FFF_OK) { stack_release(s); return rc; }
    s->magic = kStackMagic;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_live_stacks.insert(s);
    }
    *out = s;
    return FFF_OK;
}

fff_status_t fff_stack_destroy(fff_stack_t s) {
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!s || g_live_stacks.erase(s) == 0) return FFF_ERR_BAD_HANDLE;
    }
    DeviceGuard g(s->device);
    cudaDeviceSynchronize();
    stack_release(s);
    return cudaGetLastError() == cudaSuccess ? FFF_OK : FFF_ERR_CUDA;
}

fff_status_t fff_stack_set_graph(fff_stack_t s, int on) {
    if (!live_stack(s)) return FFF_ERR_BAD_HANDLE;
    if (on != 0 && on != 1) return FFF_ERR_INVALID_ARG;
    s->want_graph = on != 0;
    s->graph_failed = false;
    return FFF_OK;
}

int fff_stack_last_launch_count(fff_stack_t s) { return live_stack(s) ? s->launches : -1; }
int fff_stack_last_was_replay(fff_stack_t s) { return live_stack(s) ? (s->replayed ? 1 : 0) : -1; }

fff_status_t fff_stack_forward(fff_stack_t s, const void* x, void* y, int32_t* leaf_idx, int64_t B, void* cuda_stream) {
    if (!live_stack(s)) return FFF_ERR_BAD_HANDLE;
    if (B < 0) return FFF_ERR_INVALID_ARG;
    if (B > FFF_MAX_TOKENS) return FFF_ERR_UNSUPPORTED;
    for (fff_handle_s* h : s->layers)
        if (!live(h)) return FFF_ERR_BAD_HANDLE;
    s->replayed = false;
    if (B == 0) { s->launches = 0; return FFF_OK; }
    if (!x || !y || !aligned16(x) || !aligned16(y)) return FFF_ERR_INVALID_ARG;
    DeviceGuard g(s->device);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (B > s->cap_B) {
        if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        if (s->exec) { cudaGraphExecDestroy(s->exec); s->exec = nullptr; }
        dfree(s->buf_z); dfree(s->buf_y); dfree(s->buf_x[0]); dfree(s->buf_x[1]);
        s->buf_z = s->buf_y = s->buf_x[0] = s->buf_x[1] = nullptr;
        s->cap_B = 0;
        const size_t bytes = (size_t)B * s->D * s->esize;
        fff_status_t rc;
        if ((rc = dmalloc(&s->buf_z, bytes)) != FFF_OK || (rc = dmalloc(&s->buf_y, bytes)) != FFF_OK ||
            (rc = dmalloc(&s->buf_x[0], bytes)) != FFF_OK || (rc = dmalloc(&s->buf_x[1], bytes)) != FFF_OK)
            return rc;
        for (fff_handle_s* h : s->layers)
            if ((rc = grow_workspace(h, B)) != FFF_OK) return rc;
        s->cap_B = B;
    }
    // (a layer whose workspace has been replaced since, by fff_reserve or a larger batch of its own, is no longer where the graph writes)
    uint64_t epoch = 0;
    for (const fff_handle_s* h : s->layers) epoch += h->epoch;
    if (s->exec && s->key_epoch != epoch) {
        if (cudaDeviceSynchronize() != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        cudaGraphExecDestroy(s->exec);
        s->exec = nullptr;
    }
    const bool same_as_graph = s->exec && s->key_x == x && s->key_y == y && s->key_leaf == leaf_idx && s->key_B == B && s->key_stream == st;
    if (s->want_graph && same_as_graph) {
        if (cudaGraphLaunch(s->exec, st) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
        s->replayed = true;
        return FFF_OK;
    }
    // The second forward with the same arguments is recorded into a graph (the first ran every one-time set-up:
    // workspaces, kernel attributes); later ones replay it.
    const bool seen = s->seen_x == x && s->seen_y == y && s->seen_leaf == leaf_idx && s->seen_B == B && s->seen_stream == st;
    if (s->want_graph && !s->graph_failed && seen) {
        cudaGraph_t graph = nullptr;
        if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            const fff_status_t rc = stack_enqueue(s, x, y, leaf_idx, B, st);
            const cudaError_t ce = cudaStreamEndCapture(st, &graph);
            cudaGraphExec_t exec = nullptr;
            if (rc == FFF_OK && ce == cudaSuccess && graph && cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess) {
                cudaGraphDestroy(graph);
                if (s->exec) cudaGraphExecDestroy(s->exec);
                s->exec = exec;
                s->key_x = x; s->key_y = y; s->key_leaf = leaf_idx; s->key_B = B; s->key_stream = st;
                s->key_epoch = epoch;
                if (cudaGraphLaunch(s->exec, st) != cudaSuccess) return cudaGetLastError(), FFF_ERR_CUDA;
                s->replayed = true;
                return FFF_OK;
            }
            if (graph) cudaGraphDestroy(graph);
        }
        cudaGetLastError();
        s->graph_failed = true;            // this stack's forward cannot be recorded: plain launches from now on
    }
    s->seen_x = x; s->seen_y = y; s->seen_leaf = leaf_idx; s->seen_B = B; s->seen_stream = st;
    return stack_enqueue(s, x, y, leaf_idx, B, st);
}

}  // extern "C"
