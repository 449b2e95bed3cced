// A batch of layer calls: the layers of one chunk handed over together, so that layers of one kind share their launches.
// The plan (which layer goes where, its tiling and scratch) is made once; a run fills in the buffers and launches.
#include "batch.cuh"
#include "wgrad_tc.cuh"
#include <algorithm>
#include <cstddef>
#include <exception>
#include <mutex>
#include <new>
#include <vector>

using namespace dp;

namespace {
// Streams and events the runs of a batch fork to.  Making a set costs some 100 us, more than the first run of a small model,
// so a batch takes one that an earlier batch has given back: a set keeps its order of work, and a new batch's launches at
// worst queue behind what the old one still has running.  At most kKeptSets wait for a taker.
struct SideStreams {
    int device;
    bool beside;                 // normalisation layers run beside the convolutions
    cudaStream_t stream[BatchStreams::kCount];
    cudaEvent_t fork, begun, gate, gram_done, done[BatchStreams::kCount];
};
constexpr size_t kKeptSets = 8;
std::mutex kept_mu;
std::vector<SideStreams *> &kept_sets() { static auto *sets = new std::vector<SideStreams *>; return *sets; }   // outlives every batch

void drop_streams(SideStreams *t) {
    for (int i = 1; i < BatchStreams::kCount; ++i) {
        if (t->done[i]) cudaEventDestroy(t->done[i]);
        if (t->stream[i]) cudaStreamDestroy(t->stream[i]);
    }
    if (t->fork) cudaEventDestroy(t->fork);
    if (t->begun) cudaEventDestroy(t->begun);
    if (t->gate) cudaEventDestroy(t->gate);
    if (t->gram_done) cudaEventDestroy(t->gram_done);
    delete t;
}
// a set on the current device, or null
SideStreams *take_streams(bool beside) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    {
        std::lock_guard<std::mutex> lock(kept_mu);
        auto &sets = kept_sets();
        for (size_t i = sets.size(); i-- > 0;) {
            if (sets[i]->device != dev || sets[i]->beside != beside) continue;
            SideStreams *t = sets[i];
            sets.erase(sets.begin() + (std::ptrdiff_t)i);
            return t;
        }
    }
    SideStreams *t = new (std::nothrow) SideStreams{};
    if (!t) return nullptr;
    t->device = dev;
    t->beside = beside;
    // Beside normalisation layers, what others wait for, and short launches, take SMs before large clusters do, and those before
    // the caller's stream.  Elsewhere the normalisation layers are to fill gaps and not to come first (a chunk of 4 ResNet-50
    // examples: 167 us with these priorities and single calls on a stream of their own, 155 with neither).
    int low = 0, high = 0;
    if (beside) (void)cudaDeviceGetStreamPriorityRange(&low, &high);
    int priority[BatchStreams::kCount] = {};
    priority[BatchStreams::kClusters] = priority[BatchStreams::kClusters6] = high / 2;
    priority[BatchStreams::kSums] = priority[BatchStreams::kAffine] = high;
    bool ok = cudaEventCreateWithFlags(&t->fork, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&t->begun, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&t->gate, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&t->gram_done, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 1; ok && i < BatchStreams::kCount; ++i)
        ok = cudaStreamCreateWithPriority(&t->stream[i], cudaStreamNonBlocking, priority[i]) == cudaSuccess &&
             cudaEventCreateWithFlags(&t->done[i], cudaEventDisableTiming) == cudaSuccess;
    if (ok) return t;
    (void)cudaGetLastError();
    drop_streams(t);
    return nullptr;
}
void give_back(SideStreams *t) {
    bool idle = true;                        // a stream some unfinished capture holds is of no use to others
    for (int i = 1; i < BatchStreams::kCount; ++i) {
        cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
        idle = idle && cudaStreamIsCapturing(t->stream[i], &c) == cudaSuccess && c == cudaStreamCaptureStatusNone;
    }
    if (idle) {
        std::lock_guard<std::mutex> lock(kept_mu);
        auto &sets = kept_sets();
        if (sets.capacity() < kKeptSets) { try { sets.reserve(kKeptSets); } catch (const std::exception &) {} }
        if (sets.size() < std::min(kKeptSets, sets.capacity())) { sets.push_back(t); return; }
    }
    drop_streams(t);
}
}  // namespace

struct dp_batch {
    struct Item {
        dp_layer_desc desc;
        int epi;
        WgradPlan plan;
        int group, slot;             // table of its kind and place in it; group < 0: a call of its own
        int lane;                    // of a call of its own: 0 has a stream of the batch's, others are the caller's
        size_t scratch;              // byte offset of the layer's own scratch (factors, finished per-example gradients)
    };
    std::vector<Item> items;
    std::vector<AffineGroup> affine;             // shapes filled in, buffers per run
    std::vector<int> affine_dtype;
    std::vector<char> affine_beside;             // runs beside convolutions
    bool beside = false;                         // planned for some that do
    int singles_stream = BatchStreams::kSingles; // single calls of lane 0
    size_t affine_partial = 0;                   // byte offset of the pixel-chunk partials
    std::vector<ConvJob> convs;                  // geometry filled in, buffers per run
    std::vector<int> conv_item;                  // item of every conv
    double walk = 0.0;                           // conv_batch_walk() of all of them
    size_t singles = 0;                          // byte offset of the scratch the single calls share
    bool used[BatchStreams::kCount] = {};        // streams that have launches of their own
    size_t total = 0;
    int lanes = 1;                               // streams the single calls spread over
    int target = 0;                              // SM target they are planned for (they share the GPU when there are lanes)
    size_t lane_bytes = 0;                       // workspace of every lane but the first
    // Taken by the first run, on its device; host threads take turns at enqueueing.
    mutable std::mutex mu;
    mutable SideStreams *side = nullptr;
    mutable int lane_device = -1;
    mutable std::vector<cudaEvent_t> lane_events;            // [lanes]: the fork, then every further lane's end
};

namespace dp {

// Whether the batch has side streams, on this device.
static bool side_streams(const dp_batch &b) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (!b.side) b.side = take_streams(b.beside);
    return b.side && b.side->device == dev;
}

// Events the further lanes are forked and joined with, on this device; false: the single calls stay on one stream.
static bool lane_events(const dp_batch &b) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (b.lane_device < 0) {
        while ((int)b.lane_events.size() < b.lanes) {
            cudaEvent_t e;
            if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { (void)cudaGetLastError(); return false; }
            b.lane_events.push_back(e);
        }
        b.lane_device = dev;
    }
    return b.lane_device == dev;
}

// Rough time of a call of its own on a GPU it has to itself, in microseconds: enough to spread the calls over lanes.
static double single_cost(const dp_batch::Item &it) {
    if (it.desc.kind != DP_LAYER_CONV2D) return 6.0;
    const ConvGeom g = geom_of(&it.desc);
    return 12.0 + 2.0 * g.B * g.M * g.N * g.K / (it.plan.use_tc ? 2e8 : 2e7);
}

// Gives every call of its own a lane, the longest first, each to the lane with the least work.
static void plan_lanes(dp_batch &b, int lanes) {
    std::vector<int> singles;
    for (int i = 0; i < (int)b.items.size(); ++i)
        if (b.items[i].group < 0) singles.push_back(i);
    b.lanes = std::max(1, std::min(lanes, (int)singles.size()));
    if (b.lanes == 1) return;
    b.lane_events.reserve(b.lanes);
    b.target = sm_target_set() ? sm_target() : 0;
    std::stable_sort(singles.begin(), singles.end(), [&](int x, int y) { return single_cost(b.items[x]) > single_cost(b.items[y]); });
    std::vector<double> load(b.lanes, 0.0);
    for (const AffineGroup &g : b.affine)                    // these follow lane 0, or have a stream of their own
        for (int k = 0; b.singles_stream == BatchStreams::kAffine && k < g.n; ++k) load[0] += (double)g.seg[k].B * g.seg[k].HW * g.seg[k].C * 4.0 / 5e6;
    for (int i : singles) {
        dp_batch::Item &it = b.items[i];
        make_layer_plan(&it.desc, it.epi, it.plan);          // (for the target)
        it.lane = (int)(std::min_element(load.begin(), load.end()) - load.begin());
        load[it.lane] += single_cost(it);
        b.lane_bytes = std::max(b.lane_bytes, round_up(it.plan.total, 256));
    }
}

static bool affine_of(const dp_layer_desc &d) { return d.kind == DP_LAYER_NORM_AFFINE && affine_batch_eligible(storage_type(&d), d.C_in); }
static double affine_bytes(const dp_layer_desc &d) { return 2.0 * d.B * d.H * d.W * d.C_in * (storage_type(&d) == DP_F32 ? 4 : 2); }
// From here on layers run beside the convolutions: the layers of a ResNet-50 of fewer examples are through in the gaps between the
// launches, and shallower rings of the convolutions cost more than that.  Chunks of 3, 4, 5, 6, 8 and 12 examples (133, 178, 222,
// 267, 356 and 533 MB of these layers): 136, 154, 180, 214, 255 and 358 us, with the layers beside 144, 152, 177, 188, 242 and 330.
constexpr double kBesideBytes = 250e6;

// What the convolutions' launches leave the normalisation layers that run beside them, in bytes: some 2.8 TB/s of theirs for the
// time these take by rates measured on a chunk of ResNet-50 (53 layers x 32 examples: 263 Gflop in 550 us clipped; 16 examples:
// 133 Gflop and 1.6 GB stored in 430 us).
static double bytes_beside(const dp_batch &b) {
    double us = 0.0;
    for (const ConvJob &j : b.convs) {
        const double rate = j.dtype == DP_BF16 ? 480e6 : (j.dtype == DP_TF32 ? 200e6 : 90e6);
        us += 2.0 * j.g.B * j.g.M * j.g.N * j.g.K / rate;
        if (j.epi == DP_EPI_STORE_NORM) us += 4.0 * j.g.B * j.g.M * j.g.N / 10e6;
    }
    return us * 2.8e6;
}

static void plan_affine(dp_batch &b, size_t &off) {
    // Layers beside the convolutions as far as these last, the rest at the GPU's full rate, in a form that takes SMs of its own.
    double room = b.beside ? bytes_beside(b) : 0.0;
    std::vector<char> beside(b.items.size(), 0);
    for (size_t i = 0; i < b.items.size(); ++i) {
        const dp_layer_desc &d = b.items[i].desc;
        if (!affine_of(d) || affine_bytes(d) > room) continue;
        beside[i] = 1;
        room -= affine_bytes(d);
    }
    size_t partial_floats = 0;
    for (int form = 0; form < 4; ++form) {
        const int dtype = form & 1 ? DP_F32 : DP_BF16;
        const bool is_beside = form < 2;
        bool fresh_group = true;
        for (size_t i = 0; i < b.items.size(); ++i) {
            dp_batch::Item &it = b.items[i];
            const dp_layer_desc &d = it.desc;
            if (!affine_of(d) || storage_type(&d) != dtype || (beside[i] != 0) != is_beside) continue;
            if (fresh_group || b.affine.back().n == kGroupLayers) {
                fresh_group = false;
                AffineGroup fresh = {};
                b.affine.push_back(fresh);
                b.affine_dtype.push_back(dtype);
                b.affine_beside.push_back(is_beside);
            }
            AffineGroup &g = b.affine.back();
            it.group = (int)b.affine.size() - 1;
            it.slot = g.n++;
            AffineSeg &s = g.seg[it.slot];
            affine_batch_shape(dtype, d.B, d.H * d.W, d.C_in, is_beside, s);
            s.clip = it.epi == DP_EPI_CLIP_ACCUM;
            s.separate = groups_of(&d) == 2;
            s.part_off = (long long)partial_floats;
            partial_floats += (size_t)d.B * s.chunks * 2 * d.C_in;
            // [factors][dgamma][dbeta] unless the caller takes the gradients
            it.scratch = off;
            off = round_up(off + sizeof(float) * 2 * d.B, 256);
            if (it.epi != DP_EPI_STORE_NORM) off = round_up(off + sizeof(float) * 2 * (size_t)d.B * d.C_in, 256);
        }
    }
    b.affine_partial = off;
    off = round_up(off + sizeof(float) * partial_floats, 1024);
}

// The groups that run beside convolutions (which come after, on other streams) or the others; without streams for that, all.
enum { kBeside, kApart, kAllGroups };
static dp_status run_affine(const dp_batch &b, const dp_layer_io *io, float C_l, char *ws, int which, cudaEvent_t begun, cudaStream_t st) {
    if (b.affine.empty()) return DP_OK;
    std::vector<AffineGroup> groups = b.affine;
    for (size_t i = 0; i < b.items.size(); ++i) {
        const dp_batch::Item &it = b.items[i];
        if (it.desc.kind != DP_LAYER_NORM_AFFINE || it.group < 0) continue;
        AffineSeg &s = groups[it.group].seg[it.slot];
        s.X = io[i].X; s.dY = io[i].dY;
        s.sqnorm = io[i].sqnorm; s.sq_stride = io[i].sqnorm_stride; s.clip_out = io[i].clip_out;
        s.acc_w = io[i].acc_w; s.acc_b = io[i].acc_b;
        s.factor = reinterpret_cast<float *>(ws + it.scratch);
        if (it.epi == DP_EPI_STORE_NORM) {
            s.dgamma = io[i].G_w; s.dbeta = io[i].G_b;
        } else {
            s.dgamma = reinterpret_cast<float *>(ws + it.scratch + round_up(sizeof(float) * 2 * it.desc.B, 256));
            s.dbeta = s.dgamma + (size_t)it.desc.B * it.desc.C_in;
        }
    }
    for (size_t k = 0; k < groups.size(); ++k) {
        groups[k].C_l = C_l;
        groups[k].partial = reinterpret_cast<float *>(ws + b.affine_partial);
        if (which != kAllGroups && (b.affine_beside[k] != 0) != (which == kBeside)) continue;
        int *tickets = which == kBeside && k < kWsStreams ? reinterpret_cast<int *>(ws + kWsStreamOffset) + 2 * k : nullptr;
        const dp_status rc = launch_affine_batch(b.affine_dtype[k], groups[k], tickets, tickets ? begun : nullptr, st);
        if (tickets) begun = nullptr;                        // (the first one's)
        if (rc != DP_OK) return rc;
    }
    return DP_OK;
}

// Everything else waits until the normalisation layers' blocks are there, one on every SM, while all are still empty.  Started
// together with other launches they land where room is left: two on one SM, which has none for a convolution's block until they
// end, or on an SM that a small kernel has left with little shared memory, which is not divided anew while they run.  Chunks of
// ResNet-50 (32 examples, 32 of them replayed one behind the other) took 771 or 889 us, a run of the program either the one or the
// other, and 833 without layers beside; 759 this way (on a slower GPU 807 or 921, 851, and 786).  The wait for `begun` ends in a
// kernel: in a captured graph it is an edge that only kernels may have, and what the streams do next is not always one (with the
// streams waiting themselves: the same time).
__global__ void batch_gate_kernel() {}
static dp_status open_gate(const dp_batch &b, const BatchStreams &streams, void *const *lane_streams) {
    const cudaStream_t st = streams.s[BatchStreams::kMain];
    DP_CUDA_TRY(cudaStreamWaitEvent(st, b.side->begun, 0));
    batch_gate_kernel<<<1, 1, 0, st>>>();
    DP_LAUNCH_CHECK("batch_gate_kernel");
    DP_CUDA_TRY(cudaEventRecord(b.side->gate, st));
    for (int i = 1; i < BatchStreams::kCount; ++i)
        if (b.used[i] && i != BatchStreams::kAffine) DP_CUDA_TRY(cudaStreamWaitEvent(streams.s[i], b.side->gate, 0));
    for (int k = 1; lane_streams && k < b.lanes; ++k)
        DP_CUDA_TRY(cudaStreamWaitEvent(static_cast<cudaStream_t>(lane_streams[k - 1]), b.side->gate, 0));
    return DP_OK;
}

static void plan_convs(dp_batch &b, size_t &off) {
    for (size_t i = 0; i < b.items.size(); ++i) {
        dp_batch::Item &it = b.items[i];
        const dp_layer_desc &d = it.desc;
        if (d.kind != DP_LAYER_CONV2D || !it.plan.use_tc || (int)b.convs.size() >= kWsBatchCounters) continue;
        ConvJob j = {};
        j.g = geom_of(&d); j.dtype = d.dtype; j.epi = it.epi;
        j.kind = conv_batch_kind(d.dtype, j.g, it.epi, d.has_bias != 0);
        if (j.kind == kConvSingle) continue;
        j.separate = groups_of(&d) == 2;
        it.group = 0; it.slot = (int)b.convs.size();
        b.convs.push_back(j);
        b.conv_item.push_back((int)i);
    }
    if (b.convs.empty()) return;
    double bytes = 0.0;
    for (const auto &it : b.items) bytes += affine_of(it.desc) ? affine_bytes(it.desc) : 0.0;
    b.beside = bytes >= kBesideBytes;
    b.walk = conv_batch_walk(b.convs, b.beside);
    BatchPlanning planning(b.walk, b.beside);
    for (size_t k = 0; k < b.convs.size(); ++k) {
        dp_batch::Item &it = b.items[b.conv_item[k]];
        make_layer_plan(&it.desc, it.epi, it.plan);          // scratch sizes of the tiling a batch uses
        b.convs[k].slots = it.plan.slots; b.convs[k].w_slots = it.plan.w_slots;
        it.scratch = off;
        off = round_up(off + it.plan.total - kWsHeaderBytes, 1024);
    }
}

static dp_status run_convs(const dp_batch &b, const dp_layer_io *io, float C_l, char *ws, const BatchStreams &streams,
                           const std::function<dp_status()> &join) {
    const cudaStream_t st = streams.s[BatchStreams::kMain];
    std::vector<ConvJob> jobs = b.convs;
    for (size_t k = 0; k < jobs.size(); ++k) {
        const dp_batch::Item &it = b.items[b.conv_item[k]];
        const dp_layer_io &o = io[b.conv_item[k]];
        ConvJob &j = jobs[k];
        char *base = ws + it.scratch - kWsHeaderBytes;       // the plan's offsets count from a header
        j.X = o.X; j.dY = o.dY; j.G_w = o.G_w; j.acc_w = o.acc_w;
        j.partial = reinterpret_cast<float *>(base + it.plan.partial_off);
        j.factor = reinterpret_cast<float *>(base + it.plan.factor_off);
        j.tc_workspace = base + it.plan.tc_off;
        j.counter = reinterpret_cast<int *>(ws + kWsCounterOffset) + (kWsCounters - kWsBatchCounters) + k;
        j.clip = TcInlineClip{C_l, o.sqnorm, o.sqnorm_stride, o.clip_out};
        if (it.desc.has_bias) {
            float *db = it.epi == DP_EPI_STORE_NORM ? o.G_b : reinterpret_cast<float *>(base + it.plan.db_off);
            // a bias that is a group of its own and publishes its norm itself need not come before the weights' launch
            j.bias_apart = j.separate && bias_publishes(storage_type(&it.desc), j.g);
            const dp_status rc = launch_bias(storage_type(&it.desc), o.dY, j.g, db, j.partial, it.plan.slots, it.plan.w_slots,
                                             j.bias_apart ? streams.s[BatchStreams::kSums] : st, j.bias_apart ? o.sqnorm + 1 : nullptr,
                                             o.sqnorm_stride);
            if (rc != DP_OK) return rc;
        }
    }
    return launch_conv_batch(jobs, b.walk, b.beside, reinterpret_cast<int *>(ws), streams, join);
}

static dp_status plan_batch(dp_batch &b, int n, const dp_layer_desc *descs, const int *epilogues, int lanes) {
    b.items.resize(n);
    size_t off = kWsHeaderBytes;
    {
        SmTargetScope whole_gpu(0);
        for (int i = 0; i < n; ++i) {
            dp_batch::Item &it = b.items[i];
            it.desc = descs[i]; it.epi = epilogues[i]; it.group = it.slot = -1; it.lane = 0; it.scratch = 0;
            make_layer_plan(&it.desc, it.epi, it.plan);
            if (it.desc.impl == DP_IMPL_TENSOR_CORE && !it.plan.use_tc) return DP_ERR_UNSUPPORTED;
        }
        plan_convs(b, off);
        plan_affine(b, off);
    }
    // (ahead of normalisation layers that run apart from the convolutions, which then do not all start at once)
    b.singles_stream = b.beside ? BatchStreams::kSingles : BatchStreams::kAffine;
    plan_lanes(b, lanes);
    b.singles = off;
    size_t most = 0;
    for (const auto &it : b.items) {
        if (it.group >= 0) continue;
        most = std::max(most, it.plan.total);
        b.used[b.singles_stream] = true;
    }
    if (!b.affine.empty()) b.used[BatchStreams::kAffine] = true;
    for (const ConvJob &j : b.convs) {
        b.used[BatchStreams::kMain] = true;
        b.used[conv_cluster_stream(conv_batch_cluster(j, b.walk, b.beside), b.beside)] = true;
        if (j.kind == kConvGramSum || j.kind == kConvGramTiles || b.items[b.conv_item[&j - b.convs.data()]].desc.has_bias) b.used[BatchStreams::kSums] = true;
    }
    b.total = most > kWsHeaderBytes ? round_up(off + most - kWsHeaderBytes, 256) : off;
    return DP_OK;
}

}  // namespace dp

extern "C" dp_status dp_batch_create_lanes(int n, const dp_layer_desc *descs, const int *epilogues, int lanes, dp_batch **out) {
    if (n <= 0 || !descs || !epilogues || lanes < 1 || !out) return DP_ERR_INVALID_ARG;
    *out = nullptr;
    for (int i = 0; i < n; ++i) {
        if (!valid_desc(&descs[i]) || epilogues[i] < 0 || epilogues[i] > 2) return DP_ERR_INVALID_ARG;
        if (groups_of(&descs[i]) < 1) return DP_ERR_INVALID_ARG;
    }
    dp_batch *b = new (std::nothrow) dp_batch;
    if (!b) return DP_ERR_CUDA;
    try {
        const dp_status rc = plan_batch(*b, n, descs, epilogues, lanes);
        if (rc != DP_OK) { delete b; return rc; }
    } catch (const std::exception &) {           // out of memory
        delete b;
        return DP_ERR_CUDA;
    }
    *out = b;
    return DP_OK;
}

extern "C" dp_status dp_batch_create(int n, const dp_layer_desc *descs, const int *epilogues, dp_batch **out) {
    return dp_batch_create_lanes(n, descs, epilogues, 1, out);
}

extern "C" void dp_batch_destroy(dp_batch *b) {
    if (!b) return;
    if (b->side) give_back(b->side);
    for (cudaEvent_t e : b->lane_events) cudaEventDestroy(e);
    delete b;
}

extern "C" size_t dp_batch_workspace_bytes(const dp_batch *b) { return b ? b->total : 0; }

extern "C" int dp_batch_lanes(const dp_batch *b) { return b ? b->lanes : 0; }

extern "C" size_t dp_batch_lane_bytes(const dp_batch *b) { return b ? b->lane_bytes : 0; }

extern "C" dp_status dp_batch_run(const dp_batch *b, const dp_layer_io *io, float C_l, void *workspace, size_t workspace_bytes,
                                  void *cuda_stream) {
    return dp_batch_run_lanes(b, io, C_l, workspace, workspace_bytes, cuda_stream, 0, nullptr, nullptr, 0);
}

extern "C" dp_status dp_batch_run_lanes(const dp_batch *b, const dp_layer_io *io, float C_l, void *workspace, size_t workspace_bytes,
                                        void *cuda_stream, int further, void *const *lane_streams, void *const *lane_workspaces,
                                        size_t lane_bytes) {
    if (!b || !io || further < 0) return DP_ERR_INVALID_ARG;
    const int n = (int)b->items.size();
    for (int i = 0; i < n; ++i) {
        const LayerBuffers buf = {io[i].X, io[i].dY, io[i].G_w, io[i].G_b, io[i].sqnorm, io[i].sqnorm_stride, io[i].acc_w, io[i].acc_b, io[i].clip_out};
        const dp_status rc = check_layer(&b->items[i].desc, b->items[i].epi, buf, C_l);
        if (rc != DP_OK) return rc;
    }
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < b->total) return DP_ERR_WORKSPACE;
    bool laned = b->lanes > 1 && further >= b->lanes - 1;
    if (laned && (!lane_streams || !lane_workspaces)) return DP_ERR_INVALID_ARG;
    for (int k = 0; laned && k < b->lanes - 1; ++k)
        if (!lane_workspaces[k] || !aligned(lane_workspaces[k], 256) || lane_bytes < b->lane_bytes) return DP_ERR_WORKSPACE;
    char *ws = static_cast<char *>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    std::lock_guard<std::mutex> lock(b->mu);
    SmTargetScope whole_gpu(0);          // as the plans
    // The launches of different kinds are independent: memory-bound normalisation layers and the blocks of small launches
    // fill what the tensor-core launches leave idle.
    BatchStreams streams;
    // (without convolutions there is nothing to fork from: everything stays on the caller's stream)
    const bool forked = b->used[BatchStreams::kMain] && std::find(b->used + 1, b->used + BatchStreams::kCount, true) != b->used + BatchStreams::kCount && side_streams(*b);
    for (int i = 0; i < BatchStreams::kCount; ++i) streams.s[i] = forked && i && b->used[i] ? b->side->stream[i] : st;
    streams.gram_done = forked && b->used[BatchStreams::kSums] ? b->side->gram_done : nullptr;
    if (forked) {
        DP_CUDA_TRY(cudaEventRecord(b->side->fork, st));
        for (int i = 1; i < BatchStreams::kCount; ++i)
            if (b->used[i]) DP_CUDA_TRY(cudaStreamWaitEvent(streams.s[i], b->side->fork, 0));
    }
    laned = laned && lane_events(*b);
    if (laned) {
        DP_CUDA_TRY(cudaEventRecord(b->lane_events[0], st));
        for (int k = 1; k < b->lanes; ++k)
            DP_CUDA_TRY(cudaStreamWaitEvent(static_cast<cudaStream_t>(lane_streams[k - 1]), b->lane_events[0], 0));
    }
    // What is not a tensor-core launch of several layers.  Image stems of few examples first: their blocks hold an SM for long,
    // and behind the tensor-core launch they would be the tail of the chunk (a 38 x 38 stem of 37 examples: 130 us instead
    // of 68 for the chunk).  The rest fills gaps, so it is enqueued last, before the streams meet again; so are stems of
    // more examples than SMs, whose second round of blocks would leave SMs idle (256 of 32 x 32: 135 us first, 117 last).
    auto ahead = [](const dp_batch::Item &it) { return it.plan.use_thin && it.desc.B <= sm_count(); };
    auto singles = [&](bool first) -> dp_status {
        BatchPlanning alone(0.0, false);        // tiled as their plans were: not as layers of a grouped launch
        SmTargetScope target(b->target);
        dp_status rc = DP_OK;
        for (int i = 0; i < n && rc == DP_OK; ++i) {
            const dp_batch::Item &it = b->items[i];
            if (it.group >= 0 || ahead(it) != first) continue;
            const LayerBuffers buf = {io[i].X, io[i].dY, io[i].G_w, io[i].G_b, io[i].sqnorm, io[i].sqnorm_stride, io[i].acc_w, io[i].acc_b, io[i].clip_out};
            if (laned && it.lane) {
                char *own = static_cast<char *>(lane_workspaces[it.lane - 1]);
                rc = run_layer(&it.desc, it.epi, buf, C_l, it.plan, own, own + kWsHeaderBytes, static_cast<cudaStream_t>(lane_streams[it.lane - 1]));
            } else {
                rc = run_layer(&it.desc, it.epi, buf, C_l, it.plan, ws, ws + b->singles, streams.s[b->singles_stream]);
            }
        }
        return rc;
    };
    bool joined = false;
    auto join = [&]() -> dp_status {
        if (joined) return DP_OK;
        joined = true;
        dp_status rc;
        try {
            // (singles first: they are short, and behind the normalisation layers they would be the chunk's tail)
            rc = singles(false);
            if (rc == DP_OK) rc = run_affine(*b, io, C_l, ws, forked ? kApart : kAllGroups, nullptr, streams.s[BatchStreams::kAffine]);
        } catch (const std::exception &) {       // out of memory: the streams still have to meet
            rc = DP_ERR_CUDA;
        }
        for (int k = 1; laned && k < b->lanes; ++k) {
            DP_CUDA_TRY(cudaEventRecord(b->lane_events[k], static_cast<cudaStream_t>(lane_streams[k - 1])));
            DP_CUDA_TRY(cudaStreamWaitEvent(st, b->lane_events[k], 0));
        }
        if (!forked) return rc;
        for (int i = 1; i < BatchStreams::kCount; ++i) {
            if (!b->used[i]) continue;
            DP_CUDA_TRY(cudaEventRecord(b->side->done[i], streams.s[i]));
            DP_CUDA_TRY(cudaStreamWaitEvent(st, b->side->done[i], 0));
        }
        return rc;
    };
    dp_status rc;
    try {
        // (on every SM before the convolutions' blocks are)
        const bool beside = forked && std::find(b->affine_beside.begin(), b->affine_beside.end(), 1) != b->affine_beside.end();
        rc = beside ? run_affine(*b, io, C_l, ws, kBeside, b->side->begun, streams.s[BatchStreams::kAffine]) : DP_OK;
        if (beside && rc == DP_OK) rc = open_gate(*b, streams, laned ? lane_streams : nullptr);
        if (rc == DP_OK) rc = singles(true);
        if (rc == DP_OK) rc = run_convs(*b, io, C_l, ws, streams, join);
    } catch (const std::exception &) {           // out of memory
        rc = DP_ERR_CUDA;
    }
    if (rc != DP_OK) (void)join();       // a launch failed: whatever is enqueued still comes before what follows
    return rc;
}
