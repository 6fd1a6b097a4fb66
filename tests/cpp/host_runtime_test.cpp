// host_runtime_test.cpp — the host runtime of libpcr (csrc/*.cpp) over a stand-in for
// the CUDA runtime and the kernels' launchers, so that failing calls, stream captures
// and replays can be played through without a GPU.
//
// "Device" memory is host memory filled with rubbish when it is allocated. Work on a
// stream runs at once, or is recorded while the stream is captured. A frame's first
// pass notes whether its counters and sums start from zero, its last one leaves
// them so; what lies between dirties them.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "pc_internal.h"

using namespace pcr;

// ---- the stand-in ------------------------------------------------------------------

typedef std::vector<std::function<void()>> Ops;
struct CUgraph_st { Ops ops; };
struct CUgraphExec_st { Ops ops; };

static Ops* g_recording = nullptr;        // the captured stream's work
static std::map<std::string, int> g_fail; // call -> calls until one fails (1: the next)
static int g_dirty = 0, g_frames = 0, g_instantiated = 0, g_encoded = 0, g_branches = 0, g_misnumbered = 0;
static uint32_t g_last_frame = 0;
static size_t g_room = ~(size_t)0, g_used = 0;   // bytes the "device" has, and lent
static std::map<void*, size_t> g_blocks;

static bool fails(const char* call) {
    auto it = g_fail.find(call);
    return it != g_fail.end() && it->second > 0 && --it->second == 0;
}
static void run(std::function<void()> op) {
    if (g_recording) g_recording->push_back(op);
    else op();
}

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = nullptr;
    if (fails("malloc") || g_used + n > g_room) return cudaErrorMemoryAllocation;
    *p = aligned_alloc(256, (n + 255) & ~(size_t)255);
    std::memset(*p, 0xCD, n);
    g_blocks[*p] = n;
    g_used += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    g_used -= g_blocks.at(p);
    g_blocks.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
    if (fails("memset")) return cudaErrorInvalidValue;
    run([=] { std::memset(p, v, n); });
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    run([=] { std::memcpy(d, s, n); });
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(0x60);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0.0f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = nullptr;
    if (fails("stream")) return cudaErrorMemoryAllocation;
    *s = reinterpret_cast<cudaStream_t>(0x50);
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t f, void* a) { f(a); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_recording ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    g_recording = new Ops();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = new CUgraph_st{*g_recording};
    delete g_recording;
    g_recording = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete e; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    *e = new CUgraphExec_st{g->ops};
    ++g_instantiated;
    return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t e, cudaGraph_t g, cudaGraphExecUpdateResultInfo*) {
    // another number of kernels is another topology
    if (e->ops.size() != g->ops.size()) return cudaErrorGraphExecUpdateFailure;
    e->ops = g->ops;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
    for (auto& op : e->ops) op();
    return cudaSuccess;
}
}

namespace pcr {

static bool clean(const Scratch& s) {
    for (uint32_t i = 0; i < C_LIST; ++i)
        if (i != C_ERROR && i != C_ERRINFO && s.counters[i]) return false;
    for (uint32_t i = 0; i < kMaxViewsPerLaunch * S_COUNT; ++i)
        if (s.acc[i]) return false;
    return true;
}

cudaError_t launch_begin(const CloudView&, const ViewTable&, Scratch s, Begin what, cudaStream_t) {
    if (what == Begin::kClear) return cudaSuccess;
    run([=] {
        ++g_frames;
        if (!clean(s)) ++g_dirty;
        s.counters[C_ENTRIES] += 5;
        s.acc[S_BATCHES] += 7;
    });
    return cudaSuccess;
}
cudaError_t launch_lod_append(const CloudView&, const ViewTable&, Scratch, cudaStream_t) {
    run([] {});
    return cudaSuccess;
}
cudaError_t launch_raster(const CloudView&, const ViewTable& vt, Scratch s, RasterShape, const Branch* branch,
                          cudaStream_t, int* launched) {
    // a captured launch has no number (every replay would repeat it), others one of their own
    if ((g_recording != nullptr) != (s.frame == 0) || (s.frame && s.frame <= g_last_frame)) ++g_misnumbered;
    if (s.frame) g_last_frame = s.frame;
    if (branch) {
        ++g_branches;
        run([] {});   // another topology
    }
    if (fails("raster")) return cudaErrorLaunchFailure;
    *launched = vt.n == 1 ? 2 : 1;
    for (int i = 0; i < *launched; ++i) run([] {});
    return cudaSuccess;
}
cudaError_t launch_shade(const CloudView&, const ViewTable& vt, Scratch, RasterShape, cudaStream_t, int* launched) {
    *launched = 1;
    for (uint32_t v = 0; v < vt.n; ++v)
        if (vt.v[v].flags & PC_VIEW_HQS_PACKED) *launched = 2;
    for (int i = 0; i < *launched; ++i) run([] {});
    return cudaSuccess;
}
cudaError_t launch_resolve(const CloudView&, const ViewTable& vt, uint32_t, Scratch s, bool publish, cudaStream_t,
                           int* launched) {
    bool plain = false, dilated = false;
    for (uint32_t v = 0; v < vt.n; ++v) (vt.v[v].flags & PC_VIEW_DILATE ? dilated : plain) = true;
    *launched = (int)plain + (int)dilated;
    for (int i = 1; i < *launched; ++i) run([] {});
    run([=] {
        if (!publish) return;
        for (uint32_t i = 0; i < C_LIST; ++i)
            if (i != C_ERROR && i != C_ERRINFO) s.counters[i] = 0;
        std::memcpy(s.stats, s.acc, sizeof(unsigned long long) * vt.n * S_COUNT);
        std::memset(s.acc, 0, sizeof(unsigned long long) * vt.n * S_COUNT);
    });
    return cudaSuccess;
}
cudaError_t launch_merge_min(uint64_t*, const uint64_t*, uint64_t, cudaStream_t) { return cudaSuccess; }
int raster_occupancy(int, uint32_t) { return 4; }
uint64_t encode_device_scratch(uint64_t n, bool, bool) { return 40 * n; }
cudaError_t encode_device(const float* xyz, const uint32_t* rgba, uint64_t n, uint32_t batch_size, bool keep_order,
                          void*, pc_batch* batches, uint32_t* w1, uint32_t* w2, uint32_t* w3, uint32_t* color,
                          cudaStream_t, bool* finite) {
    ++g_encoded;
    *finite = encode_host(xyz, rgba, n, batch_size, 1, keep_order, batches, w1, w2, w3, color, nullptr) == PC_OK;
    return cudaSuccess;
}

}  // namespace pcr

// ---- scenarios -----------------------------------------------------------------------

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

static cudaStream_t const kStream = reinterpret_cast<cudaStream_t>(0x40);
alignas(16) static uint64_t g_vis[2][64];
alignas(16) static uint32_t g_rgba[2][64];

struct World {
    pc_ctx* ctx = nullptr;
    pc_cloud cloud = 0;
    std::vector<float> xyz;
    explicit World(uint32_t flags = 0, uint64_t n = 1000) : xyz(3 * n) {
        for (size_t i = 0; i < xyz.size(); ++i) xyz[i] = (float)((i * 7919u) % 1000u);
        pc_config cfg;
        pc_config_default(&cfg);
        cfg.flags = flags;
        cfg.batch_size = 128;
        CHECK(pc_create(&ctx, 0, &cfg) == PC_OK);
        CHECK(pc_upload_cloud(ctx, xyz.data(), nullptr, n, &cloud) == PC_OK);
    }
    ~World() { pc_destroy(ctx); }
    pc_status frame(std::vector<uint32_t> flags = {0u}) {
        std::vector<pc_view> v(flags.size());
        std::vector<pc_framebuffer> fb(flags.size());
        for (size_t i = 0; i < flags.size(); ++i) {
            std::memset(&v[i], 0, sizeof v[i]);
            v[i].width = v[i].height = 8;
            v[i].flags = flags[i];
            fb[i].vis = g_vis[i];
            fb[i].rgba = g_rgba[i];
        }
        return pc_render(ctx, cloud, v.data(), (uint32_t)v.size(), fb.data(), kStream);
    }
    unsigned long long batches_rendered() {
        pc_view_stats st;
        CHECK(pc_get_view_stats(ctx, kStream, 0, &st) == PC_OK);   // no error word either
        return st.batches_rendered;
    }
};

// A caller's captured frame.
static cudaGraphExec_t captured_frame(World& w, pc_status expect = PC_OK) {
    cudaGraph_t g;
    cudaGraphExec_t e;
    cudaStreamBeginCapture(kStream, cudaStreamCaptureModeRelaxed);
    CHECK(w.frame() == expect);
    cudaStreamEndCapture(kStream, &g);
    cudaGraphInstantiate(&e, g, 0);
    cudaGraphDestroy(g);
    return e;
}

// A frame whose launches fail part-way leaves nothing to the next one, whether that is
// queued, captured or an earlier capture's replay.
static void failed_frame() {
    World w;
    CHECK(w.frame() == PC_OK);
    g_fail["raster"] = 1;
    CHECK(w.frame() == PC_ECUDA);
    CHECK(w.frame() == PC_OK);
    CHECK(g_dirty == 0 && w.batches_rendered() == 7);
}
static void failed_frame_then_capture() {
    World w;
    CHECK(w.frame() == PC_OK);
    g_fail["raster"] = 1;
    CHECK(w.frame() == PC_ECUDA);
    cudaGraphExec_t e = captured_frame(w);   // nothing of it has run yet
    CHECK(w.frame() == PC_OK);
    cudaGraphLaunch(e, kStream);
    CHECK(w.frame() == PC_OK);
    CHECK(g_frames == 5 && g_dirty == 0);
    cudaGraphExecDestroy(e);
}
static void failed_frame_then_replay() {
    World w;
    CHECK(w.frame() == PC_OK);
    cudaGraphExec_t e = captured_frame(w);
    g_fail["raster"] = 1;
    CHECK(w.frame() == PC_ECUDA);
    cudaGraphLaunch(e, kStream);
    CHECK(g_frames == 3 && g_dirty == 0);
    cudaGraphExecDestroy(e);
}
static void failed_capture_replayed() {
    World w;
    CHECK(w.frame() == PC_OK);
    g_fail["raster"] = 1;
    cudaGraphExec_t e = captured_frame(w, PC_ECUDA);   // the caller replays it all the same
    cudaGraphLaunch(e, kStream);
    cudaGraphLaunch(e, kStream);
    CHECK(w.frame() == PC_OK);
    CHECK(g_frames == 4 && g_dirty == 0);
    cudaGraphExecDestroy(e);
}
static void failed_clearing_is_tried_again() {
    World w;
    CHECK(w.frame() == PC_OK);
    g_fail["raster"] = 1;
    g_fail["memset"] = 1;
    CHECK(w.frame() == PC_ECUDA);
    cudaGraphExec_t e = captured_frame(w);   // clears in the graph, which has not run
    CHECK(w.frame() == PC_OK);
    cudaGraphLaunch(e, kStream);
    CHECK(g_frames == 4 && g_dirty == 0);
    cudaGraphExecDestroy(e);
}
// The scratch of a new stream starts from zero, also when its clearing fails at first
// or is only recorded.
static void first_clearing_fails() {
    World w;
    g_fail["memset"] = 1;
    CHECK(w.frame() == PC_ECUDA);
    pc_view_stats st;
    CHECK(g_frames == 0 && pc_get_view_stats(w.ctx, kStream, 0, &st) == PC_ENOTFOUND);
    CHECK(w.frame() == PC_OK);
    CHECK(g_dirty == 0 && w.batches_rendered() == 7);
}
static void first_frame_captured() {
    World w;
    cudaGraphExec_t e = captured_frame(w);
    CHECK(w.frame() == PC_OK);
    CHECK(g_dirty == 0 && w.batches_rendered() == 7);
    cudaGraphLaunch(e, kStream);
    CHECK(g_frames == 2 && g_dirty == 0 && w.batches_rendered() == 7);
    cudaGraphExecDestroy(e);
}

// pc_upload_cloud where the encoder's scratch does not fit beside the cloud: the host
// encodes, with the same bits and no message left; where the cloud does not fit
// either, the call fails before any encoding.
static void upload_without_room() {
    const uint64_t n = 10000, cloud = 16 * n, scratch = 40 * n;
    World w(0, n);
    pc_cloud_info info;
    CHECK(pc_cloud_get_info(w.ctx, w.cloud, &info) == PC_OK);
    auto bytes = [&](pc_cloud c) {
        std::vector<pc_batch> b(info.n_batches);
        std::vector<uint32_t> words(4 * n);
        CHECK(pc_cloud_download(w.ctx, c, b.data(), &words[0], &words[n], &words[2 * n], &words[3 * n]) == PC_OK);
        std::string s((const char*)b.data(), b.size() * sizeof(pc_batch));
        return s + std::string((const char*)words.data(), words.size() * 4);
    };
    const std::string expect = bytes(w.cloud);
    const size_t used = g_used;
    // room for the scratch and the cloud, for either but not both, for the cloud alone
    for (size_t room : {scratch + 2 * cloud, scratch + cloud / 2, 2 * cloud}) {
        const int before = g_encoded;
        g_room = used + room;
        pc_cloud c = 0;
        CHECK(pc_upload_cloud(w.ctx, w.xyz.data(), nullptr, n, &c) == PC_OK);
        CHECK(g_encoded - before == (room == scratch + 2 * cloud));
        CHECK(bytes(c) == expect);
        CHECK(std::string(pc_last_error(w.ctx)).empty());
        CHECK(pc_release_cloud(w.ctx, c) == PC_OK);
        CHECK(g_used == used);
    }
    // room for a part of the cloud only: refused at once, all given back
    pc_cloud c = 0;
    g_room = used + cloud / 2;
    const uint64_t encoded = g_encoded;
    std::vector<float> bad(3 * n, 0.0f);
    bad[7] = INFINITY;   // the host encoder would say so
    CHECK(pc_upload_cloud(w.ctx, bad.data(), nullptr, n, &c) == PC_ENOMEM);
    CHECK(g_encoded == (int)encoded && g_used == used && c == 0);
    CHECK(std::string(pc_last_error(w.ctx)).find("cloud allocation") != std::string::npos);
    // what the device encoder refuses leaves nothing behind either
    g_room = ~(size_t)0;
    CHECK(pc_upload_cloud(w.ctx, bad.data(), nullptr, n, &c) == PC_EINVAL);
    CHECK(g_used == used && c == 0);
    // the empty cloud
    CHECK(pc_upload_cloud(w.ctx, nullptr, nullptr, 0, &c) == PC_OK);
    CHECK(pc_cloud_get_info(w.ctx, c, &info) == PC_OK && info.n_points == 0 && info.n_batches == 0);
}

// A few points kept in their order are the host's, more and sorted ones the device's.
static void few_points_are_encoded_on_the_host() {
    for (uint32_t flags : {0u, (uint32_t)PC_CFG_KEEP_ORDER})
        for (uint64_t n : {1, 1000, 1001}) {
            g_encoded = 0;
            World w(flags, n);
            CHECK(g_encoded == !(flags && n <= 1000));
            pc_cloud c = 0;
            w.xyz[0] = NAN;
            CHECK(pc_upload_cloud(w.ctx, w.xyz.data(), nullptr, n, &c) == PC_EINVAL && c == 0);
        }
}

// PC_CFG_GRAPHS: a program that alternates between launch layouts of one view count
// instantiates one graph for each and then only updates.
static void graphs_of_alternating_layouts() {
    World w(PC_CFG_GRAPHS);
    const std::vector<std::vector<uint32_t>> layouts = {
        {0u, 0u}, {0u, PC_VIEW_DILATE}, {PC_VIEW_DILATE, PC_VIEW_DILATE}, {PC_VIEW_HQS, 0u},
        {PC_VIEW_HQS_PACKED, 0u}, {PC_VIEW_HQS_PACKED, PC_VIEW_DILATE},
        {0u}, {PC_VIEW_FORCE_K(3)}, {PC_VIEW_NO_EARLY_DEPTH}, {PC_VIEW_FORCE_K(2) | PC_VIEW_DILATE}};
    for (const auto& l : layouts) CHECK(w.frame(l) == PC_OK);
    const int made = g_instantiated;
    CHECK(made <= (int)layouts.size());
    for (int i = 0; i < 3; ++i)
        for (const auto& l : layouts) CHECK(w.frame(l) == PC_OK);
    CHECK(g_instantiated == made && g_dirty == 0);
}

// Captured frames, a caller's and the library's own, have no frame number and run the
// two one-view kernels as two branches, or as one where a branch cannot be had.
static void captured_frames_branch() {
    {
        World w;
        CHECK(w.frame() == PC_OK && g_branches == 0);
        g_fail["stream"] = 1;
        cudaGraphExecDestroy(captured_frame(w));
        CHECK(g_branches == 0);
        cudaGraphExecDestroy(captured_frame(w));
        CHECK(w.frame() == PC_OK && w.frame() == PC_OK);
        CHECK(g_branches == 1);
    }
    g_last_frame = 0;
    World w(PC_CFG_GRAPHS);
    for (int i = 0; i < 3; ++i) CHECK(w.frame() == PC_OK && g_branches == 2 + i);
    // views without a certified batch have nothing for the second branch
    for (uint32_t f : {(uint32_t)PC_VIEW_FORCE_K(3), (uint32_t)PC_VIEW_NO_EARLY_DEPTH}) CHECK(w.frame({f}) == PC_OK);
    CHECK(w.frame({0u, 0u}) == PC_OK && g_branches == 4);
    CHECK(g_misnumbered == 0 && g_instantiated == 5 && g_dirty == 0);
}

static const std::map<std::string, void (*)()>& scenarios() {
    static const std::map<std::string, void (*)()> all = {
        {"failed_frame", failed_frame},
        {"failed_frame_then_capture", failed_frame_then_capture},
        {"failed_frame_then_replay", failed_frame_then_replay},
        {"failed_capture_replayed", failed_capture_replayed},
        {"failed_clearing_is_tried_again", failed_clearing_is_tried_again},
        {"first_clearing_fails", first_clearing_fails},
        {"first_frame_captured", first_frame_captured},
        {"upload_without_room", upload_without_room},
        {"few_points_are_encoded_on_the_host", few_points_are_encoded_on_the_host},
        {"graphs_of_alternating_layouts", graphs_of_alternating_layouts},
        {"captured_frames_branch", captured_frames_branch},
    };
    return all;
}

int main(int argc, char** argv) {
    CHECK(argc == 2);
    auto it = scenarios().find(argv[1]);
    CHECK(it != scenarios().end());
    it->second();
    std::printf("%s ok\n", argv[1]);
    return 0;
}
