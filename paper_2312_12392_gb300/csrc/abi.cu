// abi.cu -- the C ABI of include/rcp.h: scenes, renders, tuning, diagnostics.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdlib>
#include <fstream>
#include <map>
#include <memory>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "scene.h"

namespace rcp {

// Whether kernels on the current device may read and write pageable host
// memory directly (a coherent CPU-GPU link with address translation through
// the host's page tables, as on Grace).
bool host_coherent() {
    static int cached[64];
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return false;
    std::call_once(once[dev], [dev] {
        int a = 0, b = 0;
        if (cudaDeviceGetAttribute(&a, cudaDevAttrPageableMemoryAccess, dev) != cudaSuccess) a = 0;
        if (cudaDeviceGetAttribute(&b, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev) != cudaSuccess) b = 0;
        cached[dev] = a && b;
    });
    return cached[dev] != 0;
}

// How frames reach host buffers (rcp_set_host_output). A page-locked buffer is
// mapped in the GPU's own page tables: the last pass writes it directly. A
// pageable buffer is reached through the GPU's translation of host addresses
// (where the device reads pageable memory coherently): for a buffer the GPU
// wrote recently the translations are cached and the writes overlap the last
// pass for free, but for a fresh one every page misses and the frame is much
// slower than a device image and a copy (measured: ~100 against ~450
// frames/s at 1080p). AUTO therefore writes a pageable buffer directly only if
// it is one of the last kHostLru buffers written directly (same address and
// size), and otherwise packs the image on the device and copies it; a buffer
// used again is written directly from its second use on.
namespace {
std::atomic<int> g_host_output{RCP_HOST_OUTPUT_AUTO};
std::mutex g_lru_mu;
constexpr int kHostLru = 8;
std::vector<std::pair<const void*, size_t>> g_lru;  // most recent first
}  // namespace

bool page_locked(const void* p) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();  // an unregistered pointer is not an error to keep
        return false;
    }
    return a.type == cudaMemoryTypeHost && a.devicePointer == p;
}

bool use_direct_output(const void* p, size_t bytes) {
    const int mode = g_host_output.load();
    if (mode == RCP_HOST_OUTPUT_COPY) return false;
    if (page_locked(p)) return true;  // in the GPU's page tables, at the same address
    if (!host_coherent()) return false;
    std::lock_guard<std::mutex> lk(g_lru_mu);
    auto it = std::find(g_lru.begin(), g_lru.end(), std::make_pair(p, bytes));
    const bool seen = it != g_lru.end();
    if (seen) g_lru.erase(it);
    g_lru.insert(g_lru.begin(), std::make_pair(p, bytes));
    if ((int)g_lru.size() > kHostLru) g_lru.pop_back();
    return mode == RCP_HOST_OUTPUT_DIRECT || seen;
}

// Read and write back one byte in every page of [p, p + bytes): the pages are
// mapped and writable before a kernel writes there.
void touch_pages(void* p, size_t bytes) {
    static const size_t page = [] {
        const long s = sysconf(_SC_PAGESIZE);
        return s > 0 ? (size_t)s : (size_t)4096;
    }();
    volatile unsigned char* c = (volatile unsigned char*)p;
    for (size_t i = 0; i < bytes; i += page) c[i] = c[i];
    if (bytes) c[bytes - 1] = c[bytes - 1];
}


namespace {
thread_local std::string g_error;
}

void set_error(const std::string& msg) { g_error = msg; }

rcp_status cuda_fail(cudaError_t e, const char* what) {
    set_error(std::string("CUDA error in ") + what + ": " + cudaGetErrorString(e));
    if (e == cudaErrorMemoryAllocation) return RCP_ERR_OOM;
    return RCP_ERR_CUDA;
}

RenderCtx::~RenderCtx() {
    if (work.done) cudaEventSynchronize(work.done);  // before anything its work still uses goes
    if (graph) cudaGraphExecDestroy(graph);
    if (img[0]) cudaFree(img[0]);
    if (rays) cudaFree(rays);
    if (block) cudaFree(block);
    if (h_views) cudaFreeHost(h_views);
    if (d_rgb) cudaFree(d_rgb);
    if (io) cudaFree(io);
    if (io_prim) cudaFree(io_prim);
    if (base_img) cudaFree(base_img);
    if (repeat) cudaFree(repeat);
    if (work.done) cudaEventDestroy(work.done);
    if (staged) cudaEventDestroy(staged);
    for (auto e : pass_ev)
        if (e) cudaEventDestroy(e);
}

Scene::~Scene() {
    ctx.clear();
    if (spill_work.done) cudaEventDestroy(spill_work.done);
    for (void* p : {(void*)d_store, d_nodes, (void*)d_prims, (void*)d_refbox, (void*)d_part_uv, (void*)d_rbox,
                    (void*)d_spill})
        if (p) cudaFree(p);
}

SceneDev Scene::dev() const {
    SceneDev s;
    s.nodes = (const float4*)d_nodes;
    s.prims = d_prims;
    s.albedo = d_albedo;
    s.n_prims = T + S;
    s.n_records = n_records;
    s.n_nodes = n_nodes;
    s.light = light;
    s.tmin = 1e-6f * diam;
    s.eps = 1e-4f * diam;
    return s;
}

int64_t Scene::device_bytes() const {
    const int64_t N = T + S;
    return T * 36 + S * 16 + N * 16 + n_nodes * ((int64_t)sizeof(WNode) + 32) + n_records * 48 +
           (d_refbox ? n_records * 32 : 0) + (d_part_uv ? n_records * (9 * 4 + 4) : 0) + (d_rbox ? n_records * 24 : 0);
}

void make_view(ViewDev& v, const rcp_camera& cam, int W, int H, const rcp_params& p) {
    double E[3], F[3], R[3], U[3];
    for (int a = 0; a < 3; ++a) {
        E[a] = cam.eye[a];
        F[a] = (double)cam.look_at[a] - cam.eye[a];
    }
    double l = sqrt(F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
    for (double& x : F) x /= l;
    const double up[3] = {cam.up[0], cam.up[1], cam.up[2]};
    R[0] = F[1] * up[2] - F[2] * up[1];
    R[1] = F[2] * up[0] - F[0] * up[2];
    R[2] = F[0] * up[1] - F[1] * up[0];
    l = sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
    for (double& x : R) x /= l;
    U[0] = R[1] * F[2] - R[2] * F[1];
    U[1] = R[2] * F[0] - R[0] * F[2];
    U[2] = R[0] * F[1] - R[1] * F[0];
    const double tn = tan((double)cam.fov_y_deg * M_PI / 360.0);
    const double hx = tn * ((double)W / H) / W, hy = tn / H;
    const double f = p.focal_dist, k = p.k;
    for (int a = 0; a < 3; ++a) {
        v.E[a] = (float)E[a];
        v.fF[a] = (float)(f * F[a]);
        v.fR[a] = (float)(f * hx * R[a]);
        v.fU[a] = (float)(f * hy * U[a]);
        v.kR[a] = (float)(k * R[a]);
        v.kU[a] = (float)(k * U[a]);
        v.kF[a] = (float)(k * F[a]);
        v.Fw[a] = (float)F[a];
    }
    v.W = W;
    v.H = H;
    v.mapping = p.mapping;
    v.z0 = p.z0;
    v.kpx = (p.mapping == RCP_MAP_IMAGE || p.mapping == RCP_MAP_NORMAL) ? p.k : 0.f;
    v.passes = 1;
    v.base = nullptr;
    v.in = nullptr;
    v.out = nullptr;
    v.prim = nullptr;
    v.rgb = nullptr;
    v.hint = nullptr;
    v.scene = nullptr;
    v.status = nullptr;
    v.repeat = MsRepeat{};
    v.done_count = nullptr;
    v.done_flag = nullptr;
    v.tiles_x = (W + 7) / 8;
    v.pix_begin = 0;
    v.chunk_begin = 0;
    v.spp = p.spp > 0 ? p.spp : 0;
    for (int i = 0; i < 2 * RCP_MAX_SPP; ++i) v.jit[i] = i < 2 * v.spp ? p.jitter[i] : 0.5f;
}

}  // namespace rcp

using namespace rcp;


namespace {

cudaStream_t lib_stream() {
    static cudaStream_t s = nullptr;
    static std::once_flag once;
    std::call_once(once, [] { cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking); });
    return s;
}

cudaStream_t capture_stream() {
    thread_local cudaStream_t s = nullptr;
    if (!s) cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    return s;
}

bool finite3(const float* v) { return std::isfinite(v[0]) && std::isfinite(v[1]) && std::isfinite(v[2]); }

rcp_status check_view(const rcp_camera* cam, int W, int H, const rcp_params* p) {
    if (!cam || !p) {
        set_error("camera or params is NULL");
        return RCP_ERR_ARG;
    }
    if (W < 1 || H < 1 || W > 8192 || H > 8192) {
        set_error("width and height must be in [1, 8192]");
        return RCP_ERR_ARG;
    }
    if (!(p->k >= 0.f) || !std::isfinite(p->k) || !(p->focal_dist > 0.f) || !std::isfinite(p->focal_dist) ||
        !std::isfinite(p->z0)) {
        set_error("k must be >= 0 and focal_dist > 0, all finite");
        return RCP_ERR_ARG;
    }
    if (p->mapping < RCP_MAP_EYE || p->mapping > RCP_MAP_NORMAL) {
        set_error("unknown mapping");
        return RCP_ERR_ARG;
    }
    if (p->spp > RCP_MAX_SPP || (p->spp > 0 && p->mapping == RCP_MAP_IMAGE)) {
        set_error("spp must be <= 16, and image-space renders take one sample per pixel");
        return RCP_ERR_ARG;
    }
    for (int i = 0; i < 2 * (p->spp > 0 ? p->spp : 0); ++i)
        if (!(p->jitter[i] >= 0.f && p->jitter[i] < 1.f)) {
            set_error("jitter offsets must lie in [0, 1)");
            return RCP_ERR_ARG;
        }
    if (!finite3(cam->eye) || !finite3(cam->look_at) || !finite3(cam->up) || !(cam->fov_y_deg > 0.f) ||
        !(cam->fov_y_deg < 180.f)) {
        set_error("camera must be finite with 0 < fov < 180");
        return RCP_ERR_ARG;
    }
    double F[3], up[3] = {cam->up[0], cam->up[1], cam->up[2]};
    for (int a = 0; a < 3; ++a) F[a] = (double)cam->look_at[a] - cam->eye[a];
    const double c0 = F[1] * up[2] - F[2] * up[1], c1 = F[2] * up[0] - F[0] * up[2], c2 = F[0] * up[1] - F[1] * up[0];
    if (F[0] == 0 && F[1] == 0 && F[2] == 0) {
        set_error("look_at equals eye");
        return RCP_ERR_ARG;
    }
    if (c0 == 0 && c1 == 0 && c2 == 0) {
        set_error("up is parallel to the view direction");
        return RCP_ERR_ARG;
    }
    return RCP_OK;
}

int device_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || sms <= 0)
        sms = 1;
    return sms;
}

// Stack entries a walk of this tree can need: one group per level, rounded up
// to a multiple of 4.
int full_stack(const Scene& sc) {
    const int st = std::max(sc.depth, 4);
    return std::min((st + 3) & ~3, MAX_STACK);
}

LaunchCfg cfg_of(const Scene& sc) {
    LaunchCfg c;
    c.block = sc.tuning.block;
    c.blocks_per_sm = sc.tuning.blocks_per_sm;
    c.chunk = sc.tuning.chunk >= 64 ? 64 : 32;
    c.fused = sc.tuning.fused_camera != 0;
    const int full = full_stack(sc);
    c.stack = sc.tuning.stack_entries > 0 ? std::min(sc.tuning.stack_entries, full) : full;
    c.spill_entries = full - c.stack;
    c.hints = sc.tuning.hints;
    c.chain = sc.tuning.chain_passes != 0;
    return c;
}

// One call's work on buffers that serve one frame at a time but that calls on
// several streams may share: a context's (descriptors, counters, images, hints;
// keyed by shape alone) and a scene's spill region. Before its first work the
// call's stream waits for the buffers' latest work, unless that is on the same
// stream. Streams are told apart by their ids, which, unlike handles, are never
// used again. Whatever the call enqueued, also one that failed part-way, is the
// buffers' latest work from then on.
class StreamUse {
  public:
    StreamUse() = default;
    StreamUse(const StreamUse&) = delete;
    StreamUse& operator=(const StreamUse&) = delete;
    ~StreamUse() {
        if (work_) cudaEventRecord(work_->done, st_);
    }
    rcp_status begin(LastWork& work, cudaStream_t st) {
        unsigned long long id = 0;
        RCP_CUDA(cudaStreamGetId(st, &id));
        if (id != work.stream_id) RCP_CUDA(cudaStreamWaitEvent(st, work.done, 0));
        work.stream_id = id;
        work_ = &work;
        st_ = st;
        return RCP_OK;
    }

  private:
    LastWork* work_ = nullptr;
    cudaStream_t st_ = nullptr;
};

// The global-memory region of a short shared stack: spill_entries per thread
// of the largest persistent grid a launch can have (the SMs' resident
// threads, or the tuned blocks per SM). Grown before any capture, never during
// one; the graph key names the region.
rcp_status ensure_spill(Scene& sc, LaunchCfg& c, cudaStream_t st, StreamUse& use) {
    if (c.spill_entries <= 0) return RCP_OK;
    const int64_t per_sm = std::max<int64_t>(2048, (int64_t)c.blocks_per_sm * c.block);
    const int64_t need = (int64_t)device_sms() * per_sm * c.spill_entries;
    if (sc.spill_cap < need) {
        if (sc.d_spill) {
            RCP_CUDA(cudaDeviceSynchronize());  // no launch may still use the old region
            cudaFree(sc.d_spill);
            sc.d_spill = nullptr;
            sc.spill_cap = 0;
            for (auto& kv : sc.ctx) {  // graphs captured with the old region
                if (kv.second->graph) cudaGraphExecDestroy(kv.second->graph);
                kv.second->graph = nullptr;
            }
        }
        RCP_CUDA(cudaMalloc((void**)&sc.d_spill, sizeof(uint2) * need));
        sc.spill_cap = need;
    }
    c.spill = sc.d_spill;
    c.spill_cap = sc.spill_cap;
    if (!sc.spill_work.done) RCP_CUDA(cudaEventCreateWithFlags(&sc.spill_work.done, cudaEventDisableTiming));
    return use.begin(sc.spill_work, st);
}

// Render contexts are cached per launch shape, least recently used first out
// when the cache exceeds CTX_MAX entries or CTX_BYTES of device memory. A
// context is freed only after its last launch has completed.
constexpr size_t CTX_MAX = 64;
constexpr int64_t CTX_BYTES = (int64_t)16 << 30;

// Drop contexts other than `keep` until `more` bytes fit, and for a new context
// (keep null) a further entry.
void make_room(Scene& sc, const RenderCtx* keep, int64_t more) {
    for (;;) {
        int64_t held = 0;
        auto victim = sc.ctx.end();
        for (auto it = sc.ctx.begin(); it != sc.ctx.end(); ++it) {
            held += it->second->bytes;
            if (it->second.get() != keep &&
                (victim == sc.ctx.end() || it->second->last_use < victim->second->last_use))
                victim = it;
        }
        if (victim == sc.ctx.end() || (sc.ctx.size() < CTX_MAX + (keep ? 1 : 0) && held + more <= CTX_BYTES)) return;
        if (sc.last == victim->second.get()) sc.last = nullptr;
        sc.ctx.erase(victim);  // the destructor waits for the context's last launch
    }
}

// n elements more for a context, counted against the cache's limit.
template <class T>
rcp_status ctx_alloc(Scene& sc, RenderCtx& ctx, T** p, int64_t n) {
    const int64_t bytes = (int64_t)sizeof(T) * n;
    make_room(sc, &ctx, bytes);
    RCP_CUDA(cudaMalloc((void**)p, bytes));
    ctx.bytes += bytes;
    return RCP_OK;
}

// The separate camera kernel's ray buffer (2 float4 per pixel), allocated
// before the first capture that needs it.
rcp_status ensure_rays(Scene& sc, RenderCtx& ctx, const LaunchCfg& c) {
    if (c.fused || c.ms || c.multi || ctx.rays) return RCP_OK;
    return ctx_alloc(sc, ctx, &ctx.rays, 2 * ctx.total_pix);
}

std::string cfg_key(const LaunchCfg& c) {
    std::ostringstream o;
    o << c.block << "/" << c.blocks_per_sm << "/" << c.chunk << "/" << c.fused << "/" << c.stack << "/"
      << c.spill_entries << "/" << (const void*)c.spill << "/" << c.count << "/" << c.ms << "/" << c.hints
      << "/" << c.chain;
    return o.str();
}

// Lay views out for one pass: global pixel and tile offsets.
void layout_views(std::vector<ViewDev>& v, int64_t& total_pix, int64_t& total_chunks) {
    total_pix = 0;
    total_chunks = 0;
    for (auto& x : v) {
        x.pix_begin = total_pix;
        x.chunk_begin = total_chunks;
        x.tiles_x = (x.W + 7) / 8;
        total_pix += (int64_t)x.W * x.H;
        total_chunks += (int64_t)x.tiles_x * ((x.H + 3) / 4);
    }
}

// A new context's counters and hints are cleared on `st`, the stream of the
// frame that it is made for.
rcp_status get_ctx(Scene& sc, int n_views, int K, int64_t total_pix, int64_t total_chunks, cudaStream_t st,
                   RenderCtx** out) {
    std::ostringstream key;
    key << n_views << ":" << K << ":" << total_pix << ":" << total_chunks;
    auto it = sc.ctx.find(key.str());
    if (it != sc.ctx.end()) {
        it->second->last_use = ++sc.use_clock;
        *out = it->second.get();
        return RCP_OK;
    }
    const int64_t need = total_pix * (int64_t)sizeof(int2) + (int64_t)sizeof(ViewDev) * K * n_views;
    make_room(sc, nullptr, need);
    auto c = std::make_unique<RenderCtx>();
    c->n_views = n_views;
    c->K = K;
    c->total_pix = total_pix;
    c->total_chunks = total_chunks;
    c->bytes = need;
    c->last_use = ++sc.use_clock;
    // one allocation: counters and status, view descriptors, hints
    const size_t head = 256, views = (sizeof(ViewDev) * (size_t)K * n_views + 255) & ~(size_t)255;
    RCP_CUDA(cudaMalloc((void**)&c->block, head + views + sizeof(int2) * total_pix));
    c->d_rays = (unsigned long long*)c->block;
    c->d_work = (unsigned*)(c->d_rays + 2);  // K + 1 <= 17 counters
    c->d_status = (int*)(c->block + head) - 4;
    c->d_views = (ViewDev*)(c->block + head);
    c->hints = (int2*)(c->block + head + views);
    c->views.resize((size_t)K * n_views);
    RCP_CUDA(cudaEventCreateWithFlags(&c->staged, cudaEventDisableTiming));
    RCP_CUDA(cudaEventCreateWithFlags(&c->work.done, cudaEventDisableTiming));
    for (int n = 0; n <= K; ++n) RCP_CUDA(cudaEventCreate(&c->pass_ev[n]));
    RCP_CUDA(cudaStreamGetId(st, &c->work.stream_id));
    RCP_CUDA(cudaMemsetAsync(c->block, 0, head, st));
    RCP_CUDA(cudaMemsetAsync(c->hints, 0xff, sizeof(int2) * total_pix, st));  // -1: no earlier hit
    RCP_CUDA(cudaEventRecord(c->work.done, st));
    *out = c.get();
    sc.ctx[key.str()] = std::move(c);
    return RCP_OK;
}

// Enqueue the K passes of ctx (views already staged in ctx->d_views).
rcp_status enqueue_passes(const Scene& sc, RenderCtx& ctx, const LaunchCfg& cfg, unsigned long long* counters,
                          cudaStream_t st, bool capturing) {
    // inside a capture an event record only becomes a graph node with the
    // external flag; outside a capture the plain record is the valid call
    auto record = [&](cudaEvent_t e) {
        return capturing ? cudaEventRecordWithFlags(e, st, cudaEventRecordExternal) : cudaEventRecord(e, st);
    };
    const SceneDev S = sc.dev();
    LaunchCfg first = cfg;
    if (ctx.direct) {
        RCP_CUDA(record(ctx.pass_ev[0]));
        rcp_status r = launch_stage_views(ctx.views.data(), ctx.n_desc, ctx.d_views, (unsigned*)ctx.d_rays, 4 + ctx.K + 1, st);
        if (r != RCP_OK) return r;
        first.behind_stage = true;
    } else {
        RCP_CUDA(cudaMemsetAsync(ctx.d_rays, 0, sizeof(unsigned long long) * 2 + sizeof(unsigned) * (ctx.K + 1), st));
        RCP_CUDA(record(ctx.pass_ev[0]));
    }
    if (ctx.chained) {  // one descriptor per view, all K passes (image mode: pass 1, then the gathers' descriptors)
        rcp_status r = ctx.image_mode
                           ? launch_pass(S, first, ctx.d_views, ctx.n_views, ctx.total_pix, ctx.total_chunks, nullptr,
                                         ctx.d_work, ctx.d_rays, counters, st)
                           : launch_chain(S, first, ctx.d_views, ctx.n_views, ctx.total_chunks, ctx.d_work, ctx.d_rays,
                                          counters, st);
        if (r != RCP_OK) return r;
        RCP_CUDA(record(ctx.pass_ev[1]));
        if (ctx.image_mode) {
            r = launch_imagespace_chain(ctx.d_views + ctx.n_views, ctx.n_views, ctx.total_chunks, st);
            if (r != RCP_OK) return r;
            RCP_CUDA(record(ctx.pass_ev[2]));
        }
        return RCP_OK;
    }
    for (int n = 0; n < ctx.K; ++n) {
        rcp_status r = (ctx.image_mode && n > 0)
                           ? launch_imagespace(ctx.d_views + (size_t)n * ctx.n_views, ctx.n_views, ctx.total_pix, st)
                           : launch_pass(S, n == 0 ? first : cfg, ctx.d_views + (size_t)n * ctx.n_views, ctx.n_views, ctx.total_pix,
                                         ctx.total_chunks, ctx.rays, ctx.d_work + n, ctx.d_rays, counters, st);
        if (r != RCP_OK) return r;
        RCP_CUDA(record(ctx.pass_ev[n + 1]));
    }
    return RCP_OK;
}

// Enqueue a frame. One of few descriptors and launches (ctx.direct) goes
// straight onto the stream: k_stage_views and the launch or two behind it take
// less of the device's time between kernels than a copy and a graph (a 128x128
// K = 6 frame of five primitives 45.9 -> 34.5 us, 32 us of it one warp's
// chain of twelve rays). Others run through the context's CUDA graph, captured when a launch
// configuration comes a second time: the first time its launches are enqueued
// directly, since capturing and instantiating a graph takes longer than the
// few launches of a frame that may be the only one of its shape.
rcp_status run_frame(const Scene& sc, RenderCtx& ctx, const LaunchCfg& cfg, cudaStream_t st) {
    if (ctx.direct) return enqueue_passes(sc, ctx, cfg, nullptr, st, false);
    const std::string key = cfg_key(cfg) + (ctx.image_mode ? "/image" : "/trace") + (ctx.chained ? "/chain" : "");
    if (!ctx.graph || ctx.graph_key != key) {
        if (ctx.seen_key != key) {
            ctx.seen_key = key;
            return enqueue_passes(sc, ctx, cfg, nullptr, st, false);
        }
        if (ctx.graph) {
            cudaGraphExecDestroy(ctx.graph);
            ctx.graph = nullptr;
        }
        cudaStream_t cs = capture_stream();
        RCP_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        rcp_status r = enqueue_passes(sc, ctx, cfg, nullptr, cs, true);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(cs, &g);
        if (r != RCP_OK) {
            if (g) cudaGraphDestroy(g);
            return r;
        }
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
        e = cudaGraphInstantiate(&ctx.graph, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
        ctx.graph_key = key;
    }
    RCP_CUDA(cudaGraphLaunch(ctx.graph, st));
    return RCP_OK;
}

// The context's ping-pong images: renders of several launches, and inputs and
// outputs that the caller leaves to the library. A chained render has none.
rcp_status ensure_img(Scene& sc, RenderCtx& ctx) {
    if (ctx.img[0]) return RCP_OK;
    rcp_status r = ctx_alloc(sc, ctx, &ctx.img[0], 2 * ctx.total_pix);
    if (r == RCP_OK) ctx.img[1] = ctx.img[0] + ctx.total_pix;
    return r;
}

// The state of a multi-sample render that leaves out repeated tiles: two
// passes' tile flags and shadow counts and (ids) hit ids. One allocation.
struct RepeatLayout {
    size_t shadow, ids, total;  // the flags come first
};
RepeatLayout repeat_layout(const RenderCtx& ctx, bool ids) {
    const auto pad = [](size_t b) { return (b + 255) & ~(size_t)255; };
    RepeatLayout l;
    l.shadow = pad(2 * (size_t)ctx.total_chunks);
    l.ids = l.shadow + pad(sizeof(unsigned) * 2 * (size_t)ctx.total_chunks);
    l.total = l.ids + (ids ? pad(sizeof(int32_t) * 2 * (size_t)ctx.total_pix) : 0);
    return l;
}

rcp_status ensure_repeat(Scene& sc, RenderCtx& ctx, bool ids) {
    if (ctx.repeat && (ctx.repeat_ids || !ids)) return RCP_OK;
    if (ctx.repeat) {
        RCP_CUDA(cudaEventSynchronize(ctx.work.done));  // no launch may still use the smaller one
        cudaFree(ctx.repeat);
        ctx.bytes -= (int64_t)repeat_layout(ctx, ctx.repeat_ids).total;
        ctx.repeat = nullptr;
    }
    ctx.repeat_ids = ids;
    return ctx_alloc(sc, ctx, &ctx.repeat, (int64_t)repeat_layout(ctx, ids).total);
}

// The staged descriptors to the device (a direct frame's go with its launch).
rcp_status upload_views(RenderCtx& ctx, cudaStream_t st) {
    if (ctx.direct) return RCP_OK;
    if (!ctx.h_views) RCP_CUDA(cudaMallocHost((void**)&ctx.h_views, sizeof(ViewDev) * ctx.views.size()));
    RCP_CUDA(cudaEventSynchronize(ctx.staged));  // the previous copy out of the staging buffer is done
    std::copy(ctx.views.begin(), ctx.views.begin() + ctx.n_desc, ctx.h_views);
    RCP_CUDA(cudaMemcpyAsync(ctx.d_views, ctx.h_views, sizeof(ViewDev) * (size_t)ctx.n_desc, cudaMemcpyHostToDevice,
                             st));
    RCP_CUDA(cudaEventRecord(ctx.staged, st));
    return RCP_OK;
}

// Stage the view descriptors of one render (n_views views, K passes): one per
// view and pass, or, when the passes run chained (chain: the tuning asks for
// it and the render allows it), one per view that runs all K passes (an
// image-space render: one per view that traces pass 1, then one per view that
// gathers passes 2..K).
rcp_status stage_views(Scene& sc, RenderCtx& ctx, const std::vector<ViewDev>& base, const float4* const* ins,
                       float4* const* outs, int32_t* const* prims, float* const* rgbs, cudaStream_t st,
                       bool chain = false, bool allow_direct = false) {
    const int K = ctx.K, nv = ctx.n_views;
    ctx.image_mode = base[0].mapping == RCP_MAP_IMAGE && K > 1;
    // a single traced pass takes the one-pass kernel, which keeps no state
    // between passes (90 registers, nothing spilled in the walk): mid 1080p
    // K = 1 0.335 against 0.316 ms chained
    ctx.chained = chain && base[0].spp == 0 && K > 1;
    ctx.launches = ctx.chained ? (ctx.image_mode ? 2 : 1) : K;
    ctx.n_desc = ctx.chained ? nv * (ctx.image_mode ? 2 : 1) : nv * K;
    ctx.direct = allow_direct && (ctx.chained || K == 1) && ctx.n_desc <= STAGE_VIEWS;
    if (ctx.image_mode && !ctx.base_img) {
        rcp_status r = ctx_alloc(sc, ctx, &ctx.base_img, ctx.total_pix);
        if (r != RCP_OK) return r;
    }
    if (ctx.chained) {
        for (int i = 0; i < nv; ++i) {
            ViewDev v = base[i];
            v.in = ins ? ins[i] : nullptr;
            v.out = outs[i];
            v.hint = ctx.hints + base[i].pix_begin;
            v.status = ctx.d_status;
            v.prim = prims ? prims[i] : nullptr;
            v.rgb = rgbs ? rgbs[i] : nullptr;
            v.passes = K;
            if (ctx.image_mode) {
                ViewDev& w = ctx.views[nv + i];
                w = v;
                w.base = ctx.base_img + base[i].pix_begin;
                w.passes = K - 1;
                v.out = ctx.base_img + base[i].pix_begin;
                v.prim = nullptr;
                v.rgb = nullptr;
                v.passes = 1;
            }
            ctx.views[i] = v;
        }
        return upload_views(ctx, st);
    }
    if (K > 1) {
        rcp_status r = ensure_img(sc, ctx);
        if (r != RCP_OK) return r;
    }
    bool want_ids = false;
    for (int i = 0; prims && i < nv; ++i) want_ids = want_ids || prims[i];
    const bool repeats = base[0].spp > 0 && K > 2;
    RepeatLayout lay{};
    if (repeats) {
        rcp_status r = ensure_repeat(sc, ctx, want_ids);
        if (r != RCP_OK) return r;
        lay = repeat_layout(ctx, ctx.repeat_ids);
    }
    for (int n = 0; n < K; ++n) {
        for (int i = 0; i < nv; ++i) {
            ViewDev v = base[i];
            const int64_t off = base[i].pix_begin;
            float4* cur = (n == K - 1) ? outs[i] : ctx.img[n & 1] + off;
            const float4* prev = (n == 0) ? (ins ? ins[i] : nullptr) : ctx.img[(n - 1) & 1] + off;
            if (ctx.image_mode) {
                // pass 1 is traced into base_img; pass n >= 2 gathers from it
                if (n == 0) cur = ctx.base_img + off;
                if (n == 1) prev = ctx.base_img + off;
                v.base = ctx.base_img + off;
            }
            v.in = prev;
            v.out = cur;
            v.hint = ctx.hints + off;  // read and rewritten by each traced pass, per pixel
            v.status = ctx.d_status;
            v.prim = (n == K - 1 && prims && !ctx.image_mode) ? prims[i] : nullptr;
            v.rgb = (n == K - 1 && rgbs && !ctx.image_mode) ? rgbs[i] : nullptr;
            if (repeats) {  // pass n + 1 writes its flags, counts and ids at parity n & 1
                const int64_t tile = base[i].chunk_begin;
                uint8_t* flags = (uint8_t*)ctx.repeat + tile;
                unsigned* shadow = (unsigned*)(ctx.repeat + lay.shadow) + tile;
                int32_t* ids = want_ids && prims[i] ? (int32_t*)(ctx.repeat + lay.ids) + off : nullptr;
                const int64_t odd = n & 1, even = odd ^ 1;
                MsRepeat& m = v.repeat;
                m.flags_in = n > 0 ? flags + even * ctx.total_chunks : nullptr;
                m.flags_out = flags + odd * ctx.total_chunks;
                m.two_ago = n > 1 ? ctx.img[odd] + off : nullptr;
                m.has_two_ago = n > 1 && n < K - 1;
                m.ids_two_ago = ids ? ids + odd * ctx.total_pix : nullptr;
                m.ids_before = ids ? ids + even * ctx.total_pix : nullptr;
                m.shadow_before = shadow + even * ctx.total_chunks;
                m.shadow = shadow + odd * ctx.total_chunks;
                if (ids && n < K - 1) v.prim = ids + odd * ctx.total_pix;
            }
            ctx.views[(size_t)n * nv + i] = v;
        }
    }
    return upload_views(ctx, st);
}

rcp_status render_views(Scene& sc, int n_views, const rcp_camera* cams, const int* Ws, const int* Hs, int K,
                        const rcp_params* p, const float4* const* ins, float4* const* outs, int32_t* const* prims,
                        cudaStream_t st, RenderCtx** ctx_out = nullptr, const LaunchCfg* cfg_override = nullptr,
                        float* const* rgbs = nullptr) {
    if (K < 1 || K > 16) {
        set_error("K must be in [1, 16]");
        return RCP_ERR_ARG;
    }
    if (n_views < 1) {
        set_error("n_views must be >= 1");
        return RCP_ERR_ARG;
    }
    std::vector<ViewDev> base(n_views);
    for (int i = 0; i < n_views; ++i) {
        rcp_status r = check_view(&cams[i], Ws[i], Hs[i], p);
        if (r != RCP_OK) return r;
        if (!outs[i]) {
            set_error("output image is NULL");
            return RCP_ERR_ARG;
        }
        make_view(base[i], cams[i], Ws[i], Hs[i], *p);
        if (p->spp > 0 && K == 1 && ins && ins[i] == outs[i]) {
            set_error("a one-pass multi-sample render reads neighbouring pixels of d_in: d_out must not alias it");
            return RCP_ERR_ARG;
        }
        if (p->mapping == RCP_MAP_IMAGE && ins && ins[i]) {
            set_error("RCP_MAP_IMAGE renders start from I_0 (d_in must be NULL); use rcp_imagespace_pass_device");
            return RCP_ERR_ARG;
        }
    }
    if (sc.depth > MAX_STACK) {
        set_error("BVH deeper than the traversal stack");
        return RCP_ERR_STACK;
    }
    // A render orders itself against other streams and stages its descriptors on
    // the host, once per call, so it cannot become part of the caller's graph.
    // Refused before anything that would invalidate the caller's capture.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    RCP_CUDA(cudaStreamIsCapturing(st, &capture));
    if (capture != cudaStreamCaptureStatusNone) {
        set_error("renders cannot be captured: the stream is being captured");
        return RCP_ERR_CUDA;
    }
    int64_t total_pix, total_chunks;
    layout_views(base, total_pix, total_chunks);
    RenderCtx* ctx = nullptr;
    rcp_status r = get_ctx(sc, n_views, K, total_pix, total_chunks, st, &ctx);
    if (r != RCP_OK) return r;
    LaunchCfg cfg = cfg_override ? *cfg_override : cfg_of(sc);
    cfg.ms = p->spp > 0;
    StreamUse use, spill_use;
    r = use.begin(ctx->work, st);
    if (r != RCP_OK) return r;
    r = stage_views(sc, *ctx, base, ins, outs, prims, rgbs, st, cfg.chain, true);
    if (r != RCP_OK) return r;
    if (ctx->chained) cfg.fused = true;  // a chained launch makes its rays itself
    r = ensure_spill(sc, cfg, st, spill_use);
    if (r != RCP_OK) return r;
    r = ensure_rays(sc, *ctx, cfg);
    if (r != RCP_OK) return r;
    r = run_frame(sc, *ctx, cfg, st);
    sc.last = ctx;
    if (ctx_out) *ctx_out = ctx;
    return r;
}

rcp_status check_status(RenderCtx& ctx, cudaStream_t st) {
    int h = 0;
    RCP_CUDA(cudaMemcpyAsync(&h, ctx.d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h) {
        RCP_CUDA(cudaMemsetAsync(ctx.d_status, 0, sizeof(int), st));
        set_error("traversal stack overflow");
        return RCP_ERR_STACK;
    }
    return RCP_OK;
}

}  // namespace

extern "C" {

const char* rcp_last_error(void) { return g_error.c_str(); }

rcp_status rcp_set_host_output(int mode) {
    if (mode != RCP_HOST_OUTPUT_AUTO && mode != RCP_HOST_OUTPUT_DIRECT && mode != RCP_HOST_OUTPUT_COPY) {
        set_error("rcp_set_host_output: unknown mode");
        return RCP_ERR_ARG;
    }
    g_host_output.store(mode);
    return RCP_OK;
}

int rcp_get_host_output(void) { return g_host_output.load(); }
const char* rcp_version(void) { return "rcp-gb300 0.1 (sm_103a)"; }

rcp_status rcp_scene_create(const float* tri, int64_t T, const float* sph, int64_t S, const float* albedo,
                            const rcp_light* light, rcp_scene** out) {
    return rcp_scene_create_ex(tri, T, sph, S, albedo, light, nullptr, out);
}

rcp_status rcp_scene_create_ex(const float* tri, int64_t T, const float* sph, int64_t S, const float* albedo,
                               const rcp_light* light, const rcp_build_options* options, rcp_scene** out) {
    if (options && options->collapse != RCP_COLLAPSE_AREA && options->collapse != RCP_COLLAPSE_SAH) {
        set_error("rcp_scene_create_ex: unknown collapse policy");
        return RCP_ERR_ARG;
    }
    if (options && (options->split_max < 0 || options->split_max > RCP_SPLIT_MAX)) {
        set_error("rcp_scene_create_ex: split_max outside [0, 8]");
        return RCP_ERR_ARG;
    }
    if (!out || !light || T < 0 || S < 0 || (T > 0 && !tri) || (S > 0 && !sph) || (T + S > 0 && !albedo)) {
        set_error("rcp_scene_create: NULL array with a nonzero count, or negative count");
        return RCP_ERR_ARG;
    }
    if (T + S >= (int64_t)1 << 30) {
        set_error("rcp_scene_create: at most 2^30 - 1 primitives");
        return RCP_ERR_ARG;
    }
    if (light->type != RCP_LIGHT_POINT && light->type != RCP_LIGHT_DIRECTIONAL) {
        set_error("rcp_scene_create: unknown light type");
        return RCP_ERR_ARG;
    }
    *out = nullptr;
    auto sc = std::make_unique<rcp_scene>();
    sc->collapse = options ? options->collapse : RCP_COLLAPSE_AREA;
    sc->split_max = options && options->split_max > 1 ? options->split_max : 1;
    sc->T = T;
    sc->S = S;
    const int64_t N = T + S;
    cudaStream_t st = lib_stream();
    // one allocation, each part on a 256-byte boundary
    const auto pad = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t tri_b = pad(sizeof(float) * 9 * T), sph_b = pad(sizeof(float) * 4 * S), alb_b = pad(sizeof(float4) * N);
    RCP_CUDA(cudaMalloc((void**)&sc->d_store, tri_b + sph_b + alb_b + sizeof(SceneDev)));
    sc->d_tri = (float*)sc->d_store;
    sc->d_sph = (float*)(sc->d_store + tri_b);
    sc->d_albedo = (float4*)(sc->d_store + tri_b + sph_b);
    sc->d_dev = (SceneDev*)(sc->d_store + tri_b + sph_b + alb_b);
    if (T) RCP_CUDA(cudaMemcpyAsync(sc->d_tri, tri, sizeof(float) * 9 * T, cudaMemcpyHostToDevice, st));
    if (S) RCP_CUDA(cudaMemcpyAsync(sc->d_sph, sph, sizeof(float) * 4 * S, cudaMemcpyHostToDevice, st));
    // finite coordinates are checked, and the albedo widened to a float4 per
    // primitive, on the device: one host thread took 4.4 ms over a million
    // triangles for the two, these kernels and the 12 MB upload 0.2 ms
    bool bad_tri = false, bad_sph = false;
    rcp_status r = ingest_scene(*sc, albedo, &bad_tri, &bad_sph, st);
    if (r != RCP_OK) return r;
    if (bad_tri || bad_sph) {
        set_error(bad_tri ? "rcp_scene_create: non-finite vertex" : "rcp_scene_create: non-finite sphere");
        return RCP_ERR_ARG;
    }
    double lv[3] = {light->v[0], light->v[1], light->v[2]};
    if (light->type == RCP_LIGHT_DIRECTIONAL) {
        const double l = sqrt(lv[0] * lv[0] + lv[1] * lv[1] + lv[2] * lv[2]);
        if (!(l > 0) || !std::isfinite(l)) {
            set_error("rcp_scene_create: zero light direction");
            return RCP_ERR_ARG;
        }
        for (double& x : lv) x /= l;
    }
    sc->light.type = light->type;
    sc->light.x = (float)lv[0];
    sc->light.y = (float)lv[1];
    sc->light.z = (float)lv[2];
    sc->light.ambient = light->ambient;
    r = build_bvh(*sc, st);
    if (r != RCP_OK) return r;
    // the traversal reads child and record indices without range checks: a
    // tree is only handed out once every index in it is known to be in range
    r = validate_bvh(*sc, st);
    if (r != RCP_OK) return r;
    const SceneDev dv = sc->dev();
    // complete before any stream can read it
    RCP_CUDA(cudaMemcpyAsync(sc->d_dev, &dv, sizeof(SceneDev), cudaMemcpyHostToDevice, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    *out = sc.release();
    return RCP_OK;
}

rcp_status rcp_scene_update_vertices_device(rcp_scene* sc, const float* d_tri, void* stream) {
    if (!sc || (!d_tri && sc->T > 0)) {
        set_error("rcp_scene_update_vertices: NULL argument");
        return RCP_ERR_ARG;
    }
    std::lock_guard<std::mutex> lk(sc->mu);
    cudaStream_t st = (cudaStream_t)stream;
    if (sc->T) RCP_CUDA(cudaMemcpyAsync(sc->d_tri, d_tri, sizeof(float) * 9 * sc->T, cudaMemcpyDeviceToDevice, st));
    return refit_bvh(*sc, st);
}

rcp_status rcp_scene_update_vertices(rcp_scene* sc, const float* tri) {
    if (!sc || (!tri && sc->T > 0)) {
        set_error("rcp_scene_update_vertices: NULL argument");
        return RCP_ERR_ARG;
    }
    for (int64_t i = 0; i < sc->T * 9; ++i)
        if (!std::isfinite(tri[i])) {
            set_error("rcp_scene_update_vertices: non-finite vertex");
            return RCP_ERR_ARG;
        }
    std::lock_guard<std::mutex> lk(sc->mu);
    cudaStream_t st = lib_stream();
    if (sc->T) RCP_CUDA(cudaMemcpyAsync(sc->d_tri, tri, sizeof(float) * 9 * sc->T, cudaMemcpyHostToDevice, st));
    rcp_status r = refit_bvh(*sc, st);
    if (r != RCP_OK) return r;
    RCP_CUDA(cudaStreamSynchronize(st));
    return RCP_OK;
}

rcp_status rcp_scene_get_info(const rcp_scene* sc, rcp_scene_info* info) {
    if (!sc || !info) {
        set_error("rcp_scene_get_info: NULL argument");
        return RCP_ERR_ARG;
    }
    info->n_tris = sc->T;
    info->n_spheres = sc->S;
    info->n_nodes = sc->n_nodes;
    info->depth = sc->depth;
    info->max_leaf = sc->max_leaf;
    info->device_bytes = sc->device_bytes();
    info->diam = sc->diam;
    info->build_ms = sc->build_ms;
    info->collapse = sc->collapse;
    info->split_max = sc->split_max;
    info->n_records = sc->n_records;
    return RCP_OK;
}

rcp_status rcp_scene_validate(const rcp_scene* sc) {
    if (!sc) {
        set_error("rcp_scene_validate: NULL scene");
        return RCP_ERR_ARG;
    }
    return validate_bvh(*sc, lib_stream());
}

void rcp_scene_destroy(rcp_scene* sc) {
    if (!sc) return;
    cudaStreamSynchronize(lib_stream());
    delete sc;
}

rcp_status rcp_render_device(const rcp_scene* csc, const rcp_camera* cam, int W, int H, int K, const rcp_params* p,
                             const float* d_in, float* d_out, int32_t* d_prim, void* stream) {
    if (!csc) {
        set_error("rcp_render_device: NULL scene");
        return RCP_ERR_ARG;
    }
    rcp_scene* sc = const_cast<rcp_scene*>(csc);
    std::lock_guard<std::mutex> lk(sc->mu);
    const float4* ins[1] = {(const float4*)d_in};
    float4* outs[1] = {(float4*)d_out};
    int32_t* prims[1] = {d_prim};
    return render_views(*sc, 1, cam, &W, &H, K, p, ins, outs, prims, (cudaStream_t)stream);
}

rcp_status rcp_render_batch_device(const rcp_scene* csc, int n_views, const rcp_camera* cams, const int* Ws,
                                   const int* Hs, int K, const rcp_params* p, const float* const* d_ins,
                                   float* const* d_outs, int32_t* const* d_prims, void* stream) {
    if (!csc || !cams || !Ws || !Hs || !d_outs || n_views < 1) {
        set_error("rcp_render_batch_device: NULL argument or no views");
        return RCP_ERR_ARG;
    }
    rcp_scene* sc = const_cast<rcp_scene*>(csc);
    std::lock_guard<std::mutex> lk(sc->mu);
    return render_views(*sc, n_views, cams, Ws, Hs, K, p, (const float4* const*)d_ins, (float4* const*)d_outs,
                        d_prims, (cudaStream_t)stream);
}

static rcp_status ensure_io(Scene& sc, RenderCtx& ctx, bool rgb, bool prim) {
    const int64_t P = ctx.total_pix;
    rcp_status r = RCP_OK;
    if (!ctx.io) r = ctx_alloc(sc, ctx, &ctx.io, P);
    if (r == RCP_OK && rgb && !ctx.d_rgb) r = ctx_alloc(sc, ctx, &ctx.d_rgb, 3 * P);
    if (r == RCP_OK && prim && !ctx.io_prim) r = ctx_alloc(sc, ctx, &ctx.io_prim, P);
    return r;
}

rcp_status rcp_render(const rcp_scene* csc, const rcp_camera* cam, int W, int H, int K, const rcp_params* p,
                      float* out_rgb) {
    if (!csc || !out_rgb) {
        set_error("rcp_render: NULL argument");
        return RCP_ERR_ARG;
    }
    rcp_scene* sc = const_cast<rcp_scene*>(csc);
    std::lock_guard<std::mutex> lk(sc->mu);
    rcp_status r = check_view(cam, W, H, p);
    if (r != RCP_OK) return r;
    if (K < 1 || K > 16) {
        set_error("K must be in [1, 16]");
        return RCP_ERR_ARG;
    }
    cudaStream_t st = lib_stream();
    const int64_t P = (int64_t)W * H;
    RenderCtx* ctx = nullptr;
    r = get_ctx(*sc, 1, K, P, (int64_t)((W + 7) / 8) * ((H + 3) / 4), st, &ctx);
    if (r != RCP_OK) return r;
    const bool direct = p->mapping != RCP_MAP_IMAGE && use_direct_output(out_rgb, sizeof(float) * 3 * P);
    r = ensure_io(*sc, *ctx, !direct, false);
    if (r != RCP_OK) return r;
    const float4* ins[1] = {nullptr};
    float4* outs[1] = {ctx->io};
    if (direct) {
        // The last pass writes the caller's RGB straight into host memory over
        // the chip-to-chip link, while it traces: no pack kernel and no copy
        // after the frame. Each page is touched here first, so that the device
        // never meets an unmapped page (and a bad pointer faults on the host).
        touch_pages(out_rgb, sizeof(float) * 3 * P);
        float* rgbs[1] = {out_rgb};
        r = render_views(*sc, 1, cam, &W, &H, K, p, ins, outs, nullptr, st, nullptr, nullptr, rgbs);
        if (r != RCP_OK) {
            cudaStreamSynchronize(st);  // no pass may still write the caller's buffer after we return
            return r;
        }
        return check_status(*ctx, st);
    }
    r = render_views(*sc, 1, cam, &W, &H, K, p, ins, outs, nullptr, st);
    if (r != RCP_OK) return r;
    r = launch_pack_rgb(ctx->io, ctx->d_rgb, P, st);
    if (r != RCP_OK) return r;
    RCP_CUDA(cudaMemcpyAsync(out_rgb, ctx->d_rgb, sizeof(float) * 3 * P, cudaMemcpyDeviceToHost, st));
    return check_status(*ctx, st);
}

rcp_status rcp_render_pass(const rcp_scene* csc, const rcp_camera* cam, int W, int H, const rcp_params* p,
                           const float* in_rgbz, float* out_rgbz, int32_t* out_prim) {
    if (!csc || !out_rgbz) {
        set_error("rcp_render_pass: NULL argument");
        return RCP_ERR_ARG;
    }
    rcp_scene* sc = const_cast<rcp_scene*>(csc);
    std::lock_guard<std::mutex> lk(sc->mu);
    rcp_status r = check_view(cam, W, H, p);
    if (r != RCP_OK) return r;
    if (p->mapping == RCP_MAP_IMAGE) {
        set_error("rcp_render_pass: an image-space pass needs the frame's traced image; use "
                  "rcp_imagespace_pass_device");
        return RCP_ERR_ARG;
    }
    cudaStream_t st = lib_stream();
    const int64_t P = (int64_t)W * H;
    RenderCtx* ctx = nullptr;
    r = get_ctx(*sc, 1, 1, P, (int64_t)((W + 7) / 8) * ((H + 3) / 4), st, &ctx);
    if (r != RCP_OK) return r;
    r = ensure_io(*sc, *ctx, false, out_prim != nullptr);
    if (r != RCP_OK) return r;
    // I_{n-1} goes to ctx->img[1] (unused by a one-pass render) and I_n to
    // ctx->io: separate buffers, since jittered samples read neighbouring pixels
    if (in_rgbz) {
        r = ensure_img(*sc, *ctx);
        if (r != RCP_OK) return r;
    }
    if (in_rgbz) RCP_CUDA(cudaMemcpyAsync(ctx->img[1], in_rgbz, sizeof(float4) * P, cudaMemcpyHostToDevice, st));
    const float4* ins[1] = {in_rgbz ? ctx->img[1] : nullptr};
    float4* outs[1] = {ctx->io};
    int32_t* prims[1] = {out_prim ? ctx->io_prim : nullptr};
    r = render_views(*sc, 1, cam, &W, &H, 1, p, ins, outs, prims, st);
    if (r != RCP_OK) return r;
    RCP_CUDA(cudaMemcpyAsync(out_rgbz, ctx->io, sizeof(float4) * P, cudaMemcpyDeviceToHost, st));
    if (out_prim)
        RCP_CUDA(cudaMemcpyAsync(out_prim, ctx->io_prim, sizeof(int32_t) * P, cudaMemcpyDeviceToHost, st));
    return check_status(*ctx, st);
}

rcp_status rcp_imagespace_pass_device(const float* d_base, const float* d_prev, float* d_out, int W, int H,
                                      float k_px, void* stream) {
    if (!d_base || !d_prev || !d_out || W < 1 || H < 1 || W > 8192 || H > 8192 || !(k_px >= 0.f) ||
        !std::isfinite(k_px)) {
        set_error("rcp_imagespace_pass_device: NULL image, size outside [1, 8192] or k_px not finite >= 0");
        return RCP_ERR_ARG;
    }
    if (((uintptr_t)d_base | (uintptr_t)d_prev | (uintptr_t)d_out) & 15) {
        set_error("rcp_imagespace_pass_device: images must be 16-byte aligned");
        return RCP_ERR_ARG;
    }
    if (d_out == d_base || d_out == d_prev) {
        set_error("rcp_imagespace_pass_device: out must not alias base or prev");
        return RCP_ERR_ARG;
    }
    return launch_imagespace_single((const float4*)d_base, (const float4*)d_prev, (float4*)d_out, W, H, k_px,
                                    (cudaStream_t)stream);
}

rcp_status rcp_get_tuning(const rcp_scene* sc, rcp_tuning* out) {
    if (!sc || !out) {
        set_error("rcp_get_tuning: NULL argument");
        return RCP_ERR_ARG;
    }
    *out = sc->tuning;
    return RCP_OK;
}

rcp_status rcp_set_tuning(rcp_scene* sc, const rcp_tuning* t) {
    if (!sc || !t) {
        set_error("rcp_set_tuning: NULL argument");
        return RCP_ERR_ARG;
    }
    if ((t->block != 64 && t->block != 128 && t->block != 256) || (t->chunk != 32 && t->chunk != 64) ||
        t->blocks_per_sm < 0 || t->blocks_per_sm > 32 || (t->fused_camera != 0 && t->fused_camera != 1) ||
        t->stack_entries < 0 || t->stack_entries > MAX_STACK || t->hints < 0 || t->hints > 3 ||
        (t->chain_passes != 0 && t->chain_passes != 1)) {
        set_error("rcp_set_tuning: block in {64,128,256}, chunk in {32,64}, 0 <= blocks_per_sm <= 32, fused 0/1, "
                  "0 <= stack_entries <= 64, 0 <= hints <= 3, chain_passes 0/1");
        return RCP_ERR_ARG;
    }
    std::lock_guard<std::mutex> lk(sc->mu);
    sc->tuning = *t;
    return RCP_OK;
}

// K passes with work counters, chained where `chain` asks for it and the render
// allows it.
static rcp_status count_frame(rcp_scene* sc, const rcp_camera* cam, int W, int H, int K, const rcp_params* p,
                              const float* d_in, float* d_out, bool chain, rcp_counters* out) {
    std::lock_guard<std::mutex> lk(sc->mu);
    rcp_status r = check_view(cam, W, H, p);
    if (r != RCP_OK) return r;
    if (K < 1 || K > 16) {
        set_error("K must be in [1, 16]");
        return RCP_ERR_ARG;
    }
    cudaStream_t st = lib_stream();
    const int64_t P = (int64_t)W * H;
    RenderCtx* ctx = nullptr;
    r = get_ctx(*sc, 1, K, P, (int64_t)((W + 7) / 8) * ((H + 3) / 4), st, &ctx);
    if (r != RCP_OK) return r;
    std::vector<ViewDev> base(1);
    make_view(base[0], *cam, W, H, *p);
    int64_t tp, tc;
    layout_views(base, tp, tc);
    const float4* ins[1] = {(const float4*)d_in};
    if (!d_out) {
        r = ensure_io(*sc, *ctx, false, false);
        if (r != RCP_OK) return r;
    }
    float4* outs[1] = {d_out ? (float4*)d_out : ctx->io};
    StreamUse use, spill_use;
    r = use.begin(ctx->work, st);
    if (r != RCP_OK) return r;
    r = stage_views(*sc, *ctx, base, ins, outs, nullptr, nullptr, st, chain);
    if (r != RCP_OK) return r;
    DevBuf<unsigned long long> d_cnt;
    RCP_CUDA(d_cnt.alloc(8));
    RCP_CUDA(cudaMemsetAsync(d_cnt.p, 0, sizeof(unsigned long long) * 8, st));
    LaunchCfg cfg = cfg_of(*sc);
    cfg.count = true;
    cfg.ms = p->spp > 0;
    if (ctx->chained) cfg.fused = true;
    r = ensure_spill(*sc, cfg, st, spill_use);
    if (r != RCP_OK) return r;
    r = ensure_rays(*sc, *ctx, cfg);
    if (r != RCP_OK) return r;
    r = enqueue_passes(*sc, *ctx, cfg, d_cnt.p, st, false);
    if (r != RCP_OK) return r;
    unsigned long long h[8] = {0};
    RCP_CUDA(cudaMemcpyAsync(h, d_cnt.p, sizeof(h), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    out->rays = (int64_t)h[0];
    out->primary_rays = (int64_t)h[1];
    out->shadow_rays = (int64_t)h[2];
    out->nodes = (int64_t)h[3];
    out->box_tests = (int64_t)h[4];
    out->tri_tests = (int64_t)h[5];
    out->sphere_tests = (int64_t)h[6];
    return check_status(*ctx, st);
}

rcp_status rcp_count_pass(const rcp_scene* sc, const rcp_camera* cam, int W, int H, const rcp_params* p,
                          const float* d_in, float* d_out, rcp_counters* out) {
    if (!sc || !out) {
        set_error("rcp_count_pass: NULL argument");
        return RCP_ERR_ARG;
    }
    return count_frame(const_cast<rcp_scene*>(sc), cam, W, H, 1, p, d_in, d_out, false, out);
}

rcp_status rcp_count_frame(const rcp_scene* sc, const rcp_camera* cam, int W, int H, int K, const rcp_params* p,
                           const float* d_in, float* d_out, rcp_counters* out) {
    if (!sc || !out) {
        set_error("rcp_count_frame: NULL argument");
        return RCP_ERR_ARG;
    }
    if (p && ((p->mapping == RCP_MAP_IMAGE && d_in) || (p->spp > 0 && K == 1 && d_in && d_in == d_out))) {
        set_error("rcp_count_frame: d_in as for rcp_render_device");
        return RCP_ERR_ARG;
    }
    return count_frame(const_cast<rcp_scene*>(sc), cam, W, H, K, p, d_in, d_out, sc->tuning.chain_passes != 0, out);
}

rcp_status rcp_debug_trace(const rcp_scene* sc, int64_t n, const float* orig_tmin, const float* dir_tmax, int any,
                           int brute, float* t_out, int32_t* prim_out, int stack_entries, void* stream) {
    if (!sc || n < 0 || (n > 0 && (!orig_tmin || !dir_tmax || !t_out || !prim_out))) {
        set_error("rcp_debug_trace: NULL argument");
        return RCP_ERR_ARG;
    }
    if (stack_entries < 0 || stack_entries > MAX_STACK) {
        set_error("rcp_debug_trace: stack_entries outside [0, 64]");
        return RCP_ERR_ARG;
    }
    if (((uintptr_t)orig_tmin | (uintptr_t)dir_tmax) & 15) {
        set_error("rcp_debug_trace: ray arrays must be 16-byte aligned");
        return RCP_ERR_ARG;
    }
    if (sc->depth > MAX_STACK) {
        set_error("BVH deeper than the traversal stack");
        return RCP_ERR_STACK;
    }
    cudaStream_t st = (cudaStream_t)stream;
    DevBuf<int> d_status;
    RCP_CUDA(d_status.alloc(1));
    RCP_CUDA(cudaMemsetAsync(d_status.p, 0, sizeof(int), st));
    rcp_status r = launch_debug_trace(sc->dev(), n, orig_tmin, dir_tmax, any, brute, t_out, prim_out,
                                      stack_entries > 0 ? stack_entries : MAX_STACK, d_status.p, st);
    if (r != RCP_OK) return r;
    int h = 0;
    RCP_CUDA(cudaMemcpyAsync(&h, d_status.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("traversal stack overflow");
        return RCP_ERR_STACK;
    }
    return RCP_OK;
}

rcp_status rcp_last_ray_counts(const rcp_scene* sc, int64_t* primary, int64_t* shadow) {
    if (!sc || !primary || !shadow) {
        set_error("rcp_last_ray_counts: NULL argument");
        return RCP_ERR_ARG;
    }
    if (!sc->last) {
        set_error("rcp_last_ray_counts: no render yet");
        return RCP_ERR_STATE;
    }
    unsigned long long h[2];
    RCP_CUDA(cudaMemcpy(h, sc->last->d_rays, sizeof(h), cudaMemcpyDeviceToHost));
    *primary = (int64_t)h[0];
    *shadow = (int64_t)h[1];
    return RCP_OK;
}

int64_t rcp_render_h2d_bytes(int n_views, int K) {
    if (n_views < 1 || K < 1 || K > 16) return -1;
    return (int64_t)sizeof(ViewDev) * n_views * K;
}

rcp_status rcp_last_pass_times(const rcp_scene* sc, float* ms, int max_passes, int* n_passes) {
    if (!sc || !ms || !n_passes || max_passes < 1) {
        set_error("rcp_last_pass_times: NULL argument");
        return RCP_ERR_ARG;
    }
    if (!sc->last) {
        set_error("rcp_last_pass_times: no render yet");
        return RCP_ERR_STATE;
    }
    const RenderCtx& c = *sc->last;
    const int n = std::min(c.launches, max_passes);
    for (int i = 0; i < n; ++i) RCP_CUDA(cudaEventElapsedTime(&ms[i], c.pass_ev[i], c.pass_ev[i + 1]));
    *n_passes = n;
    return RCP_OK;
}

rcp_status rcp_debug_cluster_lookback_timeout(int64_t spin_limit, void* stream) {
    if (spin_limit < 1 || spin_limit > (1ll << 20)) {
        set_error("rcp_debug_cluster_lookback_timeout: spin_limit outside [1, 2^20]");
        return RCP_ERR_ARG;
    }
    return debug_cluster_timeout((int)spin_limit, (cudaStream_t)stream);
}

rcp_status rcp_debug_morton(const float* xyz, int64_t n, const float* lo, const float* hi, uint32_t* codes,
                            void* stream) {
    if (n < 0 || (n > 0 && (!xyz || !lo || !hi || !codes))) {
        set_error("rcp_debug_morton: NULL argument");
        return RCP_ERR_ARG;
    }
    rcp_status r = debug_morton(xyz, n, lo, hi, codes, (cudaStream_t)stream);
    if (r != RCP_OK) return r;
    RCP_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return RCP_OK;
}

}  // extern "C"

extern "C" rcp_status rcp_debug_sort_pairs(uint32_t* keys, uint32_t* values, int64_t n, int bits, void* stream) {
    return rcp_debug_sort_pairs_tiles(keys, values, n, bits, -1, stream);
}

extern "C" rcp_status rcp_debug_sort_pairs_tiles(uint32_t* keys, uint32_t* values, int64_t n, int bits,
                                                 int64_t resident_tiles, void* stream) {
    if (n < 0 || bits < 1 || bits > 32 || (n > 0 && (!keys || !values))) {
        set_error("rcp_debug_sort_pairs: bad argument");
        return RCP_ERR_ARG;
    }
    if (n <= 1) return RCP_OK;
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *ak = nullptr, *av = nullptr;
    void* scratch = nullptr;
    int* d_err = nullptr;
    rcp_status r = RCP_OK;
    cudaError_t e = cudaMalloc((void**)&ak, sizeof(uint32_t) * n);
    if (e == cudaSuccess) e = cudaMalloc((void**)&av, sizeof(uint32_t) * n);
    if (e == cudaSuccess) e = cudaMalloc(&scratch, radix_sort_scratch_bytes(n));
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(d_err, 0, sizeof(int), st);
    if (e != cudaSuccess) r = cuda_fail(e, "rcp_debug_sort_pairs alloc");
    if (r == RCP_OK) r = radix_sort_pairs(keys, values, ak, av, n, bits, scratch, d_err, st, resident_tiles);
    int h = 0;
    if (r == RCP_OK) {
        e = cudaMemcpyAsync(&h, d_err, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) r = cuda_fail(e, "rcp_debug_sort_pairs");
    }
    cudaFree(ak);
    cudaFree(av);
    cudaFree(scratch);
    cudaFree(d_err);
    if (r == RCP_OK && h) {
        set_error("radix sort: look-back wait ran out");
        r = RCP_ERR_TIMEOUT;
    }
    return r;
}

// ---------------------------------------------------------------- autotuner

namespace {

std::string gpu_name() {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return "unknown";
    return prop.name;
}

// A flat JSON object {"key": [block, blocks_per_sm, chunk, fused, stack_entries, hints, chain_passes, us], ...}
std::map<std::string, std::vector<double>> read_cache(const char* path) {
    std::map<std::string, std::vector<double>> m;
    if (!path) return m;
    std::ifstream f(path);
    if (!f) return m;
    std::stringstream ss;
    ss << f.rdbuf();
    const std::string s = ss.str();
    size_t i = 0;
    while ((i = s.find('"', i)) != std::string::npos) {
        const size_t j = s.find('"', i + 1);
        if (j == std::string::npos) break;
        const std::string key = s.substr(i + 1, j - i - 1);
        const size_t a = s.find('[', j), b = s.find(']', j);
        if (a == std::string::npos || b == std::string::npos || b < a) break;
        std::vector<double> v;
        std::stringstream vs(s.substr(a + 1, b - a - 1));
        std::string tok;
        while (std::getline(vs, tok, ',')) v.push_back(atof(tok.c_str()));
        if (v.size() >= 8) m[key] = v;  // entries of fewer fields predate a tuning field: searched again
        i = b + 1;
    }
    return m;
}

void write_cache(const char* path, const std::map<std::string, std::vector<double>>& m) {
    if (!path) return;
    const std::string tmp = std::string(path) + ".tmp";
    {
        std::ofstream f(tmp);
        if (!f) return;
        f << "{\n";
        size_t n = 0;
        for (auto& kv : m) {
            f << "  \"" << kv.first << "\": [";
            for (size_t q = 0; q < kv.second.size(); ++q) f << (q ? ", " : "") << kv.second[q];
            f << "]" << (++n < m.size() ? "," : "") << "\n";
        }
        f << "}\n";
    }
    rename(tmp.c_str(), path);
}

}  // namespace

extern "C" rcp_status rcp_autotune(rcp_scene* sc, const rcp_camera* cam, int W, int H, const rcp_params* p,
                                   const char* cache_path, rcp_tuning* out) {
    if (!sc) {
        set_error("rcp_autotune: NULL scene");
        return RCP_ERR_ARG;
    }
    rcp_status r = check_view(cam, W, H, p);
    if (r != RCP_OK) return r;
    int cls = 0;
    for (int64_t n = sc->T + sc->S; n > 1; n >>= 1) ++cls;
    std::ostringstream key;
    key << gpu_name() << "|prims2^" << cls << "|depth" << sc->depth << "|" << W << "x" << H << "|map" << p->mapping
        << "|spp" << p->spp;
    auto cache = read_cache(cache_path);
    auto it = cache.find(key.str());
    if (it != cache.end()) {
        const auto& v = it->second;
        rcp_tuning t{(int)v[0], (int)v[1], (int)v[2], (int)v[3], (int)v[4], (int)v[5], (int)v[6]};
        r = rcp_set_tuning(sc, &t);
        if (r == RCP_OK && out) *out = t;
        if (r == RCP_OK) return RCP_OK;
    }
    std::lock_guard<std::mutex> lk(sc->mu);
    cudaStream_t st = lib_stream();
    const int64_t P = (int64_t)W * H;
    DevBuf<float4> d_img;
    RCP_CUDA(d_img.alloc(P));
    EventPair ev;
    RCP_CUDA(ev.create());
    double best_us = 1e30;
    rcp_tuning best = sc->tuning;
    const int full = full_stack(*sc);
    std::vector<int> stacks{0};  // 0: one entry per tree level
    if (full / 2 >= 4) stacks.push_back(((full / 2) + 3) & ~3);
    // one launch per pass over block x fused camera x chunk x stack x hints;
    // chained passes (fused camera) over block x chunk x stack x hints
    std::vector<rcp_tuning> cands;
    for (int b : {64, 128, 256})
        for (int chain = 0; chain < 2; ++chain)
            for (int fused = chain; fused < 2; ++fused)
                for (int chunk : {32, 64})
                    for (int stk : stacks)
                        for (int hints : {3, 0})
                            if (stk < full) cands.push_back(rcp_tuning{b, 0, chunk, fused, stk, hints, chain});
    for (const rcp_tuning& t : cands) {
        sc->tuning = t;
        const float4* ins[1] = {nullptr};
        float4* outs[1] = {d_img.p};
        double us = 1e30;
        // K = 4 so later passes read real images and a chained launch has
        // passes to carry; best of 3
        for (int rep = 0; rep < 4 && r == RCP_OK; ++rep) {
            cudaEventRecord(ev.a, st);
            r = render_views(*sc, 1, cam, &W, &H, 4, p, ins, outs, nullptr, st);
            cudaEventRecord(ev.b, st);
            if (cudaEventSynchronize(ev.b) != cudaSuccess) r = RCP_ERR_CUDA;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, ev.a, ev.b);
            if (rep > 0) us = std::min(us, 1000.0 * ms);
        }
        if (r != RCP_OK) break;
        if (us < best_us) {
            best_us = us;
            best = t;
        }
    }
    sc->tuning = best;
    if (r != RCP_OK) return r;
    cache[key.str()] = {(double)best.block,        (double)best.blocks_per_sm, (double)best.chunk,
                        (double)best.fused_camera, (double)best.stack_entries, (double)best.hints,
                        (double)best.chain_passes, best_us};
    write_cache(cache_path, cache);
    if (out) *out = best;
    return RCP_OK;
}
