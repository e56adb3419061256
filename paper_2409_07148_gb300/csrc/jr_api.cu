// Host runtime behind the C ABI of include/jr.h: argument checks, device
// memory for scenes and chain sets, launch sequencing, error reporting.  No
// exception or abort crosses the ABI; every failure becomes a jr_status and a
// thread-local message.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/jr.h"
#include "jr_internal.h"

using namespace jr;

namespace {

thread_local std::string g_err;

jr_status fail(jr_status s, const std::string& msg) {
    g_err = msg;
    return s;
}

jr_status cuda_fail(cudaError_t e, const char* what) {
    (void)cudaGetLastError();  // clear a sticky launch error so later calls see a clean slate
    return fail(e == cudaErrorMemoryAllocation ? JR_ERR_OOM : JR_ERR_CUDA,
                std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")");
}

#define JR_CUDA(call, what)                      \
    do {                                         \
        cudaError_t e_ = (call);                 \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

// Testing hook (jr_debug_fail_alloc): when >= 0, the number of device
// allocations still to succeed before one fails with cudaErrorMemoryAllocation.
std::atomic<long long> g_fail_alloc_in{-1};

template <class T>
cudaError_t dev_alloc(T** p, size_t count) {
    long long k = g_fail_alloc_in.load();
    while (k >= 0 && !g_fail_alloc_in.compare_exchange_weak(k, k - 1)) {
    }
    if (k == 0) return cudaErrorMemoryAllocation;
    return cudaMalloc((void**)p, sizeof(T) * (count > 0 ? count : 1));
}

}  // namespace

struct jr_scene {
    Bvh4Node* nodes = nullptr;
    TriRecord* tris = nullptr;
    Material* mats = nullptr;
    SceneView view{};
    jr_scene_info info{};
    ~jr_scene() {
        cudaFree(nodes);
        cudaFree(tris);
        cudaFree(mats);
    }
};

struct jr_chains {
    const jr_scene* scene = nullptr;
    jr_params params{};
    ChainView view{};
    uint64_t steps = 0;
    int block = 128;
    uint32_t exec = JR_EXEC_AUTO;
    uint64_t epochs = 0;  // restarts from a new regeneration distribution (Philox tag 3 key)
    uint64_t flow_gen = 0;      // bumped whenever the attached flow (or its weight) changes
    uint32_t visit_budget = 0;  // traversal watchdog limits of this set's launches (0: the scene's)
    int stack_limit = 0;
    AheadView ahead{};          // look-ahead buffers (JR_EXEC_AUTO)
    double ahead_share = -1.0;  // the expected share of local steps (< 0: not read back yet)
    bool ahead_fixed = false;   // a captured graph holds the buffers' addresses: they stay as they are
    // The scene as this set's launches see it (with the set's traversal limits).
    SceneView scene_view() const {
        SceneView v = scene->view;
        if (visit_budget) v.visit_budget = visit_budget;
        if (stack_limit) v.stack_limit = stack_limit;
        return v;
    }
    ~jr_chains() {
        cudaFree(ahead.F);
        cudaFree(ahead.queue);
        cudaFree(ahead.ctl);
        cudaFree(view.wf.y);
        cudaFree(view.wf.par);
        cudaFree(view.wf.ua);
        cudaFree(view.wf.fy);
        cudaFree(view.wf.uy);
        cudaFree(view.wf.fq);
        cudaFree(view.wf.done);
        cudaFree(view.wf.queue);
        cudaFree(view.wf.qcount);
        cudaFree(view.x);
        cudaFree(view.fpu);
        cudaFree(view.fb);
        cudaFree(view.acc64);
        cudaFree(view.counters);
        cudaFree(view.status);
        cudaFree(view.drift);
    }
};

// Post-burn-in iterations of an MH chain set over all chains (the N of its estimator).
static uint64_t mh_samples(const jr_chains* c) {
    if (!(c->view.flags & JR_FLAG_MH)) return 0;
    return c->steps > c->view.burn_in ? (c->steps - c->view.burn_in) * c->view.n : 0;
}

// swizzle_nodes_kernel's moves on the host: chunk c of node i to c ^ (i & 7).  For few
// nodes, whose launch would be a seventh of the scene's creation.
constexpr size_t kHostSwizzleNodes = 256;
static void swizzle_nodes_host(Bvh4Node* nodes, size_t n) {
    for (size_t i = 0; i < n; ++i) {
        unsigned char from[sizeof(Bvh4Node)], to[sizeof(Bvh4Node)];
        std::memcpy(from, nodes + i, sizeof(from));
        for (size_t c = 0; c < sizeof(Bvh4Node) / 16; ++c) std::memcpy(to + 16 * (c ^ (i & 7)), from + 16 * c, 16);
        std::memcpy(nodes + i, to, sizeof(to));
    }
}

// Whether a scene of at most kWarpChainMaxTris triangles is a closed surface, which no path
// leaves: every edge (by the positions of its ends) is walked as often one way as the
// other.  Each way adds or takes one hash of the edge, so that the sum is 0 then, and
// otherwise with a chance of 2^-64, which costs speed only.
static bool closed_surface(const jr_scene_desc* d) {
    if (d->n_tris == 0 || d->n_tris > kWarpChainMaxTris) return false;
    const auto point = [&](uint32_t v) {
        uint64_t h = 0;
        for (int a = 0; a < 3; ++a) {
            const float x = d->verts[3 * (size_t)v + a] + 0.0f;  // -0 as 0
            uint32_t bits;
            std::memcpy(&bits, &x, sizeof(bits));
            h = (h ^ bits) * 0x9E3779B97F4A7C15ull;  // splitmix64's constants
            h ^= h >> 29;
        }
        return h;
    };
    uint64_t sum = 0;
    for (uint32_t t = 0; t < d->n_tris; ++t) {
        const uint32_t* tri = d->tris + 3 * (size_t)t;
        const uint64_t h[3] = {point(tri[0]), point(tri[1]), point(tri[2])};
        for (int k = 0; k < 3; ++k) {
            const uint64_t a = std::min(h[k], h[(k + 1) % 3]), b = std::max(h[k], h[(k + 1) % 3]);
            uint64_t e = (a ^ (b * 0xBF58476D1CE4E5B9ull)) * 0x94D049BB133111EBull;
            e ^= e >> 31;
            if (a != b) sum += h[k] == a ? e : 0 - e;
        }
    }
    return sum == 0;
}

extern "C" {

const char* jr_last_error(void) { return g_err.c_str(); }

const char* jr_version(void) { return "jr-gb300 0.1 (sm_103a)"; }

jr_status jr_scene_create(const jr_scene_desc* desc, void* stream, jr_scene** out) {
    if (!desc || !out) return fail(JR_ERR_INVALID_ARG, "jr_scene_create: null argument");
    if (desc->n_tris > 0 && (!desc->verts || !desc->tris || !desc->tri_material))
        return fail(JR_ERR_INVALID_ARG, "jr_scene_create: null triangle arrays");
    if (desc->n_materials == 0 || !desc->materials)
        return fail(JR_ERR_INVALID_ARG, "jr_scene_create: at least one material is required");
    for (uint32_t t = 0; t < desc->n_tris; ++t)
        if (desc->tri_material[t] >= desc->n_materials)
            return fail(JR_ERR_INVALID_ARG, "jr_scene_create: triangle material index out of range");
    std::vector<Material> mats(desc->n_materials);
    for (uint32_t m = 0; m < desc->n_materials; ++m) {
        const float* r = desc->materials + (size_t)JR_MATERIAL_FLOATS * m;
        Material& q = mats[m];
        q.type = (int)r[0];
        if (r[0] != (float)q.type || q.type < JR_MAT_LAMBERT || q.type > JR_MAT_DIELECTRIC)
            return fail(JR_ERR_INVALID_ARG, "jr_scene_create: unknown material type");
        q.albedo = make_float3(r[1], r[2], r[3]);
        q.emission = make_float3(r[4], r[5], r[6]);
        q.emits = (r[4] != 0.f || r[5] != 0.f || r[6] != 0.f);
        q.phong_inv_n1 = 1.0f / (r[7] + 1.0f);
        q.phong_scale = (r[7] + 2.0f) / (r[7] + 1.0f);
        q.ior = r[8];
        q.pad = 0.f;
        if (q.type == JR_MAT_PHONG && !(r[7] >= 0.f)) return fail(JR_ERR_INVALID_ARG, "jr_scene_create: Phong n < 0");
        if (q.type == JR_MAT_DIELECTRIC && !(r[8] > 0.f)) return fail(JR_ERR_INVALID_ARG, "jr_scene_create: ior <= 0");
    }
    HostBvh bvh;
    std::string err;
    bool closed = false;
    try {
        if (!build_bvh(desc->verts, desc->n_verts, desc->tris, desc->n_tris, desc->tri_material, &bvh, &err))
            return fail(JR_ERR_INVALID_ARG, "jr_scene_create: " + err);
        closed = closed_surface(desc);
    } catch (const std::bad_alloc&) {
        return fail(JR_ERR_OOM, "jr_scene_create: host allocation failed in the BVH build");
    } catch (const std::exception& ex) {
        return fail(JR_ERR_INVALID_ARG, std::string("jr_scene_create: BVH build failed: ") + ex.what());
    }
    jr_scene* s = new (std::nothrow) jr_scene();
    if (!s) return fail(JR_ERR_OOM, "jr_scene_create: host allocation failed");
    cudaStream_t st = (cudaStream_t)stream;
    const bool on_host = bvh.nodes.size() <= kHostSwizzleNodes;
    if (on_host) swizzle_nodes_host(bvh.nodes.data(), bvh.nodes.size());
    cudaError_t e;
    if ((e = dev_alloc(&s->nodes, bvh.nodes.size())) != cudaSuccess ||
        (e = dev_alloc(&s->tris, bvh.tris.size())) != cudaSuccess ||
        (e = dev_alloc(&s->mats, mats.size())) != cudaSuccess ||
        (e = cudaMemcpyAsync(s->nodes, bvh.nodes.data(), sizeof(Bvh4Node) * bvh.nodes.size(), cudaMemcpyHostToDevice,
                             st)) != cudaSuccess ||
        (!on_host && (e = launch_swizzle_nodes(s->nodes, (uint32_t)bvh.nodes.size(), st)) != cudaSuccess) ||
        (e = cudaMemcpyAsync(s->tris, bvh.tris.data(), sizeof(TriRecord) * bvh.tris.size(), cudaMemcpyHostToDevice,
                             st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(s->mats, mats.data(), sizeof(Material) * mats.size(), cudaMemcpyHostToDevice, st)) !=
            cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
        delete s;
        return cuda_fail(e, "jr_scene_create");
    }
    s->view.nodes = s->nodes;
    s->view.tris = s->tris;
    s->view.mats = s->mats;
    s->view.root = bvh.root;
    s->view.n_nodes = (int)bvh.nodes.size();
    s->view.n_tris = (uint32_t)bvh.tris.size();
    s->view.visit_budget = kNodeVisitBudget;
    s->view.stack_limit = kStackSize;
    s->view.stack_need = bvh.stack_need;
    s->view.closed = closed;
    std::memcpy(s->view.cam, desc->camera, sizeof(float) * 12);
    s->info.n_tris = desc->n_tris;
    s->info.n_nodes = (uint32_t)bvh.nodes.size();
    s->info.bvh_depth = (uint32_t)bvh.depth;
    s->info.n_materials = desc->n_materials;
    s->info.device_bytes =
        sizeof(Bvh4Node) * bvh.nodes.size() + sizeof(TriRecord) * bvh.tris.size() + sizeof(Material) * mats.size();
    *out = s;
    return JR_OK;
}

jr_status jr_scene_get_info(const jr_scene* scene, jr_scene_info* out) {
    if (!scene || !out) return fail(JR_ERR_INVALID_ARG, "jr_scene_get_info: null argument");
    *out = scene->info;
    return JR_OK;
}

void jr_scene_destroy(jr_scene* scene) { delete scene; }

static jr_status check_params(const jr_params* p, const char* who) {
    if (!p) return fail(JR_ERR_INVALID_ARG, std::string(who) + ": null params");
    if (p->width == 0 || p->height == 0 || (uint64_t)p->width * p->height > (1u << 26))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": image size out of range (1 .. 2^26 pixels)");
    if (p->max_depth > JR_MAX_DEPTH) return fail(JR_ERR_INVALID_ARG, std::string(who) + ": max_depth > 15");
    if (!(p->c_tilde > 0.f) || !std::isfinite(p->c_tilde))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": c_tilde must be finite and > 0");
    if (!(p->sigma > 0.f) || !std::isfinite(p->sigma))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": sigma must be finite and > 0");
    if (p->flags & ~(JR_FLAG_RAO_BLACKWELL | JR_FLAG_MH | JR_FLAG_MALA))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": unknown flag");
    if ((p->flags & JR_FLAG_MALA) && (p->flags & JR_FLAG_RAO_BLACKWELL))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": MALA chains splat the sampled holding time");
    if ((p->flags & JR_FLAG_MH) && (p->flags & JR_FLAG_RAO_BLACKWELL))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": the MH baseline has no holding times to Rao-Blackwellise");
    if ((p->flags & JR_FLAG_MH) && !(p->large_step >= 0.f && p->large_step <= 1.f))
        return fail(JR_ERR_INVALID_ARG, std::string(who) + ": large_step must be in [0, 1]");
    return JR_OK;
}

jr_status jr_chains_create(const jr_scene* scene, const jr_params* params, void* stream, jr_chains** out) {
    if (!scene || !out) return fail(JR_ERR_INVALID_ARG, "jr_chains_create: null argument");
    jr_status ps = check_params(params, "jr_chains_create");
    if (ps != JR_OK) return ps;
    if (params->n_chains == 0) return fail(JR_ERR_INVALID_ARG, "jr_chains_create: n_chains must be >= 1");
    if (params->chain_offset + params->n_chains > (1ull << 32))
        return fail(JR_ERR_INVALID_ARG, "jr_chains_create: chain ids must stay below 2^32");
    jr_chains* c = new (std::nothrow) jr_chains();
    if (!c) return fail(JR_ERR_OOM, "jr_chains_create: host allocation failed");
    c->scene = scene;
    c->params = *params;
    ChainView& v = c->view;
    v.n = params->n_chains;
    v.chain_offset = (uint32_t)params->chain_offset;
    v.width = params->width;
    v.height = params->height;
    v.depth = params->max_depth;
    v.dim = 2 + 2 * params->max_depth;
    v.flags = params->flags;
    v.seed = params->seed;
    v.c_tilde = params->c_tilde;
    v.sigma = params->sigma;
    v.large_step = (params->flags & JR_FLAG_MH) ? params->large_step : 0.f;
    v.burn_in = (params->flags & JR_FLAG_MH) ? params->burn_in : 0;
    const size_t npx = (size_t)params->width * params->height;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    if ((e = dev_alloc(&v.x, (size_t)v.dim * v.n)) != cudaSuccess || (e = dev_alloc(&v.fpu, 5 * v.n)) != cudaSuccess ||
        (e = dev_alloc(&v.fb, npx)) != cudaSuccess || (e = dev_alloc(&v.acc64, npx)) != cudaSuccess ||
        (e = dev_alloc(&v.counters, kCounters)) != cudaSuccess || (e = dev_alloc(&v.status, 1)) != cudaSuccess ||
        (e = cudaMemsetAsync(v.fb, 0, sizeof(float4) * npx, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(v.acc64, 0, sizeof(double4_32a) * npx, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(v.counters, 0, sizeof(unsigned long long) * kCounters, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(v.status, 0, sizeof(unsigned int), st)) != cudaSuccess ||
        ((v.flags & JR_FLAG_MALA) && (e = dev_alloc(&v.drift, (size_t)v.dim * v.n)) != cudaSuccess) ||
        (e = launch_init(scene->view, v, st)) != cudaSuccess ||
        ((v.flags & JR_FLAG_MALA) && (e = launch_mala_reeval(scene->view, v, st)) != cudaSuccess) ||
        (e = prepare_static_scratch()) != cudaSuccess) {  // jr_advance_static's array, see jr_wavefront.cu
        delete c;
        return cuda_fail(e, "jr_chains_create");
    }
    *out = c;
    return JR_OK;
}

void jr_chains_destroy(jr_chains* chains) { delete chains; }

// Wavefront buffers, allocated on the first wavefront advance of a chain set.
static jr_status ensure_wavefront(jr_chains* c, cudaStream_t st) {
    WaveView& w = c->view.wf;
    if (w.y) return JR_OK;
    const uint64_t n = c->view.n;
    cudaError_t e;
    if ((e = dev_alloc(&w.y, (size_t)c->view.dim * n)) != cudaSuccess || (e = dev_alloc(&w.par, n)) != cudaSuccess ||
        (e = dev_alloc(&w.ua, n)) != cudaSuccess || (e = dev_alloc(&w.fy, n)) != cudaSuccess ||
        (e = dev_alloc(&w.queue, n)) != cudaSuccess ||
        (e = dev_alloc(&w.qcount, kQCount)) != cudaSuccess || (e = dev_alloc(&w.uy, n)) != cudaSuccess ||
        (e = dev_alloc(&w.fq, 2 * n)) != cudaSuccess || (e = dev_alloc(&w.done, n)) != cudaSuccess ||
        (e = cudaMemsetAsync(w.done, 0, n, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(w.par, 0, n, st)) != cudaSuccess) {
        cudaFree(w.done);
        cudaFree(w.y);
        cudaFree(w.par);
        cudaFree(w.ua);
        cudaFree(w.fy);
        cudaFree(w.queue);
        cudaFree(w.qcount);
        cudaFree(w.uy);
        cudaFree(w.fq);
        w = WaveView{};
        return cuda_fail(e, "jr_advance (wavefront buffers)");
    }
    return JR_OK;
}

// The current device's SM count (0 where it cannot be had).
static uint64_t sm_count() {
    static DeviceOnce once;
    long long sms = 0;
    const cudaError_t e = once.get(
        [](int dev, long long* v) {
            int n = 0;
            const cudaError_t r = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
            *v = n;
            return r;
        },
        &sms);
    return e == cudaSuccess ? (uint64_t)sms : 0;
}

// One warp per chain: asked for, or (auto) a small scene with fewer chains
// than 32 per SM -- while one thread per chain would leave the SMs without
// even one warp each (measured on the Cornell box and a depth-6 furnace: one
// chain per warp 6.1x / 2.2x faster at 256 chains, 2.5x / 0.94x at 4 096;
// the megakernel 1.5x / 0.56x ahead at 8 192).  Only for sets without a flow
// (the wavefront takes those).
static bool warp_per_chain(const jr_chains* c) {
    if (c->view.flow.D != 0) return false;
    if (c->exec == JR_EXEC_WARP) return true;
    if (c->exec != JR_EXEC_AUTO || c->scene->view.n_tris > kWarpChainMaxTris) return false;
    return c->view.n < 32 * sm_count();
}

// Whether JR_EXEC_AUTO runs this advance in look-ahead windows (jr_ahead.cu); sets
// their buffers up on first use.  A window costs the latency of one path launch and
// of its longest run of local steps, whatever the number of steps, so it takes the
// more steps the fewer chains there are.  Measured against the best of the other
// modes (us per advance; Cornell + spheres / slit caustic / terrain):
//   2^20 chains, 2 steps     1 381, 1 416  /    842,   895  / 1 333, 1 338
//   2^18 chains, 2 steps       533,   584  /    448,   511  /   608,   606
//   2^16 chains, 8 steps       703, 1 148  /    611,   663  /   898,   911  (4: 467, 610 / 421, 381 / 567, 485)
//   30 000 chains, 16 steps    844, 1 576  /    864,   923  / 1 207, 1 234  (8: 540, 841 / 548, 496 / 682, 658)
//   3 000 chains, 64 steps   1 009, 1 901  /  1 740, 1 783  / 1 901, 2 054  (16: 485, 572 / 649, 551 / 767, 657)
// and one warp per chain in the 24-triangle box: 256 chains, 64 steps 159, 198 (16: 88,
// 69).  Such scenes with more chains than that stay in the megakernel: their paths
// are short and alike, so it loses little (2^16 chains, 16 steps: 514, 369).
// MALA Restore, whose megakernel takes the gradient of every candidate, gains from
// fewer steps on (131 072 chains, 2 steps 497, 1 052 / 542, 863 / 717, 865; 32 768
// chains, 4 steps 532, 887 / 569, 778 / 719, 729; 10 007 chains, 8 steps 594, 1 161 /
// 783, 900 / 874, 958; 3 000 chains, 32 steps 1 143, 2 738 / 1 958, 2 039 / 2 388, 2 623).
//
// It pays while few steps are local, because a local step's regeneration candidate
// is traced for nothing.  The stationary share of local steps is p_lambda /
// (p_lambda + c~) (Section 6.1); p_lambda = E_mu[p] is estimated from the initial states,
// which are samples of mu (later ones follow the jump chain, which favours large p: 40
// steps on, the 24-triangle box reads as 0.64 local instead of 0.14).  So the answer is
// the same whatever the set has done before, and after a restore.  Where the buffers
// cannot be had, or the stream is being captured before they exist, the other modes
// run.
//
// The limit, measured by c~ at shares of 0.05, 0.1, 0.2 and 0.35, as the time of the best
// of the other modes over that of look-ahead:
//   Cornell + spheres   10 007 x 32 steps  2.09 1.80 1.55 1.47  2^20 x 16  1.13 1.12 1.11 1.10
//   slit caustic                           1.53 1.62 1.68 1.67             1.54 1.50 1.53 1.50
//   terrain                                1.27 1.03 0.99 0.99             1.29 1.22 1.13 1.04
//   terrain             65 536 x 16 steps  1.13 1.06 0.94 0.92
// and MALA, 3 000 chains x 64 steps, shares of 0.03, 0.05, 0.1, 0.2: Cornell + spheres 1.95
// 1.73 1.37 1.18, terrain 1.68 1.39 1.12 1.02, slit caustic 1.09 0.93 0.89 0.94 (1 000 chains
// 1.04 0.95 0.77 0.80), from 7 000 chains up above 1 everywhere.  A quarter is where the
// scene that gains least breaks even.
//
// One warp per chain beyond 4 chains per SM (up to there a block per chain takes a
// window's local steps two or three at a time): a window settled by a warp per chain
// gains only what its path launch saves, so with less than kAheadShareSteps steps the limit
// is lower in proportion (24-triangle box, one warp per chain over look-ahead at shares
// of 0.05, 0.1, 0.15, 0.2: 1 000 chains x 32 steps 1.11 1.02 0.96 0.88, x 48 1.50 1.16 0.99
// 0.93, x 64 1.77 1.18 1.10 1.04; depth 8, 2 000 x 32 1.28 1.04 0.95 0.81, x 64 above 1).
constexpr double kAheadShare = 0.25, kAheadShareSteps = 96.0;

// Lets this thread allocate while some other stream of it captures in the global mode.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
    RelaxedCapture(const RelaxedCapture&) = delete;
    RelaxedCapture& operator=(const RelaxedCapture&) = delete;
};

static bool use_ahead(jr_chains* c, uint32_t n_steps, cudaStream_t st) {
    if (c->exec != JR_EXEC_AUTO || c->view.flow.D != 0 || (c->view.flags & JR_FLAG_MH)) return false;
    const uint64_t n = c->view.n;
    const bool mala = (c->view.flags & JR_FLAG_MALA) != 0;
    const uint32_t least = mala ? (n >= (1u << 17) ? 2 : n >= (1u << 15) ? 4 : n >= (1u << 13) ? 8 : 32)
                                : n >= (1u << 18) ? 2 : n >= (1u << 16) ? 8 : n >= (1u << 14) ? 16 : 32;
    if (n_steps < least || n > kAheadItems / least) return false;
    const bool warp = !mala && warp_per_chain(c);
    if (c->scene->view.n_tris <= kWarpChainMaxTris && !warp) return false;
    const double limit =
        warp && n > 4 * sm_count() ? kAheadShare * std::min(1.0, n_steps / kAheadShareSteps) : kAheadShare;
    if (c->ahead_share >= limit) return false;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool captured = cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    if (captured) {  // with the buffers an advance outside a capture left, or not at all
        c->ahead_fixed = c->ahead_fixed || c->ahead.window != 0;
        return c->ahead.window != 0;
    }
    RelaxedCapture relaxed;  // another stream of this thread may be capturing
    if (c->ahead_share < 0.0) {
        double sum = 0.0;
        if (cudaMemcpyAsync(&sum, c->view.counters + kCounterMuP, sizeof(sum), cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return false;
        const double p = sum / (double)n;
        const double share = p / (p + (double)c->view.c_tilde);
        c->ahead_share = share >= 0.0 ? share : 1.0;
        // A later advance of fewer steps is the wavefront's, and may be captured: its
        // buffers have to exist by then.
        if (c->ahead_share < kAheadShare && !mala && n >= kWavefrontMinChains && ensure_wavefront(c, st) != JR_OK)
            (void)cudaGetLastError();
        if (!(c->ahead_share < limit)) return false;
    }
    AheadView& a = c->ahead;
    uint64_t window = least;  // a power of two, so that advances of growing lengths rarely grow it
    while (window < n_steps) window *= 2;
    window = std::min<uint64_t>(window, kAheadItems / n);
    // Two only where a window's tail waits for the next window's paths (launch_ahead).
    const uint32_t buffers = n_steps > window && !mala && !warp ? 2 : 1;
    if (c->ahead_fixed) return a.window != 0;
    if (!a.queue && (dev_alloc(&a.queue, n) != cudaSuccess || dev_alloc(&a.ctl, kCtlCount) != cudaSuccess)) {
        (void)cudaGetLastError();
        cudaFree(a.queue);
        a.queue = nullptr;
        return false;
    }
    if (a.window < window || a.buffers < buffers) {
        // The old buffer goes first (this waits for the launches that use it), so that no
        // more than one is held; where the new one cannot be had, one of the old size may.
        const AheadView old = a;
        cudaFree(a.F);
        a.F = nullptr;
        a.window = (uint32_t)std::max<uint64_t>(window, old.window);
        a.buffers = std::max(buffers, old.buffers);
        if (dev_alloc(&a.F, (size_t)a.buffers * a.window * n) != cudaSuccess) {
            (void)cudaGetLastError();
            a.F = nullptr;
            a.window = old.window;
            a.buffers = old.buffers;
            if (a.window == 0 || dev_alloc(&a.F, (size_t)a.buffers * a.window * n) != cudaSuccess) {
                (void)cudaGetLastError();
                a.F = nullptr;
                a.window = a.buffers = 0;
            }
        }
    }
    return a.window != 0;
}

// One warp per chain has no traversal, so no traversal limits either: there the
// look-ahead paths run under the scene's own.
static cudaError_t run_ahead(jr_chains* c, uint32_t n_steps, cudaStream_t st, KernelTimer* tm) {
    const bool warp = warp_per_chain(c) && !(c->view.flags & JR_FLAG_MALA);
    return launch_ahead(warp ? c->scene->view : c->scene_view(), c->view, c->ahead, c->steps, n_steps, warp, st, tm);
}

static jr_status advance_impl(jr_chains* c, uint32_t n_steps, uint8_t* f, float* dt, int32_t* pix,
                              unsigned long long* work, void* stream, const char* who) {
    if (!c) return fail(JR_ERR_INVALID_ARG, std::string(who) + ": null chains");
    if (n_steps == 0) return JR_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const bool plain = !f && !dt && !pix && !work;
    const bool has_flow = c->view.flow.D != 0;
    if (c->view.flags & JR_FLAG_MALA) {  // Langevin moves: the megakernel, or look-ahead windows
        if (work) return fail(JR_ERR_STATE, std::string(who) + ": the counted advance does not run MALA chains");
        if (plain && use_ahead(c, n_steps, st)) JR_CUDA(run_ahead(c, n_steps, st, nullptr), who);
        else JR_CUDA(launch_step_mala(c->scene_view(), c->view, c->steps, n_steps, f, dt, pix, st), who);
        JR_CUDA(launch_fold(c->view, st), who);
        c->steps += n_steps;
        return JR_OK;
    }
    if (has_flow && !plain)
        return fail(JR_ERR_STATE, std::string(who) + ": traced and counted advances do not run with a flow attached");
    const bool wave = plain && (has_flow || c->exec == JR_EXEC_WAVEFRONT ||
                                (c->exec == JR_EXEC_AUTO && c->view.n >= kWavefrontMinChains));
    if (plain && use_ahead(c, n_steps, st)) {
        JR_CUDA(run_ahead(c, n_steps, st, nullptr), who);
    } else if (wave) {
        jr_status a = ensure_wavefront(c, st);
        if (a != JR_OK) return a;
        JR_CUDA(launch_wavefront(c->scene_view(), c->view, c->steps, n_steps, st), who);
    } else if (plain && warp_per_chain(c)) {
        JR_CUDA(launch_step_warp(c->scene_view(), c->view, c->steps, n_steps, st), who);
    } else {
        JR_CUDA(launch_step(c->scene_view(), c->view, c->steps, n_steps, f, dt, pix, work, c->block, st), who);
    }
    JR_CUDA(launch_fold(c->view, st), who);
    c->steps += n_steps;
    return JR_OK;
}

jr_status jr_advance(jr_chains* chains, uint32_t n_steps, void* stream) {
    return advance_impl(chains, n_steps, nullptr, nullptr, nullptr, nullptr, stream, "jr_advance");
}

jr_status jr_advance_traced(jr_chains* chains, uint32_t n_steps, uint8_t* flags_dev, float* dt_dev,
                            int32_t* pix_dev, void* stream) {
    return advance_impl(chains, n_steps, flags_dev, dt_dev, pix_dev, nullptr, stream, "jr_advance_traced");
}

jr_status jr_advance_timed(jr_chains* c, uint32_t n_steps, double ms_out[4], uint64_t launches_out[4], void* stream) {
    if (!c || !ms_out || !launches_out) return fail(JR_ERR_INVALID_ARG, "jr_advance_timed: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    const bool wave = c->view.flow.D != 0 || c->exec == JR_EXEC_WAVEFRONT ||
                      (c->exec == JR_EXEC_AUTO && c->view.n >= kWavefrontMinChains);
    KernelTimer tm;
    if (n_steps > 0 && (c->view.flags & JR_FLAG_MALA)) {
        if (use_ahead(c, n_steps, st)) {
            JR_CUDA(run_ahead(c, n_steps, st, &tm), "jr_advance_timed");
        } else {
            JR_CUDA(tm.mark(-1, st), "jr_advance_timed");
            JR_CUDA(launch_step_mala(c->scene_view(), c->view, c->steps, n_steps, nullptr, nullptr, nullptr, st),
                    "jr_advance_timed");
            JR_CUDA(tm.mark(KernelTimer::kStep, st), "jr_advance_timed");
        }
        JR_CUDA(launch_fold(c->view, st), "jr_advance_timed");
        c->steps += n_steps;
    } else if (n_steps > 0) {
        if (use_ahead(c, n_steps, st)) {
            JR_CUDA(run_ahead(c, n_steps, st, &tm), "jr_advance_timed");
        } else if (wave) {
            jr_status a = ensure_wavefront(c, st);
            if (a != JR_OK) return a;
            JR_CUDA(launch_wavefront(c->scene_view(), c->view, c->steps, n_steps, st, kModeStep, &tm),
                    "jr_advance_timed");
        } else {
            JR_CUDA(tm.mark(-1, st), "jr_advance_timed");
            if (warp_per_chain(c))
                JR_CUDA(launch_step_warp(c->scene_view(), c->view, c->steps, n_steps, st), "jr_advance_timed");
            else
                JR_CUDA(launch_step(c->scene_view(), c->view, c->steps, n_steps, nullptr, nullptr, nullptr, nullptr,
                                    c->block, st),
                        "jr_advance_timed");
            JR_CUDA(tm.mark(KernelTimer::kStep, st), "jr_advance_timed");
        }
        JR_CUDA(launch_fold(c->view, st), "jr_advance_timed");
        c->steps += n_steps;
    }
    JR_CUDA(cudaStreamSynchronize(st), "jr_advance_timed");
    JR_CUDA(tm.totals(ms_out, launches_out), "jr_advance_timed");
    return JR_OK;
}

jr_status jr_advance_static(jr_chains* chains, uint32_t n_steps, void* stream) {
    if (!chains) return fail(JR_ERR_INVALID_ARG, "jr_advance_static: null chains");
    if (chains->view.n > kStaticMaxChains)
        return fail(JR_ERR_INVALID_ARG, "jr_advance_static: " + std::to_string(chains->view.n) +
                                            " chains exceed the fixed scratch of " +
                                            std::to_string(kStaticMaxChains) + " chains; use jr_advance");
    if (chains->view.flow.D != 0)
        return fail(JR_ERR_STATE, "jr_advance_static: chains with a flow attached advance with jr_advance");
    if (chains->view.flags & JR_FLAG_MALA)
        return fail(JR_ERR_STATE, "jr_advance_static: MALA chains advance with jr_advance (megakernel)");
    if (n_steps == 0) return JR_OK;
    cudaStream_t st = (cudaStream_t)stream;
    JR_CUDA(launch_wavefront_static(chains->scene_view(), chains->view, chains->steps, n_steps, st),
            "jr_advance_static");
    JR_CUDA(launch_fold(chains->view, st), "jr_advance_static");
    chains->steps += n_steps;
    return JR_OK;
}

jr_status jr_set_execution(jr_chains* chains, uint32_t mode) {
    if (!chains) return fail(JR_ERR_INVALID_ARG, "jr_set_execution: null chains");
    if (mode > JR_EXEC_WARP) return fail(JR_ERR_INVALID_ARG, "jr_set_execution: unknown mode");
    chains->exec = mode;
    return JR_OK;
}

jr_status jr_set_block_size(jr_chains* chains, uint32_t block) {
    if (!chains) return fail(JR_ERR_INVALID_ARG, "jr_set_block_size: null chains");
    if (block < 32 || block > 256 || block % 32 != 0)
        return fail(JR_ERR_INVALID_ARG, "jr_set_block_size: block must be a multiple of 32 in [32, 256]");
    chains->block = (int)block;
    return JR_OK;
}

jr_status jr_chains_set_limits(jr_chains* chains, uint32_t node_visit_budget, uint32_t stack_entries) {
    if (!chains) return fail(JR_ERR_INVALID_ARG, "jr_chains_set_limits: null chains");
    if (stack_entries > (uint32_t)kStackSize)
        return fail(JR_ERR_INVALID_ARG, "jr_chains_set_limits: at most " + std::to_string(kStackSize) +
                                            " stack entries");
    chains->visit_budget = node_visit_budget;
    chains->stack_limit = (int)stack_entries;
    return JR_OK;
}

jr_status jr_debug_fail_alloc(int64_t n) {
    g_fail_alloc_in.store(n < 0 ? -1 : (long long)n);
    return JR_OK;
}

jr_status jr_advance_counted(jr_chains* chains, uint32_t n_steps, uint64_t work_out[3], void* stream) {
    if (!chains || !work_out) return fail(JR_ERR_INVALID_ARG, "jr_advance_counted: null argument");
    unsigned long long* w = nullptr;
    JR_CUDA(dev_alloc(&w, 3), "jr_advance_counted");
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(w, 0, 3 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) {
        cudaFree(w);
        return cuda_fail(e, "jr_advance_counted");
    }
    jr_status s = advance_impl(chains, n_steps, nullptr, nullptr, nullptr, w, stream, "jr_advance_counted");
    unsigned long long h[3] = {0, 0, 0};
    if (s == JR_OK) {
        if ((e = cudaMemcpyAsync(h, w, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
            (e = cudaStreamSynchronize(st)) != cudaSuccess) {
            cudaFree(w);
            return cuda_fail(e, "jr_advance_counted");
        }
        for (int k = 0; k < 3; ++k) work_out[k] = h[k];
    }
    cudaFree(w);
    return s;
}

jr_status jr_resolve(jr_chains* c, float* rgb_out, int out_is_device, void* stream) {
    if (!c || !rgb_out) return fail(JR_ERR_INVALID_ARG, "jr_resolve: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t npx = (size_t)c->view.width * c->view.height;
    if (out_is_device) {
        JR_CUDA(launch_resolve(c->view, rgb_out, mh_samples(c), st), "jr_resolve");
        return JR_OK;
    }
    float* tmp = nullptr;
    JR_CUDA(dev_alloc(&tmp, 3 * npx), "jr_resolve");
    cudaError_t e;
    if ((e = launch_resolve(c->view, tmp, mh_samples(c), st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(rgb_out, tmp, sizeof(float) * 3 * npx, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
        cudaFree(tmp);
        return cuda_fail(e, "jr_resolve");
    }
    cudaFree(tmp);
    return JR_OK;
}

jr_status jr_get_accumulator(jr_chains* c, double* out, int out_is_device, void* stream) {
    if (!c || !out) return fail(JR_ERR_INVALID_ARG, "jr_get_accumulator: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = sizeof(double4_32a) * (size_t)c->view.width * c->view.height;
    JR_CUDA(cudaMemcpyAsync(out, c->view.acc64, bytes, out_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                            st),
            "jr_get_accumulator");
    if (!out_is_device) JR_CUDA(cudaStreamSynchronize(st), "jr_get_accumulator");
    return JR_OK;
}

jr_status jr_get_stats(jr_chains* c, jr_stats* out, void* stream) {
    if (!c || !out) return fail(JR_ERR_INVALID_ARG, "jr_get_stats: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long cnt[kCounters];
    unsigned int status = 0;
    JR_CUDA(cudaMemcpyAsync(cnt, c->view.counters, sizeof(cnt), cudaMemcpyDeviceToHost, st), "jr_get_stats");
    JR_CUDA(cudaMemcpyAsync(&status, c->view.status, sizeof(status), cudaMemcpyDeviceToHost, st), "jr_get_stats");
    JR_CUDA(cudaStreamSynchronize(st), "jr_get_stats");
    out->steps_per_chain = c->steps;
    out->regenerations = cnt[0];
    out->local_steps = cnt[1];
    out->accepted = cnt[2];
    out->status_word = status;
    out->dim = c->view.dim;
    std::memcpy(&out->p_sum_large, &cnt[kCounterPSum], sizeof(double));
    if (status & (JR_STATUS_TRAVERSAL | JR_STATUS_STACK))
        return fail(JR_ERR_WATCHDOG, "jr_get_stats: a ray exhausted the traversal budget or stack");
    if (status & JR_STATUS_NONFINITE) return fail(JR_ERR_NUMERIC, "jr_get_stats: non-finite path contribution");
    return JR_OK;
}

jr_status jr_get_state(jr_chains* c, float* x_out, float* fpu_out, void* stream) {
    if (!c) return fail(JR_ERR_INVALID_ARG, "jr_get_state: null chains");
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t n = c->view.n, D = c->view.dim;
    std::vector<float> pairs;
    if (x_out) {  // the device keeps coordinate pairs (xidx); the caller gets [D][n]
        try {
            pairs.resize((size_t)D * n);
        } catch (const std::bad_alloc&) {
            return fail(JR_ERR_OOM, "jr_get_state: host allocation failed");
        }
        JR_CUDA(cudaMemcpyAsync(pairs.data(), c->view.x, sizeof(float) * D * n, cudaMemcpyDeviceToHost, st),
                "jr_get_state");
    }
    if (fpu_out)
        JR_CUDA(cudaMemcpyAsync(fpu_out, c->view.fpu, sizeof(float) * 5 * n, cudaMemcpyDeviceToHost, st),
                "jr_get_state");
    JR_CUDA(cudaStreamSynchronize(st), "jr_get_state");
    if (x_out)
        for (uint32_t d = 0; d < D; ++d)
            for (uint64_t i = 0; i < n; ++i) x_out[d * n + i] = pairs[xidx(d, i, n)];
    return JR_OK;
}

jr_status jr_set_state(jr_chains* c, const float* x_in, const float* fpu_in, void* stream) {
    if (!c || !x_in) return fail(JR_ERR_INVALID_ARG, "jr_set_state: null argument");
    for (uint64_t k = 0; k < (uint64_t)c->view.dim * c->view.n; ++k)
        if (!(x_in[k] >= 0.0f && x_in[k] < 1.0f)) return fail(JR_ERR_INVALID_ARG, "jr_set_state: x outside [0,1)");
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t n = c->view.n, D = c->view.dim;
    std::vector<float> pairs;
    try {
        pairs.resize((size_t)D * n);
    } catch (const std::bad_alloc&) {
        return fail(JR_ERR_OOM, "jr_set_state: host allocation failed");
    }
    for (uint32_t d = 0; d < D; ++d)
        for (uint64_t i = 0; i < n; ++i) pairs[xidx(d, i, n)] = x_in[d * n + i];
    JR_CUDA(cudaMemcpyAsync(c->view.x, pairs.data(), sizeof(float) * D * n, cudaMemcpyHostToDevice, st),
            "jr_set_state");
    if (c->view.flags & JR_FLAG_MALA)  // F, p and the drift from the states themselves
        JR_CUDA(launch_mala_reeval(c->scene_view(), c->view, st), "jr_set_state");
    else if (fpu_in)
        JR_CUDA(cudaMemcpyAsync(c->view.fpu, fpu_in, sizeof(float) * 5 * c->view.n, cudaMemcpyHostToDevice, st),
                "jr_set_state");
    else
        JR_CUDA(launch_reeval(c->scene_view(), c->view, st), "jr_set_state");
    JR_CUDA(cudaStreamSynchronize(st), "jr_set_state");
    return JR_OK;
}

jr_status jr_set_counters(jr_chains* c, const jr_stats* in, const double* acc_host, void* stream) {
    if (!c || !in) return fail(JR_ERR_INVALID_ARG, "jr_set_counters: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long cnt[kCounters] = {in->regenerations, in->local_steps, in->accepted, 0, 0, 0, 0, 0};
    std::memcpy(&cnt[kCounterPSum], &in->p_sum_large, sizeof(double));
    unsigned int status = in->status_word;
    // all but kCounterMuP, which belongs to the set and not to the run
    JR_CUDA(cudaMemcpyAsync(c->view.counters, cnt, sizeof(cnt[0]) * kCounterMuP, cudaMemcpyHostToDevice, st),
            "jr_set_counters");
    JR_CUDA(cudaMemcpyAsync(c->view.counters + kCounterMuP + 1, cnt + kCounterMuP + 1,
                            sizeof(cnt[0]) * (kCounters - kCounterMuP - 1), cudaMemcpyHostToDevice, st),
            "jr_set_counters");
    JR_CUDA(cudaMemcpyAsync(c->view.status, &status, sizeof(status), cudaMemcpyHostToDevice, st), "jr_set_counters");
    if (acc_host)
        JR_CUDA(cudaMemcpyAsync(c->view.acc64, acc_host, sizeof(double4_32a) * (size_t)c->view.width * c->view.height,
                                cudaMemcpyHostToDevice, st),
                "jr_set_counters");
    JR_CUDA(cudaStreamSynchronize(st), "jr_set_counters");
    c->steps = in->steps_per_chain;
    return JR_OK;
}

jr_status jr_eval_states(const jr_scene* scene, const jr_params* params, const float* x_dev, uint64_t n, float* F_dev,
                         float* p_dev, float* u_dev, float* k_dev, int32_t* hit_ids_dev, void* stream) {
    if (!scene || !params || (n > 0 && !x_dev)) return fail(JR_ERR_INVALID_ARG, "jr_eval_states: null argument");
    if (params->max_depth > JR_MAX_DEPTH) return fail(JR_ERR_INVALID_ARG, "jr_eval_states: max_depth > 15");
    if (!(params->c_tilde > 0.f)) return fail(JR_ERR_INVALID_ARG, "jr_eval_states: c_tilde must be > 0");
    JR_CUDA(launch_eval_states(scene->view, params->max_depth, params->c_tilde, x_dev, n, F_dev, p_dev, u_dev, k_dev,
                               hit_ids_dev, (cudaStream_t)stream),
            "jr_eval_states");
    return JR_OK;
}

jr_status jr_eval_grad(const jr_scene* scene, const jr_params* params, const float* x_dev, uint64_t n, float* F_dev,
                       float* dF_dev, void* stream) {
    if (!scene || !params || (n > 0 && !x_dev)) return fail(JR_ERR_INVALID_ARG, "jr_eval_grad: null argument");
    if (params->max_depth > JR_MAX_DEPTH) return fail(JR_ERR_INVALID_ARG, "jr_eval_grad: max_depth > 15");
    JR_CUDA(launch_eval_grad(scene->view, params->max_depth, x_dev, n, F_dev, dF_dev, (cudaStream_t)stream),
            "jr_eval_grad");
    return JR_OK;
}

jr_status jr_render_pt(const jr_scene* scene, const jr_params* params, uint64_t sample_begin, uint64_t n_samples,
                       double* accum_dev, void* stream) {
    if (!scene || !params || !accum_dev) return fail(JR_ERR_INVALID_ARG, "jr_render_pt: null argument");
    if (params->width == 0 || params->height == 0 || params->max_depth > JR_MAX_DEPTH)
        return fail(JR_ERR_INVALID_ARG, "jr_render_pt: bad image size or depth");
    JR_CUDA(launch_render_pt(scene->view, params->width, params->height, params->max_depth, params->seed, sample_begin,
                             n_samples, accum_dev, (cudaStream_t)stream),
            "jr_render_pt");
    return JR_OK;
}

jr_status jr_fp32_peak(double* tflops_out, double* ms_out, void* stream) {
    if (!tflops_out) return fail(JR_ERR_INVALID_ARG, "jr_fp32_peak: null output");
    JR_CUDA(measure_fma_peak(tflops_out, ms_out, (cudaStream_t)stream), "jr_fp32_peak");
    return JR_OK;
}

jr_status jr_philox(uint64_t seed, uint32_t tag, uint32_t block, uint64_t chain_begin, uint64_t step, uint64_t n,
                    uint32_t* out_dev, void* stream) {
    if (n > 0 && !out_dev) return fail(JR_ERR_INVALID_ARG, "jr_philox: null output");
    JR_CUDA(launch_philox(seed, tag, block, chain_begin, step, n, out_dev, (cudaStream_t)stream), "jr_philox");
    return JR_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batches: many chain sets (scenes of uneven size, images, depths) advanced by
// one persistent launch, optionally replayed from a captured CUDA graph.
struct jr_batch {
    std::vector<jr_chains*> sets;
    std::vector<uint64_t> dev_steps;  // the step index each set has on the device side
    std::vector<uint64_t> dev_flow_gen;  // the flow generation of each set's device descriptor
    BatchEntry* entries = nullptr;
    uint64_t* px_off = nullptr;
    unsigned int* cursor = nullptr;
    BatchItem* items = nullptr;
    size_t items_cap = 0;
    uint32_t n_items = 0;
    uint32_t max_dim = 0;
    uint64_t total_px = 0, total_chains = 0;
    int block = 128;  // chains per megakernel work item; 0: the batched wavefront
    int checks = 0;   // the watchdogs the megakernel checks: the most that any set's device descriptor needs
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint32_t graph_steps = 0;
    int graph_block = -1;
    // the batched wavefront, set up on first use: the merged scene, roots,
    // chain prefix sums, step-launch work items, the path launches' cursor
    Bvh4Node* m_nodes = nullptr;
    TriRecord* m_tris = nullptr;
    Material* m_mats = nullptr;
    int* roots = nullptr;
    uint64_t* chain_off = nullptr;
    BatchItem* wf_items = nullptr;
    unsigned int* fetch = nullptr;
    BatchWave bw{};
    bool wf_ready = false;
    void drop_graph() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
    }
    // A set's device descriptor gets view v (a captured graph holds the old variant).
    void needs(const SceneView& v) {
        if (trav_checks(v) <= checks) return;
        checks = trav_checks(v);
        drop_graph();
    }
    ~jr_batch() {
        drop_graph();
        cudaFree(entries);
        cudaFree(px_off);
        cudaFree(cursor);
        cudaFree(items);
        cudaFree(m_nodes);
        cudaFree(m_tris);
        cudaFree(m_mats);
        cudaFree(roots);
        cudaFree(chain_off);
        cudaFree(wf_items);
        cudaFree(fetch);
    }
};

namespace {

// Work items: blocks of `block` chains, most expensive first (a chain step
// costs about (depth + 1) ray casts of log(triangles) traversal depth).
jr_status build_items(jr_batch* b, int block, cudaStream_t st) {
    struct Cand {
        double cost;
        BatchItem it;
    };
    std::vector<Cand> v;
    for (uint32_t k = 0; k < b->sets.size(); ++k) {
        const jr_chains* c = b->sets[k];
        const double per_chain = (c->view.depth + 1.0) * std::log2(c->scene->info.n_tris + 2.0);
        for (uint64_t beg = 0; beg < c->view.n; beg += (uint64_t)block) {
            const uint64_t end = std::min<uint64_t>(beg + block, c->view.n);
            v.push_back({per_chain * (double)(end - beg), BatchItem{k, (uint32_t)beg, (uint32_t)end}});
        }
    }
    std::stable_sort(v.begin(), v.end(), [](const Cand& a, const Cand& c) { return a.cost > c.cost; });
    std::vector<BatchItem> h(v.size());
    for (size_t q = 0; q < v.size(); ++q) h[q] = v[q].it;
    if (h.size() > b->items_cap) {
        cudaFree(b->items);
        b->items = nullptr;
        b->items_cap = 0;
        JR_CUDA(dev_alloc(&b->items, h.size()), "jr_batch (work items)");
        b->items_cap = h.size();
    }
    JR_CUDA(cudaMemcpyAsync(b->items, h.data(), sizeof(BatchItem) * h.size(), cudaMemcpyHostToDevice, st),
            "jr_batch (work items)");
    JR_CUDA(cudaStreamSynchronize(st), "jr_batch (work items)");
    b->n_items = (uint32_t)h.size();
    b->block = block;
    return JR_OK;
}

bool batch_has_flow(const jr_batch* b) {
    for (const jr_chains* c : b->sets)
        if (c->view.flow.D != 0) return true;
    return false;
}

// The host views of the sets with a flow attached (their flow launches).
std::vector<ChainView> flow_views(const jr_batch* b) {
    std::vector<ChainView> v;
    for (const jr_chains* c : b->sets)
        if (c->view.flow.D != 0) v.push_back(c->view);
    return v;
}

// Bring the device-side step index of every set up to date with its host
// counter (a set may have been advanced on its own since the last batch), and
// a set's device descriptor with its flow when jr_chains_set_flow changed it
// (a captured graph holds the old flow's launches, so it is dropped).
jr_status sync_steps(jr_batch* b, cudaStream_t st) {
    for (size_t k = 0; k < b->sets.size(); ++k) {
        const jr_chains* c = b->sets[k];
        if (c->flow_gen != b->dev_flow_gen[k]) {
            BatchEntry h{};
            h.s = c->scene_view();
            h.c = c->view;
            h.step = c->steps;
            JR_CUDA(cudaMemcpyAsync(b->entries + k, &h, sizeof(h), cudaMemcpyHostToDevice, st), "jr_batch (flow)");
            JR_CUDA(cudaStreamSynchronize(st), "jr_batch (flow)");
            b->dev_flow_gen[k] = c->flow_gen;
            b->dev_steps[k] = c->steps;
            b->needs(h.s);
            b->drop_graph();
        }
        const uint64_t s = b->sets[k]->steps;
        if (s != b->dev_steps[k]) {
            unsigned long long v = s;
            JR_CUDA(cudaMemcpyAsync(reinterpret_cast<char*>(b->entries + k) + offsetof(BatchEntry, step), &v,
                                    sizeof(v), cudaMemcpyHostToDevice, st),
                    "jr_batch (step index)");
            JR_CUDA(cudaStreamSynchronize(st), "jr_batch (step index)");
            b->dev_steps[k] = s;
        }
    }
    return JR_OK;
}

void after_launch(jr_batch* b, uint32_t n_steps) {
    for (size_t k = 0; k < b->sets.size(); ++k) {
        b->sets[k]->steps += n_steps;
        b->dev_steps[k] += n_steps;
    }
}

// Set up the batched wavefront once: every set's wavefront buffers (and the
// device descriptors that point at them), the merged scene (each distinct
// scene copied once and rebased), the sets' roots in it, the chain prefix
// sums and the step launches' work items.
jr_status prepare_wave(jr_batch* b, cudaStream_t st) {
    if (b->wf_ready) return JR_OK;
    const uint32_t S = (uint32_t)b->sets.size();
    if (S > kBatchMaxSets)
        return fail(JR_ERR_INVALID_ARG, "jr_batch: the batched wavefront takes at most " +
                                            std::to_string(kBatchMaxSets) + " sets");
    for (jr_chains* c : b->sets) {
        jr_status a = ensure_wavefront(c, st);
        if (a != JR_OK) return a;
    }
    std::vector<BatchEntry> h(S);
    std::vector<const jr_scene*> uniq;
    std::vector<uint64_t> noff, toff, moff;  // per distinct scene
    uint64_t nn = 0, nt = 0, nm = 0;
    std::vector<int> root(S);
    std::vector<uint64_t> coff(S + 1, 0);
    std::vector<BatchItem> items;
    for (uint32_t k = 0; k < S; ++k) {
        const jr_chains* c = b->sets[k];
        h[k].s = c->scene_view();
        b->needs(h[k].s);
        h[k].c = c->view;
        h[k].step = b->dev_steps[k];
        size_t u = 0;
        while (u < uniq.size() && uniq[u] != c->scene) ++u;
        if (u == uniq.size()) {
            uniq.push_back(c->scene);
            noff.push_back(nn);
            toff.push_back(nt);
            moff.push_back(nm);
            nn += (uint64_t)c->scene->view.n_nodes;
            nt += c->scene->info.n_tris;
            nm += c->scene->info.n_materials;
        }
        root[k] = rebase_ref(c->scene->view.root, (int)noff[u], (int)toff[u]);
        coff[k + 1] = coff[k] + c->view.n;
        for (uint64_t beg = 0; beg < c->view.n; beg += 128)
            items.push_back(BatchItem{k, (uint32_t)beg, (uint32_t)std::min<uint64_t>(beg + 128, c->view.n)});
    }
    if (nt >= (1ull << 28) || nn >= (1ull << 31) || coff[S] >= (1ull << 31))
        return fail(JR_ERR_INVALID_ARG, "jr_batch: the merged scene or the chain count is too large for the "
                                        "batched wavefront (2^28 triangles, 2^31 nodes or chains)");
    const char* who = "jr_batch (batched wavefront set-up)";
    // a set-up that failed part way may have left buffers: free them first
    cudaFree(b->m_nodes);
    cudaFree(b->m_tris);
    cudaFree(b->m_mats);
    cudaFree(b->roots);
    cudaFree(b->chain_off);
    cudaFree(b->wf_items);
    cudaFree(b->fetch);
    b->m_nodes = nullptr;
    b->m_tris = nullptr;
    b->m_mats = nullptr;
    b->roots = nullptr;
    b->chain_off = nullptr;
    b->wf_items = nullptr;
    b->fetch = nullptr;
    JR_CUDA(dev_alloc(&b->m_nodes, std::max<uint64_t>(nn, 1)), who);
    JR_CUDA(dev_alloc(&b->m_tris, std::max<uint64_t>(nt, 1)), who);
    JR_CUDA(dev_alloc(&b->m_mats, std::max<uint64_t>(nm, 1)), who);
    JR_CUDA(dev_alloc(&b->roots, S), who);
    JR_CUDA(dev_alloc(&b->chain_off, S + 1), who);
    JR_CUDA(dev_alloc(&b->wf_items, std::max<size_t>(items.size(), 1)), who);
    JR_CUDA(dev_alloc(&b->fetch, 1), who);
    for (size_t u = 0; u < uniq.size(); ++u) {
        const jr_scene* sc = uniq[u];
        const uint32_t n_nodes = (uint32_t)sc->view.n_nodes, n_tris = sc->info.n_tris,
                       n_mats = sc->info.n_materials;
        if (n_nodes)
            JR_CUDA(cudaMemcpyAsync(b->m_nodes + noff[u], sc->nodes, sizeof(Bvh4Node) * n_nodes,
                                    cudaMemcpyDeviceToDevice, st),
                    who);
        if (n_tris)
            JR_CUDA(cudaMemcpyAsync(b->m_tris + toff[u], sc->tris, sizeof(TriRecord) * n_tris,
                                    cudaMemcpyDeviceToDevice, st),
                    who);
        if (n_mats)
            JR_CUDA(cudaMemcpyAsync(b->m_mats + moff[u], sc->mats, sizeof(Material) * n_mats,
                                    cudaMemcpyDeviceToDevice, st),
                    who);
        JR_CUDA(launch_rebase_scene(b->m_nodes + noff[u], n_nodes, b->m_tris + toff[u], n_tris, (int)noff[u],
                                    (int)toff[u], (int)moff[u], st),
                who);
    }
    JR_CUDA(cudaMemcpyAsync(b->entries, h.data(), sizeof(BatchEntry) * S, cudaMemcpyHostToDevice, st), who);
    JR_CUDA(cudaMemcpyAsync(b->roots, root.data(), sizeof(int) * S, cudaMemcpyHostToDevice, st), who);
    JR_CUDA(cudaMemcpyAsync(b->chain_off, coff.data(), sizeof(uint64_t) * (S + 1), cudaMemcpyHostToDevice, st), who);
    if (!items.empty())
        JR_CUDA(cudaMemcpyAsync(b->wf_items, items.data(), sizeof(BatchItem) * items.size(), cudaMemcpyHostToDevice,
                                st),
                who);
    JR_CUDA(cudaStreamSynchronize(st), who);
    BatchWave& bw = b->bw;
    bw.merged = SceneView{};
    bw.merged.nodes = b->m_nodes;
    bw.merged.tris = b->m_tris;
    bw.merged.mats = b->m_mats;
    bw.merged.root = kNoChild;
    bw.merged.n_nodes = (int)nn;
    bw.merged.n_tris = (uint32_t)nt;
    bw.merged.visit_budget = kNodeVisitBudget;
    bw.merged.stack_limit = kStackSize;
    bw.roots = b->roots;
    bw.chain_off = b->chain_off;
    bw.items = b->wf_items;
    bw.n_sets = S;
    bw.n_items = (uint32_t)items.size();
    bw.fetch = b->fetch;
    long long blocks = 0;
    bw.checks = 0;  // the merged scene is traversed under the default limits
    for (const jr_scene* sc : uniq) bw.checks = std::max(bw.checks, trav_checks(sc->view));
    JR_CUDA(batch_wavefront_grid(bw.checks, &blocks), who);
    b->wf_ready = true;
    return JR_OK;
}

// Enqueue one batch advance (no allocation, so it can be captured): the
// megakernel launch, or the batched wavefront's launches; then the fold,
// which also moves every set's device step index on by n_steps.
cudaError_t enqueue_batch(jr_batch* b, uint32_t n_steps, cudaStream_t st) {
    const uint32_t S = (uint32_t)b->sets.size();
    if (b->block == 0) {
        cudaError_t e = launch_batch_wavefront(b->bw, b->entries, n_steps, flow_views(b), st);
        if (e != cudaSuccess) return e;
        return launch_batch(b->entries, b->items, 0, b->px_off, S, b->total_px, b->cursor, b->max_dim, 128,
                            b->checks, n_steps, st);
    }
    return launch_batch(b->entries, b->items, b->n_items, b->px_off, S, b->total_px, b->cursor, b->max_dim, b->block,
                        b->checks, n_steps, st);
}

jr_status batch_launch(jr_batch* b, uint32_t n_steps, cudaStream_t st, const char* who) {
    if (b->block != 0 && batch_has_flow(b))
        return fail(JR_ERR_STATE, std::string(who) + ": a set has a flow attached; select JR_BATCH_WAVEFRONT");
    if (b->block == 0) {
        jr_status a = prepare_wave(b, st);
        if (a != JR_OK) return a;
    }
    JR_CUDA(enqueue_batch(b, n_steps, st), who);
    return JR_OK;
}

}  // namespace

extern "C" {

jr_status jr_batch_create(jr_chains* const* sets, uint32_t n_sets, void* stream, jr_batch** out) {
    if (!sets || !out || n_sets == 0) return fail(JR_ERR_INVALID_ARG, "jr_batch_create: null argument or no sets");
    cudaStream_t st = (cudaStream_t)stream;
    jr_batch* b = new (std::nothrow) jr_batch();
    if (!b) return fail(JR_ERR_OOM, "jr_batch_create: host allocation failed");
    std::vector<BatchEntry> h(n_sets);
    std::vector<uint64_t> off(n_sets + 1, 0);
    for (uint32_t k = 0; k < n_sets; ++k) {
        jr_chains* c = sets[k];
        if (!c) {
            delete b;
            return fail(JR_ERR_INVALID_ARG, "jr_batch_create: null chain set");
        }
        for (uint32_t q = 0; q < k; ++q)
            if (sets[q] == c) {
                delete b;
                return fail(JR_ERR_INVALID_ARG, "jr_batch_create: a chain set appears twice");
            }
        if (c->view.flags & JR_FLAG_MALA) {
            delete b;
            return fail(JR_ERR_STATE, "jr_batch_create: MALA chain sets advance on their own (megakernel)");
        }
        h[k].s = c->scene_view();
        b->needs(h[k].s);
        h[k].c = c->view;
        h[k].step = c->steps;
        off[k + 1] = off[k] + (uint64_t)c->view.width * c->view.height;
        b->max_dim = std::max(b->max_dim, c->view.dim);
        b->total_chains += c->view.n;
        b->sets.push_back(c);
        b->dev_steps.push_back(c->steps);
        b->dev_flow_gen.push_back(c->flow_gen);
    }
    b->total_px = off[n_sets];
    cudaError_t e;
    if ((e = dev_alloc(&b->entries, n_sets)) != cudaSuccess || (e = dev_alloc(&b->px_off, n_sets + 1)) != cudaSuccess ||
        (e = dev_alloc(&b->cursor, 1)) != cudaSuccess ||
        (e = cudaMemcpyAsync(b->entries, h.data(), sizeof(BatchEntry) * n_sets, cudaMemcpyHostToDevice, st)) !=
            cudaSuccess ||
        (e = cudaMemcpyAsync(b->px_off, off.data(), sizeof(uint64_t) * (n_sets + 1), cudaMemcpyHostToDevice, st)) !=
            cudaSuccess ||
        (e = cudaMemsetAsync(b->cursor, 0, sizeof(unsigned int), st)) != cudaSuccess) {
        delete b;
        return cuda_fail(e, "jr_batch_create");
    }
    jr_status r = build_items(b, 128, st);
    if (r == JR_OK && batch_has_flow(b)) b->block = 0;  // sets with a flow advance in the batched wavefront only
    if (r == JR_OK) r = batch_launch(b, 0, st, "jr_batch_create");  // set-up launch: no steps
    if (r != JR_OK) {
        delete b;
        return r;
    }
    *out = b;
    return JR_OK;
}

void jr_batch_destroy(jr_batch* batch) { delete batch; }

jr_status jr_batch_set_block(jr_batch* b, uint32_t block) {
    if (!b) return fail(JR_ERR_INVALID_ARG, "jr_batch_set_block: null batch");
    if (block == JR_BATCH_WAVEFRONT) {
        b->block = 0;
        return JR_OK;
    }
    if (block < 32 || block > 256 || block % 32 != 0)
        return fail(JR_ERR_INVALID_ARG,
                    "jr_batch_set_block: block must be a multiple of 32 in [32, 256], or JR_BATCH_WAVEFRONT");
    if (batch_has_flow(b))
        return fail(JR_ERR_STATE, "jr_batch_set_block: sets with a flow attached advance in the batched wavefront");
    return build_items(b, (int)block, nullptr);
}

jr_status jr_batch_advance(jr_batch* b, uint32_t n_steps, void* stream) {
    if (!b) return fail(JR_ERR_INVALID_ARG, "jr_batch_advance: null batch");
    if (n_steps == 0) return JR_OK;
    cudaStream_t st = (cudaStream_t)stream;
    jr_status r = sync_steps(b, st);
    if (r == JR_OK) r = batch_launch(b, n_steps, st, "jr_batch_advance");
    if (r == JR_OK) after_launch(b, n_steps);
    return r;
}

jr_status jr_batch_advance_graph(jr_batch* b, uint32_t n_steps, void* stream) {
    if (!b) return fail(JR_ERR_INVALID_ARG, "jr_batch_advance_graph: null batch");
    if (n_steps == 0) return JR_OK;
    cudaStream_t st = (cudaStream_t)stream;
    jr_status r = sync_steps(b, st);
    if (r == JR_OK && b->block != 0 && batch_has_flow(b))
        r = fail(JR_ERR_STATE, "jr_batch_advance_graph: a set has a flow attached; select JR_BATCH_WAVEFRONT");
    if (r == JR_OK && b->block == 0) r = prepare_wave(b, st);
    if (r != JR_OK) return r;
    if (!b->exec || b->graph_steps != n_steps || b->graph_block != b->block) {
        b->drop_graph();
        cudaStream_t cap = nullptr;
        JR_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "jr_batch_advance_graph");
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaError_t el = enqueue_batch(b, n_steps, cap);
            e = cudaStreamEndCapture(cap, &b->graph);
            if (e == cudaSuccess) e = el;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        cudaStreamDestroy(cap);
        if (e != cudaSuccess) {
            if (b->graph) cudaGraphDestroy(b->graph);
            b->graph = nullptr;
            b->exec = nullptr;
            return cuda_fail(e, "jr_batch_advance_graph (capture)");
        }
        b->graph_steps = n_steps;
        b->graph_block = b->block;
    }
    JR_CUDA(cudaGraphLaunch(b->exec, st), "jr_batch_advance_graph");
    after_launch(b, n_steps);
    return JR_OK;
}

jr_status jr_batch_autotune(jr_batch* b, uint32_t probe_steps, void* stream, jr_tune_report* out) {
    if (!b || !out || probe_steps == 0) return fail(JR_ERR_INVALID_ARG, "jr_batch_autotune: bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    const bool flows = batch_has_flow(b);  // only the batched wavefront runs flows
    const uint32_t all[] = {32, 64, 128, 256, JR_BATCH_WAVEFRONT}, wave_only[] = {JR_BATCH_WAVEFRONT};
    const uint32_t* cands = flows ? wave_only : all;
    const uint32_t n_cands = flows ? 1 : b->sets.size() <= kBatchMaxSets ? 5 : 4;
    jr_tune_report rep{};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    JR_CUDA(cudaEventCreate(&e0), "jr_batch_autotune");
    JR_CUDA(cudaEventCreate(&e1), "jr_batch_autotune");
    double best = INFINITY;
    jr_status r = JR_OK;
    for (uint32_t q = 0; q < n_cands && r == JR_OK; ++q) {
        if (cands[q] == JR_BATCH_WAVEFRONT) {
            b->block = 0;
            r = prepare_wave(b, st);  // one-time set-up, outside the timed probe
        } else {
            r = build_items(b, (int)cands[q], st);
        }
        if (r == JR_OK) r = sync_steps(b, st);
        if (r != JR_OK) break;
        cudaError_t e;
        if ((e = cudaEventRecord(e0, st)) != cudaSuccess) {
            r = cuda_fail(e, "jr_batch_autotune");
            break;
        }
        r = batch_launch(b, probe_steps, st, "jr_batch_autotune");
        if (r != JR_OK) break;
        after_launch(b, probe_steps);
        float ms = 0.f;
        if ((e = cudaEventRecord(e1, st)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess ||
            (e = cudaEventElapsedTime(&ms, e0, e1)) != cudaSuccess) {
            r = cuda_fail(e, "jr_batch_autotune");
            break;
        }
        const double ns = 1e6 * ms / ((double)b->total_chains * probe_steps);
        rep.block[rep.n] = cands[q];
        rep.ns_per_chain_step[rep.n] = ns;
        rep.n++;
        if (ns < best) {
            best = ns;
            rep.best_block = cands[q];
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (r != JR_OK) return r;
    if (rep.best_block == JR_BATCH_WAVEFRONT) {
        b->block = 0;
    } else {
        r = build_items(b, (int)rep.best_block, st);
        if (r != JR_OK) return r;
    }
    *out = rep;
    return JR_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// The learned regeneration flow (jr_flow.cu): parameters, evaluation, and the
// attachment to a chain set.
struct jr_flow {
    uint32_t D = 0, A = 0, AK = 0;
    uint8_t* perm = nullptr;       // [kFL][D]
    float* master = nullptr;       // [kFL][S] FP32, the documented layout
    __nv_bfloat16* wb = nullptr;   // packed bf16 weights
    float* bias = nullptr;         // packed FP32 biases
    unsigned char* ws = nullptr;   // inference layout
    unsigned int* status = nullptr;  // JR_STATUS_* bits of the flow's own launches
    float* adam_m = nullptr;       // optimiser moments [kFL][S]
    float* adam_v = nullptr;
    float* grad = nullptr;         // [kFL][S] gradient accumulator
    uint64_t adam_t = 0;
    uint32_t extra_tx = 0;  // testing hook, see jr_debug_flow_wait
    FlowView view(float beta) const {
        FlowView f;
        f.extra_tx = extra_tx;
        f.D = D;
        f.A = A;
        f.AK = AK;
        f.perm = perm;
        f.wb = wb;
        f.bias = bias;
        f.ws = ws;
        f.beta = beta;
        return f;
    }
    ~jr_flow() {
        cudaFree(perm);
        cudaFree(master);
        cudaFree(wb);
        cudaFree(bias);
        cudaFree(ws);
        cudaFree(status);
        cudaFree(adam_m);
        cudaFree(adam_v);
        cudaFree(grad);
    }
};

extern "C" {

uint64_t jr_flow_param_count(uint32_t dim) {
    if (dim < 2 || dim > (uint32_t)kMaxDim || dim % 2) return 0;
    return (uint64_t)kFL * flow_layer_floats(dim);
}

namespace {
// Both packed copies of the master parameters: the training layout and the
// inference layout.
cudaError_t pack_all(jr_flow* f, cudaStream_t st) {
    cudaError_t e = launch_flow_pack(f->master, f->wb, f->bias, f->AK, st);
    return e != cudaSuccess ? e : launch_flow_pack_ws(f->master, f->ws, f->AK, st);
}
}  // namespace

jr_status jr_flow_create(uint32_t dim, const int32_t* perm, const float* params, void* stream, jr_flow** out) {
    if (!perm || !params || !out) return fail(JR_ERR_INVALID_ARG, "jr_flow_create: null argument");
    if (dim < 2 || dim > (uint32_t)kMaxDim || dim % 2)
        return fail(JR_ERR_INVALID_ARG, "jr_flow_create: dim must be even, 2..32");
    std::vector<uint8_t> pm((size_t)kFL * dim);
    for (int l = 0; l < kFL; ++l) {
        std::vector<int> seen(dim, 0);
        for (uint32_t d = 0; d < dim; ++d) {
            const int32_t v = perm[l * dim + d];
            if (v < 0 || (uint32_t)v >= dim || seen[v]++)
                return fail(JR_ERR_INVALID_ARG, "jr_flow_create: perm[l] must be a permutation of 0..dim-1");
            pm[l * dim + d] = (uint8_t)v;
        }
    }
    jr_flow* f = new (std::nothrow) jr_flow();
    if (!f) return fail(JR_ERR_OOM, "jr_flow_create: host allocation failed");
    f->D = dim;
    f->A = dim / 2;
    f->AK = f->A * kFK;
    const size_t S = flow_layer_floats(dim), P = (size_t)kFL * S;
    const size_t nwb = (size_t)kFL * (kFH * kFS1 + kFH * kFS2 + (size_t)f->AK * kFS2);
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    if ((e = dev_alloc(&f->perm, pm.size())) != cudaSuccess || (e = dev_alloc(&f->master, P)) != cudaSuccess ||
        (e = dev_alloc(&f->wb, nwb)) != cudaSuccess ||
        (e = dev_alloc(&f->bias, (size_t)kFL * (2 * kFH + f->AK))) != cudaSuccess ||
        (e = dev_alloc(&f->ws, (size_t)kFL * flow_ws_layer_bytes(f->AK))) != cudaSuccess ||
        (e = dev_alloc(&f->status, 1)) != cudaSuccess ||
        (e = cudaMemsetAsync(f->status, 0, sizeof(unsigned int), st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(f->perm, pm.data(), pm.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(f->master, params, sizeof(float) * P, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
        (e = pack_all(f, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
        delete f;
        return cuda_fail(e, "jr_flow_create");
    }
    *out = f;
    return JR_OK;
}

void jr_flow_destroy(jr_flow* flow) { delete flow; }

jr_status jr_flow_set_params(jr_flow* f, const float* params, void* stream) {
    if (!f || !params) return fail(JR_ERR_INVALID_ARG, "jr_flow_set_params: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    JR_CUDA(cudaMemcpyAsync(f->master, params, sizeof(float) * kFL * flow_layer_floats(f->D), cudaMemcpyHostToDevice,
                            st),
            "jr_flow_set_params");
    JR_CUDA(pack_all(f, st), "jr_flow_set_params");
    JR_CUDA(cudaStreamSynchronize(st), "jr_flow_set_params");
    return JR_OK;
}

jr_status jr_flow_get_status(jr_flow* f, uint32_t* status_out, void* stream) {
    if (!f || !status_out) return fail(JR_ERR_INVALID_ARG, "jr_flow_get_status: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned int v = 0;
    JR_CUDA(cudaMemcpyAsync(&v, f->status, sizeof(v), cudaMemcpyDeviceToHost, st), "jr_flow_get_status");
    JR_CUDA(cudaStreamSynchronize(st), "jr_flow_get_status");
    *status_out = v;
    return JR_OK;
}

jr_status jr_debug_flow_wait(jr_flow* f, int enable) {
    if (!f) return fail(JR_ERR_INVALID_ARG, "jr_debug_flow_wait: null flow");
    f->extra_tx = enable ? 16u : 0u;
    return JR_OK;
}

jr_status jr_flow_get_params(jr_flow* f, float* params, void* stream) {
    if (!f || !params) return fail(JR_ERR_INVALID_ARG, "jr_flow_get_params: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    JR_CUDA(cudaMemcpyAsync(params, f->master, sizeof(float) * kFL * flow_layer_floats(f->D), cudaMemcpyDeviceToHost,
                            st),
            "jr_flow_get_params");
    JR_CUDA(cudaStreamSynchronize(st), "jr_flow_get_params");
    return JR_OK;
}

jr_status jr_flow_log_density(jr_flow* f, const float* x_dev, uint64_t n, float* lq_dev, void* stream) {
    if (!f || (n > 0 && (!x_dev || !lq_dev))) return fail(JR_ERR_INVALID_ARG, "jr_flow_log_density: null argument");
    if (n >= (1ull << 32)) return fail(JR_ERR_INVALID_ARG, "jr_flow_log_density: n must be below 2^32");
    JR_CUDA(launch_flow(f->view(0.f), false, const_cast<float*>(x_dev), nullptr, nullptr, n, nullptr, nullptr,
                        (uint32_t)n, nullptr, lq_dev, nullptr, f->status, (cudaStream_t)stream),
            "jr_flow_log_density");
    return JR_OK;
}

jr_status jr_flow_sample(jr_flow* f, float* xz_dev, uint64_t n, float* lq_dev, void* stream) {
    if (!f || (n > 0 && (!xz_dev || !lq_dev))) return fail(JR_ERR_INVALID_ARG, "jr_flow_sample: null argument");
    if (n >= (1ull << 32)) return fail(JR_ERR_INVALID_ARG, "jr_flow_sample: n must be below 2^32");
    JR_CUDA(launch_flow(f->view(0.f), true, xz_dev, nullptr, nullptr, n, nullptr, nullptr, (uint32_t)n, nullptr,
                        lq_dev, nullptr, f->status, (cudaStream_t)stream),
            "jr_flow_sample");
    return JR_OK;
}

jr_status jr_flow_copy_params(jr_flow* dst, const jr_flow* src, void* stream) {
    if (!dst || !src) return fail(JR_ERR_INVALID_ARG, "jr_flow_copy_params: null argument");
    if (dst->D != src->D) return fail(JR_ERR_INVALID_ARG, "jr_flow_copy_params: dimensions differ");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t P = (size_t)kFL * flow_layer_floats(src->D);
    JR_CUDA(cudaMemcpyAsync(dst->perm, src->perm, (size_t)kFL * src->D, cudaMemcpyDeviceToDevice, st),
            "jr_flow_copy_params");
    JR_CUDA(cudaMemcpyAsync(dst->master, src->master, sizeof(float) * P, cudaMemcpyDeviceToDevice, st),
            "jr_flow_copy_params");
    JR_CUDA(pack_all(dst, st), "jr_flow_copy_params");
    return JR_OK;
}

jr_status jr_chains_snapshot(jr_chains* c, float* x_dev, float* w_dev, void* stream) {
    if (!c || !x_dev || !w_dev) return fail(JR_ERR_INVALID_ARG, "jr_chains_snapshot: null argument");
    JR_CUDA(launch_snapshot(c->view, x_dev, w_dev, (cudaStream_t)stream), "jr_chains_snapshot");
    return JR_OK;
}

jr_status jr_chains_snapshot_append(jr_chains* c, float* x_ring, float* w_ring, uint64_t capacity,
                                    unsigned long long* total_dev, void* stream) {
    if (!c || !x_ring || !w_ring || !total_dev) return fail(JR_ERR_INVALID_ARG, "jr_chains_snapshot_append: null argument");
    if (capacity == 0) return fail(JR_ERR_INVALID_ARG, "jr_chains_snapshot_append: capacity must be > 0");
    JR_CUDA(launch_snapshot_append(c->view, x_ring, w_ring, capacity, total_dev, (cudaStream_t)stream),
            "jr_chains_snapshot_append");
    return JR_OK;
}

jr_status jr_flow_gradient(jr_flow* f, const float* x_dev, const float* w_dev, uint64_t n, uint64_t off,
                           uint32_t batch, float* grad_host, float* loss_host, void* stream) {
    if (!f || !x_dev || !w_dev || !grad_host) return fail(JR_ERR_INVALID_ARG, "jr_flow_gradient: null argument");
    if (batch == 0 || off + batch > n) return fail(JR_ERR_INVALID_ARG, "jr_flow_gradient: rows out of range");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t P = (size_t)kFL * flow_layer_floats(f->D);
    float* buf = nullptr;  // gradient, then the weight sum and the loss
    JR_CUDA(dev_alloc(&buf, P + 2), "jr_flow_gradient");
    cudaError_t e = cudaMemsetAsync(buf, 0, sizeof(float) * (P + 2), st);
    if (e == cudaSuccess) e = launch_flow_wsum(w_dev, nullptr, off, batch, buf + P, 1, 1, st);
    if (e == cudaSuccess) e = launch_flow_train_step(f->view(0.f), x_dev, w_dev, n, off, batch, buf, buf + P, buf + P + 1, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad_host, buf, sizeof(float) * P, cudaMemcpyDeviceToHost, st);
    float tail[2] = {0.f, 0.f};
    if (e == cudaSuccess) e = cudaMemcpyAsync(tail, buf + P, sizeof(tail), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(buf);
    if (e != cudaSuccess) return cuda_fail(e, "jr_flow_gradient");
    if (loss_host) *loss_host = tail[1];
    return JR_OK;
}

jr_status jr_flow_train(jr_flow* f, const float* x_dev, const float* w_dev, uint64_t n, uint32_t iters,
                        uint32_t batch, float lr, uint64_t seed, float* loss_host, void* stream) {
    return jr_flow_train_rows(f, x_dev, w_dev, n, n, iters, batch, lr, seed, loss_host, stream);
}

jr_status jr_flow_train_rows(jr_flow* f, const float* x_dev, const float* w_dev, uint64_t n, uint64_t n_rows,
                             uint32_t iters, uint32_t batch, float lr, uint64_t seed, float* loss_host,
                             void* stream) {
    if (!f || !x_dev || !w_dev) return fail(JR_ERR_INVALID_ARG, "jr_flow_train: null argument");
    if (n_rows > n) return fail(JR_ERR_INVALID_ARG, "jr_flow_train: n_rows exceeds the row stride");
    if (batch == 0 || batch % 64 != 0 || batch > n_rows)
        return fail(JR_ERR_INVALID_ARG, "jr_flow_train: batch must be a positive multiple of 64, at most n_rows");
    if (!(lr > 0.f)) return fail(JR_ERR_INVALID_ARG, "jr_flow_train: lr must be > 0");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t P = (size_t)kFL * flow_layer_floats(f->D);
    if (!f->grad) {
        cudaError_t e;
        if ((e = dev_alloc(&f->grad, P)) != cudaSuccess || (e = dev_alloc(&f->adam_m, P)) != cudaSuccess ||
            (e = dev_alloc(&f->adam_v, P)) != cudaSuccess ||
            (e = cudaMemsetAsync(f->adam_m, 0, sizeof(float) * P, st)) != cudaSuccess ||
            (e = cudaMemsetAsync(f->adam_v, 0, sizeof(float) * P, st)) != cudaSuccess) {
            cudaFree(f->grad);
            cudaFree(f->adam_m);
            cudaFree(f->adam_v);
            f->grad = f->adam_m = f->adam_v = nullptr;
            return cuda_fail(e, "jr_flow_train (optimiser state)");
        }
    }
    std::vector<uint64_t> offs(iters);
    uint64_t rng = seed * 0x9E3779B97F4A7C15ull + 0xD1B54A32D192ED03ull;
    for (uint32_t it = 0; it < iters; ++it) {
        rng ^= rng >> 30;  // splitmix64 (Steele, Lea, Flood 2014): the minibatch window
        rng *= 0xBF58476D1CE4E5B9ull;
        rng ^= rng >> 27;
        rng *= 0x94D049BB133111EBull;
        rng ^= rng >> 31;
        offs[it] = rng % (n_rows - batch + 1);
    }
    // [iters][2] minibatch weight sum and loss, then the windows' offsets [iters]
    float* scal = nullptr;
    JR_CUDA(dev_alloc(&scal, 4 * (size_t)std::max<uint32_t>(iters, 1)), "jr_flow_train");
    uint64_t* offs_dev = reinterpret_cast<uint64_t*>(scal + 2 * (size_t)std::max<uint32_t>(iters, 1));
    cudaError_t e = cudaMemsetAsync(scal, 0, sizeof(float) * 2 * std::max<uint32_t>(iters, 1), st);
    if (iters > 0) {
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(offs_dev, offs.data(), sizeof(uint64_t) * iters, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = launch_flow_wsum(w_dev, offs_dev, 0, batch, scal, 2, iters, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(f->grad, 0, sizeof(float) * P, st);
    }
    for (uint32_t it = 0; it < iters && e == cudaSuccess; ++it) {
        if ((e = launch_flow_train_step(f->view(0.f), x_dev, w_dev, n, offs[it], batch, f->grad, scal + 2 * it,
                                        scal + 2 * it + 1, st)) != cudaSuccess)
            break;
        e = launch_adam(f->master, f->grad, f->adam_m, f->adam_v, f->D, lr, ++f->adam_t, f->wb, f->bias, st);
    }
    if (e == cudaSuccess) e = launch_flow_pack_ws(f->master, f->ws, f->AK, st);
    std::vector<float> h(2 * (size_t)std::max<uint32_t>(iters, 1));
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h.data(), scal, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(scal);
    if (e != cudaSuccess) return cuda_fail(e, "jr_flow_train");
    if (loss_host)
        for (uint32_t it = 0; it < iters; ++it) loss_host[it] = h[2 * it + 1];
    return JR_OK;
}

}  // extern "C"

namespace {

// Without a flow, a drain's steps run in the wavefront while more than
// kDrainTailChains chains may be open (there its packed warps pay), then in launches
// of drain_kernel of 8, 16, 32 ... at most kDrainTailSteps steps, and once at most
// kRunsDrainMost are open, a block takes each tour several steps at a time (jr_runs.cu).
// A checkpoint of 2^18 chains on the slit caustic: 37.0 ms in the wavefront alone, 8.5
// ms with drain_kernel, and with the blocks from 400, 1 400, 2 500, 10 000 open tours on
// 7.9, 6.0, 5.8, 5.8 ms; 100 000 chains on the terrain 28.8, 5.9; 5.4, 4.9, 4.7, 4.8 ms.
constexpr uint32_t kDrainTailChains = 1u << 16, kDrainFirstSteps = 8, kDrainTailSteps = 4096, kRunsDrainMost = 2500;

// Drain: advance only the chains that are inside a tour until every tour has
// ended (a kill ends the tour and the chain); the steps are regular steps of
// Alg. 2 for those chains.  Returns the chains still in a tour after
// max_steps (0 when every tour completed).
jr_status drain_impl(jr_chains* c, uint32_t max_steps, uint64_t* remaining, cudaStream_t st, const char* who) {
    jr_status a = ensure_wavefront(c, st);
    if (a != JR_OK) return a;
    JR_CUDA(cudaMemsetAsync(c->view.wf.done, 0, c->view.n, st), who);
    unsigned int active = (unsigned int)std::min<uint64_t>(c->view.n, 0xffffffffu);
    uint32_t k = 0;
    // Steps are enqueued in groups that grow while tours stay open, so the
    // host waits rarely.  A step after the last tour has ended is a no-op; the
    // drain mark (1 + the last step after which a tour was open) gives the
    // steps the drain really took, as if the host had checked after every step.
    JR_CUDA(cudaMemsetAsync(c->view.counters + 3, 0, sizeof(unsigned long long), st), who);
    const uint64_t s0 = c->steps;
    uint32_t group = 1;
    const bool flow = c->view.flow.D != 0;  // u(y) of each candidate comes from the wavefront's flow launches
    while (active > 0 && k < max_steps && (flow || active > kDrainTailChains)) {
        const uint32_t g = flow ? std::min(group, max_steps - k) : 1u;
        // one launch sequence per group: a single closing finish launch, not one per step
        JR_CUDA(launch_wavefront(c->scene_view(), c->view, s0 + k, g, st, kModeDrain), who);
        k += g;
        JR_CUDA(cudaMemcpyAsync(&active, c->view.wf.qcount + kQActive, sizeof(active), cudaMemcpyDeviceToHost, st),
                who);
        JR_CUDA(cudaStreamSynchronize(st), who);
        group = std::min<uint32_t>(2 * group, 16);
    }
    // Few open tours: each runs without waiting for the others, in launches of growing
    // length until only the longest are left, which a block each then takes several
    // steps at a time.
    for (uint32_t len = kDrainFirstSteps; active > 0 && k < max_steps; len = std::min(2 * len, kDrainTailSteps)) {
        const bool runs = k > 0 && active <= kRunsDrainMost;
        const uint32_t g = std::min(runs ? kDrainTailSteps : len, max_steps - k);
        unsigned long long* ctl = c->view.counters + kCounterDrain;
        if (runs) JR_CUDA(launch_runs_drain(c->scene_view(), c->view, s0 + k, g, ctl, st), who);
        else JR_CUDA(launch_drain(c->scene_view(), c->view, s0 + k, g, ctl, st), who);
        k += g;
        unsigned long long open = 0;
        JR_CUDA(cudaMemcpyAsync(&open, ctl + 1, sizeof(open), cudaMemcpyDeviceToHost, st), who);
        JR_CUDA(cudaStreamSynchronize(st), who);
        active = (unsigned int)open;
    }
    if (k > 0) {
        unsigned long long mark = 0;
        JR_CUDA(cudaMemcpyAsync(&mark, c->view.counters + 3, sizeof(mark), cudaMemcpyDeviceToHost, st), who);
        JR_CUDA(cudaStreamSynchronize(st), who);
        c->steps = active > 0 ? s0 + k : std::max<uint64_t>(mark, s0) + 1;
    }
    JR_CUDA(launch_fold(c->view, st), who);
    if (remaining) *remaining = active;
    return JR_OK;
}

// Restart: every chain starts a new tour from the current mu.
jr_status restart_impl(jr_chains* c, cudaStream_t st, const char* who) {
    jr_status a = ensure_wavefront(c, st);
    if (a != JR_OK) return a;
    c->epochs += 1;
    JR_CUDA(launch_wavefront(c->scene_view(), c->view, c->epochs, 1, st, kModeRestart), who);
    return JR_OK;
}

}  // namespace

extern "C" {

jr_status jr_complete_tours(jr_chains* c, uint32_t max_steps, uint64_t* remaining, void* stream) {
    if (!c) return fail(JR_ERR_INVALID_ARG, "jr_complete_tours: null chains");
    if (c->view.flags & JR_FLAG_MH) return fail(JR_ERR_STATE, "jr_complete_tours: an MH chain set has no tours");
    if (c->view.flags & JR_FLAG_MALA)
        return fail(JR_ERR_STATE, "jr_complete_tours: the drain runs in the wavefront, which has no MALA moves");
    cudaStream_t st = (cudaStream_t)stream;
    jr_status r = drain_impl(c, max_steps, remaining, st, "jr_complete_tours");
    if (r == JR_OK) r = restart_impl(c, st, "jr_complete_tours");
    return r;
}

jr_status jr_chains_set_flow(jr_chains* c, const jr_flow* f, float beta, uint32_t max_drain_steps,
                             uint64_t* remaining, void* stream) {
    if (!c) return fail(JR_ERR_INVALID_ARG, "jr_chains_set_flow: null chains");
    if (c->view.flags & (JR_FLAG_MH | JR_FLAG_MALA))
        return fail(JR_ERR_STATE, "jr_chains_set_flow: MH and MALA chains regenerate from the uniform mu only");
    // A flow of lower dimension models the leading coordinates only (the rest
    // stay uniform); it must cover the path's start record, coordinates 0..3.
    if (f && !(f->D == c->view.dim || (f->D >= 4 && f->D < c->view.dim)))
        return fail(JR_ERR_INVALID_ARG, "jr_chains_set_flow: the flow's dimension must equal the chains' or lie in 4 .. D - 1");
    if (f && !(beta >= 0.f && beta < 1.f))
        return fail(JR_ERR_INVALID_ARG, "jr_chains_set_flow: beta must be in [0, 1)");
    cudaStream_t st = (cudaStream_t)stream;
    uint64_t rem = 0;
    jr_status r = drain_impl(c, max_drain_steps, &rem, st, "jr_chains_set_flow");  // finish the tours of the old mu
    if (r != JR_OK) return r;
    if (remaining) *remaining = rem;
    c->view.flow = f ? f->view(beta) : FlowView{};
    c->flow_gen += 1;
    return restart_impl(c, st, "jr_chains_set_flow");
}

}  // extern "C"
