// Host side of the library (host.cpp) against a stand-in for the CUDA runtime
// and the kernel launchers, for what no GPU test can bring about: allocations
// that fail in the middle of a set-up call, and copies that no wait orders
// before a launch on another stream.  Prints "ok" or what went wrong.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include <string>
#include <vector>
#include "internal.h"
#include "rascas_gb300.h"

namespace {
int g_fail_at = -1, g_launches = 0, g_bad_order = 0;
std::set<void*> g_live;               // device buffers
std::set<cudaStream_t> g_pending;     // streams with copies that nothing has waited for
rg::Params g_params;                  // of the last propagation
const cudaStream_t kLegacy = nullptr;

void copied(cudaStream_t st) { g_pending.insert(st == cudaStreamLegacy ? kLegacy : st); }
cudaError_t launch(cudaStream_t st) {
    ++g_launches;
    for (cudaStream_t s : g_pending)
        if (s != st) ++g_bad_order;
    return cudaSuccess;
}
bool live(const void* p) { return g_live.count(const_cast<void*>(p)) != 0; }
}  // namespace

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 2; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaMalloc(void** p, size_t b) {
    if (g_fail_at >= 0 && g_fail_at-- == 0) { *p = nullptr; return cudaErrorMemoryAllocation; }
    *p = std::calloc(1, b ? b : 1);
    g_live.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) { g_live.erase(p); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t b, cudaMemcpyKind k) {
    std::memcpy(d, s, b);
    if (k != cudaMemcpyDeviceToHost) copied(kLegacy);   // pageable memory: may still be under way
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t b, cudaMemcpyKind, cudaStream_t st) {
    std::memcpy(d, s, b);
    copied(st);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t b, cudaStream_t st) { std::memset(d, v, b); copied(st); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { g_pending.erase(st == cudaStreamLegacy ? kLegacy : st); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)0x20; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
}

namespace rg {
#define PROPAGATE const Params& P, const PacketsIn&, const PacketsOut&, const TraceOut&, int, int, cudaStream_t st
cudaError_t launch_propagate(PROPAGATE) { g_params = P; return launch(st); }
cudaError_t launch_propagate_fad(PROPAGATE) { g_params = P; return launch(st); }
cudaError_t launch_peel(const Params&, int, cudaStream_t st) { return launch(st); }
cudaError_t launch_peel_fad(const Params&, int, cudaStream_t st) { return launch(st); }
#define RAYS const Params&, long long, const double*, const double*, const double*, double*, int32_t*, double*, int, int32_t*, RayInit*, int, cudaStream_t st
cudaError_t launch_ray_tau(RAYS) { return launch(st); }
cudaError_t launch_ray_tau_fad(RAYS) { return launch(st); }
cudaError_t launch_ray_columns(const Params&, long long, const double*, const double*, double*, double*, double, double,
                               int32_t*, RayInit*, int, cudaStream_t st) { return launch(st); }
cudaError_t launch_grad_unpack(long long, const float4*, float*, cudaStream_t st) { return launch(st); }
cudaError_t launch_pack_fields(long long, const float*, const float*, const float*, const float*, const float*, const float*,
                               const float*, float4*, cudaStream_t st) { return launch(st); }
cudaError_t launch_leaf_links(const Geo&, int*, cudaStream_t st) { return launch(st); }
cudaError_t launch_eval_voigt(long long, const float*, const double*, float*, int, cudaStream_t st) { return launch(st); }
cudaError_t launch_sample_upar(const Params&, long long, const double*, const float*, const uint64_t*, float*, int32_t*,
                               cudaStream_t st) { return launch(st); }
cudaError_t noalloc_scratch(void** p, size_t* b) { static char s[1 << 16]; *p = s; *b = sizeof s; return cudaSuccess; }
cudaError_t probe_issue_rates(int, void*, double*) { return cudaSuccess; }
size_t packet_save_bytes(int) { return 64; }
int propagate_block_size() { return 128; }
int propagate_blocks_per_sm(int, bool) { return 1; }
int propagate_batch_blocks_per_sm(int, int) { return 1; }
}  // namespace rg

namespace {
int bad(const std::string& what) { std::printf("%s\n", what.c_str()); return 1; }

// an octree of one level, or of two (64 leaves)
struct Tree {
    std::vector<int32_t> son;
    std::vector<float> f;
    rascas_octree t{};
    explicit Tree(bool deep) {
        const int n = deep ? 64 : 8;
        if (!deep) for (int c = 0; c < 8; ++c) son.push_back(-1 - c);
        else {
            for (int c = 0; c < 8; ++c) son.push_back(c + 1);
            for (int c = 0; c < 64; ++c) son.push_back(-1 - c);
        }
        f.assign(n, 1.0f);
        t.noct = (int)son.size() / 8; t.nleaf = n; t.son = son.data();
        t.n_HI = t.vx = t.vy = t.vz = t.T = t.n_dust = f.data();
        t.box_cm = 1.0;
    }
};

rascas_detector detector(int nbin, int npix) {
    rascas_detector d{};
    d.nu_lo = 1.0; d.nu_hi = 2.0; d.nbin = nbin; d.ndir = 1; d.dirs[0][2] = 1.0; d.npix = npix; d.fov = 1.0; d.cube = 1;
    return d;
}

struct Run {
    rascas_ctx* c = nullptr;
    double pos[3] = {0.5, 0.5, 0.5}, dir[3] = {0, 0, 1}, nu[1] = {1.5}, tau[1];
    uint64_t id[1] = {0};
    rascas_packets_in in{pos, dir, nu, id};
    explicit Run(void* stream) {
        rascas_create(&c, 0);
        rascas_set_stream(c, stream);
        rascas_line l{};
        l.nu0 = 1.5; l.A_ul = 1.0; l.f_lu = 1.0; l.mass_g = 1e-24; l.abundance = 1.0; l.nchan = 1; l.chan_A[0] = 1.0; l.chan_nu[0] = 1.5;
        rascas_set_lines(c, &l, 1, nullptr);
        rascas_physics p{};
        p.x_gauss = 8.0; p.tau_stop = 50.0;
        rascas_set_physics(c, &p);
    }
    ~Run() { rascas_destroy(c); }
    int domain() { rascas_domain d{}; d.kind = RASCAS_DOMAIN_CUBE; for (double& x : d.centre) x = 0.5; d.size = 0.5; return rascas_set_domain(c, &d); }
    int load(bool deep) { Tree t(deep); return rascas_load_octree(c, &t.t, RASCAS_HOST); }
    int detect(int nbin, int npix) { const rascas_detector d = detector(nbin, npix); return rascas_set_detector(c, &d); }
    int propagate() { return rascas_propagate(c, &in, 1, nullptr, RASCAS_HOST, nullptr); }
    int batch(bool deep) {
        Tree t(deep);
        rascas_model m{};
        m.tree = t.t; m.domain.kind = RASCAS_DOMAIN_CUBE; for (double& x : m.domain.centre) x = 0.5; m.domain.size = 0.5;
        m.nu_lo = 1.0; m.nu_hi = 2.0; m.packets = in; m.npackets = 1;
        return rascas_load_batch(c, &m, 1, deep ? 80 : 10, RASCAS_HOST);
    }
};
}  // namespace

int main() {
    // allocation k of a set-up call fails: the context has lost what the call
    // was to replace, says so, launches nothing on freed memory, and recovers
    for (int k = 0; k < 5; ++k) {
        Run r((void*)0x10);
        if (r.load(false) || r.domain() || r.propagate()) return bad("octree: set-up");
        g_fail_at = k;
        if (r.load(true) != RASCAS_E_OOM) return bad("octree: no E_OOM");
        g_fail_at = -1;
        const int n = g_launches;
        if (r.propagate() != RASCAS_E_STATE || g_launches != n) return bad("octree: propagated after a failed load");
        if (r.load(true) || r.propagate() || !live(g_params.g.rec) || !live(g_params.g.link)) return bad("octree: not recovered");
    }
    for (int k = 0; k < 4; ++k) {
        Run r((void*)0x10);
        if (r.load(false) || r.domain() || r.detect(10, 2) || r.propagate()) return bad("detector: set-up");
        g_fail_at = k;
        if (r.detect(100, 20) != RASCAS_E_OOM) return bad("detector: no E_OOM");
        g_fail_at = -1;
        if (r.propagate() || g_params.ndir != 0 || g_params.g.spec) return bad("detector: tallies after a failed call");
        if (r.detect(100, 20) || r.propagate() || g_params.npix != 20 || !live(g_params.pimg) || !live(g_params.pcube))
            return bad("detector: not recovered");
        rascas_detector d = detector(10, 40);
        d.dirs[0][2] = 0.0;
        if (rascas_set_detector(r.c, &d) != RASCAS_E_ARG || r.propagate() || g_params.npix != 20 || g_params.ndir != 1)
            return bad("detector: a refused call changed the context");
    }
    for (int k = 0; k < 7; ++k) {   // the packet buffers keep their size
        Run r((void*)0x10);
        if (r.batch(false) || rascas_propagate_batch(r.c, RASCAS_BATCH_PER_MODEL, nullptr)) return bad("batch: set-up");
        g_fail_at = k;
        const int e = r.batch(true);
        g_fail_at = -1;
        const int n = g_launches;
        if (e == RASCAS_OK) continue;   // fewer allocations than k
        if (e != RASCAS_E_OOM || rascas_propagate_batch(r.c, RASCAS_BATCH_PER_MODEL, nullptr) != RASCAS_E_STATE || g_launches != n)
            return bad("batch: propagated after a failed load");
        if (r.batch(true) || rascas_propagate_batch(r.c, RASCAS_BATCH_PER_MODEL, nullptr)) return bad("batch: not recovered");
    }
    // every copy of a set-up call is waited for before a launch on another stream
    for (void* stream : {(void*)0x10, (void*)nullptr}) {
        Run r(stream);
        g_pending.clear();
        g_bad_order = 0;
        std::vector<float> f(64, 2.0f);
        if (r.load(true) || r.domain() || r.detect(10, 2) || r.propagate()) return bad("order: set-up");
        if (rascas_update_fields(r.c, f.data(), f.data(), f.data(), f.data(), f.data(), f.data(), nullptr, RASCAS_HOST) ||
            rascas_ray_tau(r.c, 1, r.pos, r.dir, r.nu, r.tau, nullptr, nullptr, 0, nullptr, RASCAS_HOST) || r.domain() || r.propagate())
            return bad("order: fields");
        if (r.batch(true) || rascas_propagate_batch(r.c, RASCAS_BATCH_PER_MODEL, nullptr)) return bad("order: batch");
        if (g_bad_order) return bad("order: a launch on another stream than copies that nothing waited for");
    }
    std::printf("ok\n");
    return 0;
}
