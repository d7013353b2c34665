// The host side of the multi-domain batch (csrc/batch.cu) over a CUDA runtime that is faked here: "device" memory
// is host memory, an allocation can be made to fail, and a launch is recorded (in a capture) or checked (outside
// of one, or when its graph is replayed): its tile and run arrays must be live allocations that hold what the
// kernel would read, every pass must cover every cell of its members once, and passes must follow the AA phases.
// No GPU is touched.  Usage: batch_host <scenario>; prints "ok" and exits 0.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include "ctx_internal.h"

#define REQUIRE(c)                                                          \
    do {                                                                    \
        if (!(c)) {                                                         \
            std::printf("line %d: %s\n", __LINE__, #c);                     \
            std::exit(1);                                                   \
        }                                                                   \
    } while (0)

namespace {

std::map<const char*, size_t> live;   // allocations
int allocs_left = -1;                 // cudaMalloc calls that still succeed (-1: all)
int instantiated = 0;
int device_sms = 152;
int last_runs = 0;                    // of the last density pass

struct Pass {
    bool collide;
    lbm::BatchDomTable tab;
    const void* items;
    int n, parity, shape, near;
};
struct Graph {
    std::vector<Pass> passes;
};
Graph* capture = nullptr;

std::map<const float*, lbm_ctx*> by_base;
std::map<const float*, long long> collided, summed;   // cells

bool check_near = false;

// next to a wall of its domain (no member has a mask)
bool at_wall(const lbm::BatchDom& d, int x, int y, int z) {
    return (d.wall_x && (x == 0 || x == d.nx - 1)) || (d.wall_y && (y == 0 || y == d.ny - 1)) ||
           (d.wall_z && (z == 0 || z == d.nz - 1));
}
void check_tile(const Pass& p, const lbm::BatchTile& t, const lbm::BatchDom& d, int w, int h) {
    const int n = std::min(t.zc, d.nz - t.z0);
    REQUIRE(t.near == 0 || (p.near != lbm::NEAR_NONE && n <= 32 && (n == 32 || t.near >> n == 0)));
    REQUIRE(t.near == 0 || p.near == lbm::NEAR_SOME || n == 1);
    for (int j = 0; j < n; ++j) {
        bool need = false;
        for (int y = t.y0; y < std::min(t.y0 + h, d.ny); ++y)
            for (int x = t.x0; x < std::min(t.x0 + w, d.nx); ++x) need |= at_wall(d, x, y, t.z0 + j);
        REQUIRE(need == (j < 32 && ((t.near >> j) & 1u)));
    }
}
void check_run(const Pass& p, const lbm::BatchRun& r, const lbm::BatchDom& d) {
    REQUIRE(!r.near || p.near);
    for (int c = (int)r.begin; c < (int)r.end && !r.near; ++c)
        REQUIRE(!at_wall(d, c % d.nx, c / d.nx % d.ny, c / d.nx / d.ny));
}

void check(const Pass& p) {
    const size_t item = p.collide ? sizeof(lbm::BatchTile) : sizeof(lbm::BatchRun);
    auto it = live.upper_bound((const char*)p.items);
    REQUIRE(p.items && it != live.begin());
    --it;
    REQUIRE((const char*)p.items + p.n * item <= it->first + it->second);
    for (int k = 0; k < p.n; ++k) {
        if (p.collide) {
            const lbm::BatchTile& t = ((const lbm::BatchTile*)p.items)[k];
            const lbm::BatchDom& d = p.tab.d[t.d];
            const lbm::BatchShape& s = lbm::BATCH_SHAPES[p.shape];
            const int w = t.narrow ? lbm::BATCH_NARROW_BX : s.bx, h = s.bx * s.by / w;
            REQUIRE(by_base.count(d.base));
            REQUIRE(t.x0 >= 0 && t.x0 < d.nx && t.y0 >= 0 && t.y0 < d.ny && t.z0 >= 0 && t.z0 < d.nz);
            const long long cells = (long long)std::min(w, d.nx - t.x0) * std::min(h, d.ny - t.y0) *
                                    std::min(t.zc, d.nz - t.z0);
            const long long n = by_base[d.base]->kp.ncell;
            REQUIRE(p.parity == (int)(collided[d.base] / n % 2));
            REQUIRE(collided[d.base] / n == summed[d.base] / n && summed[d.base] % n == 0);
            collided[d.base] += cells;
            if (check_near) check_tile(p, t, d, w, h);
        } else {
            const lbm::BatchRun& r = ((const lbm::BatchRun*)p.items)[k];
            const lbm::BatchDom& d = p.tab.d[r.d];
            REQUIRE(by_base.count(d.base) && r.begin < r.end);
            const long long n = by_base[d.base]->kp.ncell;
            REQUIRE(r.end <= n && collided[d.base] % n == 0);
            REQUIRE(p.parity == (int)(collided[d.base] / n % 2));
            summed[d.base] += r.end - r.begin;
            last_runs = p.n;
            if (check_near) check_run(p, r, d);
        }
    }
}

cudaError_t enqueue(const Pass& p) {
    if (capture) capture->passes.push_back(p);
    else check(p);
    return cudaSuccess;
}

template <class T>
T handle() { return (T) new char; }

}  // namespace

// ---------------------------------------------------------------- the runtime
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { std::abort(); }   // no member has a mask
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { std::abort(); }
cudaError_t __cudaGetKernel(void*, const void*) { std::abort(); }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, cudaStream_t) { std::abort(); }

cudaError_t cudaMalloc(void** p, size_t n) {
    if (allocs_left == 0) return cudaErrorMemoryAllocation;
    if (allocs_left > 0) --allocs_left;
    *p = std::malloc(n);
    live[(const char*)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    REQUIRE(live.erase((const char*)p) == 1);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = device_sms, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (char*)e, cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = handle<cudaStream_t>(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete (char*)s, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return capture = new Graph, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)capture;
    capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    ++instantiated;
    return *e = (cudaGraphExec_t) new Graph(*(Graph*)g), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete (Graph*)g, cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return delete (Graph*)e, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
    for (const Pass& p : ((Graph*)e)->passes) check(p);
    return cudaSuccess;
}
lbm_status lbm_sync(lbm_ctx*) { return LBM_OK; }
const char* lbm_last_error(const lbm_ctx*) { return ""; }
}

namespace lbm {
void set_thread_error(const char*) {}
#define FAKE_LAUNCHERS(Q)                                                                                      \
    cudaError_t launch_collide_batch_q##Q(const KParams&, const BatchDomTable& tab, const BatchTile* t, int n, \
                                          int parity, int near, int shape, cudaStream_t) {                     \
        return enqueue({true, tab, t, n, parity, shape, near});                                                \
    }                                                                                                          \
    cudaError_t launch_psi_runs_q##Q(const KParams&, const BatchDomTable& tab, const BatchRun* r, int n,       \
                                     int parity, int near, cudaStream_t) {                                     \
        return enqueue({false, tab, r, n, parity, 0, near});                                                   \
    }
FAKE_LAUNCHERS(19)
FAKE_LAUNCHERS(27)
}  // namespace lbm

// ---------------------------------------------------------------- scenarios
namespace {

struct Domains {
    std::vector<std::unique_ptr<lbm_ctx>> own;
    std::vector<lbm_ctx*> ctx;
    std::vector<std::unique_ptr<float>> base;
    void add(int Q, int nx, int ny, int nz, bool wall_z, float G = -1.0f, bool wall_x = false, bool wall_y = false) {
        own.emplace_back(new lbm_ctx);
        lbm_ctx* c = own.back().get();
        std::memset(&c->kp, 0, sizeof c->kp);
        c->Q = Q;
        c->kp.nx = nx;
        c->kp.ny = ny;
        c->kp.nz = nz;
        c->kp.wall_x = wall_x;
        c->kp.wall_y = wall_y;
        c->kp.wall_z = wall_z;
        c->kp.ncell = c->kp.plane = (long long)nx * ny * nz;
        c->kp.multiphase = 1;
        c->kp.G = G;
        base.emplace_back(new float);
        c->kp.fq[0] = base.back().get();
        c->initialised = true;
        by_base[c->kp.fq[0]] = c;
        ctx.push_back(c);
    }
    // every member has taken `steps` steps by its counter and by the passes that ran
    void stepped(long long steps) const {
        for (const lbm_ctx* c : ctx) {
            REQUIRE(c->t == steps && c->parity == (int)(steps % 2));
            REQUIRE(collided[c->kp.fq[0]] == steps * c->kp.ncell && summed[c->kp.fq[0]] == steps * c->kp.ncell);
        }
    }
};

Domains three() {   // three chains, one of 70 members (two launches), one with walls
    Domains d;
    for (int k = 0; k < 70; ++k) d.add(19, 20 + k % 3, 9, 6, k % 4 == 0);
    d.add(27, 47, 10, 12, true);
    d.add(19, 33, 8, 10, false, -0.5f);
    return d;
}

// A rebuild that runs out of device memory at any of its allocations: the call reports it, no step launches what was
// not built or counts steps that were not taken, and the batch goes on once there is memory.
void failed_rebuild() {
    for (int at = 0;; ++at) {
        collided.clear();
        summed.clear();
        Domains d = three();
        lbm_batch* b = nullptr;
        REQUIRE(lbm_batch_create(d.ctx.data(), (int)d.ctx.size(), nullptr, &b) == LBM_OK);
        REQUIRE(lbm_batch_step(b, 5) == LBM_OK);
        d.stepped(5);
        // re-tiled by a call of its own
        allocs_left = at < 100 ? at : -1;
        lbm_status s = LBM_OK;
        for (int g = 0; g < 5 && s == LBM_OK; ++g) s = lbm_batch_set_group(b, g, 1, 2);
        REQUIRE(s == LBM_OK || s == LBM_ERR_OOM);
        const bool failed = s != LBM_OK;
        allocs_left = failed ? 0 : -1;
        if (failed) {
            REQUIRE(lbm_batch_step(b, 3) == LBM_ERR_OOM);
            d.stepped(5);
        }
        allocs_left = -1;
        REQUIRE(lbm_batch_step(b, 3) == LBM_OK);
        d.stepped(8);
        // a member that got a wall-less layout of other walls: grouped anew at the next step
        d.ctx[1]->kp.wall_y = 1;
        allocs_left = at;
        s = lbm_batch_step(b, 2);
        REQUIRE(s == LBM_OK || s == LBM_ERR_OOM);
        if (s != LBM_OK) {
            d.stepped(8);
            allocs_left = 0;
            REQUIRE(lbm_batch_step(b, 2) == LBM_ERR_OOM);
            d.stepped(8);
            allocs_left = -1;
            REQUIRE(lbm_batch_step(b, 2) == LBM_OK);
        }
        allocs_left = -1;
        d.stepped(10);
        lbm_batch_destroy(b);
        REQUIRE(live.empty());
        by_base.clear();
        if (!failed && s == LBM_OK) return;
        REQUIRE(at < 100);
    }
}

// A member that needs solid handling since it was last stepped (here: a wall, in use: a mask), tuned or given a
// shape before it is stepped again: its groups follow first.
void retiled_after_change(bool tune) {
    Domains d;
    d.add(19, 33, 9, 14, false);
    d.add(27, 33, 9, 14, false);
    lbm_batch* b = nullptr;
    REQUIRE(lbm_batch_create(d.ctx.data(), 2, nullptr, &b) == LBM_OK);
    REQUIRE(lbm_batch_step(b, 2) == LBM_OK);
    d.ctx[1]->kp.wall_y = 1;
    if (tune) REQUIRE(lbm_batch_tune(b, 1, nullptr, 0) == LBM_OK);
    else REQUIRE(lbm_batch_set_group(b, 1, 1, 4) == LBM_OK);
    int32_t groups = 0;
    REQUIRE(lbm_batch_info(b, &groups, nullptr, nullptr) == LBM_OK && groups == 3);
    d.stepped(tune ? 26 : 2);
    REQUIRE(lbm_batch_step(b, 3) == LBM_OK);
    d.stepped(tune ? 29 : 5);
    lbm_batch_destroy(b);
}

// Calls of an odd number of steps begin in the other AA phase each time: graphs are recorded once per phase, not
// once per call, and every call takes exactly its steps.
void odd_calls() {
    for (int n : {2, 3, 5, 7, 19, 33, 65, 67, 129}) {
        collided.clear();
        summed.clear();
        Domains d = three();
        lbm_batch* b = nullptr;
        REQUIRE(lbm_batch_create(d.ctx.data(), (int)d.ctx.size(), nullptr, &b) == LBM_OK);
        instantiated = 0;
        long long steps = 0;
        for (int k = 0; k < 12; ++k) {
            REQUIRE(lbm_batch_step(b, n) == LBM_OK);
            d.stepped(steps += n);
        }
        const int most = (n % 2 ? 2 : 1) * (n >= 64 ? 2 : 1);
        if (instantiated > most) std::printf("%d graphs for calls of %d steps\n", instantiated, n);
        REQUIRE(instantiated <= most);
        lbm_batch_destroy(b);
        by_base.clear();
    }
}

// Every plane of a tile that holds cells next to a wall has its bit and no other has one, tiles with bits are at most
// 32 planes high (single planes in launches of the kind that takes no others), and runs that are not marked hold no
// such cell: for all walls, extents about 32 planes, tile shapes and z-chunks.
void near_planes() {
    check_near = true;
    for (int Q : {19, 27})
        for (int walls = 0; walls < 8; ++walls) {
            collided.clear();
            summed.clear();
            Domains d;
            int k = 0;
            for (int nz : {1, 2, 3, 31, 34, 70}) {
                d.add(Q, (const int[]){5, 32, 44, 50, 33, 64}[k], (const int[]){9, 1, 4, 6, 13, 8}[k], nz, walls & 4, -1.0f,
                      walls & 1, walls & 2);
                ++k;
            }
            lbm_batch* b = nullptr;
            REQUIRE(lbm_batch_create(d.ctx.data(), (int)d.ctx.size(), nullptr, &b) == LBM_OK);
            long long steps = 0;
            for (int shape = 0; shape < LBM_BATCH_SHAPES; ++shape)
                for (int plain : {0, 1, 7, 40, 1 << 30})
                    for (int solid : {0, 1, 33}) {
                        REQUIRE(lbm_batch_set_group(b, 0, shape, plain) == LBM_OK);
                        if (walls) REQUIRE(lbm_batch_set_group(b, 1, shape, solid) == LBM_OK);
                        REQUIRE(lbm_batch_step(b, 1) == LBM_OK);
                        d.stepped(++steps);
                    }
            lbm_batch_destroy(b);
            by_base.clear();
        }
}

// Work is cut for the SMs that the device has: 2432 x 256 cells in runs for eight blocks each.
void sm_count() {
    for (int sms : {152, 76, 304}) {
        device_sms = sms;
        collided.clear();
        summed.clear();
        Domains d;
        d.add(19, 128, 64, 76, false);
        lbm_batch* b = nullptr;
        REQUIRE(lbm_batch_create(d.ctx.data(), 1, nullptr, &b) == LBM_OK);
        REQUIRE(lbm_batch_step(b, 1) == LBM_OK);
        d.stepped(1);
        REQUIRE(last_runs == (sms == 76 ? 608 : sms == 152 ? 1216 : 2432));
        lbm_batch_destroy(b);
        by_base.clear();
    }
}

}  // namespace

int main(int argc, char** argv) {
    const std::string which = argc > 1 ? argv[1] : "";
    if (which == "failed_rebuild") failed_rebuild();
    else if (which == "tune_after_change") retiled_after_change(true);
    else if (which == "set_group_after_change") retiled_after_change(false);
    else if (which == "odd_calls") odd_calls();
    else if (which == "near_planes") near_planes();
    else if (which == "sm_count") sm_count();
    else return 2;
    std::printf("ok\n");
    return 0;
}
