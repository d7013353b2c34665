// Multi-domain batch (lbm_batch_*): many independent domains advanced together.
//
// Members are grouped by (lattice, solid handling, physical parameters); the members of one lattice and physics
// form a chain.  Per time step a chain costs one collide-stream launch and one density/psi launch whose
// blocks are tiles and runs of all its members (up to 64 members per launch), instead of two launches per
// domain.  The physical parameters (rates, equation of state, forces) and the launch's member table
// (geometry and buffer addresses) are passed by value in the kernel parameters, so a block reads them from the
// constant bank as the single-domain kernel does.  The per-cell arithmetic is the single-domain code, so a
// member's result is bitwise the same as stepping it alone.  The chains run side by side on streams of their
// own; runs of steps are replayed from CUDA graphs of 2 and 16 steps, within which the kernels of a chain
// overlap at their ends as lbm_step's do, and at whose ends the chains are joined.
// us a step, one launch a group and pass with all groups joined after every pass, in a device-side loop / this:
// 4 x 32^3 D3Q19 17.2 / 8.8; 40^3 droplets and impacts on both lattices 34.0 / 19.4; 8 x 64^3 93.9 / 85.1; ten mixed
// jobs of 48^3 - 109^3 318 / 290; 24 mixed jobs of 48^3 - 160^3 1665 / 1636.  (Advancing members in bins that fit the L2
// one after the other: 6 x 96^3 196 against 213 us in calls of 100 steps, but 210 against 214 in calls of 20, and
// ten mixed jobs 290 - 304 against 290: not worth it.)  lbm_batch_tune times the candidate tile shapes
// and z-chunks per chain on the live state.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "ctx_internal.h"
#include "lbm_internal.h"

using lbm::BatchDom;
using lbm::BatchDomTable;
using lbm::BatchRun;
using lbm::div_magic;
using lbm::BatchTile;
using lbm::KParams;

namespace {

// What the caller sees and tunes: members' tiles of one lattice, physics and solid handling.
struct Group {
    int Q = 19, solids = 0;
    KParams phys{};                 // physical parameters shared by the members (geometry zeroed)
    std::vector<int> members;       // members with tiles in this group
    int zchunk = 0;                 // 0 = automatic
    int shape = 0;                  // tile shape: index into lbm::BATCH_SHAPES
    int ntiles = 0;                 // collide tiles
};

// One launch pair (collide, density/psi) of a chain: up to BATCH_LAUNCH_DOMS members, their tiles and runs.
struct Launch {
    BatchDomTable tab{};
    BatchTile* tiles = nullptr;     // device
    BatchRun* runs = nullptr;       // device
    int nt = 0, nr = 0;
    int near = lbm::NEAR_NONE;      // which tiles and runs have cells with solid neighbours
};

// A chain: the members of one lattice and physics, advanced by their own sequence of launches.  Their tiles
// with and without solid neighbours go into the same launches.
struct Chain {
    int Q = 19, plain = -1, solid = -1;   // its groups (solid: -1 if no member has walls or solids)
    std::vector<int> members;
    std::vector<unsigned long long> masks;   // the members' mask_id when the launches were built
    std::vector<Launch> launches;
    bool built = false;                   // the launches are whole: none may run before (a build may fail half-way)
};

// Steps of the two graphs a batch replays (the longer one only in calls that replay it four times): a graph
// launch costs the GPU about 2 us between the last kernel of one and the first of the next.
constexpr int GRAPH_STEPS[2] = {2, 16};

bool has_solid_work(const lbm_ctx* c) { return c->nbmask != nullptr || c->kp.wall_x || c->kp.wall_y || c->kp.wall_z; }

// The physical part of a member's parameters: geometry, addresses and tiling fields zeroed, so
// that members with equal physics compare equal byte for byte.
KParams physics_of(const KParams& k) {
    KParams p;
    std::memcpy(&p, &k, sizeof(KParams));
    p.nx = p.ny = p.nz = 0;
    p.wall_x = p.wall_y = p.wall_z = 0;
    p.plane = p.ncell = 0;
    for (float*& q : p.fq) q = nullptr;
    for (float*& q : p.gq) q = nullptr;
    p.zchunk = 0;
    p.paired = p.hx = 0;        // storage layout (FP16 only), not physics
    return p;
}

BatchDom dom_of(const lbm_ctx* c) {
    BatchDom d{};
    d.nx = c->kp.nx;
    d.ny = c->kp.ny;
    d.nz = c->kp.nz;
    d.wall_x = c->kp.wall_x;
    d.wall_y = c->kp.wall_y;
    d.wall_z = c->kp.wall_z;
    d.plane = c->kp.plane;
    d.base = c->kp.fq[0];
    d.psi = c->psi;
    d.nbmask = c->nbmask;
    d.status = c->status;
    div_magic((uint32_t)c->kp.nx, d.mx, d.sx);
    div_magic((uint32_t)c->kp.ny, d.my, d.sy);
    return d;
}

}  // namespace

struct lbm_batch {
    std::vector<lbm_ctx*> members;
    std::vector<KParams> seen;      // member parameters the groups were built from
    std::vector<BatchDom> table;    // member geometry and addresses the groups were built from
    std::vector<Group> groups;
    std::vector<Chain> chains;
    int sms = 152;                  // of the device
    cudaStream_t stream = nullptr;
    cudaStream_t cap = nullptr;     // capture stream
    cudaGraphExec_t exec[2][2] = {};   // [AA phase a call starts from][k]: GRAPH_STEPS[k] steps (nullptr: not recorded)
    std::vector<cudaStream_t> side; // one per chain: the chains run concurrently
    cudaEvent_t fork = nullptr;
    std::vector<cudaEvent_t> done;
    std::string err;
};

namespace {

lbm_status bfail(lbm_batch* b, lbm_status s, const std::string& m) {
    if (b) b->err = m;
    else lbm::set_thread_error(m.c_str());
    return s;
}

#define BCK(b, call)                                                                                 \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess)                                                                       \
            return bfail(b, e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA,            \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                        \
    } while (0)

void drop_graph(lbm_batch* b) {
    for (auto& phase : b->exec)
        for (cudaGraphExec_t& e : phase) {
            if (e) cudaGraphExecDestroy(e);
            e = nullptr;
        }
}

void free_chain(Chain& c) {
    for (Launch& L : c.launches) {
        if (L.tiles) cudaFree(L.tiles);
        if (L.runs) cudaFree(L.runs);
    }
    c.launches.clear();
    c.built = false;
}

constexpr int ZC_WHOLE = 1 << 30;   // a z-chunk candidate: every column marches through all its planes
constexpr int ZC_AUTO_MAX = 32;   // automatic z-chunks: longer marches gain little, and in a mix of
                                  // uneven members shorter blocks balance the last wave

// flags[(z * nyb + yb) * nxb + xb] = 1 if a cell of the blockDim.x x blockDim.y column (xb, yb) in
// plane z has a solid neighbour or is solid (its neighbour mask is nonzero).
__global__ void tile_flags_kernel(const uint32_t* __restrict__ nbmask, int nx, int ny, uint8_t* flags) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    bool any = false;
    if (x < nx && y < ny) any = nbmask[((long long)z * ny + y) * nx + x] != 0u;
    any = __syncthreads_or(any);
    if (threadIdx.x == 0 && threadIdx.y == 0)
        flags[((long long)z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = any ? 1 : 0;
}

// Mask flags of a member for tw x th columns (cached on the context until its fields are
// re-initialised or another tile shape asks).
lbm_status member_tile_flags(lbm_batch* b, lbm_ctx* c, int tw, int th) {
    const KParams& k = c->kp;
    const long long nxb = (k.nx + tw - 1) / tw, nyb = (k.ny + th - 1) / th;
    const size_t n = (size_t)(nxb * nyb * k.nz);
    if (!c->nbmask || (c->tile_flags.size() == n && c->tile_flags_tw == tw && c->tile_flags_th == th)) return LBM_OK;
    uint8_t* d = nullptr;
    BCK(b, cudaMalloc((void**)&d, n));
    c->tile_flags.assign(n, 1);
    c->tile_flags_tw = tw;
    c->tile_flags_th = th;
    tile_flags_kernel<<<dim3((unsigned)nxb, (unsigned)nyb, (unsigned)k.nz), dim3(tw, th), 0, b->stream>>>(
        c->nbmask, k.nx, k.ny, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->tile_flags.data(), d, n, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    cudaFree(d);
    if (e != cudaSuccess) {
        c->tile_flags.clear();
        return bfail(b, LBM_ERR_CUDA, std::string("tile flags: ") + cudaGetErrorString(e));
    }
    return LBM_OK;
}

// Tiles of the members of a chain: tw x th cells in (x, y) (the groups' shape) and a chunk of at most zc z planes (the
// group's fixed zchunk, a member's own, or automatic).  A tile with planes that need solid handling (a cell with
// a solid neighbour: mask, or the first / last plane, row or column next to a wall) names them in its bits, and
// its march switches from plane to plane; only those planes pay for the solid tests.  (As marches of their own
// they paid for their start, too: figures at collide_batch_kernel.)  The first and the last plane of a column are tiles of
// their own where the plane beside them needs no solid handling, as at walls in z: four 40^3 domains 16.4 us a step
// (D3Q19) and 22.4 (D3Q27) so, 17.6 and 28.4 as part of the column's first and last chunks.
//
// Where a row leaves 1 .. 16 cells past its last full tile width (tw = 32), those cells form narrow
// columns, 16 cells wide and twice as high, which the same blocks step (BatchTile::narrow): a
// 32-wide tile there would leave 16 to 31 of its 32 lanes per row idle.
//
// The density/psi pass covers a member as runs of consecutive cells of whole planes: it needs no stencil, so
// nothing ties its threads to rows, and rows that do not fill a tile's width leave no lanes idle.  Rows, th
// at a time, in which some column has solid neighbours form runs of their own.  us a step of four 96^3 domains
// with a post along z, runs with and without by planes / by rows: D3Q19 153 / 145, D3Q27 221 / 212.
#ifndef LBM_BATCH_NARROW
#define LBM_BATCH_NARROW 1
#endif
#ifndef LBM_BATCH_LPT
#define LBM_BATCH_LPT 1
#endif

struct Column {
    int x0, y0, w, h, narrow;
};

// the columns of a member for tiles tw x th: full-width columns, then the narrow ones (if any)
std::vector<Column> member_columns(const KParams& k, int tw, int th) {
    std::vector<Column> cols;
    const int r = k.nx % tw;
    const bool narrow = LBM_BATCH_NARROW && tw > lbm::BATCH_NARROW_BX && r > 0 && r <= lbm::BATCH_NARROW_BX;
    const int wmain = narrow ? k.nx - r : k.nx;
    for (int y0 = 0; y0 < k.ny; y0 += th)
        for (int x0 = 0; x0 < wmain; x0 += tw) cols.push_back({x0, y0, tw, th, 0});
    if (narrow) {
        const int hn = tw * th / lbm::BATCH_NARROW_BX;
        for (int y0 = 0; y0 < k.ny; y0 += hn) cols.push_back({wmain, y0, lbm::BATCH_NARROW_BX, hn, 1});
    }
    return cols;
}

// Automatic z-chunk of a chain: blocks of zc planes over all its columns.  Few column-planes: the shortest
// time of the latency / throughput model that choose_zchunk (kernels_impl.cuh) explains; many: four waves
// of resident blocks, at most ZC_AUTO_MAX planes.
int auto_zchunk(const lbm_batch* b, const Chain& c, int resident, int tw, int th) {
    const double sms = b->sms, cap = sms * resident, ratio = c.Q == 19 ? 6.1 : 5.0;
    double planes = 0.0;
    long long cols = 0;
    for (int i : c.members) {
        const long long n = (long long)member_columns(b->members[i]->kp, tw, th).size();
        cols += n;
        planes += (double)n * b->members[i]->kp.nz;
    }
    if (planes >= 17.0 * cap) {
        const double chunks = std::max(1.0, std::ceil(4.0 * cap / std::max(cols, 1LL)));
        return std::min(ZC_AUTO_MAX, std::max(1, (int)std::ceil(planes / std::max(cols, 1LL) / chunks)));
    }
    int best = 1;
    double best_cost = 1e300;
    for (int zc = 1; zc <= ZC_AUTO_MAX; ++zc) {
        double blocks = 0.0;
        for (int i : c.members) {
            const KParams& k = b->members[i]->kp;
            blocks += (double)member_columns(k, tw, th).size() * ((k.nz + zc - 1) / zc);
        }
        const double waves = blocks / cap, B = (zc + 2) * ratio;
        const double A = blocks / sms * (zc + 1) * (1.0 + 0.15 * (std::ceil(waves) / waves - 1.0));
        const double cost = std::max(B, A + 0.35 * B);
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = zc;
        }
    }
    return best;
}

lbm_status build_chain(lbm_batch* b, Chain& c) {
    free_chain(c);
    c.masks.clear();
    for (int i : c.members) c.masks.push_back(b->members[i]->mask_id);
    Group& plain = b->groups[c.plain];
    Group* solid = c.solid >= 0 ? &b->groups[c.solid] : nullptr;
    if (plain.shape < 0 || plain.shape >= lbm::BATCH_NSHAPES) return bfail(b, LBM_ERR_ARG, "unknown tile shape");
    const lbm::BatchShape& sh = lbm::BATCH_SHAPES[plain.shape];
    const int tw = sh.bx, th = sh.by;
    const int fw = lbm::BATCH_NARROW_BX, fh = th;   // mask flags grid: both column kinds are unions of its cells
    const int zauto = auto_zchunk(b, c, c.Q == 19 ? sh.minb19 : sh.minb27, tw, th);
    double cells = 0.0;
    for (int i : c.members) cells += (double)b->members[i]->kp.ncell;
    // 2048 cells a run, fewer where that would leave SMs without their eight blocks
    const uint32_t run_cells = 256u * (uint32_t)std::min(8.0, std::max(1.0, cells / (b->sms * 8.0 * 256.0)));
    std::vector<uint8_t> need;      // per plane of one column: needs solid handling
    std::vector<uint8_t> rows;      // per plane and th rows: some column needs solid handling
    for (size_t j0 = 0; j0 < c.members.size(); j0 += lbm::BATCH_LAUNCH_DOMS) {
        const int nd = (int)std::min(c.members.size() - j0, (size_t)lbm::BATCH_LAUNCH_DOMS);
        c.launches.emplace_back();
        Launch& L = c.launches.back();
        std::vector<BatchTile> t;
        std::vector<BatchRun> runs;
        for (int d = 0; d < nd; ++d) {   // d: slot in the launch's member table
            L.tab.d[d] = b->table[c.members[j0 + d]];
            lbm_ctx* ctx = b->members[c.members[j0 + d]];
            const KParams& k = ctx->kp;
            const bool solid_work = has_solid_work(ctx);
            lbm_status fs = member_tile_flags(b, ctx, fw, fh);
            if (fs != LBM_OK) return fs;
            auto chunk = [&](const Group& g) {   // the batch's tuned choice, the member's own setting, automatic
                const int zc = g.zchunk > 0 ? g.zchunk : (k.zchunk > 0 ? k.zchunk : zauto);
                return std::min(zc, k.nz);
            };
            const int zc[2] = {chunk(plain), chunk(solid ? *solid : plain)};
            const int nxf = (k.nx + fw - 1) / fw, nyf = (k.ny + fh - 1) / fh;
            need.resize(k.nz);
            const int nrow = (k.ny + th - 1) / th;
            rows.assign((size_t)nrow * k.nz, 0);
            const size_t member_t0 = t.size();
            for (const Column& col : member_columns(k, tw, th)) {
                const bool side = (k.wall_x && (col.x0 == 0 || col.x0 + col.w >= k.nx)) ||
                                  (k.wall_y && (col.y0 == 0 || col.y0 + col.h >= k.ny));
                const int fx0 = col.x0 / fw, fx1 = std::min(nxf, (col.x0 + col.w + fw - 1) / fw);
                const int fy0 = col.y0 / fh, fy1 = std::min(nyf, (col.y0 + col.h + fh - 1) / fh);
                for (int z = 0; z < k.nz; ++z) {
                    bool s2 = solid_work && (side || (k.wall_z && (z == 0 || z == k.nz - 1)));
                    if (solid_work && ctx->nbmask)
                        for (int fy = fy0; fy < fy1 && !s2; ++fy)
                            for (int fx = fx0; fx < fx1 && !s2; ++fx)
                                s2 = ctx->tile_flags[((size_t)z * nyf + fy) * nxf + fx] != 0;
                    need[z] = s2 ? 1 : 0;
                    for (int y = col.y0; s2 && y < std::min(col.y0 + col.h, k.ny); y += th) rows[(size_t)z * nrow + y / th] = 1;
                }
                auto tile = [&](int z0, int n, uint32_t near) {
                    t.push_back({d, col.x0, col.y0, z0, n, col.narrow, near});
                    (near ? *solid : plain).ntiles += 1;
                };
                auto any = [&](int z0, int n) { return std::find(&need[z0], &need[z0] + n, 1) != &need[z0] + n; };
                const int first = k.nz > 1 && need[0] && !need[1] ? 1 : 0;
                const int last = k.nz - (k.nz > 2 && need[k.nz - 1] && !need[k.nz - 2] ? 1 : 0);
                if (first) tile(0, 1, 1u);
                for (int z0 = first; z0 < last;) {
                    int n = std::min(zc[0], last - z0);
                    uint32_t near = 0;
                    if (any(z0, n)) {   // by the solid group's z-chunk
                        n = std::min(std::min(zc[1], 32), last - z0);
                        for (int j = 0; j < n; ++j) near |= (uint32_t)need[z0 + j] << j;
                    }
                    tile(z0, n, near);
                    if (near) L.near = lbm::NEAR_SOME;
                    z0 += n;
                }
                if (last < k.nz) tile(last, 1, 1u);
                if ((first || last < k.nz) && L.near == lbm::NEAR_NONE) L.near = lbm::NEAR_ENDS;
            }
            // z-chunk-major order within the member (as the single-domain grid): blocks resident at
            // the same time work on neighbouring columns of the same planes
            std::stable_sort(t.begin() + member_t0, t.end(), [](const BatchTile& a, const BatchTile& b2) {
                return a.z0 != b2.z0 ? a.z0 < b2.z0 : (a.y0 != b2.y0 ? a.y0 < b2.y0 : a.x0 < b2.x0);
            });
            // the rows in the order of the cells: those before block j of th rows
            auto cells_before = [&](int j) {
                return ((uint32_t)(j / nrow) * (uint32_t)k.ny + (uint32_t)(j % nrow * th)) * (uint32_t)k.nx;
            };
            const int blocks = nrow * k.nz;
            for (int j0 = 0; j0 < blocks;) {
                int j1 = j0 + 1;
                while (j1 < blocks && rows[j1] == rows[j0]) ++j1;
                const uint32_t end = cells_before(j1);
                for (uint32_t a = cells_before(j0); a < end; a += std::min(run_cells, end - a))
                    runs.push_back({d, a, a + std::min(run_cells, end - a), rows[j0]});
                j0 = j1;
            }
        }
        // longest marches first within a launch: blocks start roughly in index order, so the short ones
        // fill the last wave instead of a few long ones running on alone
        if (LBM_BATCH_LPT)
            std::stable_sort(t.begin(), t.end(), [](const BatchTile& a, const BatchTile& b2) { return a.zc > b2.zc; });
        // against the collide pass's direction: the pass starts on what that one left in the L2
        std::reverse(runs.begin(), runs.end());
        if (t.size() > 0x7fffffff || runs.size() > 0x7fffffff) return bfail(b, LBM_ERR_ARG, "too many tiles");
        // Wall planes in a kernel whose plain tiles keep their registers, or in one that takes any tile: the latter
        // is faster on D3Q27 in launches of many waves (us a step with walls in z: four 96^3, 3744 tiles, 220.9 / 218.8, ten of
        // 48^3 - 102^3 311.8 / 305.6; but four 72^3, 3060 tiles, 101.6 / 104.0 and four 40^3 21.3 / 22.4; D3Q19 four 96^3
        // 147.4 / 149.1).
        if (L.near == lbm::NEAR_ENDS && c.Q == 27 && t.size() > 4.5 * b->sms * sh.minb27) L.near = lbm::NEAR_SOME;
        L.nt = (int)t.size();
        L.nr = (int)runs.size();
        if (L.nt > 0) {
            BCK(b, cudaMalloc((void**)&L.tiles, t.size() * sizeof(BatchTile)));
            BCK(b, cudaMemcpyAsync(L.tiles, t.data(), t.size() * sizeof(BatchTile), cudaMemcpyHostToDevice, b->stream));
        }
        if (L.nr > 0) {
            BCK(b, cudaMalloc((void**)&L.runs, runs.size() * sizeof(BatchRun)));
            BCK(b, cudaMemcpyAsync(L.runs, runs.data(), runs.size() * sizeof(BatchRun), cudaMemcpyHostToDevice, b->stream));
        }
        BCK(b, cudaStreamSynchronize(b->stream));   // t and runs go
    }
    c.built = true;
    return LBM_OK;
}

// Rebuilds the tiles of every chain (only of the one with group `only`, if that is not negative).
lbm_status build_chains(lbm_batch* b, int only = -1) {
    drop_graph(b);
    for (Chain& c : b->chains) {
        if (only >= 0 && c.plain != only && c.solid != only) continue;
        b->groups[c.plain].ntiles = 0;
        if (c.solid >= 0) b->groups[c.solid].ntiles = 0;
        lbm_status s = build_chain(b, c);
        if (s != LBM_OK) return s;
    }
    return LBM_OK;
}

cudaError_t collide_chain(const lbm_batch* b, const Chain& c, int parity, cudaStream_t st) {
    const Group& g = b->groups[c.plain];
    for (const Launch& L : c.launches) {
        cudaError_t e = c.Q == 19 ? lbm::launch_collide_batch_q19(g.phys, L.tab, L.tiles, L.nt, parity, L.near, g.shape, st)
                                  : lbm::launch_collide_batch_q27(g.phys, L.tab, L.tiles, L.nt, parity, L.near, g.shape, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t psi_chain(const lbm_batch* b, const Chain& c, int parity, cudaStream_t st) {
    const Group& g = b->groups[c.plain];
    if (!g.phys.multiphase) return cudaSuccess;
    for (const Launch& L : c.launches) {
        cudaError_t e = c.Q == 19 ? lbm::launch_psi_runs_q19(g.phys, L.tab, L.runs, L.nr, parity, L.near, st)
                                  : lbm::launch_psi_runs_q27(g.phys, L.tab, L.runs, L.nr, parity, L.near, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// (Re)build the groups, chains and tiles from the members' current parameters.  Members with walls or
// solids join both the plain group (interior tiles) and the solid-handling group of their physics.
lbm_status regroup(lbm_batch* b) {
    drop_graph(b);
    for (Chain& c : b->chains) free_chain(c);
    b->chains.clear();
    b->groups.clear();
    const int n = (int)b->members.size();
    b->seen.resize(n);
    b->table.resize(n);
    auto group_of = [&](int Q, int solids, const KParams& phys) -> int {
        for (size_t g = 0; g < b->groups.size(); ++g)
            if (b->groups[g].Q == Q && b->groups[g].solids == solids &&
                std::memcmp(&b->groups[g].phys, &phys, sizeof(KParams)) == 0)
                return (int)g;
        Group g;
        g.Q = Q;
        g.solids = solids;
        g.phys = phys;
        b->groups.push_back(g);
        return (int)b->groups.size() - 1;
    };
    for (int i = 0; i < n; ++i) {
        const lbm_ctx* c = b->members[i];
        if ((unsigned long long)c->Q * (unsigned long long)c->kp.plane > 0xFFFFFFFFull)
            return bfail(b, LBM_ERR_ARG, "a batch member holds 2^32 or more population values "
                                         "(Q x cells rounded up to 64); step it alone");
        std::memcpy(&b->seen[i], &c->kp, sizeof(KParams));
        b->table[i] = dom_of(c);
        const KParams phys = physics_of(c->kp);
        const int plain = group_of(c->Q, 0, phys), solid = has_solid_work(c) ? group_of(c->Q, 1, phys) : -1;
        b->groups[plain].members.push_back(i);
        if (solid >= 0) b->groups[solid].members.push_back(i);
        Chain* k = nullptr;
        for (Chain& c2 : b->chains)
            if (c2.plain == plain) k = &c2;
        if (!k) {
            b->chains.emplace_back();
            k = &b->chains.back();
            k->Q = c->Q;
            k->plain = plain;
        }
        if (solid >= 0) k->solid = solid;
        k->members.push_back(i);
    }
    return build_chains(b);
}

// Has any member changed (got or lost a solid mask) since the groups were built?
bool members_changed(const lbm_batch* b) {
    for (size_t i = 0; i < b->members.size(); ++i) {
        const BatchDom d = dom_of(b->members[i]);
        if (std::memcmp(&b->seen[i], &b->members[i]->kp, sizeof(KParams)) != 0 ||
            std::memcmp(&b->table[i], &d, sizeof(BatchDom)) != 0)
            return true;
    }
    return false;
}

// Brings groups, chains and tiles in line with members that were re-initialised: regroups if one got or lost a
// solid mask, re-tiles the chains with a member whose mask was given anew (it lies in the same buffers, and
// which planes of a column need solid handling depends on its cells) or that an earlier call failed to build;
// tuned shapes and z-chunks stay then.
lbm_status refresh(lbm_batch* b) {
    if (members_changed(b)) return regroup(b);
    for (Chain& c : b->chains) {
        bool same = c.built;
        for (size_t j = 0; same && j < c.members.size(); ++j) same = c.masks[j] == b->members[c.members[j]]->mask_id;
        if (!same) {
            lbm_status s = build_chains(b, c.plain);
            if (s != LBM_OK) return s;
        }
    }
    return LBM_OK;
}

// `steps` steps of every member from AA phase `parity` (psi of the current state valid).  Within a chain a step
// needs the one before it (psi reads populations that neighbouring tiles wrote, collide the psi halo); the chains
// have nothing in common, so each runs all these steps on a stream of its own, joined at the end.
cudaError_t step_all(lbm_batch* b, int parity, int steps, cudaStream_t st) {
    auto steps_of = [&](const Chain& c, cudaStream_t s) {
        cudaError_t e = cudaSuccess;
        for (int k = 0; k < steps && e == cudaSuccess; ++k) {
            const int p = parity ^ (k & 1);
            e = collide_chain(b, c, p, s);
            if (e == cudaSuccess) e = psi_chain(b, c, p ^ 1, s);
        }
        return e;
    };
    const size_t n = b->chains.size();
    if (n == 1) return steps_of(b->chains[0], st);
    cudaError_t e = cudaSuccess;
    if (!b->fork) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    while (e == cudaSuccess && b->side.size() < n) {
        cudaStream_t s2 = nullptr;
        cudaEvent_t ev = nullptr;
        e = cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking);
        if (e == cudaSuccess) {
            b->side.push_back(s2);
            e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
            if (e == cudaSuccess) b->done.push_back(ev);
        }
    }
    if (e == cudaSuccess) e = cudaEventRecord(b->fork, st);
    for (size_t k = 0; k < n && e == cudaSuccess; ++k) {
        e = cudaStreamWaitEvent(b->side[k], b->fork, 0);
        if (e == cudaSuccess) e = steps_of(b->chains[k], b->side[k]);
        if (e == cudaSuccess) e = cudaEventRecord(b->done[k], b->side[k]);
    }
    for (size_t k = 0; k < n && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(st, b->done[k], 0);
    return e;
}

// b->exec[parity][k]: GRAPH_STEPS[k] steps as one graph.  One set per AA phase: calls of an odd number of steps start
// from the other phase each time.  Recorded anew whenever the phase changed / kept, us a call of 65 steps: 4 chains of
// one 24^3 member each 1386 / 903, 24 chains 5230 / 2484; of 5 steps 185 / 93 and 792 / 290.
lbm_status record_graph(lbm_batch* b, int k, int parity) {
    if (!b->cap) BCK(b, cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
    BCK(b, cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = step_all(b, parity, GRAPH_STEPS[k], b->cap);
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(b->cap, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec[parity][k], g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        b->exec[parity][k] = nullptr;
        return bfail(b, LBM_ERR_CUDA, std::string("graph: ") + cudaGetErrorString(e));
    }
    return LBM_OK;
}

void advance_members(lbm_batch* b, int n) {
    for (lbm_ctx* c : b->members) {
        c->t += n;
        c->parity ^= (n & 1);
    }
}

}  // namespace

extern "C" {

lbm_status lbm_batch_create(lbm_ctx* const* ctxs, int32_t n, void* cuda_stream, lbm_batch** out) {
    if (!out) return bfail(nullptr, LBM_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!ctxs || n < 1) return bfail(nullptr, LBM_ERR_ARG, "a batch needs at least one context");
    for (int i = 0; i < n; ++i) {
        if (!ctxs[i]) return bfail(nullptr, LBM_ERR_ARG, "NULL context in the batch");
        if (!ctxs[i]->initialised) return bfail(nullptr, LBM_ERR_STATE, "every context must be initialised");
        if (ctxs[i]->f16)
            return bfail(nullptr, LBM_ERR_ARG, "contexts with the FP16 store cannot join a batch");
        if (ctxs[i]->onepass)
            return bfail(nullptr, LBM_ERR_ARG, "contexts with the one-pass layout cannot join a batch");
        if (ctxs[i]->parity != ctxs[0]->parity)
            return bfail(nullptr, LBM_ERR_STATE, "all contexts must have taken an equal number of steps mod 2");
        for (int j = 0; j < i; ++j)
            if (ctxs[j] == ctxs[i]) return bfail(nullptr, LBM_ERR_ARG, "a context appears twice in the batch");
    }
    lbm_batch* b = new lbm_batch();
    b->members.assign(ctxs, ctxs + n);
    b->stream = (cudaStream_t)cuda_stream;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0)
        b->sms = sms;
    lbm_status s = regroup(b);
    if (s == LBM_OK && cudaStreamSynchronize(b->stream) != cudaSuccess) s = bfail(b, LBM_ERR_CUDA, "batch set-up");
    if (s != LBM_OK) {
        lbm::set_thread_error(b->err.c_str());
        lbm_batch_destroy(b);
        return s;
    }
    *out = b;
    return LBM_OK;
}

lbm_status lbm_batch_step(lbm_batch* b, int32_t n) {
    if (!b) return LBM_ERR_ARG;
    if (n < 0) return bfail(b, LBM_ERR_ARG, "n must be >= 0");
    const int parity = b->members[0]->parity;
    for (const lbm_ctx* c : b->members) {
        if (c->parity != parity) return bfail(b, LBM_ERR_STATE, "members were stepped apart: AA phases differ");
        if (c->sticky != LBM_OK) return bfail(b, c->sticky, "a member has a sticky error: " + c->err);
    }
    lbm_status rs = refresh(b);
    if (rs != LBM_OK) return rs;
    cudaGraphExec_t* exec = b->exec[parity];
    int left = n;
    for (int k = 1; k >= 0; --k) {
        if (left < GRAPH_STEPS[k] || (k == 1 && !exec[1] && n < 4 * GRAPH_STEPS[1])) continue;
        if (!exec[k]) {
            lbm_status s = record_graph(b, k, parity);
            if (s != LBM_OK) return s;
        }
        for (; left >= GRAPH_STEPS[k]; left -= GRAPH_STEPS[k]) BCK(b, cudaGraphLaunch(exec[k], b->stream));
    }
    if (left > 0) BCK(b, step_all(b, parity ^ ((n - left) & 1), left, b->stream));
    advance_members(b, n);
    return LBM_OK;
}

lbm_status lbm_batch_sync(lbm_batch* b) {
    if (!b) return LBM_ERR_ARG;
    BCK(b, cudaStreamSynchronize(b->stream));
    lbm_status first = LBM_OK;
    for (lbm_ctx* c : b->members) {
        lbm_status s = lbm_sync(c);
        if (s != LBM_OK && first == LBM_OK) {
            first = s;
            b->err = lbm_last_error(c);
        }
    }
    return first;
}

}  // extern "C"

namespace {

// The group with the same lattice and physics and the other solid handling (-1 if none).  A member
// with solids has its solid-free tiles in one and the others in the other; both must be cut into the
// same columns (the same tile shape), or their tiles would not partition the member's cells.
int partner_group(const lbm_batch* b, int k) {
    const Group& g = b->groups[k];
    for (int j = 0; j < (int)b->groups.size(); ++j) {
        const Group& h = b->groups[j];
        if (j != k && h.Q == g.Q && h.solids != g.solids && std::memcmp(&h.phys, &g.phys, sizeof(KParams)) == 0)
            return j;
    }
    return -1;
}

// Times every chain's collide launches over `trial_steps` steps with each group set to candidate
// (shape_of(g, ci), zchunk_of(g, ci)) in turn, ci < ncand; times[ci][g] receives the total of the chains with
// group g.  The members advance by ncand x (trial_steps + 1) steps.
template <class SF, class ZF>
lbm_status time_candidates(lbm_batch* b, int trial_steps, int ncand, SF shape_of, ZF zchunk_of,
                           std::vector<std::vector<double>>& times) {
    const size_t G = b->groups.size();
    std::vector<const Chain*> chains;
    for (const Chain& c : b->chains) chains.push_back(&c);
    const size_t C = chains.size();
    times.assign(ncand, std::vector<double>(G, 0.0));
    std::vector<cudaEvent_t> ev(2 * C * trial_steps);
    for (auto& e : ev) BCK(b, cudaEventCreate(&e));
    lbm_status result = LBM_OK;
    for (int ci = 0; ci < ncand && result == LBM_OK; ++ci) {
        for (size_t k = 0; k < G; ++k) {
            b->groups[k].shape = shape_of((int)k, ci);
            b->groups[k].zchunk = zchunk_of((int)k, ci);
        }
        result = build_chains(b);
        if (result != LBM_OK) break;
        int parity = b->members[0]->parity;
        // one untimed step, then events around every chain's collide launches
        cudaError_t e = step_all(b, parity, 1, b->stream);
        parity ^= 1;
        for (int s = 0; s < trial_steps && e == cudaSuccess; ++s) {
            for (size_t k = 0; k < C && e == cudaSuccess; ++k) {
                e = cudaEventRecord(ev[2 * (s * C + k)], b->stream);
                if (e == cudaSuccess) e = collide_chain(b, *chains[k], parity, b->stream);
                if (e == cudaSuccess) e = cudaEventRecord(ev[2 * (s * C + k) + 1], b->stream);
            }
            for (size_t k = 0; k < C && e == cudaSuccess; ++k) e = psi_chain(b, *chains[k], parity ^ 1, b->stream);
            parity ^= 1;
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        if (e != cudaSuccess) {
            result = bfail(b, LBM_ERR_CUDA, std::string("tuning: ") + cudaGetErrorString(e));
            break;
        }
        advance_members(b, trial_steps + 1);
        for (size_t k = 0; k < C; ++k)
            for (int s = 0; s < trial_steps; ++s) {
                float ms = 0.f;
                cudaEventElapsedTime(&ms, ev[2 * (s * C + k)], ev[2 * (s * C + k) + 1]);
                times[ci][chains[k]->plain] += ms;
                if (chains[k]->solid >= 0) times[ci][chains[k]->solid] += ms;
            }
    }
    for (auto& e : ev) cudaEventDestroy(e);
    return result;
}

}  // namespace

extern "C" {

lbm_status lbm_batch_tune(lbm_batch* b, int32_t trial_steps, int32_t* zchunk_out, int32_t max_groups) {
    if (!b) return LBM_ERR_ARG;
    if (trial_steps < 1) return bfail(b, LBM_ERR_ARG, "trial_steps must be >= 1");
    lbm_status rs = refresh(b);
    if (rs != LBM_OK) return rs;
    const int G = (int)b->groups.size();
    std::vector<std::vector<double>> t;
    // stage 1: every tile shape (on all groups at once) with automatic z-chunks; a group and its
    // partner take the shape that minimises their summed time
    lbm_status r = time_candidates(
        b, trial_steps, lbm::BATCH_NSHAPES, [](int, int ci) { return ci; }, [](int, int) { return 0; }, t);
    if (r != LBM_OK) return r;
    std::vector<int> shape(G, 0), zchunk(G, 0);
    for (int k = 0; k < G; ++k) {
        const int p = partner_group(b, k);
        double best = 1e300;
        for (int ci = 0; ci < lbm::BATCH_NSHAPES; ++ci) {
            const double v = t[ci][k] + (p >= 0 ? t[ci][p] : 0.0);
            if (v < best) {
                best = v;
                shape[k] = ci;
            }
        }
    }
    // stage 2: the z-chunks for the chosen shapes, per group
    const int zc[] = {0, 1, 4, 8, 16, 32, ZC_WHOLE};
    const int nz = (int)(sizeof(zc) / sizeof(zc[0]));
    r = time_candidates(
        b, trial_steps, nz, [&](int k, int) { return shape[k]; }, [&](int, int ci) { return zc[ci]; }, t);
    if (r != LBM_OK) return r;
    for (int k = 0; k < G; ++k) {
        double best = 1e300;
        for (int ci = 0; ci < nz; ++ci)
            if (t[ci][k] < best) {
                best = t[ci][k];
                zchunk[k] = zc[ci];
            }
    }
    for (int k = 0; k < G; ++k) {
        b->groups[k].shape = shape[k];
        b->groups[k].zchunk = zchunk[k];
        if (zchunk_out && k < max_groups) zchunk_out[k] = zchunk[k];
    }
    return build_chains(b);
}

lbm_status lbm_batch_group(const lbm_batch* b, int32_t group, int32_t* lattice, int32_t* solids, int32_t* shape,
                           int32_t* zchunk) {
    if (!b) return LBM_ERR_ARG;
    if (group < 0 || group >= (int32_t)b->groups.size()) return LBM_ERR_ARG;
    const Group& g = b->groups[group];
    if (lattice) *lattice = g.Q;
    if (solids) *solids = g.solids;
    if (shape) *shape = g.shape;
    if (zchunk) *zchunk = g.zchunk;
    return LBM_OK;
}

lbm_status lbm_batch_set_group(lbm_batch* b, int32_t group, int32_t shape, int32_t zchunk) {
    if (!b) return LBM_ERR_ARG;
    if (group < 0 || group >= (int32_t)b->groups.size()) return bfail(b, LBM_ERR_ARG, "no such group");
    if (shape < 0 || shape >= lbm::BATCH_NSHAPES) return bfail(b, LBM_ERR_ARG, "shape must lie in [0, LBM_BATCH_SHAPES)");
    if (zchunk < 0) return bfail(b, LBM_ERR_ARG, "zchunk must be >= 0");
    if (members_changed(b)) {   // the chain's tiles may need a group that is not there yet
        lbm_status s = regroup(b);
        if (s != LBM_OK) return s;
        if (group >= (int32_t)b->groups.size()) return bfail(b, LBM_ERR_ARG, "no such group");
    }
    b->groups[group].shape = shape;
    b->groups[group].zchunk = zchunk;
    const int p = partner_group(b, group);
    if (p >= 0) b->groups[p].shape = shape;   // the partner takes the same columns
    return build_chains(b, group);
}

lbm_status lbm_batch_info(const lbm_batch* b, int32_t* ngroups, int32_t* ntiles, int32_t* graph_mode) {
    if (!b) return LBM_ERR_ARG;
    if (ngroups) *ngroups = (int32_t)b->groups.size();
    if (ntiles) {
        long long t = 0;
        for (const Group& g : b->groups) t += g.ntiles;
        *ntiles = (int32_t)std::min<long long>(t, 0x7fffffff);
    }
    if (graph_mode) *graph_mode = b->exec[0][0] || b->exec[0][1] || b->exec[1][0] || b->exec[1][1] ? 2 : 0;
    return LBM_OK;
}

void lbm_batch_destroy(lbm_batch* b) {
    if (!b) return;
    (void)cudaStreamSynchronize(b->stream);
    drop_graph(b);
    for (Chain& c : b->chains) free_chain(c);
    if (b->cap) cudaStreamDestroy(b->cap);
    for (cudaStream_t s2 : b->side) cudaStreamDestroy(s2);
    for (cudaEvent_t ev : b->done) cudaEventDestroy(ev);
    if (b->fork) cudaEventDestroy(b->fork);
    delete b;
}

const char* lbm_batch_last_error(const lbm_batch* b) { return b ? b->err.c_str() : lbm_last_error(nullptr); }

}  // extern "C"
