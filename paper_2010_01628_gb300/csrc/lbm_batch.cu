// lbm_batch.cu -- batched parameter sweeps: many independent domains of
// uneven sizes advanced together, one launch per pass of a step over the nodes
// of all of them (lbm_step replays 16 steps per graph).
//
// Work decomposition: every domain is cut into tiles of `threads` consecutive
// nodes (x fastest), one CTA per tile.  The first tiles and the parameters (size,
// boundaries, omega, g, Hartmann field, colour densities and surface tension,
// Shan-Chen interaction strength...) of up to BATCH_TAB domains are kernel
// parameters: a CTA finds its domain by a binary search in the constant bank and
// starts its pulls at once (the same tables in global memory put two dependent
// loads before them: 64-domain Shan-Chen sweep 18.6 GLUPS instead of 27.4).
// More domains take more launches, or one with the tables in device memory
// (batch_many).  The colour-gradient and Shan-Chen steps take two passes (order
// parameter or pseudopotential, then collision).
//
// A launch per pass beats a persistent kernel that holds both passes and
// synchronises the grid between them: each pass keeps its own register count
// (32-48 instead of the joint 64), may use the read-only load path, and the
// launch boundary as a graph node costs less than a grid barrier did.
// Persistent -> per pass, FP32, GB300, GLUPS: 64 domains of 32..96^3: MHD 19.8
// -> 21.9 (7.0 TB/s at 320 B per update: HBM-bound), Shan-Chen 20.8 -> 27.4,
// colour gradient 14.1 -> 16.0, fluid 41.1 -> 46.4 (HBM-bound); 4 domains of
// 32^3 (latency-bound): 11.4 -> 18.8, 9.8 -> 15.9, 8.0 -> 10.8, 20 -> 30.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "lbm_cgm.cuh"
#include "lbm_fluid.cuh"
#include "lbm_internal.h"
#include "lbm_mhd.cuh"
#include "lbm_sc.cuh"

namespace lbm {

struct BatchDomain {
    FluidArgs fl;     // box, omega, g, lid
    MhdArgs mh;       // box, omega, tau_m, g, b_wall
    CgmArgs cg;       // box, omega, alpha_r, alpha_b, A, beta, g, rho_ref g
    ScArgs sc;        // box, omega, G, g, rho_ref g, lid
    size_t off;       // element offset of the domain's plane 0 in a state copy
    size_t soff;      // offset of the domain's node 0 in each scratch plane (colour gradient)
    FastDiv div_nx, div_ny;
};

struct BarrierState {
    unsigned int count;
    unsigned int gen;
    int err;
    int pad;
};

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Sense-counting grid barrier with a bounded wait.  `expected` is the number
// of CTAs that must arrive.  Returns false (and every CTA should return) if the
// wait timed out here or an error was raised elsewhere.
__device__ bool grid_barrier(BarrierState* bs, unsigned expected, unsigned long long timeout_ns) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned* vgen = &bs->gen;
        volatile int* verr = &bs->err;
        const unsigned g = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(&bs->count, 1u) + 1u;
        int res = 1;
        if (arrived == expected) {
            atomicExch(&bs->count, 0u);
            __threadfence();
            atomicAdd(&bs->gen, 1u);
        } else {
            const unsigned long long t0 = globaltimer_ns();
            while (*vgen == g) {
                if (*verr != 0) {
                    res = 0;
                    break;
                }
                if (globaltimer_ns() - t0 > timeout_ns) {
                    atomicCAS(&bs->err, 0, (int)LBM_ERR_TIMEOUT);
                    res = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        ok = res;
    }
    __syncthreads();
    return ok != 0;
}

// Domains [first, first + nd) of the batch, as a kernel parameter.
constexpr int BATCH_TAB = 128;
template <class Args>
struct BatchRec {
    Args a;          // starts with its Box
    size_t off;      // element offset of the domain's plane 0 in a state copy
    size_t soff;     // offset of its node 0 in each scratch plane
    FastDiv div_nx, div_ny;  // node -> row -> plane
};
template <class Args>
struct BatchTab {
    int nd;
    uint32_t tile0[BATCH_TAB];
    BatchRec<Args> rec[BATCH_TAB];
};
// All domains of the batch, in global memory.
template <class Args>
struct BatchRecAt {
    BatchRec<Args> r;
    uint32_t tile0;
};
template <class Args>
struct BatchMany {
    const BatchRecAt<Args>* rec;
    const uint32_t* domain;  // of each tile
};

template <int PHYS> struct BatchArgs;
template <> struct BatchArgs<LBM_PHYS_FLUID> { using T = FluidArgs; };
template <> struct BatchArgs<LBM_PHYS_MHD> { using T = MhdArgs; };
template <> struct BatchArgs<LBM_PHYS_CGM> { using T = CgmArgs; };
template <> struct BatchArgs<LBM_PHYS_SC> { using T = ScArgs; };

// One pass of one step.  scratch (colour gradient, Shan-Chen): phi (psi) of
// every domain's nodes, then rho_r, each `scratch_n` values long.  WALLS: false
// when every domain is periodic in all three directions (the node code then
// carries no bounce-back).
// CTAs of 256 threads per SM the passes are held to.  Unbounded, the
// parameters picked from the constant bank at a run-time index fill up to 128
// registers (FP32 Shan-Chen sweep 19.7 GLUPS, 27.4 at these bounds; colour gradient
// 14.4, 15.2 at 4 and 16.0 at 5 CTAs).  In FP64 MHD (136 registers) and the colour
// gradient (156) left one CTA per SM, whose start and end nothing covered: 64 x 64^3
// 12.2 -> 11.6 ms and 19.1 -> 18.5 ms a step at two.
constexpr int batch_ctas(int phys, int pass, size_t elem) {
    if (elem != 4) return phys == LBM_PHYS_MHD || phys == LBM_PHYS_CGM ? 2 : 1;
    if (phys == LBM_PHYS_MHD) return 4;
    if (phys == LBM_PHYS_SC) return pass == 0 ? 6 : 5;
    if (phys == LBM_PHYS_CGM) return 5;
    return 6;
}
template <class Args>
__device__ __forceinline__ const BatchRec<Args>& batch_domain(const BatchTab<Args>& tab, uint32_t& tile0) {
    int lo = 0, hi = tab.nd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab.tile0[mid] <= blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    tile0 = tab.tile0[lo];
    return tab.rec[lo];
}
template <class Args>
__device__ __forceinline__ const BatchRec<Args>& batch_domain(const BatchMany<Args>& tab, uint32_t& tile0) {
    const BatchRecAt<Args>& at = tab.rec[__ldg(tab.domain + blockIdx.x)];
    tile0 = at.tile0;
    return at.r;
}
template <int PHYS, int PASS, typename S, typename C, bool WALLS, class Tab>
__global__ void __launch_bounds__(256, batch_ctas(PHYS, PASS, sizeof(S)))
    batch_pass_kernel(const S* __restrict__ src, S* __restrict__ dst, C* __restrict__ scratch, size_t scratch_n,
                      const __grid_constant__ Tab tab) {
    uint32_t tile0;
    const auto& D = batch_domain(tab, tile0);
    const Box& b = D.a.box;
    const uint32_t cell = (blockIdx.x - tile0) * blockDim.x + threadIdx.x;
    if (cell >= (uint32_t)b.n) return;
    const uint32_t row = fast_div(cell, D.div_nx);
    const int x = (int)(cell - row * (uint32_t)b.nx);
    const int z = (int)fast_div(row, D.div_ny);
    const int y = (int)(row - (uint32_t)z * (uint32_t)b.ny);
    if constexpr (PHYS == LBM_PHYS_SC && PASS == 0)
        sc_psi_node<S, C, WALLS>(src + D.off, scratch + D.soff, D.a, x, y, z);
    else if constexpr (PHYS == LBM_PHYS_SC)
        sc_collide_node<S, C, WALLS>(src + D.off, dst + D.off, scratch + D.soff, D.a, x, y, z);
    else if constexpr (PHYS == LBM_PHYS_CGM && PASS == 0)
        cgm_phi_node<S, C, WALLS>(src + D.off, scratch + D.soff, scratch + scratch_n + D.soff, D.a, x, y, z);
    else if constexpr (PHYS == LBM_PHYS_CGM)
        cgm_collide_node<S, C, WALLS>(src + D.off, dst + D.off, scratch + D.soff, scratch + scratch_n + D.soff,
                                           D.a, x, y, z);
    else if constexpr (PHYS == LBM_PHYS_MHD)
        mhd_node<S, C, WALLS>(src + D.off, dst + D.off, D.a, x, y, z);
    else
        fluid_node<S, C, WALLS>(src + D.off, dst + D.off, D.a, x, y, z);
}

// Diagnostic, of use on its own: no step contains a grid barrier.  One that waits
// for a CTA more than the grid has, so every wait runs into its (short) limit; used
// to check that bounded waits end and report LBM_ERR_TIMEOUT.
__global__ void barrier_selftest_kernel(BarrierState* bs, unsigned long long timeout_ns) {
    grid_barrier(bs, gridDim.x + 1, timeout_ns);
}

}  // namespace lbm

using lbm::BarrierState;
using lbm::BatchDomain;

struct BatchState {
    int nd = 0;
    std::vector<lbm_ctx*> views;
    std::vector<BatchDomain> doms;
    bool many = false;                // tables in device memory, one launch a pass
    std::vector<unsigned char> tabs;  // a BatchTab per launch of a pass, or (many) all records
    std::vector<uint32_t> tiles;      // CTAs of each launch
    std::vector<uint32_t> domain;     // many: domain of each tile
    // many: device copies, by threads / 32; written once, as a caller's graph may
    // hold steps of an earlier CTA size
    struct {
        void* rec = nullptr;
        uint32_t* domain = nullptr;
    } device[256 / 32 + 1];
    uint32_t ntiles = 0;
    int threads = 256;
    size_t state_elems = 0;
    size_t scratch_n = 0;  // values per scratch plane (colour gradient: all domains' nodes)
    bool walls = true;     // false: every domain periodic in x, y and z
};

namespace {

// Whether a batch keeps its tables in device memory: more domains than one
// launch's parameters hold, and few nodes a launch.  One launch of all domains
// then beats a launch of 32 KB of parameters per 128 of them; large domains hide
// the launches, and in FP32 the parameters' constant bank is the faster table.
// us per step, 16-step graphs, parameters -> device memory: 1000 x 8^3 fluid FP32
// 24.6 -> 11.2, colour gradient 83 -> 38, 4000 x 6^3 Shan-Chen 170 -> 39, 129 x 8^3
// Shan-Chen FP64 80 -> 53; 512 x 16^3 (2^19 nodes a launch) FP32 0.92 .. 1.03, 1000
// x 20^3 (10^6) 0.93 .. 1.06, 130 x 64^3 1.00 .. 1.13; FP64 0.92 .. 1.01 at every size.
bool batch_many(int ndomains, size_t cells, lbm_precision prec) {
    const size_t launches = (size_t)(ndomains + lbm::BATCH_TAB - 1) / lbm::BATCH_TAB;
    return launches > 1 && (prec == LBM_FP64 || cells < launches << 19);
}

const lbm::FluidArgs& args_of(const BatchDomain& d, lbm::FluidArgs*) { return d.fl; }
const lbm::MhdArgs& args_of(const BatchDomain& d, lbm::MhdArgs*) { return d.mh; }
const lbm::CgmArgs& args_of(const BatchDomain& d, lbm::CgmArgs*) { return d.cg; }
const lbm::ScArgs& args_of(const BatchDomain& d, lbm::ScArgs*) { return d.sc; }

template <int PHYS>
using TabOf = lbm::BatchTab<typename lbm::BatchArgs<PHYS>::T>;
template <int PHYS>
using RecOf = lbm::BatchRecAt<typename lbm::BatchArgs<PHYS>::T>;
template <int PHYS>
size_t table_bytes_of(const BatchState* B) {
    static_assert(sizeof(TabOf<PHYS>) <= 32000, "kernel parameters are limited to 32,764 bytes");
    return B->many ? B->nd * sizeof(RecOf<PHYS>) : B->tiles.size() * sizeof(TabOf<PHYS>);
}
size_t table_bytes(const lbm_ctx* c) {
    switch (c->physics) {
        case LBM_PHYS_MHD: return table_bytes_of<LBM_PHYS_MHD>(c->batch);
        case LBM_PHYS_CGM: return table_bytes_of<LBM_PHYS_CGM>(c->batch);
        case LBM_PHYS_SC: return table_bytes_of<LBM_PHYS_SC>(c->batch);
        default: return table_bytes_of<LBM_PHYS_FLUID>(c->batch);
    }
}
uint32_t tiles_of(const BatchDomain& d, int threads) { return (uint32_t)((d.fl.box.n + threads - 1) / threads); }

template <int PHYS>
void fill_tables(BatchState* B) {
    using Args = typename lbm::BatchArgs<PHYS>::T;
    std::fill(B->tiles.begin(), B->tiles.end(), 0u);
    for (int d = 0; d < B->nd; ++d) {
        const BatchDomain& D = B->doms[d];
        const int launch = B->many ? 0 : d / lbm::BATCH_TAB;
        const uint32_t tile0 = B->tiles[launch], n = tiles_of(D, B->threads);
        lbm::BatchRec<Args>* r;
        if (B->many) {
            RecOf<PHYS>& at = ((RecOf<PHYS>*)B->tabs.data())[d];
            at.tile0 = tile0;
            std::fill_n(B->domain.begin() + tile0, n, (uint32_t)d);
            r = &at.r;
        } else {
            TabOf<PHYS>& t = ((TabOf<PHYS>*)B->tabs.data())[launch];
            const int k = d % lbm::BATCH_TAB;
            t.nd = k + 1;
            t.tile0[k] = tile0;
            r = &t.rec[k];
        }
        r->a = args_of(D, (Args*)nullptr);
        r->off = D.off;
        r->soff = D.soff;
        r->div_nx = D.div_nx;
        r->div_ny = D.div_ny;
        B->tiles[launch] += n;
    }
}

// Tiles and tables of the current CTA size.  A step allocates nothing: it runs
// behind a C entry point.
cudaError_t configure(lbm_ctx* c) {
    BatchState* B = c->batch;
    switch (c->physics) {
        case LBM_PHYS_MHD: fill_tables<LBM_PHYS_MHD>(B); break;
        case LBM_PHYS_CGM: fill_tables<LBM_PHYS_CGM>(B); break;
        case LBM_PHYS_SC: fill_tables<LBM_PHYS_SC>(B); break;
        default: fill_tables<LBM_PHYS_FLUID>(B); break;
    }
    B->ntiles = 0;
    for (uint32_t t : B->tiles) B->ntiles += t;
    c->block_x = B->threads;  // part of the launch shape that graphs are kept for
    auto& dev = B->device[B->threads / 32];
    if (!B->many || dev.domain) return cudaSuccess;
    void* rec = lbm_internal_dev_alloc(c, B->tabs.size());
    uint32_t* domain = (uint32_t*)lbm_internal_dev_alloc(c, sizeof(uint32_t) * B->ntiles);
    cudaError_t e = rec && domain ? cudaSuccess : cudaErrorMemoryAllocation;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(rec, B->tabs.data(), B->tabs.size(), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(domain, B->domain.data(), sizeof(uint32_t) * B->ntiles, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess) {
        dev.rec = rec;
        dev.domain = domain;
    } else {
        lbm_internal_dev_free(c, rec);
        lbm_internal_dev_free(c, domain);
    }
    return e;
}

template <int PHYS, typename S, typename C, bool WALLS, class Tab>
void step_launch(lbm_ctx* c, uint32_t tiles, const Tab& tab) {
    const S* src = (const S*)c->buf[c->cur];
    S* dst = (S*)c->buf[c->cur ^ 1];
    BatchState* B = c->batch;
    if constexpr (PHYS == LBM_PHYS_SC || PHYS == LBM_PHYS_CGM)
        launch_step(c, lbm::batch_pass_kernel<PHYS, 0, S, C, WALLS, Tab>, tiles, B->threads, 0, src, dst, (C*)c->phi,
                    B->scratch_n, tab);
    launch_step(c, lbm::batch_pass_kernel<PHYS, 1, S, C, WALLS, Tab>, tiles, B->threads, 0, src, dst, (C*)c->phi,
                B->scratch_n, tab);
}

template <int PHYS, typename S, typename C, bool WALLS>
cudaError_t steps_t(lbm_ctx* c, long n, bool dry) {
    BatchState* B = c->batch;
    for (long s = 0; s < n; ++s) {
        if (B->many)
            step_launch<PHYS, S, C, WALLS>(
                c, B->ntiles,
                lbm::BatchMany<typename lbm::BatchArgs<PHYS>::T>{(const RecOf<PHYS>*)B->device[B->threads / 32].rec,
                                                                 B->device[B->threads / 32].domain});
        else
            for (size_t k = 0; k < B->tiles.size(); ++k)
                step_launch<PHYS, S, C, WALLS>(c, B->tiles[k], ((const TabOf<PHYS>*)B->tabs.data())[k]);
        if (!dry) c->cur ^= 1;
    }
    return cudaGetLastError();
}

template <int PHYS>
cudaError_t steps_phys(lbm_ctx* c, long n, bool dry) {
    if (c->prec == LBM_FP64)
        return c->batch->walls ? steps_t<PHYS, double, double, true>(c, n, dry)
                               : steps_t<PHYS, double, double, false>(c, n, dry);
    return c->batch->walls ? steps_t<PHYS, float, float, true>(c, n, dry)
                           : steps_t<PHYS, float, float, false>(c, n, dry);
}

}  // namespace

namespace lbm {

cudaError_t batch_step(lbm_ctx* c, long n, bool dry) {
    switch (c->physics) {
        case LBM_PHYS_MHD: return steps_phys<LBM_PHYS_MHD>(c, n, dry);
        case LBM_PHYS_CGM: return steps_phys<LBM_PHYS_CGM>(c, n, dry);
        case LBM_PHYS_SC: return steps_phys<LBM_PHYS_SC>(c, n, dry);
        default: return steps_phys<LBM_PHYS_FLUID>(c, n, dry);
    }
}

cudaError_t batch_apply_config(lbm_ctx* c, int threads) {
    if (threads < BATCH_MIN_THREADS || threads > 256 || threads % 32 != 0) return cudaErrorInvalidValue;
    const int before = c->batch->threads;
    c->batch->threads = threads;
    const cudaError_t e = configure(c);
    if (e != cudaSuccess) {  // the former size's tables are there
        c->batch->threads = before;
        configure(c);
    }
    return e;
}

void batch_destroy(lbm_ctx* c) {
    BatchState* B = c->batch;
    if (!B) return;
    for (lbm_ctx* v : B->views) delete v;
    for (auto& dev : B->device) {
        lbm_internal_dev_free(c, dev.rec);
        lbm_internal_dev_free(c, dev.domain);
    }
    delete B;
    c->batch = nullptr;
}

}  // namespace lbm

// ---------------------------------------------------------------------------
extern "C" {

lbm_status lbm_batch_create(lbm_ctx** out, int ndomains, const lbm_grid* grids, const lbm_relax* relax,
                            const lbm_forcing* forcing, lbm_physics physics, const lbm_physparams* phys,
                            lbm_precision precision, void* cuda_stream) {
    if (!out || ndomains < 1 || !grids || !relax) return LBM_ERR_ARG;
    *out = nullptr;
    if (physics != LBM_PHYS_FLUID && physics != LBM_PHYS_MHD && physics != LBM_PHYS_CGM && physics != LBM_PHYS_SC)
        return LBM_ERR_UNSUPPORTED;
    if (precision != LBM_FP32 && precision != LBM_FP64) return LBM_ERR_UNSUPPORTED;
    if ((physics == LBM_PHYS_MHD || physics == LBM_PHYS_CGM || physics == LBM_PHYS_SC) && !phys) return LBM_ERR_ARG;
    const int planes = physics == LBM_PHYS_MHD ? 40 : (physics == LBM_PHYS_CGM ? 24 : 19);
    const size_t elem = precision == LBM_FP64 ? 8 : 4;
    size_t total = 0, max_plane = 0, cells = 0, max_tiles = 0;
    for (int d = 0; d < ndomains; ++d) {
        const lbm_grid& g = grids[d];
        if (g.nx < 1 || g.ny < 1 || g.nz < 1) return LBM_ERR_ARG;
        const double n = (double)g.nx * g.ny * g.nz;
        if (n >= 2147483648.0) return LBM_ERR_ARG;
        if (!(relax[d].omega > 0.0 && relax[d].omega < 2.0)) return LBM_ERR_ARG;
        if (relax[d].omega_bulk != 1.0 || relax[d].omega_3 != 1.0 || relax[d].omega_4 != 1.0)
            return LBM_ERR_UNSUPPORTED;
        if (physics == LBM_PHYS_MHD && !(phys[d].tau_m > 0.5)) return LBM_ERR_ARG;
        if (physics == LBM_PHYS_CGM &&
            !(phys[d].alpha_r >= 0.0 && phys[d].alpha_r < 1.0 && phys[d].alpha_b >= 0.0 && phys[d].alpha_b < 1.0))
            return LBM_ERR_ARG;
        if (physics == LBM_PHYS_SC && !std::isfinite(phys[d].G)) return LBM_ERR_ARG;
        if (forcing && forcing[d].rho_ref != 0.0 && physics != LBM_PHYS_CGM && physics != LBM_PHYS_SC)
            return LBM_ERR_UNSUPPORTED;
        if (g.wall_model != LBM_WALL_BOUNCE_BACK || relax[d].moment_space != LBM_MOMENTS_CENTRAL)
            return LBM_ERR_UNSUPPORTED;
        if ((physics == LBM_PHYS_MHD || physics == LBM_PHYS_CGM) && (g.periodic_mask & 2u) == 0 &&
            (g.lid_u[0] != 0.0 || g.lid_u[1] != 0.0 || g.lid_u[2] != 0.0))
            return LBM_ERR_UNSUPPORTED;
        const size_t nn = (size_t)g.nx * g.ny * g.nz;
        total += ((size_t)planes * nn + 63) / 64 * 64;  // each domain block starts 256-byte aligned
        max_plane = std::max(max_plane, (size_t)g.nx * g.ny);
        cells += nn;
        max_tiles += (nn + lbm::BATCH_MIN_THREADS - 1) / lbm::BATCH_MIN_THREADS;
    }
    lbm_ctx* c = new (std::nothrow) lbm_ctx();
    BatchState* B = new (std::nothrow) BatchState();
    if (!c || !B) {
        delete c;
        delete B;
        return LBM_ERR_OOM;
    }
    c->batch = B;
    c->owns = true;
    c->grid = grids[0];
    c->relax = relax[0];
    if (forcing) c->forcing = forcing[0];
    c->physics = physics;
    if (phys) c->phys = phys[0];
    c->prec = precision;
    c->stream = (cudaStream_t)cuda_stream;
    cudaGetDevice(&c->device);
    c->elem = elem;
    c->planes = planes;
    c->box.nx = c->box.ny = c->box.nz = 0;
    c->box.n = cells;
    B->nd = ndomains;
    lbm_status st = LBM_OK;
    try {
        B->doms.reserve(ndomains);
        B->views.reserve(ndomains);
        B->many = batch_many(ndomains, cells, precision);
        B->tiles.resize(B->many ? 1 : (ndomains + lbm::BATCH_TAB - 1) / lbm::BATCH_TAB);
        B->tabs.resize(table_bytes(c));
        if (B->many) B->domain.resize(max_tiles);
    } catch (const std::bad_alloc&) {
        st = LBM_ERR_OOM;
    }
    if (st == LBM_OK) st = lbm_internal_alloc_batch(c, total, cells, max_plane);
    if (st != LBM_OK) {
        lbm::batch_destroy(c);
        lbm_internal_release(c);
        delete c;
        return st;
    }
    B->state_elems = total;
    B->scratch_n = cells;
    B->walls = false;
    for (int d = 0; d < ndomains; ++d) B->walls = B->walls || (grids[d].periodic_mask & 7u) != 7u;
    cudaError_t e = cudaSuccess;
    size_t off = 0, uoff = 0, soff = 0;
    for (int d = 0; d < ndomains && e == cudaSuccess; ++d) {
        const lbm_grid& g = grids[d];
        BatchDomain D;
        std::memset(&D, 0, sizeof(D));
        D.fl.box.nx = g.nx;
        D.fl.box.ny = g.ny;
        D.fl.box.nz = g.nz;
        D.fl.box.periodic = g.periodic_mask & 7u;
        D.fl.box.n = (size_t)g.nx * g.ny * g.nz;
        D.div_nx = lbm::make_fast_div((uint32_t)g.nx);
        D.div_ny = lbm::make_fast_div((uint32_t)g.ny);
        D.fl.omega = relax[d].omega;
        for (int a = 0; a < 3; ++a) {
            D.fl.g[a] = forcing ? forcing[d].g[a] : 0.0;
            D.fl.lid[a] = (g.periodic_mask & 2u) ? 0.0 : g.lid_u[a];
        }
        D.mh.box = D.fl.box;
        D.mh.omega = relax[d].omega;
        if (physics == LBM_PHYS_MHD) {
            D.mh.tau_m = phys[d].tau_m;
            D.mh.inv_tau_m = 1.0 / phys[d].tau_m;
            D.mh.jfac = 1.0 / (phys[d].tau_m * lbm::CSM2);
            for (int a = 0; a < 3; ++a) {
                D.mh.g[a] = D.fl.g[a];
                D.mh.bw[a] = phys[d].b_wall[a];
            }
        }
        if (physics == LBM_PHYS_CGM) {
            D.cg.box = D.fl.box;
            D.cg.omega = relax[d].omega;
            D.cg.alpha_r = phys[d].alpha_r;
            D.cg.alpha_b = phys[d].alpha_b;
            D.cg.A = phys[d].A;
            D.cg.beta = phys[d].beta;
            for (int a = 0; a < 3; ++a) {
                D.cg.g[a] = D.fl.g[a];
                D.cg.rg[a] = forcing ? forcing[d].rho_ref * forcing[d].g[a] : 0.0;
            }
        }
        if (physics == LBM_PHYS_SC) {
            D.sc.box = D.fl.box;
            D.sc.omega = relax[d].omega;
            D.sc.G = phys[d].G;
            for (int a = 0; a < 3; ++a) {
                D.sc.g[a] = D.fl.g[a];
                D.sc.rg[a] = forcing ? forcing[d].rho_ref * forcing[d].g[a] : 0.0;
                D.sc.lid[a] = D.fl.lid[a];
            }
        }
        D.off = off;
        D.soff = soff;
        B->doms.push_back(D);
        // a view context per domain (init/fields/reduce/populations)
        lbm_ctx* v = new (std::nothrow) lbm_ctx();
        if (!v) {
            e = cudaErrorMemoryAllocation;
            break;
        }
        *v = *c;
        v->batch = nullptr;
        v->owns = false;
        v->parent = c;
        v->grid = g;
        v->relax = relax[d];
        if (forcing) v->forcing = forcing[d];
        else std::memset(&v->forcing, 0, sizeof(v->forcing));
        if (phys) v->phys = phys[d];
        v->box = D.fl.box;
        v->buf[0] = (char*)c->buf[0] + off * elem;
        v->buf[1] = (char*)c->buf[1] + off * elem;
        v->uprev = (char*)c->uprev + uoff * (precision == LBM_FP64 ? 8 : 4);  // compute-type velocities
        v->phi = c->phi ? (char*)c->phi + soff * (precision == LBM_FP64 ? 8 : 4) : nullptr;
        v->block_x = g.nx >= 256 ? 256 : (g.nx >= 128 ? 128 : (g.nx >= 64 ? 64 : 32));
        B->views.push_back(v);
        off += ((size_t)planes * D.fl.box.n + 63) / 64 * 64;
        uoff += 3 * D.fl.box.n;
        soff += D.fl.box.n;
    }
    if (e == cudaSuccess) e = configure(c);
    // rest state for every domain
    for (int d = 0; d < ndomains && e == cudaSuccess; ++d) {
        lbm_ctx* v = B->views[d];
        e = lbm_internal_init_rest(v);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        lbm::batch_destroy(c);
        lbm_internal_release(c);
        delete c;
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
    }
    *out = c;
    return LBM_OK;
}

lbm_status lbm_batch_domain(lbm_ctx* c, int d, lbm_ctx** view) {
    if (!c || !c->batch || !view || d < 0 || d >= c->batch->nd) return LBM_ERR_ARG;
    c->batch->views[d]->cur = c->cur;
    *view = c->batch->views[d];
    return LBM_OK;
}

lbm_status lbm_batch_step(lbm_ctx* c, long n) {
    if (!c || !c->batch || n < 0) return LBM_ERR_ARG;
    if (n == 0) return LBM_OK;
    const cudaError_t e = lbm_internal_run_steps(c, n);
    for (lbm_ctx* v : c->batch->views) v->cur = c->cur;
    if (e != cudaSuccess) {
        c->err = std::string("lbm_batch_step: ") + cudaGetErrorString(e);
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}

lbm_status lbm_batch_info(const lbm_ctx* c, int* threads, int* grid, int* graph, long* tiles) {
    if (!c || !c->batch) return LBM_ERR_ARG;
    if (threads) *threads = c->batch->threads;
    if (grid) *grid = (int)c->batch->ntiles;
    if (graph) *graph = c->graphs.failed ? 0 : 1;
    if (tiles) *tiles = (long)c->batch->ntiles;
    return LBM_OK;
}

lbm_status lbm_barrier_selftest(double timeout_s, int* observed) {
    if (!observed || !(timeout_s > 0.0) || timeout_s > 10.0) return LBM_ERR_ARG;
    BarrierState* bs = nullptr;
    if (cudaMalloc(&bs, sizeof(BarrierState)) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_OOM;
    }
    cudaError_t e = cudaMemset(bs, 0, sizeof(BarrierState));
    if (e == cudaSuccess) {
        lbm::barrier_selftest_kernel<<<4, 64>>>(bs, (unsigned long long)(timeout_s * 1e9));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    BarrierState h;
    if (e == cudaSuccess) e = cudaMemcpy(&h, bs, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(bs);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    *observed = h.err;
    return LBM_OK;
}

}  // extern "C"

size_t lbm_internal_batch_state_elems(const lbm_ctx* c) { return c->batch ? c->batch->state_elems : 0; }
