// lbm_mhd.cu -- magnetohydrodynamic step (Sec. III.F of arXiv:2010.01628):
// the single-phase CM step driven by the Lorentz force F = j x b, coupled to
// vector-valued magnetic populations (per-node update in lbm_mhd.cuh).
#include "lbm_mhd.cuh"
#include "lbm_internal.h"
#include "lbm_reduce.cuh"

namespace lbm {

template <typename S, typename C, bool WALLS, bool FLAT>
__global__ void __launch_bounds__(256) mhd_step_kernel(const S* __restrict__ src, S* __restrict__ dst, MhdArgs p,
                                                       FastDiv div_nx) {
    int x, y;
    if (!plane_node<FLAT>(p.box, div_nx, 0, p.box.ny, x, y)) return;
    mhd_node<S, C, WALLS>(src, dst, p, x, y, blockIdx.z);
}

template <typename S, typename C>
__global__ void mhd_init_kernel(S* __restrict__ dst, FieldsIn in, Box b, int z0, int nzs,
                                bool uniform) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, zs = blockIdx.z;
    if (x >= b.nx || zs >= nzs) return;
    const size_t k = ((size_t)zs * b.ny + y) * b.nx + x;
    const uint32_t self = ((uint32_t)(z0 + zs) * (uint32_t)b.ny + (uint32_t)y) * (uint32_t)b.nx + (uint32_t)x;
    C rho = (C)1, drho = (C)0, ux = (C)0, uy = (C)0, uz = (C)0;
    C bb[3] = {(C)0, (C)0, (C)0};
    if (!uniform) {
        drho = (C)(in.rho[k] - 1.0);
        rho = (C)in.rho[k];
        ux = (C)in.value(in.u[0], k);
        uy = (C)in.value(in.u[1], k);
        uz = (C)in.value(in.u[2], k);
        bb[0] = (C)in.value(in.B[0], k);
        bb[1] = (C)in.value(in.B[1], k);
        bb[2] = (C)in.value(in.B[2], k);
    }
    C f[Q];
    equilibrium_shifted<C>(rho, drho, ux, uy, uz, f);
    scatter19<S, C>(dst, b.n, self, f);
    S* gdst = dst + (size_t)Q * b.n;
    store_geq<S, C, 0>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 1>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 2>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 3>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 4>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 5>(gdst, b.n, self, ux, uy, uz, bb);
    store_geq<S, C, 6>(gdst, b.n, self, ux, uy, uz, bb);
}

template <typename S, typename C, bool WALLS>
__global__ void mhd_fields_kernel(const S* __restrict__ src, FieldsOut out, MhdArgs p, int z0, int nzs) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, zs = blockIdx.z;
    const Box& b = p.box;
    if (x >= b.nx || zs >= nzs) return;
    const int z = z0 + zs;
    const size_t k = ((size_t)zs * b.ny + y) * b.nx + x;
    const uint32_t self = ((uint32_t)z * (uint32_t)b.ny + (uint32_t)y) * (uint32_t)b.nx + (uint32_t)x;
    const Nbr q = make_nbr(b, x, y, z);
    C f[Q];
    gather19<S, C, WALLS>(src, b, q, x, y, z, self, (C)0, (C)0, (C)0, f);
    const C bw[3] = {(C)p.bw[0], (C)p.bw[1], (C)p.bw[2]};
    C g[7][3];
    gather_mag<S, C, WALLS>(src + (size_t)Q * b.n, b, q, x, y, z, self, bw, g);
    const Moments<C> mo = moments19(f);
    C bb[3];
    const Macro<C> a = mhd_macro<C>(mo, g, p, bb);
    if (out.rho) out.rho[k] = (double)a.rho;
    if (out.u[0]) out.u[0][k] = (double)a.ux;
    if (out.u[1]) out.u[1][k] = (double)a.uy;
    if (out.u[2]) out.u[2][k] = (double)a.uz;
    if (out.B[0]) out.B[0][k] = (double)bb[0];
    if (out.B[1]) out.B[1][k] = (double)bb[1];
    if (out.B[2]) out.B[2][k] = (double)bb[2];
}

template <typename S, typename C, bool WALLS>
__global__ void __launch_bounds__(RED_THREADS) mhd_reduce_kernel(const S* __restrict__ src, MhdArgs p,
                                                                 C* __restrict__ uprev, bool have_prev, bool record,
                                                                 double* __restrict__ partials,
                                                                 NodeDiv div) {
    const Box& b = p.box;
    RedAcc acc;
    acc.zero();
    const C bw[3] = {(C)p.bw[0], (C)p.bw[1], (C)p.bw[2]};
    for (uint32_t self = blockIdx.x * RED_THREADS + threadIdx.x; self < (uint32_t)b.n;
         self += gridDim.x * RED_THREADS) {
        int x, y, z;
        node_of(self, b, div, x, y, z);
        C up[3];
        load_prev(uprev, b.n, self, have_prev, up);
        const Nbr q = make_nbr(b, x, y, z);
        C f[Q];
        gather19<S, C, WALLS>(src, b, q, x, y, z, self, (C)0, (C)0, (C)0, f);
        C g[7][3];
        gather_mag<S, C, WALLS>(src + (size_t)Q * b.n, b, q, x, y, z, self, bw, g);
        const Moments<C> mo = moments19(f);
        C bb[3];
        const Macro<C> a = mhd_macro<C>(mo, g, p, bb);
        reduce_node<C>(acc, a.rho, a.ux, a.uy, a.uz, up, uprev, b.n, self, have_prev, record);
    }
    block_reduce_store(acc, partials);
}

// ---------------------------------------------------------------------------
static MhdArgs mhd_args(const lbm_ctx* c) {
    MhdArgs p;
    p.box = c->box;
    p.omega = c->relax.omega;
    p.tau_m = c->phys.tau_m;
    p.inv_tau_m = 1.0 / c->phys.tau_m;
    p.jfac = 1.0 / (c->phys.tau_m * CSM2);
    for (int a = 0; a < 3; ++a) {
        p.g[a] = c->forcing.g[a];
        p.bw[a] = c->phys.b_wall[a];
    }
    return p;
}

template <typename S, typename C, bool WALLS, bool FLAT>
static cudaError_t steps_t(lbm_ctx* c, long n, bool dry) {
    const MhdArgs p = mhd_args(c);
    const int bx = c->block_x;
    const dim3 grid = step_grid(c->box, bx, c->box.ny, FLAT);
    for (long s = 0; s < n; ++s) {
        launch_step(c, mhd_step_kernel<S, C, WALLS, FLAT>, grid, bx, 0, (const S*)c->buf[c->cur],
                    (S*)c->buf[c->cur ^ 1], p, make_fast_div((uint32_t)c->box.nx));
        if (!dry) c->cur ^= 1;
    }
    return cudaGetLastError();
}
template <typename S, typename C>
static cudaError_t step_t(lbm_ctx* c, long n, bool dry) {
    const bool flat = step_flat(c->box, c->block_x);
    if ((c->box.periodic & 7u) != 7u)
        return flat ? steps_t<S, C, true, true>(c, n, dry) : steps_t<S, C, true, false>(c, n, dry);
    return flat ? steps_t<S, C, false, true>(c, n, dry) : steps_t<S, C, false, false>(c, n, dry);
}

template <typename S, typename C>
static cudaError_t init_t(lbm_ctx* c, const FieldsIn& in, int z0, int nzs, bool uniform) {
    const int bx = c->block_x;
    dim3 grid((unsigned)((c->box.nx + bx - 1) / bx), (unsigned)c->box.ny, (unsigned)nzs);
    mhd_init_kernel<S, C><<<grid, bx, 0, c->stream>>>((S*)c->buf[c->cur], in, c->box, z0, nzs, uniform);
    return cudaGetLastError();
}

template <typename S, typename C>
static cudaError_t fields_t(lbm_ctx* c, const FieldsOut& out, int z0, int nzs) {
    const MhdArgs p = mhd_args(c);
    const int bx = c->block_x;
    dim3 grid((unsigned)((c->box.nx + bx - 1) / bx), (unsigned)c->box.ny, (unsigned)nzs);
    if ((c->box.periodic & 7u) != 7u)
        mhd_fields_kernel<S, C, true><<<grid, bx, 0, c->stream>>>((const S*)c->buf[c->cur], out, p, z0, nzs);
    else
        mhd_fields_kernel<S, C, false><<<grid, bx, 0, c->stream>>>((const S*)c->buf[c->cur], out, p, z0, nzs);
    return cudaGetLastError();
}

template <typename S, typename C>
static cudaError_t reduce_t(lbm_ctx* c, bool record) {
    const MhdArgs p = mhd_args(c);
    if ((c->box.periodic & 7u) != 7u)
        mhd_reduce_kernel<S, C, true><<<RED_BLOCKS, RED_THREADS, 0, c->stream>>>(
            (const S*)c->buf[c->cur], p, (C*)c->uprev, c->have_prev, record, c->partials, node_div(c->box));
    else
        mhd_reduce_kernel<S, C, false><<<RED_BLOCKS, RED_THREADS, 0, c->stream>>>(
            (const S*)c->buf[c->cur], p, (C*)c->uprev, c->have_prev, record, c->partials, node_div(c->box));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return reduce_finalize(c);
}

cudaError_t mhd_step(lbm_ctx* c, long n, bool dry) {
    return c->prec == LBM_FP64 ? step_t<double, double>(c, n, dry) : step_t<float, float>(c, n, dry);
}
cudaError_t mhd_init(lbm_ctx* c, const FieldsIn& in, int z0, int nzs, bool uniform) {
    return c->prec == LBM_FP64 ? init_t<double, double>(c, in, z0, nzs, uniform)
                               : init_t<float, float>(c, in, z0, nzs, uniform);
}
cudaError_t mhd_fields(lbm_ctx* c, const FieldsOut& out, int z0, int nzs) {
    return c->prec == LBM_FP64 ? fields_t<double, double>(c, out, z0, nzs) : fields_t<float, float>(c, out, z0, nzs);
}
cudaError_t mhd_reduce(lbm_ctx* c, bool record) {
    return c->prec == LBM_FP64 ? reduce_t<double, double>(c, record) : reduce_t<float, float>(c, record);
}

}  // namespace lbm
