// Image-space kernels of one SDP-BSREM subiteration (Table I):
//   - the fused update: gather backprojection b = A_i^T w, RDP gradient (Eq. gradRD, 8-point
//     in-plane neighbourhood), the smoothness map nu (Sec. III, Eq. nuki), the preconditioner
//     S (Eq. preconditioner) and the clamp P_t (Eq. OperatorPt), with the FP64 sum of the new
//     iterate in the epilogue;
//   - the mu reduction that feeds mean(mu), the plain sum behind mean(f), and the stand-alone
//     RDP value / gradient and nu maps.
// Pixel-driven: one thread handles one pixel and one group of G planes; neighbours come
// through L1; the gather's (pixel, view) weights are shared by all groups through shared memory.
#include "image.cuh"
#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

int sm_count();

void update_fp32_scalars(UpdateArgs &a)
{
    a.fs_lam = (float)a.lam_alpha;
    a.fs_bm = (float)a.beta_over_M;
    a.fs_gamma_r = (float)a.gamma_r;
    a.fs_eps = (float)a.eps;
    a.fs_t = (float)a.t;
    a.fs_U = (float)a.U;
    a.fs_nu1 = (float)a.nu1;
    a.fs_nu2 = (float)a.nu2;
    a.fs_ips = (float)a.invp_scale;
    a.fs_scale = (float)a.g.scale;
}

// the scalar in the kernel's arithmetic: the host-converted FP32 copy, or the double
template <typename T>
__device__ __forceinline__ T scal(double d, float f)
{
    if constexpr (sizeof(T) == 4) return f;
    else return d;
}

// f^{k,i} = P_t(f - lambda_k alpha_{k,i} nu S(f) (A_i^T w + (beta/M) grad R(f)))
// Virtual block: tpv tiles of TP consecutive pixels x NG plane groups (thread = pixel * NG +
// group); the (pixel, view) weights of each tile are computed once into shared memory.  A
// persistent grid strides over the virtual blocks of one scan or of a batch of scans.
template <int G, int KC, int AR, bool SUB = false, bool TOF = false>
__global__ void __launch_bounds__(256, G == 1 ? 4 : 3) update_kernel(
    const __grid_constant__ UpdateArgs one, const Batch bt)
{
    using T = typename ArithT<AR>::T;
    __shared__ BpTable<KC, AR> tb;
    grid_dependency_wait();                      // as in update_kernel_x8
    grid_dependents_launch();
    const int total = total_vblocks(one, bt);
    __shared__ UpdateArgs sh_args;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        int vloc, nv;
        const UpdateArgs &a = scan_args(one, bt, vb, vloc, nv, sh_args);
        const GeoDev &g = a.g;
        const int N = g.N, NG = g.NG, Pp = g.Pp, npix = N * N;
        const int TP = 256 / NG;
        const int pl = threadIdx.x / NG, grp = threadIdx.x % NG;
        const int VC = max(1, min(a.nviews, BpTable<KC, AR>::CAP / TP));
        const bool dyn = a.nu_mode == 1 || a.nu_mode == 2;
        const double q = (double)npix * g.P;
        // per-scan scalars in the kernel's arithmetic: an FP64 division in every thread of every
        // virtual block is costly at GB300's FP64 rate
        const T inv_mean_f = dyn ? (T)q / (T)*a.sum_f : T(1);
        const T mean_mu = dyn ? (T)*a.sum_mu / (T)q : T(1);
        const T lam = scal<T>(a.lam_alpha, a.fs_lam), bm = scal<T>(a.beta_over_M, a.fs_bm);
        const T U = scal<T>(a.U, a.fs_U), tt = scal<T>(a.t, a.fs_t);
        const T nu1 = scal<T>(a.nu1, a.fs_nu1), nu2 = scal<T>(a.nu2, a.fs_nu2), halfU = T(0.5) * U;
        const T *w = reinterpret_cast<const T *>(a.w);
        const T *f = reinterpret_cast<const T *>(a.f);
        const T *invp = reinterpret_cast<const T *>(a.invp);
        const T scale = scal<T>(g.scale, a.fs_scale);
        const int ntiles = (npix + TP - 1) / TP;
        T part = T(0);
        for (int tile = vloc * a.tpv; tile < min(ntiles, (vloc + 1) * a.tpv); ++tile) {
            const int j0 = tile * TP, j = j0 + pl;
            const bool active = pl < TP && j < npix;
            // 1. stencil first, folded into fc, coef = lambda alpha nu S and rg = (beta/M) grad R,
            //    so that the backprojection's accumulators do not coexist with the stencil state
            T fc[G], coef[G], rg[G];
            if (active) {
                const int ix = j % N, iy = j / N;
                T gr[G], gx[G], gy[G], rv[G], gz[G];
#pragma unroll
                for (int p = 0; p < G; ++p) gz[p] = T(0);
                const T gam_r = scal<T>(a.gamma_r, a.fs_gamma_r), eps_t = scal<T>(a.eps, a.fs_eps);
                if (dyn) stencil<G, AR, true, true, false>(g, f, grp, ix, iy, gam_r, eps_t, fc, gr, gx, gy, rv, a.z3, gz);
                else stencil<G, AR, true, false, false>(g, f, grp, ix, iy, gam_r, eps_t, fc, gr, gx, gy, rv, a.z3, gz);
                T nu[G];
                if (a.nu_mode == 3) {
                    load_group<G, T>(reinterpret_cast<const T *>(a.nu_frozen) + (unsigned)j * (unsigned)Pp + grp * G, nu);
                } else if (!dyn) {
#pragma unroll
                    for (int p = 0; p < G; ++p) nu[p] = T(1);
                } else {
#pragma unroll
                    for (int p = 0; p < G; ++p) nu[p] = nu_of<T>(gx[p], gy[p], gz[p], inv_mean_f, mean_mu, nu1, nu2);
                    if (a.nu_mode == 2)
                        store_group<G, T>(reinterpret_cast<T *>(a.nu_frozen) + (unsigned)j * (unsigned)Pp + grp * G, nu);
                }
                T ipv[G];
                if (a.vox) {
                    load_group<G, T>(invp + (unsigned)j * (unsigned)Pp + grp * G, ipv);
#pragma unroll
                    for (int p = 0; p < G; ++p) ipv[p] *= scal<T>(a.invp_scale, a.fs_ips);
                } else {
                    const T ip = invp[j] * scal<T>(a.invp_scale, a.fs_ips);
#pragma unroll
                    for (int p = 0; p < G; ++p) ipv[p] = ip;
                }
#pragma unroll
                for (int p = 0; p < G; ++p) {
                    const T S = (fc[p] < halfU ? fc[p] : U - fc[p]) * ipv[p];
                    coef[p] = lam * nu[p] * S;
                    rg[p] = bm * gr[p];
                }
            }
            // 2. gather backprojection A_i^T w with the tile's shared (pixel, view) weights
            GroupSum<G, AR> bp;
            bp.zero();
            for (int u0 = 0; u0 < a.nviews; u0 += VC) {
                const int nvc = min(VC, a.nviews - u0);
                __syncthreads();
                bp_fill<KC, AR, 0, SUB>(g, a.slot0, u0, nvc, j0, TP, tb);
                __syncthreads();
                if (!active) continue;
                if constexpr (TOF)
                    bp_accumulate_tof<G, KC, AR>(g, tb, w, TP, nvc, pl, grp, bp, j % N, j / N,
                                                 a.slot0, u0);
                else
                    bp_accumulate<G, KC, AR>(g, tb, w, TP, nvc, pl, grp, bp);
            }
            if (!active) continue;
            // 3. step and clamp P_t (TV variant: the unclamped z and the metric W = coef, for the
            //    proximal step that follows)
            T out[G], wv[G];
#pragma unroll
            for (int p = 0; p < G; ++p) {
                const T d = scale * bp.value(p) + rg[p];
                T ft = fc[p] - coef[p] * d;
                if (!a.tv) ft = ft <= T(0) ? tt : (ft >= U ? U - tt : ft);
                const bool valid = grp * G + p < g.P;
                out[p] = valid ? ft : T(0);
                wv[p] = valid ? coef[p] : T(1);
                part += out[p];
            }
            const unsigned o = (unsigned)j * (unsigned)Pp + grp * G;
            store_group<G, T>(reinterpret_cast<T *>(a.fout) + o, out);
            if (a.tv) {
                store_group<G, T>(reinterpret_cast<T *>(a.zbuf) + o, out);
                store_group<G, T>(reinterpret_cast<T *>(a.wbuf) + o, wv);
            }
        }
        double v[1] = {(double)part};
        grid_reduce<1>(v, a.red, a.sum_fout, vloc, nv);
    }
}

// Stand-alone gather backprojection (also the sensitivity, proj == nullptr); one pixel tile
// per virtual block.
template <int G, int KC, int AR, bool SUB = false, bool TOF = false>
__global__ void __launch_bounds__(256) back_kernel(const __grid_constant__ BackArgs a)
{
    using T = typename ArithT<AR>::T;
    __shared__ BpTable<KC, AR> tb;
    const GeoDev &g = a.g;
    const int N = g.N, NG = g.NG, npix = N * N;
    const int TP = 256 / NG;
    const int pl = threadIdx.x / NG, grp = threadIdx.x % NG;
    const int VC = max(1, min(a.nviews, BpTable<KC, AR>::CAP / TP));
    const T *proj = reinterpret_cast<const T *>(a.proj);
    const int ntiles = (npix + TP - 1) / TP;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int j0 = tile * TP, j = j0 + pl;
        const bool active = pl < TP && j < npix;
        GroupSum<G, AR> acc;
        acc.zero();
        for (int u0 = 0; u0 < a.nviews; u0 += VC) {
            const int nvc = min(VC, a.nviews - u0);
            __syncthreads();
            bp_fill<KC, AR, 0, SUB>(g, a.slot0, u0, nvc, j0, TP, tb);
            __syncthreads();
            if (!active) continue;
            if constexpr (TOF)
                bp_accumulate_tof<G, KC, AR>(g, tb, proj, TP, nvc, pl, grp, acc, j % N, j / N,
                                             a.slot0, u0);
            else
                bp_accumulate<G, KC, AR>(g, tb, proj, TP, nvc, pl, grp, acc);
        }
        if (!active) continue;
        T b[G];
        const T scale = (T)g.scale;
#pragma unroll
        for (int p = 0; p < G; ++p) b[p] = (grp * G + p < g.P) ? scale * acc.value(p) : T(0);
        store_group<G, T>(reinterpret_cast<T *>(a.img) + (size_t)j * g.Pp + (size_t)grp * G, b);
    }
}

// KIND 0: sum f; 1: sum mu; 2: nu map; 3: RDP gradient; 4: RDP value.  Virtual block: 256 x ipt
// (pixel, plane group) items, item = thread + 256 k.
template <int G, int AR, int KIND>
__global__ void __launch_bounds__(256) image_kernel(const __grid_constant__ ImageArgs one,
                                                    const Batch bt)
{
    using T = typename ArithT<AR>::T;
    __shared__ ImageArgs sh_args;
    __shared__ double red_sh[1][32];
    VblockRuns runs(total_vblocks(one, bt));
    const ImageArgs *ap = nullptr;
    int done = 0, vloc = 0, nv = 0;
    KeptScan kept;
    for (int vb; (vb = runs.next()) >= 0;) {
        if (scan_args_kept(one, bt, vb, vloc, nv, sh_args, kept, ap)) done = 0;
        const ImageArgs &a = *ap;
        const GeoDev &g = a.g;
        const int N = g.N, NG = g.NG, Pp = g.Pp;
        const unsigned items = (unsigned)N * (unsigned)N * (unsigned)NG;    // < 2^32 (geometry limits)
        const double q = (double)N * N * g.P;
        const T *f = reinterpret_cast<const T *>(a.f);
        const T inv_mean_f = (KIND == 1 || KIND == 2) ? (T)q / (T)*a.sum_f : T(1);
        const T mean_mu = KIND == 2 ? (T)*a.sum_mu / (T)q : T(1);
        T part = T(0);
        for (int k = 0; k < a.ipt; ++k) {
            const unsigned tid = ((unsigned)vloc * (unsigned)a.ipt + (unsigned)k) * 256u + threadIdx.x;
            if (tid >= items) break;
            const int grp = NG == 1 ? 0 : (int)(tid % (unsigned)NG);
            const int j = NG == 1 ? (int)tid : (int)(tid / (unsigned)NG);
            const int ix = j % N, iy = j / N;
            T fc[G], gr[G], gx[G], gy[G], rv[G], out[G], gz[G];
#pragma unroll
            for (int p = 0; p < G; ++p) gz[p] = T(0);
            if constexpr (KIND == 0) {
                load_group<G, T>(f + (size_t)j * Pp + (size_t)grp * G, fc);
#pragma unroll
                for (int p = 0; p < G; ++p) part += (grp * G + p < g.P) ? fc[p] : T(0);
            } else if constexpr (KIND == 1 || KIND == 2) {
                stencil<G, AR, false, true, false>(g, f, grp, ix, iy, T(0), T(0), fc, gr, gx, gy, rv, a.z3, gz);
#pragma unroll
                for (int p = 0; p < G; ++p) {
                    T mu = grad_norm3(gx[p], gy[p], gz[p]) * inv_mean_f;
                    mu = mu < T(0.01) ? T(0.01) : mu;
                    if constexpr (KIND == 1) {
                        part += (grp * G + p < g.P) ? mu : T(0);
                    } else {
                        out[p] = grp * G + p < g.P ? clampT<T>(fast_div(mean_mu, mu), (T)a.nu1, (T)a.nu2) : T(0);
                    }
                }
                if constexpr (KIND == 2)
                    store_group<G, T>(reinterpret_cast<T *>(a.out) + (size_t)j * Pp + (size_t)grp * G, out);
            } else if constexpr (KIND == 3) {
                stencil<G, AR, true, false, false>(g, f, grp, ix, iy, (T)a.gamma_r, (T)a.eps, fc, gr, gx, gy, rv, a.z3, gz);
#pragma unroll
                for (int p = 0; p < G; ++p) out[p] = grp * G + p < g.P ? gr[p] : T(0);
                store_group<G, T>(reinterpret_cast<T *>(a.out) + (size_t)j * Pp + (size_t)grp * G, out);
            } else if (a.tv) {
                // R_TV: |(f_{j+x} - f_j, f_{j+y} - f_j)|, a component 0 across the last column / row
                T fx[G], fy[G];
                load_group<G, T>(f + (size_t)j * Pp + (size_t)grp * G, fc);
                if (ix + 1 < N) load_group<G, T>(f + (size_t)(j + 1) * Pp + (size_t)grp * G, fx);
                if (iy + 1 < N) load_group<G, T>(f + (size_t)(j + N) * Pp + (size_t)grp * G, fy);
#pragma unroll
                for (int p = 0; p < G; ++p) {
                    const T dx = ix + 1 < N ? fx[p] - fc[p] : T(0);
                    const T dy = iy + 1 < N ? fy[p] - fc[p] : T(0);
                    part += (grp * G + p < g.P) ? sqrt(dx * dx + dy * dy) : T(0);
                }
            } else {
                stencil<G, AR, false, false, true>(g, f, grp, ix, iy, (T)a.gamma_r, (T)a.eps, fc, gr, gx, gy, rv, a.z3, gz);
#pragma unroll
                for (int p = 0; p < G; ++p) part += (grp * G + p < g.P) ? rv[p] : T(0);
            }
        }
        if constexpr (KIND == 0 || KIND == 1 || KIND == 4) {
            double v[1] = {(double)part};
            reduce_partial<1>(v, a.red, vloc, red_sh);
            ++done;
            if (runs.ends() || vloc + 1 == nv) {
                reduce_finish<1>(a.red, a.result, done, nv, red_sh);
                done = 0;
            }
        }
    }
}

// The mu pass alone (batches, and scans whose pass does not join the projection).
__global__ void __launch_bounds__(256) mu_kernel_x8(const __grid_constant__ ImageArgs one, const Batch bt)
{
    const int total = total_vblocks(one, bt);
    __shared__ ImageArgs sh_args;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        int vloc, nv;
        const ImageArgs &a = scan_args(one, bt, vb, vloc, nv, sh_args);
        mu_x8_vblock(a, vloc, nv);
    }
}

// pixel tiles per virtual block so that a scan never needs more partial sums than its reducer
int resident_blocks(const void *fn);

template <int G, int KC>
static const void *update_fn(int arith, int sub, int tof)
{
    if (tof && sub) {                            // TOF on ring-sampled bins: KC = 4
        if (arith == AR_FP32) return (const void *)update_kernel<G, 4, AR_FP32, true, true>;
        if (arith == AR_KAHAN) return (const void *)update_kernel<G, 4, AR_KAHAN, true, true>;
        return (const void *)update_kernel<G, 4, AR_FP64, true, true>;
    }
    if (tof) {                                   // TOF geometries: generic kernel
        if (arith == AR_FP32) return (const void *)update_kernel<G, KC, AR_FP32, false, true>;
        if (arith == AR_KAHAN) return (const void *)update_kernel<G, KC, AR_KAHAN, false, true>;
        return (const void *)update_kernel<G, KC, AR_FP64, false, true>;
    }
    if (sub) {                                   // sub-ray geometries: KC = 4, generic kernel
        if (arith == AR_FP32) return (const void *)update_kernel<G, 4, AR_FP32, true>;
        if (arith == AR_KAHAN) return (const void *)update_kernel<G, 4, AR_KAHAN, true>;
        return (const void *)update_kernel<G, 4, AR_FP64, true>;
    }
    if constexpr (G == 1) {                      // single-plane FP32: the TV variant only
        if (arith == AR_FP32) return (const void *)update_kernel<G, KC, AR_FP32>;
        if (arith == AR_KAHAN) return (const void *)update_kernel<G, KC, AR_KAHAN>;
    }
    return (const void *)update_kernel<G, KC, AR_FP64>;
}

// Pixel tiles per virtual block: each virtual block ends in a block reduction and a grid-wide
// ticket, so the tiles are grouped into one wave of virtual blocks over the resident block
// slots (and never more virtual blocks than the reducer has partial sums for).
void update_shape(UpdateArgs &a, int arith)
{
    if (plane1_path(a.g, arith) && !a.tv) { update_shape_p1(a, arith); return; }
    const int TP = 256 / a.g.NG;
    const int ntiles = update_x8_path(a, arith) ? update_x8_tiles(a) : (a.g.N * a.g.N + TP - 1) / TP;
    const int sub = a.g.table, tof = a.g.T > 1;
    const void *fn = update_x8_path(a, arith) ? update_x8_fn(a, arith)
                     : a.g.G == 1 ? (a.g.K <= 2 ? update_fn<1, 2>(arith, sub, tof) : update_fn<1, 4>(arith, sub, tof))
                                  : (a.g.K <= 2 ? update_fn<8, 2>(arith, sub, tof) : update_fn<8, 4>(arith, sub, tof));
    const int slots = sm_count() * resident_blocks(fn);
    a.tpv = std::max({1, (ntiles + a.red.capacity - 1) / a.red.capacity, (ntiles + slots - 1) / slots});
    if (update_x8_path(a, arith) && (a.z3 || a.vox) && !a.tv && a.g.T == 1) a.tpv = update_x8_tpv(a);
    a.nvb = (ntiles + a.tpv - 1) / a.tpv;
}

// items per thread: at most ~4 virtual blocks per SM (each ends in a block reduction; 2 for
// single-plane images, of which a batch runs many) and never more virtual blocks than reduction
// slots
void image_shape(ImageArgs &a)
{
    const long long items = (long long)a.g.N * a.g.N * a.g.NG;
    const long long nblk = (items + 255) / 256;
    const int cap = a.red.capacity > 0 ? a.red.capacity : (1 << 30);
    const long long target = (long long)sm_count() * (a.g.G == 1 ? 2 : 4);
    a.ipt = (int)std::max<long long>({1, (nblk + cap - 1) / cap, (nblk + target - 1) / target});
    a.nvb = (int)((nblk + a.ipt - 1) / a.ipt);
}

static int persistent_grid(int nvb) { return std::max(1, std::min(nvb, sm_count() * 8)); }

template <int G, int KC>
static pet_status update_dispatch(const UpdateArgs &a, const Batch &b, int arith, int grid, cudaStream_t st,
                                  bool pdl)
{
    if (a.g.T > 1 && a.g.table) {                // TOF on ring-sampled bins: KC = 4
        if (arith == AR_FP32) launch_pdl(update_kernel<G, 4, AR_FP32, true, true>, grid, st, pdl, a, b);
        else if (arith == AR_KAHAN) launch_pdl(update_kernel<G, 4, AR_KAHAN, true, true>, grid, st, pdl, a, b);
        else launch_pdl(update_kernel<G, 4, AR_FP64, true, true>, grid, st, pdl, a, b);
        return PET_OK;
    }
    if (a.g.T > 1) {                             // TOF geometries: generic kernel
        if (arith == AR_FP32) launch_pdl(update_kernel<G, KC, AR_FP32, false, true>, grid, st, pdl, a, b);
        else if (arith == AR_KAHAN) launch_pdl(update_kernel<G, KC, AR_KAHAN, false, true>, grid, st, pdl, a, b);
        else launch_pdl(update_kernel<G, KC, AR_FP64, false, true>, grid, st, pdl, a, b);
        return PET_OK;
    }
    if (a.g.table) {                             // sub-ray / ring geometries: KC = 4, generic kernel
        if (arith == AR_FP32) launch_pdl(update_kernel<G, 4, AR_FP32, true>, grid, st, pdl, a, b);
        else if (arith == AR_KAHAN) launch_pdl(update_kernel<G, 4, AR_KAHAN, true>, grid, st, pdl, a, b);
        else launch_pdl(update_kernel<G, 4, AR_FP64, true>, grid, st, pdl, a, b);
        return PET_OK;
    }
    if constexpr (G == 1) {                      // single-plane FP32: the TV variant only
        if (arith == AR_FP32) { launch_pdl(update_kernel<G, KC, AR_FP32>, grid, st, pdl, a, b); return PET_OK; }
        if (arith == AR_KAHAN) { launch_pdl(update_kernel<G, KC, AR_KAHAN>, grid, st, pdl, a, b); return PET_OK; }
    }
    if (arith != AR_FP64) return fail(PET_ERR_INVALID, "update: no FP32 kernel for this scan");
    launch_pdl(update_kernel<G, KC, AR_FP64>, grid, st, pdl, a, b);
    return PET_OK;
}

static pet_status update_any(const UpdateArgs &a, const Batch &b, int arith, int grid, cudaStream_t st,
                            bool pdl)
{
    LaunchScope ls(PET_K_UPDATE, st);
    if (plane1_path(a.g, arith) && !a.tv) {
        update_p1_dispatch(a, b, arith, grid, st, pdl);
    } else if (update_x8_path(a, arith)) {
        update_x8_dispatch(a, b, arith, grid, st, pdl);
    } else if (a.g.G == 1) {
        if (a.g.K <= 2) PET_TRY((update_dispatch<1, 2>(a, b, arith, grid, st, pdl)));
        else PET_TRY((update_dispatch<1, 4>(a, b, arith, grid, st, pdl)));
    } else {
        if (a.g.K <= 2) PET_TRY((update_dispatch<8, 2>(a, b, arith, grid, st, pdl)));
        else PET_TRY((update_dispatch<8, 4>(a, b, arith, grid, st, pdl)));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "update_kernel launch");
    return PET_OK;
}

pet_status launch_update(const UpdateArgs &a0, int arith, cudaStream_t st, bool after_kernel)
{
    UpdateArgs a = a0;
    update_shape(a, arith);
    update_fp32_scalars(a);
    return update_any(a, Batch{nullptr, nullptr, 0, 0}, arith, persistent_grid(a.nvb), st, after_kernel);
}

pet_status launch_update_batch(const UpdateArgs &shape, const Batch &b, int arith, cudaStream_t st)
{
    return update_any(shape, b, arith, b.grid, st, false);
}

template <int G, int KC>
static pet_status back_dispatch(const BackArgs &a, int arith, int grid, cudaStream_t st)
{
    if (a.g.T > 1 && a.g.table) {
        if (arith == AR_FP32) back_kernel<G, 4, AR_FP32, true, true><<<grid, 256, 0, st>>>(a);
        else if (arith == AR_KAHAN) back_kernel<G, 4, AR_KAHAN, true, true><<<grid, 256, 0, st>>>(a);
        else back_kernel<G, 4, AR_FP64, true, true><<<grid, 256, 0, st>>>(a);
        return PET_OK;
    }
    if (a.g.T > 1) {
        if (arith == AR_FP32) back_kernel<G, KC, AR_FP32, false, true><<<grid, 256, 0, st>>>(a);
        else if (arith == AR_KAHAN) back_kernel<G, KC, AR_KAHAN, false, true><<<grid, 256, 0, st>>>(a);
        else back_kernel<G, KC, AR_FP64, false, true><<<grid, 256, 0, st>>>(a);
        return PET_OK;
    }
    if (a.g.table) {
        if (arith == AR_FP32) back_kernel<G, 4, AR_FP32, true><<<grid, 256, 0, st>>>(a);
        else if (arith == AR_KAHAN) back_kernel<G, 4, AR_KAHAN, true><<<grid, 256, 0, st>>>(a);
        else back_kernel<G, 4, AR_FP64, true><<<grid, 256, 0, st>>>(a);
        return PET_OK;
    }
    if (arith == AR_FP32) back_kernel<G, KC, AR_FP32><<<grid, 256, 0, st>>>(a);
    else if (arith == AR_KAHAN) back_kernel<G, KC, AR_KAHAN><<<grid, 256, 0, st>>>(a);
    else back_kernel<G, KC, AR_FP64><<<grid, 256, 0, st>>>(a);
    return PET_OK;
}

pet_status launch_back(const BackArgs &a, int arith, cudaStream_t st)
{
    const int TP = 256 / a.g.NG;
    const int ntiles = (a.g.N * a.g.N + TP - 1) / TP;
    const int grid = persistent_grid(ntiles);
    LaunchScope ls(PET_K_OTHER, st);
    if (back_quad_path(a, arith)) {
        back_quad_dispatch(a, arith, st);
    } else if (a.g.G == 1) {
        if (a.g.K <= 2) PET_TRY((back_dispatch<1, 2>(a, arith, grid, st)));
        else PET_TRY((back_dispatch<1, 4>(a, arith, grid, st)));
    } else {
        if (a.g.K <= 2) PET_TRY((back_dispatch<8, 2>(a, arith, grid, st)));
        else PET_TRY((back_dispatch<8, 4>(a, arith, grid, st)));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "back_kernel launch");
    return PET_OK;
}

template <int KIND>
static pet_status image_any(const ImageArgs &a, const Batch &b, int arith, int grid, cudaStream_t st)
{
    LaunchScope ls(KIND == 1 ? PET_K_MU_SUM : (KIND == 4 ? PET_K_RDP_VALUE : PET_K_OTHER), st);
    // FP32 and Kahan modes share the FP32 image arithmetic
    if (a.g.G == 1) {
        if (arith == AR_FP64) image_kernel<1, AR_FP64, KIND><<<grid, 256, 0, st>>>(a, b);
        else image_kernel<1, AR_FP32, KIND><<<grid, 256, 0, st>>>(a, b);
    } else {
        if (arith == AR_FP64) image_kernel<8, AR_FP64, KIND><<<grid, 256, 0, st>>>(a, b);
        else image_kernel<8, AR_FP32, KIND><<<grid, 256, 0, st>>>(a, b);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "image_kernel launch");
    return PET_OK;
}

template <int KIND>
static pet_status launch_image(const ImageArgs &a0, int arith, cudaStream_t st)
{
    ImageArgs a = a0;
    image_shape(a);
    return image_any<KIND>(a, Batch{nullptr, nullptr, 0, 0}, arith, persistent_grid(a.nvb), st);
}

pet_status launch_sum(const ImageArgs &a, int arith, cudaStream_t st) { return launch_image<0>(a, arith, st); }
// Shape of the mu pass: the packed kernel (8-plane groups, FP32) takes a.ipt pixel tiles per
// virtual block, one wave of virtual blocks over the resident block slots; otherwise the
// items-per-thread shape of image_kernel.
void mu_shape(ImageArgs &a, int arith)
{
    if (a.g.G != 8 || arith == AR_FP64 || a.z3) {
        image_shape(a);
        return;
    }
    const int TP = 256 / a.g.NG;
    const int ntiles = (a.g.N * a.g.N + TP - 1) / TP;
    const int slots = sm_count() * resident_blocks((const void *)mu_kernel_x8);
    const int cap = a.red.capacity > 0 ? a.red.capacity : (1 << 30);
    a.ipt = std::max({1, (ntiles + cap - 1) / cap, (ntiles + slots - 1) / slots});
    a.nvb = (ntiles + a.ipt - 1) / a.ipt;
}

static pet_status mu_any(const ImageArgs &a, const Batch &b, int arith, int grid, cudaStream_t st)
{
    if (a.g.G != 8 || arith == AR_FP64 || a.z3) return image_any<1>(a, b, arith, grid, st);
    LaunchScope ls(PET_K_MU_SUM, st);
    mu_kernel_x8<<<grid, 256, 0, st>>>(a, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "mu_kernel_x8 launch");
    return PET_OK;
}

pet_status launch_mu_sum(const ImageArgs &a0, int arith, cudaStream_t st)
{
    ImageArgs a = a0;
    mu_shape(a, arith);
    return mu_any(a, Batch{nullptr, nullptr, 0, 0}, arith, persistent_grid(a.nvb), st);
}
pet_status launch_nu_map(const ImageArgs &a, int arith, cudaStream_t st) { return launch_image<2>(a, arith, st); }
pet_status launch_rdp_grad(const ImageArgs &a, int arith, cudaStream_t st) { return launch_image<3>(a, arith, st); }
pet_status launch_rdp_value(const ImageArgs &a, int arith, cudaStream_t st) { return launch_image<4>(a, arith, st); }
pet_status launch_mu_sum_batch(const ImageArgs &shape, const Batch &b, int arith, cudaStream_t st)
{
    return mu_any(shape, b, arith, b.grid, st);
}
pet_status launch_rdp_value_batch(const ImageArgs &shape, const Batch &b, int arith, cudaStream_t st)
{
    return image_any<4>(shape, b, arith, b.grid, st);
}

}  // namespace pet
