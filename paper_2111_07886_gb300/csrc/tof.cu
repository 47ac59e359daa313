// Time-of-flight forward projector (the TOF data of the clinical reconstructions, Sec. IV-C):
// y_(i,t) = sum_j A_ij h_t(tau_j) f_j, A_ij the one-line Siddon lengths of bin i = (v, b),
// h_t the Gaussian timing kernel integrated over TOF bin t at the position tau_j of pixel j's
// centre along the line.  One thread walks one (ray, TOF bin, plane group) over the part of
// the ray where h_t can be non-zero (|tau - tau_t| <= the kernel's window), with the same
// column-by-column walk and exact lengths as the non-TOF projector, each length weighted by h_t
// at its pixel's centre.  Epilogues as in fwd_kernel: plain, ratio (with the per-bin detection
// factors), or the objective's FP64 sums.  Outputs are [nviews][NB][T][Pp].  One scan, or a batch
// of TOF scans (per-scan arguments and virtual blocks, as in fwd_kernel).
#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

// FP32 kernels take h_t from a table of h(u) = h_t(c_t + u) (the kernel relative to the TOF
// bin's centre c_t, the same for every bin) over the window |u| <= W: values and derivatives at
// TAB nodes, cubic Hermite interpolation in between (error below 1e-7 of the peak for the node
// spacing of at most sigma / 16; the table is built per block with the tail-mass form of h).
constexpr int TOF_TAB = 2048;

__device__ __forceinline__ void tof_fill_table(const GeoDev &g, float2 *tab)
{
    const float Wt = g.tof_wf, dt_ = (2.f * Wt) / (float)(TOF_TAB - 1);
    const float k = g.tof_kf, hd = 0.5f * g.tof_df;
    const float dphi = 1.1283791670955126f * k;   // 2 k / sqrt(pi)
    for (int i = threadIdx.x; i < TOF_TAB; i += blockDim.x) {
        const float u = -Wt + (float)i * dt_;
        const float z0 = (-hd - u) * k, z1 = (hd - u) * k;
        // h(u) = Phi(sqrt2 z1) - Phi(sqrt2 z0); h'(u) = k / sqrt(pi) (e^{-z0^2} - e^{-z1^2})
        tab[i] = make_float2(tof_h<float>(z0, z1), 0.5f * dphi * (expf(-z0 * z0) - expf(-z1 * z1)));
    }
}

// h at table coordinate x in [0, TOF_TAB - 1)
__device__ __forceinline__ float tof_table(const float2 *tab, float x, float dt_)
{
    const int i = (int)x;
    const float f = x - (float)i;
    const float2 p0 = tab[i], p1 = tab[i + 1];
    const float f2 = f * f, f3 = f2 * f;
    const float h00 = 2.f * f3 - 3.f * f2 + 1.f, h01 = 3.f * f2 - 2.f * f3;
    const float h10 = f3 - 2.f * f2 + f, h11 = f3 - f2;
    return h00 * p0.x + h01 * p1.x + dt_ * (h10 * p0.y + h11 * p1.y);
}

template <int G, int AR, int MODE>
__global__ void __launch_bounds__(256) tof_fwd_kernel(const __grid_constant__ FwdArgs one,
                                                      const Batch bt)
{
    using T = typename ArithT<AR>::T;
    constexpr bool D = AR == AR_FP64;
    __shared__ float2 tab[D ? 1 : TOF_TAB];
    __shared__ float tab_key[3];                       // the TOF kernel the table holds
    __shared__ FwdArgs sh_args;
    if (threadIdx.x == 0) tab_key[0] = tab_key[1] = tab_key[2] = -1.f;
    __syncthreads();
    const int total = total_vblocks(one, bt);
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        int vloc, nv;
        const FwdArgs &a = scan_args(one, bt, vb, vloc, nv, sh_args);
        const GeoDev &g = a.g;
        const int NG = g.NG, NB = g.NB, N = g.N, Pp = g.Pp, TT = g.T;
        const long long items = (long long)a.nviews * NB * TT * NG;
        const T d = D ? (T)g.tof_d : (T)g.tof_df, kk = D ? (T)g.tof_k : (T)g.tof_kf;
        const T W = (D ? (T)g.tof_w : (T)g.tof_wf) + T(1);   // + 1: pixel centres vs the line
        const float Wt = g.tof_wf, dt_ = (2.f * Wt) / (float)(TOF_TAB - 1), idt = 1.f / dt_;
        if constexpr (!D) {
            // (re)build the table when this scan's kernel differs from the one it holds
            // (block-uniform: every thread reads the same arguments)
            if (tab_key[0] != g.tof_df || tab_key[1] != g.tof_kf || tab_key[2] != g.tof_wf) {
                __syncthreads();
                tof_fill_table(g, tab);
                __syncthreads();
                if (threadIdx.x == 0) { tab_key[0] = g.tof_df; tab_key[1] = g.tof_kf; tab_key[2] = g.tof_wf; }
                __syncthreads();
            }
        }
        double obj[2] = {0.0, 0.0};
        for (int k = 0; k < a.tpv; ++k) {
            const long long it = ((long long)vloc * a.tpv + k) * 256 + threadIdx.x;
            if (it >= items) continue;
            const int grp = (int)(it % NG);
            const long long rt = it / NG;
            const int t = (int)(rt % TT);
            const int ray = (int)(rt / TT);              // subset-local u * NB + b
            const int slot = a.slot0 + ray / NB, b = ray % NB;
            const ViewGeo &vw = g.views[slot];
            const RayGeo &rg = g.rays[(size_t)a.slot0 * NB + ray];
            // driving columns whose line point lies within the window of TOF bin t
            const T r = g.ring ? (T)g.bins[b].c0
                               : (T)(2 * b - (NB - 1)) * T(0.5) * (D ? (T)g.rho : (T)(float)g.rho);
            const T tauA = D ? (T)vw.tdr * r + (T)vw.tdc : (T)vw.tdrf * r + (T)vw.tdcf;
            const T tdd = D ? (T)vw.tdd : (T)vw.tddf;
            const T ct = (T)(2 * t - (TT - 1)) * T(0.5) * d;
            T lo_d = (ct - W - tauA) / tdd, hi_d = (ct + W - tauA) / tdd;
            if (lo_d > hi_d) { const T x = lo_d; lo_d = hi_d; hi_d = x; }
            const int k0 = max(0, (int)ceil(lo_d) - rg.d0);
            const int k1 = min(rg.nd, (int)floor(hi_d) - rg.d0 + 1);
            const int ds = vw.xdrive ? 1 : N;
            const int cs = vw.xdrive ? N : 1;
            // pixel (d, r) of the walk is (ix, iy) = (d, r) or (r, d)
            const T tpd = D ? (T)(vw.xdrive ? vw.taux : vw.tauy) : (T)(vw.xdrive ? vw.tauxf : vw.tauyf);
            const T tpr = D ? (T)(vw.xdrive ? vw.tauy : vw.taux) : (T)(vw.xdrive ? vw.tauyf : vw.tauxf);
            const T tp0 = D ? (T)vw.tau0 : (T)vw.tau0f;
            const T e0 = (T)(2 * t - TT) * T(0.5) * d;  // lower edge of the TOF bin
            auto hw = [&](int dd, int rr) -> T {
                const T tau = tp0 + (T)dd * tpd + (T)rr * tpr;
                if constexpr (D) {
                    return tof_h<T>((e0 - tau) * kk, (e0 + d - tau) * kk);
                } else {
                    const float x = (tau - ct + Wt) * idt;
                    if (!(x >= 0.f && x < (float)(TOF_TAB - 1))) return 0.f;
                    return tof_table(tab, x, dt_);
                }
            };
            const T *img = reinterpret_cast<const T *>(a.img) + (size_t)grp * G;
            GroupSum<G, AR> acc;
            acc.zero();
            if constexpr (D) {
                const double step = vw.step, ast = fabs(vw.step), L = vw.L, im = vw.inv_minor;
                for (int kd = k0; kd < k1; ++kd) {
                    const int dd = rg.d0 + kd;
                    const double lo = fma((double)kd, step, rg.lo);
                    const double hi = lo + ast;
                    const double f0 = floor(lo), f1 = floor(hi);
                    const int r0 = (int)f0, r1 = (int)f1;
                    double l1 = (r1 != r0) ? (hi - f1) * im : 0.0;
                    double l0 = L - l1;
                    const bool ok0 = (unsigned)r0 < (unsigned)N, ok1 = (unsigned)r1 < (unsigned)N;
                    l0 = ok0 ? l0 * hw(dd, r0) : 0.0;
                    l1 = (ok1 && l1 > 0.0) ? l1 * hw(dd, r1) : 0.0;
                    T x0[G], x1[G];
                    load_group<G, T>(img + (unsigned)(dd * ds + (ok0 ? r0 : 0) * cs) * (unsigned)Pp, x0);
                    load_group<G, T>(img + (unsigned)(dd * ds + (ok1 ? r1 : 0) * cs) * (unsigned)Pp, x1);
                    acc.add2terms(l0, x0, l1, x1);
                }
            } else {
                const long long stp = vw.stepq, ast = vw.absstepq;
                const float L = vw.Lf, im = vw.inv_minorf * kQ32;
                long long lo = rg.loq + (long long)k0 * stp;
                for (int kd = k0; kd < k1; ++kd) {
                    const int dd = rg.d0 + kd;
                    const long long hi = lo + ast;
                    const int r0 = (int)(lo >> 32), r1 = (int)(hi >> 32);
                    float l1 = (r1 != r0) ? __uint2float_rn((unsigned)(hi & 0xFFFFFFFFLL)) * im : 0.f;
                    float l0 = L - l1;
                    const bool ok0 = (unsigned)r0 < (unsigned)N, ok1 = (unsigned)r1 < (unsigned)N;
                    l0 = ok0 ? l0 * hw(dd, r0) : 0.f;
                    l1 = (ok1 && l1 > 0.f) ? l1 * hw(dd, r1) : 0.f;
                    T x0[G], x1[G];
                    load_group<G, T>(img + (unsigned)(dd * ds + (ok0 ? r0 : 0) * cs) * (unsigned)Pp, x0);
                    load_group<G, T>(img + (unsigned)(dd * ds + (ok1 ? r1 : 0) * cs) * (unsigned)Pp, x1);
                    acc.add2terms(l0, x0, l1, x1);
                    lo += stp;
                }
            }
            const size_t o = ((size_t)ray * TT + t) * Pp + (size_t)grp * G;
            const T scale = (T)g.scale;
            if constexpr (MODE == FWD_PLAIN) {
                T y[G];
#pragma unroll
                for (int p = 0; p < G; ++p) y[p] = scale * acc.value(p);
                store_group<G, T>(reinterpret_cast<T *>(a.out) + o, y);
            } else {
                int cnt[G];
                float gam[G];
                load_group_i<G>(a.counts + o, cnt);
                load_group<G, float>(a.gamma + o, gam);
                const float *mp = a.mult ? a.mult + o : nullptr;
                if constexpr (MODE == FWD_RATIO) {
                    T w[G];
#pragma unroll
                    for (int p = 0; p < G; ++p) {
                        const T m = mp ? (T)__ldg(mp + p) : T(1);
                        const T y = scale * (acc.value(p) * m) + (T)gam[p];
                        w[p] = (grp * G + p < g.P) ? m * (T(1) - (T)cnt[p] / y) : T(0);
                    }
                    store_group<G, T>(reinterpret_cast<T *>(a.out) + o, w);
                } else {
                    T s_af = T(0);
                    double s_gl = 0.0;
#pragma unroll
                    for (int p = 0; p < G; ++p) {
                        if (grp * G + p < g.P) {
                            const T v = acc.value(p);
                            const T af = scale * (mp ? v * (T)__ldg(mp + p) : v);
                            s_af += af;
                            if (cnt[p] != 0) s_gl += (double)cnt[p] * log((double)af + (double)gam[p]);
                        }
                    }
                    obj[0] += (double)s_af;
                    obj[1] += s_gl;
                }
            }
        }
        if constexpr (MODE == FWD_OBJECTIVE) grid_reduce<2>(obj, a.red, a.result, vloc, nv);
    }
}

// ------------------------------------------------------------------------------------------
// FP32 TOF projection of stacks.  The kernel above walks every (ray, TOF bin, group) by itself: with a
// timing kernel wider than a TOF bin, the same pixel is fetched and its h_t evaluated by up to T
// threads times NG groups (540 us for the 12-view subset of the 256 x 256 x 89, 13-bin scan, bound
// by those fetches through L2).  Here a block takes RB neighbouring rays and up to TOF_HG
// half-groups of four planes, and walks the rays once, 32 driving steps at a time:
//   1. a warp per ray lists the pixels the line crosses in these steps (offset, length, position);
//   2. all threads compute the weights length x h_t of every listed pixel and TOF bin;
//   3. thread (ray, slice of TOF_TW bins, half-group) reads each pixel once (16 bytes) and adds it to
//      its slice's sums, two pixels (about a driving step) per compensated step.
// ------------------------------------------------------------------------------------------
constexpr int TOF_TW = 7, TOF_WP = 8, TOF_THREADS = 256, TOF_HG = 24, TOF_STEPS = 32;

// dynamic shared memory of a block at most, and of one ray: 2 TOF_STEPS entries of ts slices x 8
// weight pairs, an offset, and (length, position)
constexpr int TOF_SMEM_MAX = 72 * 1024;
static __host__ __device__ __forceinline__ int tof_ray_smem(int ts) { return 2 * TOF_STEPS * (ts * TOF_WP * 8 + 8 + 4); }

// threads per ray, rays per block and half-group blocks of a shape
struct TofShape { int ts, hgb, nhb, rb; };
static __host__ __device__ __forceinline__ TofShape tof_shape(int NG, int T)
{
    TofShape s;
    s.ts = (T + TOF_TW - 1) / TOF_TW;
    s.hgb = 2 * NG < TOF_HG ? 2 * NG : TOF_HG;
    if (s.hgb > TOF_THREADS / s.ts) s.hgb = TOF_THREADS / s.ts;
    s.nhb = (2 * NG + s.hgb - 1) / s.hgb;
    s.rb = TOF_THREADS / (s.ts * s.hgb);
    if (s.rb > 8) s.rb = 8;
    const int most = TOF_SMEM_MAX / tof_ray_smem(s.ts);
    if (s.rb > most) s.rb = most;
    return s;
}
// Enough planes and TOF bins that a third of a block's threads have sums to hold; below, the walk per TOF
// bin.  Iterations of 128 x 128 scans (12 views per subset), this kernel and the walk: 17 planes x 9 TOF bins
// 1359 and 1473 us, 33 x 21 2526 and 3125, 48 x 7 1470 and 1736.  The line is on the safe side: at 16
// planes x 9 bins 1328 and 1356 us, 16 x 13 1437 and 1467, 40 x 5 1352 and 1664; 8 x 21 1752 and 1721.
bool tof_stack_shape(int NG, int T)
{
    const TofShape s = tof_shape(NG, T);
    return s.rb * s.ts * s.hgb >= TOF_THREADS / 3;
}

template <int AR, int MODE>
__global__ void __launch_bounds__(TOF_THREADS, 2) tof_fwd_stack(const __grid_constant__ FwdArgs one, const Batch bt)
{
    extern __shared__ __align__(16) unsigned char tof_sh[];
    __shared__ float2 tab[TOF_TAB];
    __shared__ float tab_key[3];                       // the TOF kernel the table holds
    __shared__ FwdArgs sh_args;
    __shared__ int count[8], steps_of[8], first_of[8];
    constexpr int E = 2 * TOF_STEPS;
    if (threadIdx.x == 0) tab_key[0] = tab_key[1] = tab_key[2] = -1.f;
    __syncthreads();
    const int total = total_vblocks(one, bt);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        int vloc, nv;
        const FwdArgs &a = scan_args(one, bt, vb, vloc, nv, sh_args);
        const GeoDev &g = a.g;
        const int NB = g.NB, N = g.N, T = g.T;
        const unsigned Pp = (unsigned)g.Pp;
        const TofShape sh = tof_shape(g.NG, T);
        f2x *wts = reinterpret_cast<f2x *>(tof_sh);                            // [rb][E][ts][8]
        float2 *lt = reinterpret_cast<float2 *>(wts + sh.rb * E * sh.ts * TOF_WP);  // [rb][E]
        unsigned *off = reinterpret_cast<unsigned *>(lt + sh.rb * E);          // [rb][E]
        const float d = g.tof_df, W = g.tof_wf + 1.f;      // + 1: pixel centres vs the line
        const float Wt = g.tof_wf, dt_ = (2.f * Wt) / (float)(TOF_TAB - 1), idt = 1.f / dt_;
        if (tab_key[0] != g.tof_df || tab_key[1] != g.tof_kf || tab_key[2] != g.tof_wf) {
            __syncthreads();
            tof_fill_table(g, tab);
            __syncthreads();
            if (threadIdx.x == 0) { tab_key[0] = g.tof_df; tab_key[1] = g.tof_kf; tab_key[2] = g.tof_wf; }
            __syncthreads();
        }
        const int per_ray = sh.ts * sh.hgb;
        const int tiles_v = (NB + sh.rb - 1) / sh.rb, ntiles = a.nviews * tiles_v * sh.nhb;
        const int rl = threadIdx.x / per_ray, in_ray = threadIdx.x - rl * per_ray;
        const int slice = in_ray / sh.hgb;
        double obj[2] = {0.0, 0.0};
        for (int k = 0; k < a.tpv; ++k) {
            // half-group block, then view, then the view's tiles from its centre outwards (the long
            // rays first, so that the launch ends on short ones)
            const int tile = vloc * a.tpv + k;
            if (tile >= ntiles) break;
            __syncthreads();                            // the previous tile's step counts are read
            const int hb = tile % sh.nhb, rest = tile / sh.nhb, u = rest % a.nviews, tr = rest / a.nviews;
            const int tb = (tiles_v - 1) / 2 + ((tr & 1) ? (tr + 1) / 2 : -(tr / 2));
            const int slot = a.slot0 + u;
            const ViewGeo &vw = g.views[slot];
            // pixel (d, r) of the walk is (ix, iy) = (d, r) or (r, d)
            const float tpd = vw.xdrive ? vw.tauxf : vw.tauyf, tpr = vw.xdrive ? vw.tauyf : vw.tauxf;
            const unsigned ds = (vw.xdrive ? 1u : (unsigned)N) * Pp, cs = (vw.xdrive ? (unsigned)N : 1u) * Pp;
            // driving steps of each ray whose line point lies within the window of some TOF bin
            if (threadIdx.x < (unsigned)sh.rb) {
                const int b = tb * sh.rb + (int)threadIdx.x;
                int k0 = 0, n = 0;
                if (b < NB) {
                    const RayGeo &rg = g.rays[(size_t)slot * NB + b];
                    const float r = g.ring ? (float)g.bins[b].c0 : (float)(2 * b - (NB - 1)) * 0.5f * (float)g.rho;
                    const float tauA = vw.tdrf * r + vw.tdcf, tdd = vw.tddf;
                    const float ce = (float)(T - 1) * 0.5f * d + W;
                    float lo_d = (-ce - tauA) / tdd, hi_d = (ce - tauA) / tdd;
                    if (lo_d > hi_d) { const float x = lo_d; lo_d = hi_d; hi_d = x; }
                    k0 = max(0, (int)ceilf(lo_d) - rg.d0);
                    n = max(0, min(rg.nd, (int)floorf(hi_d) - rg.d0 + 1) - k0);
                }
                first_of[threadIdx.x] = k0;
                steps_of[threadIdx.x] = n;
            }
            __syncthreads();
            int nmax = 0;
            for (int q = 0; q < sh.rb; ++q) nmax = max(nmax, steps_of[q]);
            const int hg = hb * sh.hgb + in_ray - slice * sh.hgb;    // half-group of four planes
            const bool work = rl < sh.rb && hg < 2 * g.NG && tb * sh.rb + rl < NB;
            const float *img = reinterpret_cast<const float *>(a.img) + hg * 4;
            f2x sm[TOF_TW][2], er[TOF_TW][2];
#pragma unroll
            for (int t = 0; t < TOF_TW; ++t) sm[t][0] = sm[t][1] = er[t][0] = er[t][1] = 0ull;
            for (int c0 = 0; c0 < nmax; c0 += TOF_STEPS) {
                // 1. the pixels of each ray in these steps
                for (int q = wid; q < sh.rb; q += TOF_THREADS / 32) {
                    const int n = min(TOF_STEPS, steps_of[q] - c0);
                    bool ok0 = false, ok1 = false;
                    float l0 = 0.f, l1 = 0.f, tau0 = 0.f, tau1 = 0.f;
                    unsigned o0 = 0, o1 = 0;
                    if (lane < n) {
                        const RayGeo &rg = g.rays[(size_t)slot * NB + tb * sh.rb + q];
                        const int kd = first_of[q] + c0 + lane, dd = rg.d0 + kd;
                        const long long lo = rg.loq + (long long)kd * vw.stepq, hi = lo + vw.absstepq;
                        const int r0 = (int)(lo >> 32), r1 = (int)(hi >> 32);
                        l1 = r1 != r0 ? __uint2float_rn((unsigned)(hi & 0xFFFFFFFFLL)) * (vw.inv_minorf * kQ32) : 0.f;
                        l0 = vw.Lf - l1;
                        ok0 = (unsigned)r0 < (unsigned)N;
                        ok1 = l1 > 0.f && (unsigned)r1 < (unsigned)N;
                        const float taud = fmaf((float)dd, tpd, vw.tau0f);
                        tau0 = fmaf((float)r0, tpr, taud);
                        tau1 = fmaf((float)r1, tpr, taud);
                        o0 = (unsigned)dd * ds + (unsigned)r0 * cs;
                        o1 = o0 + cs;
                    }
                    const unsigned m0 = __ballot_sync(0xffffffffu, ok0), m1 = __ballot_sync(0xffffffffu, ok1);
                    const unsigned below = (1u << lane) - 1u;
                    int at = q * E + __popc(m0 & below) + __popc(m1 & below);
                    if (ok0) { off[at] = o0; lt[at] = make_float2(l0, tau0); ++at; }
                    if (ok1) { off[at] = o1; lt[at] = make_float2(l1, tau1); }
                    if (lane == 0) count[q] = __popc(m0) + __popc(m1);
                }
                __syncthreads();
                // 2. the weights length x h_t, h_t from the table (cubic Hermite)
                const int TT = sh.ts * TOF_TW;
                for (int q = 0; q < sh.rb; ++q)
                    for (int i = threadIdx.x; i < count[q] * TT; i += TOF_THREADS) {
                        const int e = i / TT, t = i - e * TT;
                        const float2 p = lt[q * E + e];
                        // (the position minus the TOF bin's centre, as tof_fwd_kernel rounds it)
                        const float x = (fmaf((float)(1 - T + 2 * t) * -0.5f, d, p.y) + Wt) * idt;
                        float h = 0.f;
                        if (t < T && x >= 0.f && x < (float)(TOF_TAB - 1)) h = p.x * tof_table(tab, x, dt_);
                        wts[((q * E + e) * sh.ts + t / TOF_TW) * TOF_WP + t % TOF_TW] = vsplat(h);
                    }
                __syncthreads();
                // 3. the sums
                if (work) {
                    const int n = count[rl];
                    const f2x *we = wts + (rl * E * sh.ts + slice) * TOF_WP;
                    auto pixels = [&](auto number, int e) {
                        constexpr int U = decltype(number)::value;
                        f2x x0[U], x1[U];
#pragma unroll
                        for (int i = 0; i < U; ++i) {
                            const float *px = img + off[rl * E + e + i];
                            asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(x0[i]), "=l"(x1[i]) : "l"(px));
                        }
                        auto weights = [&](int i, f2x(&wv)[TOF_TW]) {
                            const ulonglong2 *wp = reinterpret_cast<const ulonglong2 *>(we + i * sh.ts * TOF_WP);
                            const ulonglong2 w01 = wp[0], w23 = wp[1], w45 = wp[2];
                            wv[0] = w01.x; wv[1] = w01.y; wv[2] = w23.x; wv[3] = w23.y;
                            wv[4] = w45.x; wv[5] = w45.y; wv[6] = wp[3].x;
                        };
#pragma unroll
                        for (int i = 0; i < U; i += 2) {
                            f2x w0[TOF_TW], w1[TOF_TW];
                            weights(e + i, w0);
                            if (U > 1) weights(e + i + 1, w1);
#pragma unroll
                            for (int t = 0; t < TOF_TW; ++t)
#pragma unroll
                                for (int q = 0; q < 2; ++q) {
                                    const f2x *xq = q ? x1 : x0;
                                    if (U > 1) add2x<AR>(w0[t], xq[i], w1[t], xq[i + (U > 1)], sm[t][q], er[t][q]);
                                    else add2x<AR>(w0[t], xq[i], 0ull, 0ull, sm[t][q], er[t][q]);
                                }
                        }
                    };
                    int e = 0;
                    for (; e + 4 <= n; e += 4) pixels(std::integral_constant<int, 4>{}, e);
                    for (; e < n; ++e) pixels(std::integral_constant<int, 1>{}, e);
                }
                __syncthreads();                        // the lists are free again
            }
            if (!work) continue;
            const int ray = u * NB + tb * sh.rb + rl;
            const float scale = (float)g.scale;
#pragma unroll
            for (int tl = 0; tl < TOF_TW; ++tl) {
                const int t = slice * TOF_TW + tl;
                if (t >= T) break;
                float v[4];
                vunpk(vadd(sm[tl][0], er[tl][0]), v[0], v[1]);
                vunpk(vadd(sm[tl][1], er[tl][1]), v[2], v[3]);
                const size_t o = ((size_t)ray * T + t) * Pp + (size_t)hg * 4;
                float out[4];
                if constexpr (MODE == FWD_PLAIN) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) out[c] = scale * v[c];
                } else {
                    const int4 cn = __ldg(reinterpret_cast<const int4 *>(a.counts + o));
                    const float4 gm = __ldg(reinterpret_cast<const float4 *>(a.gamma + o));
                    const int cnt[4] = {cn.x, cn.y, cn.z, cn.w};
                    const float gam[4] = {gm.x, gm.y, gm.z, gm.w};
                    float s_af = 0.f;
                    double s_gl = 0.0;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const bool valid = hg * 4 + c < g.P;
                        const float m = a.mult ? __ldg(a.mult + o + c) : 1.f;
                        const float af = scale * (v[c] * m);
                        if constexpr (MODE == FWD_RATIO) {
                            out[c] = valid ? m * (1.f - (float)cnt[c] / (af + gam[c])) : 0.f;
                        } else if (valid) {
                            s_af += af;
                            if (cnt[c] != 0) s_gl += (double)cnt[c] * log((double)af + (double)gam[c]);
                        }
                    }
                    obj[0] += (double)s_af;
                    obj[1] += s_gl;
                }
                if constexpr (MODE != FWD_OBJECTIVE)
                    *reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.out) + o) =
                        make_float4(out[0], out[1], out[2], out[3]);
            }
        }
        if constexpr (MODE == FWD_OBJECTIVE) grid_reduce<2>(obj, a.red, a.result, vloc, nv);
    }
}

int sm_count();
int resident_blocks(const void *fn);

template <int G>
static const void *tof_fwd_fn(int mode, int arith)
{
#define PET_TOF_FN(AR)                                                                      \
    (mode == FWD_PLAIN ? (const void *)tof_fwd_kernel<G, AR, FWD_PLAIN>                     \
     : mode == FWD_RATIO ? (const void *)tof_fwd_kernel<G, AR, FWD_RATIO>                   \
                         : (const void *)tof_fwd_kernel<G, AR, FWD_OBJECTIVE>)
    if (arith == AR_FP64) return PET_TOF_FN(AR_FP64);
    if (arith == AR_FP32) return PET_TOF_FN(AR_FP32);
    return PET_TOF_FN(AR_KAHAN);
#undef PET_TOF_FN
}

template <int AR>
static auto tof_stack_any(int mode) -> void (*)(const FwdArgs, const Batch)
{
    return mode == FWD_PLAIN ? tof_fwd_stack<AR, FWD_PLAIN>
           : mode == FWD_RATIO ? tof_fwd_stack<AR, FWD_RATIO> : tof_fwd_stack<AR, FWD_OBJECTIVE>;
}
static const void *tof_stack_fn(int mode, int arith)
{
    return arith == AR_KAHAN ? (const void *)tof_stack_any<AR_KAHAN>(mode) : (const void *)tof_stack_any<AR_FP32>(mode);
}

static cudaError_t tof_stack_launch(const FwdArgs &a, const Batch &b, int mode, int arith, int grid, size_t smem,
                                    cudaStream_t st)
{
    auto fn = arith == AR_KAHAN ? tof_stack_any<AR_KAHAN>(mode) : tof_stack_any<AR_FP32>(mode);
    cudaError_t e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, TOF_SMEM_MAX);
    if (e != cudaSuccess) return e;
    fn<<<grid, TOF_THREADS, smem, st>>>(a, b);
    return cudaGetLastError();
}

// 256 (ray, TOF bin, group) items per block; the objective groups blocks into one wave of
// virtual blocks (each ends in a reduction step), never more than its reducer holds.
void forward_shape_tof(FwdArgs &a, int mode, int arith)
{
    const bool stack = a.g.tofk && arith != AR_FP64;
    const TofShape sh = tof_shape(a.g.NG, a.g.T);
    const long long items = (long long)a.nviews * a.g.NB * a.g.T * a.g.NG;
    const long long blocks = stack ? (long long)a.nviews * ((a.g.NB + sh.rb - 1) / sh.rb) * sh.nhb
                                   : std::max(1LL, (items + 255) / 256);
    a.S = 1;
    a.R = 1;
    a.tpv = 1;
    if (mode == FWD_OBJECTIVE) {
        // (asked without the stack kernel's dynamic shared memory: its registers allow two blocks per SM, whose
        // 2 x 90 KB fit)
        const void *fn = stack ? tof_stack_fn(mode, arith) : a.g.G == 1 ? tof_fwd_fn<1>(mode, arith) : tof_fwd_fn<8>(mode, arith);
        const long long slots = (long long)sm_count() * resident_blocks(fn);
        long long tpv = (blocks + slots - 1) / slots;
        if (a.red.capacity > 0) tpv = std::max(tpv, (blocks + a.red.capacity - 1) / a.red.capacity);
        a.tpv = (int)std::max(1LL, tpv);
    }
    a.nvb = (int)((blocks + a.tpv - 1) / a.tpv);
}

template <int G, int AR>
static void tof_launch_mode(const FwdArgs &a, const Batch &b, int mode, int grid, cudaStream_t st)
{
    if (mode == FWD_PLAIN) tof_fwd_kernel<G, AR, FWD_PLAIN><<<grid, 256, 0, st>>>(a, b);
    else if (mode == FWD_RATIO) tof_fwd_kernel<G, AR, FWD_RATIO><<<grid, 256, 0, st>>>(a, b);
    else tof_fwd_kernel<G, AR, FWD_OBJECTIVE><<<grid, 256, 0, st>>>(a, b);
}

template <int G>
static void tof_launch(const FwdArgs &a, const Batch &b, int mode, int arith, int grid, cudaStream_t st)
{
    if (arith == AR_FP64) tof_launch_mode<G, AR_FP64>(a, b, mode, grid, st);
    else if (arith == AR_FP32) tof_launch_mode<G, AR_FP32>(a, b, mode, grid, st);
    else tof_launch_mode<G, AR_KAHAN>(a, b, mode, grid, st);
}

pet_status launch_forward_tof(const FwdArgs &a0, int mode, int arith, cudaStream_t st)
{
    FwdArgs a = a0;
    if ((long long)a.nviews * a.g.NB == 0) return PET_OK;
    forward_shape_tof(a, mode, arith);
    const int grid = std::max(1, std::min(a.nvb, sm_count() * 8));
    LaunchScope ls(mode == FWD_RATIO ? PET_K_FORWARD_RATIO
                   : (mode == FWD_OBJECTIVE ? PET_K_OBJ_FORWARD : PET_K_OTHER), st);
    const Batch b{nullptr, nullptr, 0, grid};
    if (a.g.tofk && arith != AR_FP64) {
        const cudaError_t es = tof_stack_launch(a, b, mode, arith, grid, (size_t)tof_shape(a.g.NG, a.g.T).rb * tof_ray_smem(tof_shape(a.g.NG, a.g.T).ts), st);
        return es == cudaSuccess ? PET_OK : cuda_fail(es, "tof_fwd_stack launch");
    }
    if (a.g.G == 1) tof_launch<1>(a, b, mode, arith, grid, st);
    else tof_launch<8>(a, b, mode, arith, grid, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "tof_fwd_kernel launch");
    return PET_OK;
}

// Batched launch: every scan of the batch has TOF bins and the plane-group size of `shape`.
pet_status launch_forward_tof_batch(const FwdArgs &shape, const Batch &b, int mode, int arith,
                                    cudaStream_t st)
{
    LaunchScope ls(mode == FWD_RATIO ? PET_K_FORWARD_RATIO
                   : (mode == FWD_OBJECTIVE ? PET_K_OBJ_FORWARD : PET_K_OTHER), st);
    if (shape.g.tofk && arith != AR_FP64) {
        const cudaError_t es = tof_stack_launch(shape, b, mode, arith, b.grid, TOF_SMEM_MAX, st);
        return es == cudaSuccess ? PET_OK : cuda_fail(es, "tof_fwd_stack batch launch");
    }
    if (shape.g.G == 1) tof_launch<1>(shape, b, mode, arith, b.grid, st);
    else tof_launch<8>(shape, b, mode, arith, b.grid, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "tof_fwd_kernel batch launch");
    return PET_OK;
}

}  // namespace pet
