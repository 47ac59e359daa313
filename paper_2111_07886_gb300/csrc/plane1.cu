// FP32 projector and update of single-plane scans (2-D reconstructions, alone and in batches).
//
// With one plane a pixel is 4 bytes, so what bounds these kernels is not the walk's arithmetic but
// how many cache lines one warp load touches, and how many threads a small image gives:
//   - forward: neighbouring lanes walk neighbouring rays of a view, so at one driving step they
//     read neighbouring pixels of the cross axis.  Views driven along x have that axis along y:
//     they read a transposed copy of the image, which follows every single-plane FP32 image
//     [N*N] in memory (the update writes both), so both kinds of view read a few consecutive
//     sectors per warp;
//   - update: a (pixel, view) entry serves one thread only, so it is computed in registers where
//     it is used instead of going through a shared-memory table and two barriers; small images
//     split the neighbours and views of a pixel over C lanes.
// Sub-ray bins (R lines per bin) are taken in closed form: per driving step the lengths of a
// bin's R equally spaced lines in one pixel are the difference of a piecewise quadratic
// cumulative function at the pixel's two edges (line_length_below), exact in Q32.32 integers.
#include "image.cuh"
#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

int sm_count();
int resident_blocks(const void *fn);

// Single-plane FP32 scans without TOF run the kernels of this file.
bool plane1_path(const GeoDev &g, int arith) { return g.G == 1 && arith != AR_FP64 && g.T == 1; }

constexpr int P1_PAD = 4;           // zero bins on both sides of a row of w (see update_kernel_p1)
int plane1_pad() { return P1_PAD; }

// Bins whose lines are summed in closed form (kernels.cuh)
static __host__ __device__ __forceinline__ bool closed_sums(const GeoDev &g) { return g.table && g.R >= SUB_CLOSED_MIN; }

// One compensated (Kahan) or plain step of a running sum.
template <int AR>
__device__ __forceinline__ void p1_add(float y, float &s, float &e)
{
    if constexpr (AR == AR_KAHAN) {
        y += e;
        const float t = s + y;
        e = y - (t - s);
        s = t;
    } else {
        s += y;
    }
}

// The same for w0 x0 + w1 x1: one driving step of a ray, or two bins of a (pixel, view) entry.
template <int AR>
__device__ __forceinline__ void p1_add2(float w0, float x0, float w1, float x1, float &s, float &e)
{
    if constexpr (AR == AR_KAHAN) {
        const float y = fmaf(w1, x1, fmaf(w0, x0, e)), t = s + y;
        e = y - (t - s);
        s = t;
    } else {
        s = fmaf(w1, x1, fmaf(w0, x0, s));
    }
}

// `steps` driving steps of one line from cross coordinate lo (Q32.32), reading rows of stride N from
// img + base; the loads of four steps are issued together, and every step is one compensated step of
// the sum.  The carry of the 32-bit fractions says whether a step crosses into the next pixel (a
// step rises by at most one pixel, and by exactly one only at 45 degrees, where all do).
template <int AR>
__device__ __forceinline__ void p1_walk(const float *__restrict__ img, unsigned N, unsigned base, long long lo,
                                        long long stp, long long ast, float L, float im, int steps, float &s,
                                        float &e)
{
    const unsigned rise = (unsigned)ast;
    const bool all = (ast >> 32) != 0;
    auto step = [&](float &l0, float &x0, float &l1, float &x1) {
        const unsigned r = (unsigned)(int)(lo >> 32), fr = (unsigned)lo, up = fr + rise;
        const bool cross = all || up < fr;
        l1 = cross ? __uint2float_rn(up) * im : 0.f;
        l0 = L - l1;
        const float *q = img + (int)(base + r);     // r may be -1
        x0 = x1 = 0.f;
        if (r < N) x0 = __ldg(q);
        if (cross && r + 1u < N) x1 = __ldg(q + 1);
        lo += stp;
        base += N;
    };
    for (; steps >= 4; steps -= 4) {
        float l0[4], x0[4], l1[4], x1[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) step(l0[j], x0[j], l1[j], x1[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) p1_add2<AR>(l0[j], x0[j], l1[j], x1[j], s, e);
    }
    for (; steps > 0; --steps) {
        float l0, x0, l1, x1;
        step(l0, x0, l1, x1);
        p1_add2<AR>(l0, x0, l1, x1, s, e);
    }
}

// Thread layout: 256 threads = S chunks x R rays (thread = chunk * R + ray), rays in view order so
// that a warp's lanes are neighbouring bins; chunk c walks driving steps [c Lc, (c + 1) Lc).  The S
// partial sums of a ray are combined in chunk order.  A virtual block takes a.tpv ray tiles.
template <int AR, int MODE, bool SUB>
__device__ __forceinline__ void fwd_p1_vblock(const FwdArgs &a, int vloc, float *comb_s, float *comb_e,
                                              double (*red_sh)[32])
{
    const GeoDev &g = a.g;
    const int NB = g.NB, N = g.N, S = a.S, R = a.R;
    const int nrays = a.nviews * NB;
    const int ntiles = (nrays + R - 1) / R;
    const int c = threadIdx.x / R, rl = threadIdx.x - c * R;
    const bool lane_ok = c < S;
    double obj[2] = {0.0, 0.0};
    const int t_end = min(ntiles, (vloc + 1) * a.tpv);
    for (int tile = vloc * a.tpv; tile < t_end; ++tile) {
        const int ray = tile * R + rl;
        const bool live = lane_ok && ray < nrays;
        float s = 0.f, e = 0.f;
        int cnt = 0;
        float gam = 0.f, m = 1.f;
        if (MODE != FWD_PLAIN && live && c == 0) {          // read before the walk, used after it
            cnt = __ldg(a.counts + ray);
            gam = __ldg(a.gamma + ray);
            if (a.mult) m = __ldg(a.mult + ray);
        }
        if (live) {
            const ViewGeo &vw = g.views[a.slot0 + ray / NB];
            const RayGeo &rg = g.rays[(size_t)a.slot0 * NB + ray];
            // views driven along x read the transposed copy behind the image: the cross axis is
            // contiguous and the driving axis has stride N on every view
            const float *img = reinterpret_cast<const float *>(a.img);
            const unsigned copy = vw.xdrive ? (unsigned)N * (unsigned)N : 0u;
            const int Lc = (rg.nd + S - 1) / S;
            const int k0 = c * Lc, k1 = min(rg.nd, k0 + Lc);
            const long long stp = vw.stepq, ast = vw.absstepq;
            const float L = vw.Lf, im = vw.inv_minorf * kQ32;
            const unsigned base = copy + (unsigned)(rg.d0 + k0) * (unsigned)N;
            const long long lo = rg.loq + (long long)k0 * stp;
            if constexpr (SUB) {
                const int nsr = g.R;
                if (nsr >= SUB_CLOSED_MIN && !vw.axis && 2ll * nsr * (rg.shq < 0 ? -rg.shq : rg.shq) < SUB_CLOSED_SPAN) {
                    const LineFan fan = line_fan(nsr, rg.shq, ast, vw.inv_minorf, vw.inv_minorl);
                    long long b = lo - (long long)(nsr - 1) * (rg.shq < 0 ? -rg.shq : rg.shq);
                    unsigned row = base;
                    for (int k = k0; k < k1; ++k) {
                        float bl = 0.f;
                        const int rlo = max(0, (int)(b >> 32));
                        const int rtop = (int)((b + fan.span) >> 32), rhi = min(N - 1, rtop);
                        long long below = line_length_below(fan, ((long long)rlo << 32) - b);
                        for (int r = rlo; r <= rhi; ++r) {
                            const long long up = r == rtop ? fan.total
                                                           : line_length_below(fan, ((long long)(r + 1) << 32) - b);
                            bl = fmaf(fan_length(fan, up - below), __ldg(img + row + (unsigned)r), bl);
                            below = up;
                        }
                        p1_add<AR>(bl, s, e);
                        b += stp;
                        row += (unsigned)N;
                    }
                } else {
                    for (int sr = 0; sr < nsr; ++sr)
                        p1_walk<AR>(img, (unsigned)N, base, lo + (long long)(2 * sr + 1 - nsr) * rg.shq, stp, ast,
                                    L, im, k1 - k0, s, e);
                }
            } else {
                p1_walk<AR>(img, (unsigned)N, base, lo, stp, ast, L, im, k1 - k0, s, e);
            }
        }
        if (S > 1) {
            __syncthreads();
            comb_s[threadIdx.x] = s;
            comb_e[threadIdx.x] = e;
            __syncthreads();
            if (live && c == 0)
                for (int cc = 1; cc < S; ++cc) {
                    if constexpr (AR == AR_KAHAN) e += comb_e[cc * R + rl];
                    p1_add<AR>(comb_s[cc * R + rl], s, e);
                }
        }
        if (live && c == 0) {
            const float tot = s + e, scale = (float)g.scale;
            if constexpr (MODE == FWD_PLAIN) {
                reinterpret_cast<float *>(a.out)[ray] = SUB && closed_sums(g) ? fmaf(scale, s, scale * e) : scale * tot;
            } else {
                const float af = scale * (tot * m);
                if constexpr (MODE == FWD_RATIO) {
                    const int u = ray / NB, b = ray - u * NB;
                    float *out = reinterpret_cast<float *>(a.out) + (size_t)u * (NB + 2 * a.pad) + a.pad;
                    float y = af + gam;
                    if (SUB && closed_sums(g)) {
                        // scale m (s + e) + gamma with the rounding of the result only (the closed sums
                        // are exact to that): sm + sml is scale m
                        const float sm = scale * m, sml = fmaf(scale, m, -sm);
                        y = fmaf(sm, s, fmaf(sm, e, fmaf(sml, s, gam)));
                    }
                    out[b] = m * (1.f - (float)cnt / y);
                    // the zero bins on both sides of the row (see update_kernel_p1)
                    if (b == 0)
                        for (int q = 1; q <= a.pad; ++q) out[-q] = 0.f;
                    if (b == NB - 1)
                        for (int q = 0; q < a.pad; ++q) out[NB + q] = 0.f;
                } else {
                    // the likelihood terms in FP64 in every mode: ln((double) Af + gamma)
                    obj[0] += (double)af;
                    if (cnt != 0) obj[1] += (double)cnt * log((double)af + (double)gam);
                }
            }
        }
    }
    if constexpr (MODE == FWD_OBJECTIVE) reduce_partial<2>(obj, a.red, vloc, red_sh);
}

template <int AR, int MODE, bool SUB>
__global__ void __launch_bounds__(256, 4) fwd_kernel_p1(const __grid_constant__ FwdArgs one, const Batch bt)
{
    grid_dependency_wait();                      // before any memory access
    grid_dependents_launch();
    __shared__ float comb_s[256], comb_e[256];
    __shared__ FwdArgs sh_args;
    __shared__ double red_sh[2][32];
    VblockRuns runs(total_vblocks(one, bt));
    const FwdArgs *a = nullptr;
    int done = 0, vloc = 0, nv = 0;
    KeptScan kept;
    for (int vb; (vb = runs.next()) >= 0;) {
        if (scan_args_kept(one, bt, vb, vloc, nv, sh_args, kept, a)) done = 0;
        fwd_p1_vblock<AR, MODE, SUB>(*a, vloc, comb_s, comb_e, red_sh);
        ++done;
        if constexpr (MODE == FWD_OBJECTIVE)
            if (runs.ends() || vloc + 1 == nv) {
                reduce_finish<2>(a->red, a->result, done, nv, red_sh);
                done = 0;
            }
    }
}

// The subset projection and the mu pass in one launch (as fwd_mu_kernel)
template <int AR, bool SUB>
__global__ void __launch_bounds__(256, 4) fwd_mu_kernel_p1(const __grid_constant__ FwdArgs fwd,
                                                           const __grid_constant__ ImageArgs mu, int nfwd)
{
    grid_dependency_wait();
    grid_dependents_launch();
    __shared__ float comb_s[256], comb_e[256];
    const int vb = (int)blockIdx.x;
    if (vb < nfwd) fwd_p1_vblock<AR, FWD_RATIO, SUB>(fwd, vb, comb_s, comb_e, nullptr);
    else mu_p1_vblock(mu, vb - nfwd, mu.nvb);
}

// What a patch's (pixel, view) entries need of a view: t - h at the patch's first pixel, its slopes
// and 2 h (Q32.32 bins), the row's first bin in w, and the trapezoid.
struct __align__(16) P1View {
    long long x, cx, cy, h2;
    unsigned row;
    float ws, L;               // length per 2^-24 bin, L
    int axis;
};
constexpr int P1_VIEWS = 32;   // views of the subset a warp holds at a time

// Neighbour q of pixel (ix, iy), row by row without the centre: numerator and 1 / denominator of the
// RDP gradient term (without its factor 2), and the part in the Matlab-style gradient (a missing axial
// neighbour counts as the centre).
__device__ __forceinline__ void p1_neighbour(const float *f, int N, int ix, int iy, int q, float fc, float gamma_r,
                                             float eps, float &num, float &rden, float &gx, float &gy)
{
    const int r = q < 4 ? q : q + 1, dy = r / 3 - 1, dx = r - 3 * (dy + 1) - 1;
    const int x = ix + dx, y = iy + dy;
    float fk = fc;
    num = rden = 0.f;
    if ((unsigned)x < (unsigned)N && (unsigned)y < (unsigned)N) {
        fk = __ldg(f + y * N + x);
        const float d = fc - fk, ad = fabsf(d), den = fc + fk + gamma_r * ad + eps;
        num = d * (gamma_r * ad + fc + 3.f * fk + 2.f * eps);
        rden = __fdividef(1.f, den * den);
    }
    if (dy == 0) gx += (float)dx * fk;
    else if (dx == 0) gy += (float)dy * fk;
}

// The KC lengths and row values of pixel (ix, iy) and view u of the subset: sub-ray bins, and views
// along an axis (membership from the forward walk's own coordinates).
template <int KC, int AR, bool SUB>
__device__ __forceinline__ void p1_any_entry(const UpdateArgs &a, int u, int ix, int iy, float (&l)[KC], float (&x)[KC])
{
    const GeoDev &g = a.g;
    const auto ent = bp_entry<KC, AR, 0, SUB>(g, a.slot0 + u, 0, true, ix, iy);
    const float *row = reinterpret_cast<const float *>(a.w) + (size_t)u * (g.NB + 2 * P1_PAD) + P1_PAD + ent.off;
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        l[k] = ent.w[k];
        x[k] = __ldg(row + k);
    }
}

// The patches of one virtual block that fall to warp `wid`; returns this lane's sum of new pixels.
// CT: the lanes per pixel, or 0 for a.C (sub-ray bins: their entries are too much code to repeat).
template <int KC, int AR, bool SUB, int CT>
__device__ __forceinline__ float p1_patches(const UpdateArgs &a, P1View *vt, int vloc, int wid, int lane,
                                            float inv_mean_f, float mean_mu)
{
    const GeoDev &g = a.g;
    const int N = g.N, NB = g.NB, npix = N * N, stride = NB + 2 * P1_PAD;
    const bool dyn = a.nu_mode == 1 || a.nu_mode == 2;
    const int C = CT ? CT : a.C;
    const int PX = 32 / C, TX = C == 1 ? 8 : (C == 8 ? 2 : 4), TY = PX / TX;
    const int c = lane / PX, pl = lane - c * PX, py = pl / TX, px = pl - py * TX;
    const int ntx = (N + TX - 1) / TX, npatch = ntx * ((N + TY - 1) / TY);
    const float *w = reinterpret_cast<const float *>(a.w);
    const float *f = reinterpret_cast<const float *>(a.f);
    const float U = a.fs_U, tt = a.fs_t, scale = a.fs_scale;
    float part = 0.f;
    for (int k = 0; k < a.tpv; ++k) {
        const int patch = (vloc * a.tpv + k) * 8 + wid;
        if (patch >= npatch) break;
        const int x0 = (patch % ntx) * TX, y0 = (patch / ntx) * TY;
        const int ix = x0 + px, iy = y0 + py, j = iy * N + ix;
        const bool active = ix < N && iy < N;
        // stencil: each lane takes the neighbours c, c + C, ..., and the terms are added in row order
        float fc = 0.f, gr = 0.f, gx = 0.f, gy = 0.f;
        if (active) fc = __ldg(f + j);
#pragma unroll
        for (int q8 = 0; q8 < 8 / C; ++q8) {
            float num = 0.f, rden = 0.f;
            if (active) p1_neighbour(f, N, ix, iy, q8 * C + c, fc, a.fs_gamma_r, a.fs_eps, num, rden, gx, gy);
#pragma unroll
            for (int cc = 0; cc < C; ++cc) {
                const float n1 = C == 1 ? num : __shfl_sync(0xffffffffu, num, cc * PX + pl);
                const float r1 = C == 1 ? rden : __shfl_sync(0xffffffffu, rden, cc * PX + pl);
                gr = fmaf(n1, r1, gr);
            }
        }
#pragma unroll
        for (int o = PX; o < 32; o *= 2) {
            gx += __shfl_xor_sync(0xffffffffu, gx, o);
            gy += __shfl_xor_sync(0xffffffffu, gy, o);
        }
        // gather: chunk c sets up the entries of the views c, c + C, ...; every lane of the pixel adds
        // them in view order, two bins per compensated step, whatever C is
        float s = 0.f, e = 0.f;
        auto add = [&](const float (&l)[KC], const float (&x)[KC], int views) {
            if (C == 1) {
#pragma unroll
                for (int q = 0; q < KC; q += 2) p1_add2<AR>(l[q], x[q], l[q + 1], x[q + 1], s, e);
            } else {
#pragma unroll
                for (int cc = 0; cc < C; ++cc) {
                    if (cc >= views) break;
#pragma unroll
                    for (int q = 0; q < KC; q += 2) {
                        const int from = cc * PX + pl;
                        p1_add2<AR>(__shfl_sync(0xffffffffu, l[q], from), __shfl_sync(0xffffffffu, x[q], from),
                                    __shfl_sync(0xffffffffu, l[q + 1], from), __shfl_sync(0xffffffffu, x[q + 1], from), s, e);
                    }
                }
            }
        };
        if constexpr (SUB) {
            for (int u0 = 0; u0 < a.nviews; u0 += C) {
                float l[KC] = {}, x[KC] = {};
                if (active && u0 + c < a.nviews) p1_any_entry<KC, AR, SUB>(a, u0 + c, ix, iy, l, x);
                add(l, x, a.nviews - u0);
            }
        } else {
            for (int u0 = 0; u0 < a.nviews; u0 += P1_VIEWS) {
                const int nvc = min(P1_VIEWS, a.nviews - u0);
                __syncwarp();
                if (lane < nvc) {
                    const ViewGeo &vw = g.views[a.slot0 + u0 + lane];
                    P1View v;
                    v.x = vw.t0q - vw.hq + (long long)x0 * vw.cxq + (long long)y0 * vw.cyq;
                    v.cx = vw.cxq;
                    v.cy = vw.cyq;
                    v.h2 = 2 * vw.hq;
                    v.row = (unsigned)(u0 + lane) * (unsigned)stride + P1_PAD;
                    v.ws = vw.wslopef * (kQ32 * 256.f);
                    v.L = vw.Lf;
                    v.axis = vw.axis;
                    vt[lane] = v;
                }
                __syncwarp();
#pragma unroll 4
                for (int r = 0; r < nvc; r += C) {
                    float l[KC] = {}, x[KC] = {};
                    const int u = r + c;
                    if (u < nvc) {
                        const P1View v = vt[u];
                        if (!v.axis) {
                            // the entry of bp_weights, bit by bit: with d = b0 - (t - h) in [0, 1) the
                            // distance of bin b0 + q from the nearer foot of the trapezoid is
                            // min(d + q, 2 h - d - q), taken in 2^-24 bins
                            const long long t = v.x + px * v.cx + py * v.cy;
                            const unsigned lo = (unsigned)t, d = 0u - lo;
                            const int up = (int)(t >> 32) + (lo != 0u);                     // ceil
                            const int rising = (int)(d >> 8), falling = (int)((v.h2 - (long long)d) >> 8);
                            const int b0 = min(max(up, -P1_PAD), NB + P1_PAD - KC);
                            const float *row = w + (v.row + (unsigned)b0);
#pragma unroll
                            for (int q = 0; q < KC; ++q) {
                                // KC = 2 holds geometries with 2 h < 2: the rising side ends before bin 1
                                const int fall = falling - (q << 24);
                                const int dd = KC == 2 && q == 1 ? fall : min(rising + (q << 24), fall);
                                l[q] = fminf(v.L, __int2float_rn(max(0, dd)) * v.ws);
                                x[q] = __ldg(row + q);
                            }
                        } else if (active) {
                            p1_any_entry<KC, AR, false>(a, u0 + u, ix, iy, l, x);
                        }
                    }
                    add(l, x, nvc - r);
                }
            }
        }
        // step
        if (c == 0 && active) {
            float nu = 1.f;
            if (a.nu_mode == 3) {
                nu = __ldg(reinterpret_cast<const float *>(a.nu_frozen) + j);
            } else if (dyn) {
                // central differences inside, one-sided at the border
                gx *= ix > 0 && ix < N - 1 ? 0.5f : 1.f;
                gy *= iy > 0 && iy < N - 1 ? 0.5f : 1.f;
                const float x2 = fmaf(gx, gx, __fmul_rn(gy, gy));
                float mu = (x2 > 0.f ? x2 * rsqrtf(x2) : 0.f) * inv_mean_f;
                mu = mu < 0.01f ? 0.01f : mu;
                nu = clampT<float>(fast_div(mean_mu, mu), a.fs_nu1, a.fs_nu2);
                if (a.nu_mode == 2) reinterpret_cast<float *>(a.nu_frozen)[j] = nu;
            }
            const float ip = __ldg(reinterpret_cast<const float *>(a.invp) + j) * a.fs_ips;
            const float coef = a.fs_lam * nu * ((fc < 0.5f * U ? fc : U - fc) * ip);
            const float rg = __fmul_rn(a.fs_bm, 2.f * gr);
            float ft = fmaf(-coef, SUB && closed_sums(g) ? fmaf(scale, s, fmaf(scale, e, rg)) : fmaf(scale, s + e, rg), fc);
            ft = ft <= 0.f ? tt : (ft >= U ? U - tt : ft);
            part += ft;
            reinterpret_cast<float *>(a.fout)[j] = ft;
            reinterpret_cast<float *>(a.fout)[npix + ix * N + iy] = ft;   // the transposed copy
        }
    }
    return part;
}

// f^{k,i} = P_t(f - lambda_k alpha_{k,i} nu S(f) (A_i^T w + (beta/M) grad R(f))) for one plane.
// A warp works alone, without block barriers: it takes a patch of 32 / C pixels (8 x 4, 4 x 4,
// 4 x 2 or 2 x 2, so that one view's bins are a few sectors of the row of w) with C lanes per
// pixel, lane = chunk * (32 / C) + pixel.  Its lanes first set up one view each for the patch, then
// chunk c sets up the neighbours and the (pixel, view) entries c, c + C, ...; their terms go through
// shuffles and are added in the order of the rows and views, so that the result has the same bits for
// every C, those of one thread per pixel (sums of the chunks, each rounded, and positions in 2^-26
// bins cost up to 1.9 times the error against 64 bits in batches of scans that amplify rounding; the
// exact order costs 24 mixed scans x 10 iterations 68.2 ms instead of 67.8).
// Rows of w carry P1_PAD zero bins on both sides: an entry at the edge of the sinogram needs no test
// per bin.  A virtual block is 8 warps x a.tpv patches; only its sum ends in barriers.
template <int KC, int AR, bool SUB>
__global__ void __launch_bounds__(256, 4) update_kernel_p1(const __grid_constant__ UpdateArgs one, const Batch bt)
{
    __shared__ __align__(16) P1View views[SUB ? 1 : 8][P1_VIEWS];
    __shared__ UpdateArgs sh_args;
    __shared__ double red_sh[1][32];
    __shared__ float part_sh[256];
    grid_dependency_wait();
    grid_dependents_launch();
    VblockRuns runs(total_vblocks(one, bt));
    const UpdateArgs *ap = nullptr;
    int done = 0, vloc = 0, nv = 0;
    KeptScan kept;
    float inv_mean_f = 1.f, mean_mu = 1.f;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int vb; (vb = runs.next()) >= 0;) {
        const bool fresh = scan_args_kept(one, bt, vb, vloc, nv, sh_args, kept, ap);
        const UpdateArgs &a = *ap;
        const GeoDev &g = a.g;
        const int npix = g.N * g.N;
        const bool dyn = a.nu_mode == 1 || a.nu_mode == 2;
        if (fresh) {
            done = 0;
            if (dyn) {
                inv_mean_f = (float)npix / (float)*a.sum_f;
                mean_mu = (float)*a.sum_mu / (float)npix;
            }
        }
        float part = 0.f;
        P1View *vt = views[SUB ? 0 : wid];
        if constexpr (SUB) part = p1_patches<KC, AR, SUB, 0>(a, vt, vloc, wid, lane, inv_mean_f, mean_mu);
        else switch (a.C) {
        case 1: part = p1_patches<KC, AR, SUB, 1>(a, vt, vloc, wid, lane, inv_mean_f, mean_mu); break;
        case 2: part = p1_patches<KC, AR, SUB, 2>(a, vt, vloc, wid, lane, inv_mean_f, mean_mu); break;
        case 4: part = p1_patches<KC, AR, SUB, 4>(a, vt, vloc, wid, lane, inv_mean_f, mean_mu); break;
        default: part = p1_patches<KC, AR, SUB, 8>(a, vt, vloc, wid, lane, inv_mean_f, mean_mu);
        }
        // the block's 256 partial sums, added in FP64 by one warp (the FP64 pipe is narrow)
        part_sh[threadIdx.x] = part;
        __syncthreads();
        if (wid == 0) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) v += (double)part_sh[q * 32 + lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) a.red.partials[vloc] = v;
        }
        ++done;
        if (runs.ends() || vloc + 1 == nv) {
            reduce_finish<1>(a.red, a.sum_fout, done, nv, red_sh);
            done = 0;
        }
        __syncthreads();                     // part_sh is free again
    }
}

// ------------------------------------------------------------------------------------------
// Shapes and launches
// ------------------------------------------------------------------------------------------
template <int AR>
static const void *fwd_p1_fn(int mode, int sub)
{
    if (sub) return mode == FWD_PLAIN ? (const void *)fwd_kernel_p1<AR, FWD_PLAIN, true>
                    : mode == FWD_RATIO ? (const void *)fwd_kernel_p1<AR, FWD_RATIO, true>
                                        : (const void *)fwd_kernel_p1<AR, FWD_OBJECTIVE, true>;
    return mode == FWD_PLAIN ? (const void *)fwd_kernel_p1<AR, FWD_PLAIN, false>
           : mode == FWD_RATIO ? (const void *)fwd_kernel_p1<AR, FWD_RATIO, false>
                               : (const void *)fwd_kernel_p1<AR, FWD_OBJECTIVE, false>;
}

// Chunks per ray as for stacks (forward_shape): one wave of 2048 threads per SM where the rays allow it,
// at most 16 of at least 16 driving steps each.  A step of closed sums is about ten times the work of a
// line's, so there up to 32 chunks of 8 steps (the 256 x 256 ring scan with 32 rays per bin: an iteration
// takes 1.50 ms with 16 chunks and 1.30 with 32).
void forward_shape_p1(FwdArgs &a, int mode, int arith)
{
    const bool closed = closed_sums(a.g);
    const long long nrays = std::max(1LL, (long long)a.nviews * a.g.NB);
    const long long want = (long long)sm_count() * 2048;
    int S = (int)std::min<long long>(closed ? 32 : 16, (want + nrays - 1) / nrays);
    S = std::max(1, std::min(S, a.g.N / (closed ? 8 : 16)));
    if (a.g.tuneS > 0 && mode != FWD_OBJECTIVE) S = a.g.tuneS;
    while (256 % S) --S;
    a.S = S;
    a.R = 256 / S;
    const long long ntiles = (nrays + a.R - 1) / a.R;
    a.tpv = 1;
    if (mode == FWD_OBJECTIVE) {
        const void *fn = arith == AR_KAHAN ? fwd_p1_fn<AR_KAHAN>(mode, a.g.table) : fwd_p1_fn<AR_FP32>(mode, a.g.table);
        const long long slots = (long long)sm_count() * resident_blocks(fn);
        long long tpv = (ntiles + slots - 1) / slots;
        if (a.red.capacity > 0) tpv = std::max(tpv, (ntiles + a.red.capacity - 1) / a.red.capacity);
        a.tpv = (int)std::max(1LL, tpv);
    }
    a.nvb = (int)((ntiles + a.tpv - 1) / a.tpv);
}

template <int AR, bool SUB>
static void fwd_p1_launch(const FwdArgs &a, const Batch &b, int mode, int grid, cudaStream_t st, bool pdl)
{
    if (mode == FWD_PLAIN) launch_pdl(fwd_kernel_p1<AR, FWD_PLAIN, SUB>, grid, st, pdl, a, b);
    else if (mode == FWD_RATIO) launch_pdl(fwd_kernel_p1<AR, FWD_RATIO, SUB>, grid, st, pdl, a, b);
    else launch_pdl(fwd_kernel_p1<AR, FWD_OBJECTIVE, SUB>, grid, st, pdl, a, b);
}

void forward_p1_dispatch(const FwdArgs &a, const Batch &b, int mode, int arith, int grid, cudaStream_t st,
                         bool pdl)
{
    if (a.g.table) {
        if (arith == AR_KAHAN) fwd_p1_launch<AR_KAHAN, true>(a, b, mode, grid, st, pdl);
        else fwd_p1_launch<AR_FP32, true>(a, b, mode, grid, st, pdl);
    } else {
        if (arith == AR_KAHAN) fwd_p1_launch<AR_KAHAN, false>(a, b, mode, grid, st, pdl);
        else fwd_p1_launch<AR_FP32, false>(a, b, mode, grid, st, pdl);
    }
}

void forward_mu_p1(const FwdArgs &a, const ImageArgs &m, int arith, cudaStream_t st)
{
    const int grid = a.nvb + m.nvb;
    if (a.g.table) {
        if (arith == AR_KAHAN) launch_pdl(fwd_mu_kernel_p1<AR_KAHAN, true>, grid, st, true, a, m, a.nvb);
        else launch_pdl(fwd_mu_kernel_p1<AR_FP32, true>, grid, st, true, a, m, a.nvb);
    } else {
        if (arith == AR_KAHAN) launch_pdl(fwd_mu_kernel_p1<AR_KAHAN, false>, grid, st, true, a, m, a.nvb);
        else launch_pdl(fwd_mu_kernel_p1<AR_FP32, false>, grid, st, true, a, m, a.nvb);
    }
}

template <int AR>
static const void *update_p1_fn(const GeoDev &g)
{
    if (g.table) return (const void *)update_kernel_p1<4, AR, true>;
    return g.K <= 2 ? (const void *)update_kernel_p1<2, AR, false> : (const void *)update_kernel_p1<4, AR, false>;
}

// Lanes per pixel C: the fewest that give 8 warps per SM (16 for sub-ray bins, whose entries are about
// ten times the work), at least two views each.  24 mixed 2-D scans: 67.8 ms with 8 warps, 72.8 with
// 16; an iteration of the 256 x 256 ring scan with 32 rays per bin: 1.53 and 1.17 ms.
void update_shape_p1(UpdateArgs &a, int arith)
{
    const int N = a.g.N;
    auto patches = [&](int C) {
        const int TX = C == 1 ? 8 : (C == 8 ? 2 : 4), TY = 32 / C / TX;
        return (N + TX - 1) / TX * ((N + TY - 1) / TY);
    };
    int C = 1;
    while (C < 8 && patches(C) < (a.g.table ? 16 : 8) * sm_count() && a.nviews >= 4 * C) C *= 2;
    a.C = C;
    const int slots = sm_count() * resident_blocks(arith == AR_KAHAN ? update_p1_fn<AR_KAHAN>(a.g) : update_p1_fn<AR_FP32>(a.g));
    const int nt = (patches(C) + 7) / 8;
    a.tpv = std::max({1, (nt + a.red.capacity - 1) / a.red.capacity, (nt + slots - 1) / slots});
    a.nvb = (nt + a.tpv - 1) / a.tpv;
}

template <int AR>
static void update_p1_launch(const UpdateArgs &a, const Batch &b, int grid, cudaStream_t st, bool pdl)
{
    if (a.g.table) launch_pdl(update_kernel_p1<4, AR, true>, grid, st, pdl, a, b);
    else if (a.g.K <= 2) launch_pdl(update_kernel_p1<2, AR, false>, grid, st, pdl, a, b);
    else launch_pdl(update_kernel_p1<4, AR, false>, grid, st, pdl, a, b);
}

void update_p1_dispatch(const UpdateArgs &a, const Batch &b, int arith, int grid, cudaStream_t st, bool pdl)
{
    if (arith == AR_KAHAN) update_p1_launch<AR_KAHAN>(a, b, grid, st, pdl);
    else update_p1_launch<AR_FP32>(a, b, grid, st, pdl);
}

}  // namespace pet
