// The FP32 update of stacks (8-plane groups): one packed kernel for the in-plane and the 3-D prior,
// 1/p per pixel or per voxel, and the TV variant, and its precomputed backprojection entries.
#include <math.h>

#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

int sm_count();
constexpr int X8_Z3 = 1, X8_VOX = 2, X8_TV = 4, X8_TOF = 8;

// TOF: a (pixel, view) entry is X8_HD words (row offset, first TOF bin | count << 8, KC lengths) and
// h_t for up to g.tof_hw TOF bins; X8_TOF_WORDS of them in shared memory.  A tile is a TX x TY patch,
// as square as 256 / NG pixels allow: a view's rows [bin][T] of a patch overlap in two directions.
constexpr int X8_TOF_WORDS = 6144;
struct X8Patch { int tx, ty, es; };
template <int KC>
static __host__ __device__ __forceinline__ X8Patch x8_patch(const GeoDev &g)
{
    X8Patch p;
    p.es = (KC <= 2 ? 4 : 8) + (g.tof_hw + 3) / 4 * 4;
    int n = 256 / g.NG;
    if (n > X8_TOF_WORDS / p.es) n = X8_TOF_WORDS / p.es;
    p.ty = 1;
    while ((p.ty + 1) * (p.ty + 1) <= n) ++p.ty;
    p.tx = n / p.ty;
    return p;
}

// One TOF entry of pixel (ix, iy) and view u of the subset: the row offset and lengths of bp_entry,
// the TOF bins whose centre lies within the kernel's window of the pixel's position along the view's
// lines, and h_t of each (each bin edge's erfc evaluated once; the tail form of tof_h).
template <int KC, int AR>
__device__ __forceinline__ void tof_entry(const GeoDev &g, int slot0, int u, int ix, int iy, float *out)
{
    const bool in = ix < g.N && iy < g.N;
    const auto ent = bp_entry<KC, AR, 0>(g, slot0, u, in, ix, iy);
    const ViewGeo &vw = g.views[slot0 + u];
    const float tau = vw.tau0f + (float)ix * vw.tauxf + (float)iy * vw.tauyf;
    const float d = g.tof_df, kk = g.tof_kf, W = g.tof_wf;
    const float tc = tau / d + 0.5f * (float)(g.T - 1);
    const int t_lo = max(0, (int)ceilf(tc - W / d)), t_hi = min(g.T - 1, (int)floorf(tc + W / d));
    const int n = min(in ? max(0, t_hi - t_lo + 1) : 0, g.tof_hw);
    out[0] = __uint_as_float(ent.off);
    out[1] = __int_as_float(n > 0 ? t_lo | n << 8 : 0);      // t_lo < T <= 64 when n > 0
#pragma unroll
    for (int k = 0; k < KC; ++k) out[2 + k] = ent.w[k];
    float *h = out + (KC <= 2 ? 4 : 8);
    float z0 = ((float)(2 * t_lo - g.T) * 0.5f * d - tau) * kk, c0 = erfcf(fabsf(z0));
    for (int t = 0; t < n; ++t) {
        const float z1 = ((float)(2 * (t_lo + t) + 2 - g.T) * 0.5f * d - tau) * kk, c1 = erfcf(fabsf(z1));
        h[t] = z0 >= 0.f ? 0.5f * (c0 - c1) : (z1 <= 0.f ? 0.5f * (c1 - c0) : 1.f - 0.5f * (c0 + c1));
        z0 = z1;
        c0 = c1;
    }
}

// Adds an entry's rows [bin][T] to a thread's sums: two bins of a TOF bin per compensated step.
template <int KC, int AR>
__device__ __forceinline__ void tof_gather(const GeoDev &g, const float *w, const float *ent, f2x (&sm)[4], f2x (&er)[4])
{
    const unsigned Pp = (unsigned)g.Pp, TT = (unsigned)g.T;
    const int tn = __float_as_int(ent[1]), n = tn >> 8;
    float l[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) l[k] = ent[2 + k];
    const float *h = ent + (KC <= 2 ? 4 : 8);
    const float *row = w + (__float_as_uint(ent[0]) * TT + (unsigned)(tn & 255) * Pp);
    auto bins = [&](auto count, int t) {
        constexpr int U = decltype(count)::value;
        f2x x[U][KC][4];
#pragma unroll
        for (int i = 0; i < U; ++i)
#pragma unroll
            for (int kb = 0; kb < KC; ++kb) load8x(row + ((unsigned)kb * TT + (unsigned)i) * Pp, x[i][kb]);
#pragma unroll
        for (int i = 0; i < U; ++i)
#pragma unroll
            for (int kb = 0; kb < KC; kb += 2) {
                const f2x W0 = vsplat(h[t + i] * l[kb]), W1 = vsplat(h[t + i] * l[kb + 1]);
#pragma unroll
                for (int k = 0; k < 4; ++k) add2x<AR>(W0, x[i][kb][k], W1, x[i][kb + 1][k], sm[k], er[k]);
            }
        row += U * Pp;
    };
    constexpr int U = KC <= 2 ? 4 : 2;               // TOF bins whose rows are loaded together
    int t = 0;
    for (; t + U <= n; t += U) bins(std::integral_constant<int, U>{}, t);
    for (; t < n; ++t) bins(std::integral_constant<int, 1>{}, t);
}

// FP32 update for 8-plane groups held as four f32x2 pairs.  Same step as update_kernel, with:
//   - the 3x3 stencil loading every neighbour with missing ones (image border) replaced by the
//     centre value: their RDP term is exactly zero (d = 0) and the Matlab-style gradient becomes
//     the one-sided difference, as in the generic stencil;
//   - the RDP pair term written as d (den + 2 f_k + eps) / den^2 (the numerator
//     gamma_R |d| + f_j + 3 f_k + 2 eps equals den + 2 f_k + eps), from one reciprocal of den;
//   - nu = P_{nu1}^{nu2}(mean(mu) / mu) from 1 / mu = min(100, mean(f) / |grad f|);
//   - the step folded into two per-plane constants before the gather,
//     f^{k,i} = P_t(A + B b) with A = f - c (beta/M) grad R, B = -c scale, c = lambda alpha nu S,
//     so that only A, B and the sums of b = A_i^T w stay live across the gather.
// FL: X8_Z3, the 3-D prior: RDP over the 26 neighbours and nu from the 3-D gradient (each in-plane
// position's group is used as it is and shifted by one plane up and down); X8_VOX, 1/p per voxel
// (scans with per-bin detection factors); X8_TV, the TV variant (no RDP term, the unclamped z and
// the metric W written for the proximal step); X8_TOF, time of flight (see x8_patch).
// With any of these the stencil, nu and the step are the general kernel's operations in its order (GEN):
// the neighbours row by row with one division per pair, and f - c (scale b + (beta/M) grad R) from c
// read again after the gather, rounded once at f's ulp.  Folded into A + B b, the step rounds twice:
// 0.41 instead of 0.29 ulp rms per subiteration, and 2.9e-7 instead of 2.7e-7 from the 64-bit result
// after one iteration of the 256 x 256 x 89 scan with both the 3-D prior and attenuation (4.19 ms,
// 4.76 in this form, with its sums shared out as update_x8_tpv says).
// UV: views whose rows are loaded together in the gather.  Four take 128 registers, two blocks per
// SM and 8 loads in flight per thread; one takes 80 and three blocks.  The rates per tile are about
// the same (four 2.6 % faster), so what decides is how evenly the tiles fill the resident blocks
// (x8_views); the sums are the same bits.
template <int KC, int AR, int FL, int UV = 4>
__global__ void __launch_bounds__(256, UV == 1 ? 3 : 2) update_kernel_x8(
    const __grid_constant__ UpdateArgs one, const Batch bt)
{
    static_assert(AR != AR_FP64, "FP32 arithmetic only");
    // 16 KB of (pixel, view) entries: the rest of the SM's shared memory stays L1 for the gather
    using Table = BpTable<KC, AR, 1024 / (KC > 2 ? 2 : 1)>;
    constexpr bool TOF = FL & X8_TOF, Z3 = FL & X8_Z3, VOX = FL & X8_VOX, TV = FL & X8_TV, GEN = FL != 0;
    __shared__ typename std::conditional<TOF, X8Patch, Table>::type tb;
    __shared__ __align__(16) float tofs[TOF ? X8_TOF_WORDS : 4];
    // launched behind the projection (see launch_update): nothing is read before it has completed
    grid_dependency_wait();
    // the next subiteration's projection (launched after this kernel with programmatic stream
    // serialization) may be scheduled as this kernel's blocks retire; it waits for completion
    grid_dependents_launch();
    const int total = total_vblocks(one, bt);
    __shared__ UpdateArgs sh_args;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        int vloc, nv;
        const UpdateArgs &a = scan_args(one, bt, vb, vloc, nv, sh_args);
        const GeoDev &g = a.g;
        const int N = g.N, NG = g.NG, npix = N * N;
        const unsigned Pp = (unsigned)g.Pp;
        const X8Patch pa = TOF ? x8_patch<KC>(g) : X8Patch{0, 0, 0};
        const int TP = TOF ? pa.tx * pa.ty : 256 / NG;
        const int pl = threadIdx.x / NG, grp = threadIdx.x % NG;
        const int VC = max(1, min(a.nviews, TOF ? X8_TOF_WORDS / (TP * pa.es) : Table::CAP / TP));
        const int ntx = TOF ? (N + pa.tx - 1) / pa.tx : 1;
        const bool dyn = a.nu_mode == 1 || a.nu_mode == 2;
        const double q = (double)npix * g.P;
        // per-scan scalars in FP32 (an FP64 division per thread is costly at GB300's FP64 rate)
        const float mean_f = dyn ? (float)*a.sum_f / (float)q : 1.f;
        const float inv_mean_f = GEN && dyn ? (float)q / (float)*a.sum_f : 1.f;
        const float mean_mu = dyn ? (float)*a.sum_mu / (float)q : 1.f;
        const float U = a.fs_U, tt = a.fs_t;
        // eps >= 1e-30 keeps 1/den finite, so that a zero-difference term stays exactly zero
        const float eps = GEN ? a.fs_eps : fmaxf(a.fs_eps, 1e-30f);
        const float *f = reinterpret_cast<const float *>(a.f) + grp * 8;
        const float *w = reinterpret_cast<const float *>(a.w) + grp * 8;
        const float *invp = reinterpret_cast<const float *>(a.invp);
        const int ntiles = TOF ? ntx * ((N + pa.ty - 1) / pa.ty) : (npix + TP - 1) / TP;
        // the subset's precomputed entries (one contiguous block per tile) when two tiles' entries
        // fit the table: double-buffered, the next tile's block copied with cp.async while this
        // tile is gathered and the next one's stencil runs (one barrier per tile)
        const bool pre = !TOF && a.bptab && 2 * a.nviews * TP <= Table::CAP;
        const int t0 = vloc * a.tpv, t1 = min(ntiles, (vloc + 1) * a.tpv);
        auto copy_tile = [&](int tile) {
            const int tbytes = a.nviews * TP * (int)sizeof(typename Table::E);
            const char *src = static_cast<const char *>(a.bptab) + (size_t)tile * tbytes;
            if constexpr (!TOF) {
                char *dst = reinterpret_cast<char *>(tb.e) + ((tile - t0) & 1) * tbytes;
                for (int o = threadIdx.x * 16; o < tbytes; o += 256 * 16) cp_async16(dst + o, src + o);
                cp_async_commit();
            }
        };
        if (pre && t0 < t1) copy_tile(t0);
        float part = 0.f;
        for (int tile = t0; tile < t1; ++tile) {
            const int j0 = tile * TP;
            const int qy = TOF ? pl / pa.tx : 0, qx = TOF ? pl - qy * pa.tx : 0;
            const int px0 = TOF ? (tile % ntx) * pa.tx : 0, py0 = TOF ? (tile / ntx) * pa.ty : 0;
            const int ix = TOF ? px0 + qx : (j0 + pl) % N, iy = TOF ? py0 + qy : (j0 + pl) / N;
            const int j = TOF ? iy * N + ix : j0 + pl;
            const bool active = pl < TP && (TOF ? ix < N && iy < N : j < npix);
            f2x A[4], B[4];
            if (active) {
                const unsigned jc = (unsigned)j;
                const unsigned xm = ix > 0 ? jc - 1 : jc, xp = ix < N - 1 ? jc + 1 : jc;
                const unsigned ym = iy > 0 ? jc - N : jc, yp = iy < N - 1 ? jc + N : jc;
                const f2x GR = vsplat(a.fs_gamma_r), EP = vsplat(eps), TWO = vsplat(2.f);
                f2x c[4], ce[4], gr[4], g2[4], nb0[4], nb1[4], nu[4];
                load8x(f + jc * Pp, c);
#pragma unroll
                for (int k = 0; k < 4; ++k) { if (!GEN) ce[k] = vadd(c[k], EP); gr[k] = 0ull; }
                auto rdp = [&](const f2x(&x)[4]) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const f2x d = vsub(c[k], x[k]), ad = vabs(d);
                        if constexpr (GEN) {
                            const f2x EP2 = vadd(EP, EP), THREE = vsplat(3.f);
                            const f2x den = Z3 ? vadd(vfma(GR, ad, vadd(c[k], x[k])), EP)
                                               : vfma(GR, ad, vadd(vadd(c[k], x[k]), EP));
                            const f2x t = Z3 ? vadd(vfma(THREE, x[k], vfma(GR, ad, c[k])), EP2)
                                             : vfma(GR, ad, vfma(THREE, x[k], vadd(c[k], EP2)));
                            gr[k] = vfma(vmul(d, t), vrcp_finite(vmul(den, den)), gr[k]);
                        } else {
                            const f2x den = vfma(GR, ad, vadd(ce[k], x[k]));
                            const f2x num = vadd(den, vfma(TWO, x[k], EP));
                            const f2x r = vrcp(den);
                            gr[k] = vfma(vmul(d, vmul(num, r)), r, gr[k]);
                        }
                    }
                };
                // 3-D: the planes z - 1 (dn) and z + 1 (up) of a position's group x; a missing plane
                // counts as the centre pixel's own value (its term is then exactly zero)
                const int nlive = g.P - grp * 8;             // real planes from this group on
                auto shifted = [&](const f2x(&x)[4], unsigned jn, f2x(&dn)[4], f2x(&up)[4]) {
                    float v[8], cv[8];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        vunpk(x[k], v[2 * k], v[2 * k + 1]);
                        vunpk(c[k], cv[2 * k], cv[2 * k + 1]);
                    }
                    const float lo = grp > 0 ? __ldg(f + jn * Pp - 1) : cv[0];
                    const float hi = nlive > 8 ? __ldg(f + jn * Pp + 8) : cv[7];
                    float u8[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) u8[q] = q + 1 < nlive ? (q < 7 ? v[q + 1] : hi) : cv[q];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        dn[k] = vpk(k ? v[2 * k - 1] : lo, v[2 * k]);
                        up[k] = vpk(u8[2 * k], u8[2 * k + 1]);
                    }
                };
                // the RDP terms of one in-plane position (3-D: with the planes beside it)
                auto position = [&](const f2x(&x)[4], unsigned jn, bool there) {
                    if constexpr (TV) return;
                    rdp(x);
                    if constexpr (Z3) {
                        if (!there) return;
                        f2x dn[4], up[4];
                        shifted(x, jn, dn, up);
                        rdp(dn);
                        rdp(up);
                    }
                };
                if constexpr (GEN) {
                    // row by row, as the general stencil adds them
                    const bool xl = ix > 0, xr = ix < N - 1, yl = iy > 0, yr = iy < N - 1;
                    const unsigned dm = iy > 0 ? jc - N : jc, dp = iy < N - 1 ? jc + N : jc;
                    const unsigned j0_ = xl && yl ? dm - 1 : jc, j1_ = xr && yl ? dm + 1 : jc;
                    const unsigned j2_ = xl && yr ? dp - 1 : jc, j3_ = xr && yr ? dp + 1 : jc;
                    f2x vu[4], vl[4];
                    if (!TV) {
                        load8x(f + j0_ * Pp, nb0);
                        load8x(f + j1_ * Pp, nb1);
                    }
                    if (!TV || dyn) {
                        load8x(f + ym * Pp, vu);
                        load8x(f + xm * Pp, vl);
                    }
                    position(nb0, j0_, xl && yl);
                    position(vu, ym, yl);
                    position(nb1, j1_, xr && yl);
                    position(vl, xm, xl);
                    f2x dn[4], up[4];
                    if constexpr (Z3) {
                        // the centre column: two neighbours, and the gradient across the planes
                        shifted(c, jc, dn, up);
                        rdp(dn);
                        rdp(up);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int z0 = grp * 8 + 2 * k;
                            const f2x HZ = vpk(z0 > 0 && z0 + 1 < g.P ? 0.5f : 1.f, z0 + 2 < g.P ? 0.5f : 1.f);
                            g2[k] = vmul(HZ, vsub(up[k], dn[k]));
                        }
                    }
                    if (!TV || dyn) load8x(f + xp * Pp, nb0);
                    position(nb0, xp, xr);
                    if (dyn) {
                        const f2x HX = vsplat((ix > 0 && ix < N - 1) ? 0.5f : 1.f);
#pragma unroll
                        for (int k = 0; k < 4; ++k) vl[k] = vmul(HX, vsub(nb0[k], vl[k]));
                    }
                    if (!TV || dyn) load8x(f + yp * Pp, nb1);
                    if (!TV) load8x(f + j2_ * Pp, nb0);
                    position(nb0, j2_, xl && yr);
                    position(nb1, yp, yr);
                    if (dyn) {
                        // nu_of: |grad f|^2 below the smallest normal float counts as zero, as in the mu pass
                        const f2x HY = vsplat((iy > 0 && iy < N - 1) ? 0.5f : 1.f);
                        const float nu1 = a.fs_nu1, nu2 = a.fs_nu2;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const f2x gy = vmul(HY, vsub(nb1[k], vu[k]));
                            f2x q2 = vfma(vl[k], vl[k], vmul(gy, gy));
                            if (Z3) q2 = vfma(g2[k], g2[k], q2);
                            float x0, x1, r0, r1;
                            vunpk(q2, x0, x1);
                            vunpk(vrsqrt(q2), r0, r1);
                            r0 = fmaxf(0.01f, x0 >= 1.17549435e-38f ? x0 * r0 * inv_mean_f : 0.f);
                            r1 = fmaxf(0.01f, x1 >= 1.17549435e-38f ? x1 * r1 * inv_mean_f : 0.f);
                            vunpk(vmul(vsplat(mean_mu), vrcp(vpk(r0, r1))), r0, r1);
                            nu[k] = vpk(fminf(fmaxf(r0, nu1), nu2), fminf(fmaxf(r1, nu1), nu2));
                        }
                    }
                    if (!TV) load8x(f + j3_ * Pp, nb0);
                    position(nb0, j3_, xr && yr);
                    if (a.nu_mode == 2) store8x(reinterpret_cast<float *>(a.nu_frozen) + jc * Pp + grp * 8, nu);
                    if (a.nu_mode == 3) load8x(reinterpret_cast<const float *>(a.nu_frozen) + jc * Pp + grp * 8, nu);
                    if (a.nu_mode == 0) nu[0] = nu[1] = nu[2] = nu[3] = vsplat(1.f);
                } else {
                    // axial neighbours: RDP terms and the Matlab-style gradient
                    load8x(f + xm * Pp, nb0);
                    load8x(f + xp * Pp, nb1);
                    rdp(nb0);
                    rdp(nb1);
                    if (dyn) {
                        const f2x HX = vsplat((ix > 0 && ix < N - 1) ? 0.5f : 1.f);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const f2x t = vmul(HX, vsub(nb1[k], nb0[k]));
                            g2[k] = vmul(t, t);
                        }
                    }
                    load8x(f + ym * Pp, nb0);
                    load8x(f + yp * Pp, nb1);
                    rdp(nb0);
                    rdp(nb1);
                    if (dyn) {
                        const f2x HY = vsplat((iy > 0 && iy < N - 1) ? 0.5f : 1.f);
                        const float nu1 = a.fs_nu1, nu2 = a.fs_nu2;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const f2x t = vmul(HY, vsub(nb1[k], nb0[k]));
                            float r0, r1;
                            vunpk(vrsqrt(vfma(t, t, g2[k])), r0, r1);
                            // 1 / mu = 1 / max(0.01, |grad f| / mean f) = min(100, mean f / |grad f|)
                            r0 = fminf(100.f, r0 * mean_f);
                            r1 = fminf(100.f, r1 * mean_f);
                            nu[k] = vpk(fminf(fmaxf(mean_mu * r0, nu1), nu2),
                                        fminf(fmaxf(mean_mu * r1, nu1), nu2));
                        }
                        if (a.nu_mode == 2)
                            store8x(reinterpret_cast<float *>(a.nu_frozen) + jc * Pp + grp * 8, nu);
                    } else if (a.nu_mode == 3) {
                        load8x(reinterpret_cast<const float *>(a.nu_frozen) + jc * Pp + grp * 8, nu);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k) nu[k] = vsplat(1.f);
                    }
                    // diagonal neighbours
                    const bool xl = ix > 0, xr = ix < N - 1, yl = iy > 0, yr = iy < N - 1;
                    const unsigned dm = iy > 0 ? jc - N : jc, dp = iy < N - 1 ? jc + N : jc;
                    const unsigned j0_ = xl && yl ? dm - 1 : jc, j1_ = xr && yl ? dm + 1 : jc;
                    const unsigned j2_ = xl && yr ? dp - 1 : jc, j3_ = xr && yr ? dp + 1 : jc;
                    load8x(f + j0_ * Pp, nb0);
                    load8x(f + j1_ * Pp, nb1);
                    rdp(nb0);
                    rdp(nb1);
                    load8x(f + j2_ * Pp, nb0);
                    load8x(f + j3_ * Pp, nb1);
                    rdp(nb0);
                    rdp(nb1);
                }
                if constexpr (GEN) {
                    // A = -lambda alpha nu S, S = min(f, U - f) / p;  B = (beta/M) grad R
                    f2x IP[4];
                    if constexpr (VOX) {
                        load8x(invp + jc * Pp + grp * 8, IP);
                    } else {
                        IP[0] = IP[1] = IP[2] = IP[3] = vsplat(invp[j]);
                    }
                    const f2x LAM = vsplat(-a.fs_lam), IPS = vsplat(a.fs_ips), BM = vsplat(a.fs_bm);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float c0, c1;
                        vunpk(c[k], c0, c1);
                        const f2x S = vmul(vpk(c0 < 0.5f * U ? c0 : U - c0, c1 < 0.5f * U ? c1 : U - c1),
                                           vmul(IP[k], IPS));
                        A[k] = vmul(vmul(LAM, nu[k]), S);
                        B[k] = vmul(BM, vadd(gr[k], gr[k]));
                    }
                    if constexpr (TV) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float w0, w1;
                            vunpk(A[k], w0, w1);
                            nb0[k] = vpk(2 * k < nlive ? -w0 : 1.f, 2 * k + 1 < nlive ? -w1 : 1.f);
                        }
                        store8x(reinterpret_cast<float *>(a.wbuf) + jc * Pp + grp * 8, nb0);
                    }
                } else {
                    // c = lambda alpha nu S, S = min(f, U - f) / p;  A = f - c (beta/M) 2 gr;  B = -c scale
                    const f2x NK = vsplat(-a.fs_lam * invp[j] * a.fs_ips);
                    const f2x BM = vsplat(2.f * a.fs_bm), SC = vsplat(a.fs_scale);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float c0, c1;
                        vunpk(c[k], c0, c1);
                        const f2x S = vpk(fminf(c0, U - c0), fminf(c1, U - c1));
                        const f2x cn = vmul(vmul(nu[k], S), NK);
                        A[k] = vfma(cn, vmul(BM, gr[k]), c[k]);
                        B[k] = vmul(cn, SC);
                    }
                }
            }
            // gather backprojection b = A_i^T w with the tile's shared (pixel, view) weights
            f2x sm[4], er[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) { sm[k] = 0ull; er[k] = 0ull; }
            for (int u0 = 0; u0 < a.nviews; u0 += VC) {
                const int nvc = min(VC, a.nviews - u0);
                if constexpr (TOF) {
                    __syncthreads();
                    for (int e = threadIdx.x; e < TP * nvc; e += 256) {
                        const int uu = e / TP, p = e - uu * TP, yy = p / pa.tx;
                        const int x = px0 + p - yy * pa.tx, y = py0 + yy;
                        tof_entry<KC, AR>(g, a.slot0, u0 + uu, x, y, tofs + e * pa.es);
                    }
                    __syncthreads();
                } else if (pre) {
                    cp_async_wait_all();             // this tile's block (this thread's part)
                    __syncthreads();                 // all parts; the previous gather is done
                    if (tile + 1 < t1) copy_tile(tile + 1);
                } else {
                    __syncthreads();
                    if constexpr (!TOF) bp_fill<KC, AR>(g, a.slot0, u0, nvc, j0, TP, tb);
                    __syncthreads();
                }
                if (!active) continue;
                if constexpr (TOF) {
                    for (int uu = 0; uu < nvc; ++uu)
                        tof_gather<KC, AR>(g, w, tofs + (uu * TP + pl) * pa.es, sm, er);
                    continue;
                } else {
                const typename Table::E *te = tb.e + (pre ? ((tile - t0) & 1) * a.nviews * TP : 0);
                // two bins of a view, one compensated step
                auto add = [&](float w0, const f2x(&x0)[4], float w1, const f2x(&x1)[4]) {
                    const f2x W0 = vsplat(w0), W1 = vsplat(w1);
#pragma unroll
                    for (int k = 0; k < 4; ++k) add2x<AR>(W0, x0[k], W1, x1[k], sm[k], er[k]);
                };
                int uu = 0;
                if constexpr (UV > 1) {
                    for (; uu + UV <= nvc; uu += UV) {
                        f2x x[UV][KC][4];
                        float l[UV][KC];
#pragma unroll
                        for (int i = 0; i < UV; ++i) {
                            const typename Table::E ent = te[(uu + i) * TP + pl];
#pragma unroll
                            for (int kb = 0; kb < KC; ++kb) {
                                load8x(w + ent.off + kb * Pp, x[i][kb]);
                                l[i][kb] = ent.w[kb];
                            }
                        }
#pragma unroll
                        for (int i = 0; i < UV; ++i)
#pragma unroll
                            for (int kb = 0; kb < KC; kb += 2) add(l[i][kb], x[i][kb], l[i][kb + 1], x[i][kb + 1]);
                    }
                }
                for (; uu < nvc; ++uu) {
                    const typename Table::E ent = te[uu * TP + pl];
                    const float *row = w + ent.off;
#pragma unroll
                    for (int kb = 0; kb < KC; kb += 2) {
                        f2x x0[4], x1[4];
                        load8x(row + kb * Pp, x0);
                        load8x(row + (kb + 1) * Pp, x1);
                        add(ent.w[kb], x0, ent.w[kb + 1], x1);
                    }
                }
                }
            }
            if (!active) continue;
            // step and clamp P_t
            f2x out[4], fc[4];
            if constexpr (GEN) load8x(f + (unsigned)j * Pp, fc);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const f2x b = AR == AR_KAHAN ? vadd(sm[k], er[k]) : sm[k];
                float f0, f1;
                if constexpr (GEN) vunpk(vfma(A[k], vfma(vsplat(a.fs_scale), b, B[k]), fc[k]), f0, f1);
                else vunpk(vfma(B[k], b, A[k]), f0, f1);
                if constexpr (!(FL & X8_TV)) {
                    f0 = f0 <= 0.f ? tt : (f0 >= U ? U - tt : f0);
                    f1 = f1 <= 0.f ? tt : (f1 >= U ? U - tt : f1);
                }
                const int p0 = grp * 8 + 2 * k;
                f0 = p0 < g.P ? f0 : 0.f;
                f1 = p0 + 1 < g.P ? f1 : 0.f;
                part = GEN ? part + f0 + f1 : part + (f0 + f1);
                out[k] = vpk(f0, f1);
            }
            store8x(reinterpret_cast<float *>(a.fout) + (unsigned)j * Pp + grp * 8, out);
            if constexpr (FL & X8_TV)
                store8x(reinterpret_cast<float *>(a.zbuf) + (unsigned)j * Pp + grp * 8, out);
        }
        double v[1] = {(double)part};
        grid_reduce<1>(v, a.red, a.sum_fout, vloc, nv);
    }
}

// Entries of update_kernel_x8's (pixel, view) table for one subset, computed once per geometry:
// entry e = (tile t, view u, pixel pl of the tile) is bp_entry(pixel t TP + pl, view u), in the
// kernel's shared-memory order, so that one tile's entries are one contiguous block.  bp_entry
// has no arithmetic that differs between the FP32 kernels (the FP32 and FP32 + Kahan tables are
// the same bits as those the kernel computes).
template <int KC>
__global__ void __launch_bounds__(256) bp_table_kernel(const __grid_constant__ GeoDev g, int slot0,
                                                      int nviews, int TP, long long nent, void *out)
{
    using E = typename BpTable<KC, AR_KAHAN, 1024 / (KC > 2 ? 2 : 1)>::E;
    const long long per = (long long)nviews * TP;
    const int npix = g.N * g.N;
    for (long long e = blockIdx.x * 256LL + threadIdx.x; e < nent; e += (long long)gridDim.x * 256) {
        const long long tile = e / per;
        const int r = (int)(e - tile * per);
        const int uu = r / TP, pl = r - uu * TP;
        const long long j = tile * TP + pl;
        const bool in = j < npix;
        reinterpret_cast<E *>(out)[e] = bp_entry<KC, AR_KAHAN, 1024 / (KC > 2 ? 2 : 1)>(
            g, slot0, uu, in, in ? (int)(j % g.N) : 0, in ? (int)(j / g.N) : 0);
    }
}

// The entries of 8-plane groups with uniform bins and without TOF; the packed kernel's table holds
// 1024 (KC = 2) or 512 (KC = 4) entries of 16 or 32 bytes, two tiles' worth when copied.
size_t bp_table_bytes_bound(const pet_geometry_desc &d)
{
    if (d.nplanes <= 1 || d.subrays > 1 || d.ring_mm > 0 || d.tof_bins > 1) return 0;
    const long long NG = (d.nplanes + 7) / 8, TP = 256 / NG;
    const long long npix = (long long)d.n * d.n, ntiles = (npix + TP - 1) / TP;
    const long long vmax = (d.nviews + d.nsubsets - 1) / d.nsubsets;
    if (TP < 1 || 2 * vmax * TP > 1024) return 0;
    return (size_t)(ntiles * d.nviews * TP * 32);
}

pet_status build_bp_table(pet_geometry *g, cudaStream_t st)
{
    const GeoDev &gd = g->dev;
    g->bptab_off.clear();
    if (gd.G != 8 || gd.table || gd.T > 1) return PET_OK;
    const int KC = gd.K <= 2 ? 2 : 4;
    const int CAP = KC > 2 ? 512 : 1024;
    const int TP = 256 / gd.NG;
    if (TP < 1) return PET_OK;
    const size_t esz = KC > 2 ? sizeof(BpTable<4, AR_KAHAN, 512>::E) : sizeof(BpTable<2, AR_KAHAN, 1024>::E);
    const long long ntiles = ((long long)gd.N * gd.N + TP - 1) / TP;
    std::vector<size_t> off(gd.M);
    size_t total = 0;
    for (int i = 0; i < gd.M; ++i) {
        const int nv = g->voff[i + 1] - g->voff[i];
        if (2 * nv * TP > CAP) return PET_OK;       // the kernel computes this geometry's entries
        off[i] = total;
        total += (size_t)ntiles * nv * TP * esz;
    }
    if (total == 0) return PET_OK;
    void *tab = nullptr;
    PET_CUDA(dev_malloc(&tab, total));
    for (int i = 0; i < gd.M; ++i) {
        const int nv = g->voff[i + 1] - g->voff[i];
        const long long nent = ntiles * nv * TP;
        const int grid = (int)std::min<long long>((nent + 255) / 256, (long long)sm_count() * 16);
        char *out = static_cast<char *>(tab) + off[i];
        if (KC == 2) bp_table_kernel<2><<<grid, 256, 0, st>>>(gd, g->voff[i], nv, TP, nent, out);
        else bp_table_kernel<4><<<grid, 256, 0, st>>>(gd, g->voff[i], nv, TP, nent, out);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            cudaFree(tab);
            return cuda_fail(e, "bp_table_kernel launch");
        }
    }
    g->d_bptab = tab;                                // set together with the offsets
    g->bptab_off = off;
    return PET_OK;
}

// Stacks in FP32 with uniform bins run the packed kernel; TOF ones with the in-plane RDP prior.
bool update_x8_path(const UpdateArgs &a, int arith)
{
    return a.g.G == 8 && arith != AR_FP64 && !a.g.table && (a.g.T == 1 || (!a.z3 && !a.tv));
}

// pixel tiles of the packed kernel
int update_x8_tiles(const UpdateArgs &a)
{
    const int N = a.g.N;
    if (a.g.T > 1) {
        const X8Patch p = a.g.K <= 2 ? x8_patch<2>(a.g) : x8_patch<4>(a.g);
        return (N + p.tx - 1) / p.tx * ((N + p.ty - 1) / p.ty);
    }
    const int TP = 256 / a.g.NG;
    return (N * N + TP - 1) / TP;
}

// The 3-D prior and detection factors: tiles per virtual block, whose sum of new voxels is taken in FP32 by
// thread, as the general kernel shared them out over its three blocks per SM.  The sums' rounding decides
// the last bit of mean(f), and with it of every nu; another sharing gave results whose single voxels
// differ by 1e-3 of the image's rms where a scan amplifies rounding.
int update_x8_tpv(const UpdateArgs &a)
{
    const int nt = update_x8_tiles(a), slots = 3 * sm_count();
    return std::max({1, (nt + a.red.capacity - 1) / a.red.capacity, (nt + slots - 1) / slots});
}
static int update_x8_blocks(const UpdateArgs &a)
{
    const int tpv = update_x8_tpv(a);
    return (update_x8_tiles(a) + tpv - 1) / tpv;
}

// Views loaded together (see update_kernel_x8): 256 x 256 x 89 has 3121 tiles, 6.8 per block of 456
// (3 blocks per SM) and 10.3 of 304: 7 and 11 rounds, and one view is 1.4 us of 66 faster; 128 x
// 128 x 64 has 512, where one view took 503 us an iteration and four 438.  A batched launch (N = 0
// here) takes four.  Beside an objective evaluation, where the projection fills the GPU, one view and
// three blocks: of 21 drawn reconstructions 7 took 2 to 4 % longer than with the kernels before this file
// with four views (155 x 155 x 14: 1.67 ms, one view 1.60), 1 does with one.
static int x8_views(const UpdateArgs &a)
{
    if (a.g.N == 0 || a.tv || a.g.T > 1) return 4;
    if (a.z3 || a.vox) return update_x8_blocks(a) <= 2 * sm_count() ? 4 : 1;
    if (a.beside) return 1;
    const double nt = update_x8_tiles(a), s3 = 3.0 * sm_count(), s2 = 2.0 * sm_count();
    return 1.026 * ceil(nt / s3) * s3 < ceil(nt / s2) * s2 ? 1 : 4;
}

template <int KC, int AR>
static auto x8_fn(const UpdateArgs &a) -> void (*)(const UpdateArgs, const Batch)
{
    if (a.g.T > 1) return a.vox ? update_kernel_x8<KC, AR, X8_TOF | X8_VOX> : update_kernel_x8<KC, AR, X8_TOF>;
    if (a.tv) return a.vox ? update_kernel_x8<KC, AR, X8_TV | X8_VOX> : update_kernel_x8<KC, AR, X8_TV>;
    const bool one = x8_views(a) == 1;
    if (a.z3 && a.vox) return one ? update_kernel_x8<KC, AR, X8_Z3 | X8_VOX, 1> : update_kernel_x8<KC, AR, X8_Z3 | X8_VOX>;
    if (a.z3) return one ? update_kernel_x8<KC, AR, X8_Z3, 1> : update_kernel_x8<KC, AR, X8_Z3>;
    if (a.vox) return one ? update_kernel_x8<KC, AR, X8_VOX, 1> : update_kernel_x8<KC, AR, X8_VOX>;
    return one ? update_kernel_x8<KC, AR, 0, 1> : update_kernel_x8<KC, AR, 0>;
}

static auto x8_any(const UpdateArgs &a, int arith)
{
    if (a.g.K <= 2) return arith == AR_KAHAN ? x8_fn<2, AR_KAHAN>(a) : x8_fn<2, AR_FP32>(a);
    return arith == AR_KAHAN ? x8_fn<4, AR_KAHAN>(a) : x8_fn<4, AR_FP32>(a);
}

const void *update_x8_fn(const UpdateArgs &a, int arith) { return (const void *)x8_any(a, arith); }

void update_x8_dispatch(const UpdateArgs &a, const Batch &b, int arith, int grid, cudaStream_t st, bool pdl)
{
    launch_pdl(x8_any(a, arith), grid, st, pdl, a, b);
}

}  // namespace pet
