// Image-space device helpers shared by the update, mu and image kernels: the 3x3 (or 3x3x3)
// stencil of the RDP and of the Matlab-style gradient, and the smoothness map nu.
#pragma once

#include "kernels.cuh"

namespace pet {

// 1 / x (x > 0) by Newton's iteration r <- r + r (1 - x r) from the FP32 reciprocal, whose relative
// error of 2^-22 it squares twice: 6 FP64-pipe operations where a division takes about ten.  Values
// whose FP32 reciprocal is not a normal number are divided.
__device__ __forceinline__ double reciprocal(double x)
{
    if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
    double r = (double)__frcp_rn((float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// Loads the 3x3 in-plane neighbourhood of pixel (ix, iy) for one plane group.
//   RG: gr_p = 2 sum_k (f_j - f_k)(gamma_R |f_j - f_k| + f_j + 3 f_k + 2 eps) / den^2
//       (den = f_j + f_k + gamma_R |f_j - f_k| + eps; FP32 kernels use the fast reciprocal)
//   MU: gx_p, gy_p of the Matlab-style gradient: central differences inside, one-sided at
//       the edges (the missing side counts as the centre value)
//   RV: rv_p = sum_k (f_j - f_k)^2 / den
// z3: the neighbourhood is the 26 voxels around (ix, iy, plane) in the volume (neighbours
// outside it are absent), and MU also gives gz_p, the gradient across the planes (central
// inside, one-sided at the first and last plane, 0 for one plane).  Each position's plane group
// is loaded with the planes just below and above it.
template <int G, int AR, bool RG, bool MU, bool RV>
__device__ __forceinline__ void stencil(const GeoDev &g, const typename ArithT<AR>::T *f, int grp,
                                        int ix, int iy, typename ArithT<AR>::T gamma_r,
                                        typename ArithT<AR>::T eps,
                                        typename ArithT<AR>::T (&fc)[G],
                                        typename ArithT<AR>::T (&gr)[G],
                                        typename ArithT<AR>::T (&gx)[G],
                                        typename ArithT<AR>::T (&gy)[G],
                                        typename ArithT<AR>::T (&rv)[G],
                                        bool z3 = false, typename ArithT<AR>::T *gz = nullptr)
{
    using T = typename ArithT<AR>::T;
    const int N = g.N, Pp = g.Pp;
    const T *base = f + grp * G;
    const unsigned jc = (unsigned)iy * (unsigned)N + (unsigned)ix;   // images hold < 2^32 elements
    load_group<G, T>(base + jc * (unsigned)Pp, fc);
    const T hx = (ix > 0 && ix < N - 1) ? T(0.5) : T(1);
    const T hy = (iy > 0 && iy < N - 1) ? T(0.5) : T(1);
#pragma unroll
    for (int p = 0; p < G; ++p) { gr[p] = T(0); gx[p] = T(0); gy[p] = T(0); rv[p] = T(0); }
    if constexpr (MU) {
        // a missing neighbour on one side is replaced by the centre value
        const T sx = (ix == 0 ? -hx : T(0)) + (ix == N - 1 ? hx : T(0));
        const T sy = (iy == 0 ? -hy : T(0)) + (iy == N - 1 ? hy : T(0));
#pragma unroll
        for (int p = 0; p < G; ++p) { gx[p] = sx * fc[p]; gy[p] = sy * fc[p]; }
    }
    // one (centre, neighbour) pair of Eq. RDP / Eq. gradRD; FP64: the numerator
    // gamma_R |d| + c + 3 k + 2 eps as den + 2 k + eps, over den^2 by the reciprocal of den
    auto pair = [&](int p, T c, T k) {
        const T d = c - k;
        const T ad = d < T(0) ? -d : d;
        const T den = c + k + gamma_r * ad + eps;
        if constexpr (RG) {
            if constexpr (AR == AR_FP64) {
                const double r = reciprocal(den);
                gr[p] = fma(d * r, (den + fma(2.0, k, eps)) * r, gr[p]);
            } else {
                gr[p] += __fdividef(d * (gamma_r * ad + c + T(3) * k + T(2) * eps), den * den);
            }
        }
        if constexpr (RV) {
            if constexpr (AR == AR_FP64) rv[p] += d * d / den;
            else rv[p] += __fdividef(d * d, den);
        }
    };
    const int z0 = grp * G;                  // plane of element 0 of the group
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int dx = q % 3 - 1, dy = q / 3 - 1;
        if (q == 4 && !z3) continue;
        if (!RG && !RV && dx != 0 && dy != 0) continue;    // gradient only: axial neighbours
        const int x = ix + dx, y = iy + dy;
        if (x < 0 || y < 0 || x >= N || y >= N) continue;
        const unsigned jn = (unsigned)((int)jc + dy * N + dx) * (unsigned)Pp;
        T fk[G];
        if (q == 4) {
#pragma unroll
            for (int p = 0; p < G; ++p) fk[p] = fc[p];
        } else {
            load_group<G, T>(base + jn, fk);
        }
        if (z3) {
            // the planes just below and above this position's group
            const T lo = z0 > 0 ? f[jn + z0 - 1] : T(0);
            const T hi = z0 + G < g.P ? f[jn + z0 + G] : T(0);
#pragma unroll
            for (int p = 0; p < G; ++p) {
                const int z = z0 + p;
                if (z >= g.P) continue;
                if (RG || RV) {
                    if (q != 4) pair(p, fc[p], fk[p]);
                    if (z > 0) pair(p, fc[p], p > 0 ? fk[p - 1] : lo);
                    if (z + 1 < g.P) pair(p, fc[p], p + 1 < G ? fk[p + 1] : hi);
                }
                if constexpr (MU) {
                    if (q == 4 && gz) {
                        const T dn = z > 0 ? (p > 0 ? fk[p - 1] : lo) : fc[p];
                        const T up = z + 1 < g.P ? (p + 1 < G ? fk[p + 1] : hi) : fc[p];
                        gz[p] = (z > 0 && z + 1 < g.P ? T(0.5) : T(1)) * (up - dn);
                    }
                }
            }
        } else if constexpr (RG && AR != AR_FP64 && G % 2 == 0) {
            // packed FP32x2: two planes per instruction; 1/den^2 from the fast reciprocal
            const float2 GR = make_float2(gamma_r, gamma_r), THREE = make_float2(3.f, 3.f);
#pragma unroll
            for (int p = 0; p < G; p += 2) {
                const float2 c2 = make_float2(fc[p], fc[p + 1]), k2 = make_float2(fk[p], fk[p + 1]);
                const float2 d = sub2(c2, k2);
                const float2 ad = make_float2(fabsf(d.x), fabsf(d.y));
                const float2 den = fma2(GR, ad, add2(add2(c2, k2), make_float2(eps, eps)));
                const float2 t = fma2(GR, ad, fma2(THREE, k2, add2(c2, make_float2(2.f * eps, 2.f * eps))));
                const float2 num = mul2(d, t);
                const float2 den2 = mul2(den, den);
                const float2 qq = make_float2(__fdividef(num.x, den2.x), __fdividef(num.y, den2.y));
                gr[p] += qq.x;
                gr[p + 1] += qq.y;
            }
        } else if constexpr (RG || RV) {
#pragma unroll
            for (int p = 0; p < G; ++p) pair(p, fc[p], fk[p]);
        }
        if constexpr (MU) {
            if (q == 4) continue;
            if (dy == 0) {
                const T sgn = dx < 0 ? -hx : hx;
#pragma unroll
                for (int p = 0; p < G; ++p) gx[p] += sgn * fk[p];
            } else if (dx == 0) {
                const T sgn = dy < 0 ? -hy : hy;
#pragma unroll
                for (int p = 0; p < G; ++p) gy[p] += sgn * fk[p];
            }
        }
    }
    if constexpr (RG) {
#pragma unroll
        for (int p = 0; p < G; ++p) gr[p] *= T(2);
    }
}

template <typename T>
__device__ __forceinline__ T clampT(T v, T lo, T hi) { return v < lo ? lo : (v > hi ? hi : v); }

template <typename T>
__device__ __forceinline__ T fast_div(T a, T b)
{
    if constexpr (sizeof(T) == 8) return a / b;
    else return __fdividef(a, b);
}

// |(gx, gy)|: FP32 kernels use x rsqrt(x) (two instructions, a few ulp)
template <typename T>
__device__ __forceinline__ T grad_norm(T gx, T gy)
{
    const T x = gx * gx + gy * gy;
    if constexpr (sizeof(T) == 8) return sqrt(x);
    else return x > 0.f ? x * rsqrtf(x) : 0.f;
}

// |(gx, gy, gz)|
template <typename T>
__device__ __forceinline__ T grad_norm3(T gx, T gy, T gz)
{
    const T x = gx * gx + gy * gy + gz * gz;
    if constexpr (sizeof(T) == 8) return sqrt(x);
    else return x > 0.f ? x * rsqrtf(x) : 0.f;
}

// mu = max(0.01, |grad f| / mean(f)); nu = P_{nu1}^{nu2}(mean(mu) / mu)
template <typename T>
__device__ __forceinline__ T nu_of(T gx, T gy, T gz, T inv_mean_f, T mean_mu, T nu1, T nu2)
{
    T mu = grad_norm3(gx, gy, gz) * inv_mean_f;
    mu = mu < T(0.01) ? T(0.01) : mu;
    return clampT<T>(fast_div(mean_mu, mu), nu1, nu2);
}

// FP32 mu pass for 8-plane groups: sum over voxels of mu = max(0.01, |grad f| / mean(f))
// (Matlab-style gradient: central differences inside, one-sided at the border, where the
// missing neighbour is the centre value).  Thread layout of the update kernel (pixel x plane
// group, TP = 256 / NG pixels per tile); a virtual block takes a.ipt tiles.
__device__ __forceinline__ void mu_x8_vblock(const ImageArgs &a, int vloc, int nv)
{
    const GeoDev &g = a.g;
    const int N = g.N, NG = g.NG, npix = N * N;
    const unsigned Pp = (unsigned)g.Pp;
    const int TP = 256 / NG;
    const int pl = threadIdx.x / NG, grp = threadIdx.x % NG;
    const int ntiles = (npix + TP - 1) / TP;
    const float inv_mean_f = (float)((double)npix * g.P) / (float)*a.sum_f;
    const float *f = reinterpret_cast<const float *>(a.f) + grp * 8;
    const int nvalid = min(8, g.P - grp * 8);             // real planes of this group
    float part = 0.f;
    for (int tile = vloc * a.ipt; tile < min(ntiles, (vloc + 1) * a.ipt); ++tile) {
        const int j = tile * TP + pl;
        if (pl >= TP || j >= npix) continue;
        const int ix = j % N, iy = j / N;
        const unsigned jc = (unsigned)j;
        f2x w_[4], e_[4], n_[4], s_[4];
        load8x(f + (ix > 0 ? jc - 1 : jc) * Pp, w_);
        load8x(f + (ix < N - 1 ? jc + 1 : jc) * Pp, e_);
        load8x(f + (iy > 0 ? jc - N : jc) * Pp, n_);
        load8x(f + (iy < N - 1 ? jc + N : jc) * Pp, s_);
        const f2x HX = vsplat((ix > 0 && ix < N - 1) ? 0.5f : 1.f);
        const f2x HY = vsplat((iy > 0 && iy < N - 1) ? 0.5f : 1.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const f2x gx = vmul(HX, vsub(e_[k], w_[k])), gy = vmul(HY, vsub(s_[k], n_[k]));
            const f2x x2 = vfma(gx, gx, vmul(gy, gy));
            float x0, x1, r0, r1;
            vunpk(x2, x0, x1);
            vunpk(vrsqrt(x2), r0, r1);
            // |grad f|^2 below the smallest normal float (|grad f| < 1.1e-19, met on decayed
            // backgrounds) counts as zero: mu = 0.01 there, and the flushed rsqrt would be inf
            const float m0 = fmaxf(0.01f, x0 >= 1.17549435e-38f ? x0 * r0 * inv_mean_f : 0.f);
            const float m1 = fmaxf(0.01f, x1 >= 1.17549435e-38f ? x1 * r1 * inv_mean_f : 0.f);
            part += (2 * k < nvalid ? m0 : 0.f) + (2 * k + 1 < nvalid ? m1 : 0.f);
        }
    }
    double v[1] = {(double)part};
    grid_reduce<1>(v, a.red, a.result, vloc, nv);
}

// sum of mu for single-plane FP32 images: 256 a.ipt pixels of a virtual block
__device__ __forceinline__ void mu_p1_vblock(const ImageArgs &a, int vloc, int nv)
{
    const GeoDev &g = a.g;
    const int N = g.N, npix = N * N;
    const float *f = reinterpret_cast<const float *>(a.f);
    const float inv_mean_f = (float)npix / (float)*a.sum_f;
    float part = 0.f;
    for (int k = 0; k < a.ipt; ++k) {
        const int j = (vloc * a.ipt + k) * 256 + (int)threadIdx.x;
        if (j >= npix) break;
        const int ix = j % N, iy = j / N;
        float fc[1], gr[1], gx[1], gy[1], rv[1];
        stencil<1, AR_FP32, false, true, false>(g, f, 0, ix, iy, 0.f, 0.f, fc, gr, gx, gy, rv);
        part += fmaxf(0.01f, grad_norm3(gx[0], gy[0], 0.f) * inv_mean_f);
    }
    double v[1] = {(double)part};
    grid_reduce<1>(v, a.red, a.result, vloc, nv);
}

}  // namespace pet
