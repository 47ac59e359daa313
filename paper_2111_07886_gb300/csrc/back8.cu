// FP32 stand-alone backprojection of large stacks with uniform bins (no TOF), two by two pixels per thread.
//
// A thread that gathers one pixel reads KC = 2 rows per view and group.  The lines of one view that
// meet a 2 x 2 block of pixels are at most KQ = 3 neighbouring bins (4 for bins below 0.94
// pixels), so a thread that holds the four pixels' sums reads 3 rows where four threads read 8.
// The kernel waits for those reads' latency, not for their bytes: 2.67 times fewer take 589 us instead
// of 634 (all 288 views of a 256 x 256 x 89 stack).
// Its (block, view) entries hold the rows' offset and the KQ x 4 lengths, as pairs (w, w) for the
// f32x2 FMAs, in shared memory; tiles are about square, so that a view's rows are shared in both
// directions.  Sums: a view is added by FMAs onto the compensation term, and every fourth view one
// compensated step moves it into the sum (no registers beyond those of a plain compensated sum; a step
// per view takes 675 us).  What that rounds is less than what one rounding of scale (s + e) saves:
// 4.9e-8 from the 64-bit result, 5.7e-8 with a step per view and a rounded sum scaled.
#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

int sm_count();

template <int KQ> struct __align__(16) QuadEntry {
    f2x w[KQ * 4];             // [bin][pixel], pixel = 2 dy + dx
    unsigned off, pad[3];
};
constexpr int QUAD_BYTES = 32 * 1024;
template <int KQ> __host__ __device__ constexpr int quad_cap() { return QUAD_BYTES / (int)sizeof(QuadEntry<KQ>); }

// a tile's 2 x 2 blocks, about square
__host__ __device__ __forceinline__ void quad_tile(int NG, int cap, int &tx, int &ty)
{
    const int TP = 256 / NG < cap ? 256 / NG : cap;
    ty = 1;
    while ((ty + 1) * (ty + 1) <= TP) ++ty;
    tx = TP / ty;
}

// One entry: pixels (x, y), (x + 1, y), (x, y + 1), (x + 1, y + 1) against view u of the subset.
template <int KQ>
__device__ __forceinline__ void quad_entry(const GeoDev &g, int slot0, int u, int x, int y, QuadEntry<KQ> &e)
{
    int b0[4], first = 0x7fffffff;
    float wk[4][2];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int px = x + (p & 1), py = y + (p >> 1);
        b0[p] = 0;
        wk[p][0] = wk[p][1] = 0.f;
        if (px < g.N && py < g.N) {
            bp_weights<2, AR_KAHAN>(g, g.views[slot0 + u], slot0 + u, px, py, b0[p], wk[p]);
            first = min(first, b0[p]);
        }
    }
    const int bc = min(max(first, 0), g.NB - KQ);      // all KQ rows of the entry exist
    e.off = ((unsigned)u * (unsigned)g.NB + (unsigned)bc) * (unsigned)g.Pp;
#pragma unroll
    for (int k = 0; k < KQ; ++k)
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const int s = bc + k - b0[p];
            e.w[k * 4 + p] = vsplat(s == 0 ? wk[p][0] : (s == 1 ? wk[p][1] : 0.f));
        }
}

template <int KQ, int AR>
__global__ void __launch_bounds__(256, 2) back_quad_kernel(const __grid_constant__ BackArgs a)
{
    using E = QuadEntry<KQ>;
    constexpr int CAP = quad_cap<KQ>();
    __shared__ E tb[CAP];
    const GeoDev &g = a.g;
    const int N = g.N, NG = g.NG;
    int tx, ty;
    quad_tile(NG, CAP, tx, ty);
    const int nq = tx * ty;                                           // blocks of a tile
    const int ntx = (N + 2 * tx - 1) / (2 * tx), ntiles = ntx * ((N + 2 * ty - 1) / (2 * ty));
    const int q = threadIdx.x / NG, grp = threadIdx.x - q * NG, qy = q / tx, qx = q - qy * tx;
    const int VC = min(a.nviews, CAP / nq);
    const unsigned Pp = (unsigned)g.Pp;
    const float *proj = reinterpret_cast<const float *>(a.proj) + grp * 8;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (tile % ntx) * 2 * tx, y0 = (tile / ntx) * 2 * ty;
        const int x = x0 + 2 * qx, y = y0 + 2 * qy;
        const bool active = q < nq && x < N && y < N;
        f2x sm[4][4], er[4][4];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int k = 0; k < 4; ++k) sm[p][k] = er[p][k] = 0ull;
        auto merge = [&]() {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (AR == AR_KAHAN) {
                        const f2x t = vadd(sm[p][k], er[p][k]);
                        er[p][k] = vsub(er[p][k], vsub(t, sm[p][k]));
                        sm[p][k] = t;
                    }
                }
        };
        for (int u0 = 0; u0 < a.nviews; u0 += VC) {
            const int nvc = min(VC, a.nviews - u0);
            __syncthreads();
            for (int i = threadIdx.x; i < nq * nvc; i += 256) {
                const int uu = i / nq, b = i - uu * nq, by = b / tx;
                quad_entry<KQ>(g, a.slot0, u0 + uu, x0 + 2 * (b - by * tx), y0 + 2 * by, tb[i]);
            }
            __syncthreads();
            if (!active) continue;
            for (int uu = 0; uu < nvc; ++uu) {
                const E &e = tb[uu * nq + q];
                const float *row = proj + e.off;
#pragma unroll
                for (int b = 0; b < KQ; ++b) {
                    f2x v[4];
                    load8x(row + b * Pp, v);
                    const ulonglong2 w01 = reinterpret_cast<const ulonglong2 *>(e.w)[2 * b];
                    const ulonglong2 w23 = reinterpret_cast<const ulonglong2 *>(e.w)[2 * b + 1];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        er[0][k] = vfma(w01.x, v[k], er[0][k]);
                        er[1][k] = vfma(w01.y, v[k], er[1][k]);
                        er[2][k] = vfma(w23.x, v[k], er[2][k]);
                        er[3][k] = vfma(w23.y, v[k], er[3][k]);
                    }
                }
                if ((uu & 3) == 3) merge();
            }
            merge();
        }
        if (!active) continue;
        const f2x scale = vsplat((float)g.scale);       // scale (s + e), rounded once
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const int px = x + (p & 1), py = y + (p >> 1);
            if (px >= N || py >= N) continue;
            float o[8];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                vunpk(vfma(scale, sm[p][k], vmul(scale, er[p][k])), o[2 * k], o[2 * k + 1]);
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = grp * 8 + c < g.P ? o[c] : 0.f;
            store_group<8, float>(reinterpret_cast<float *>(a.img) + ((unsigned)(py * N + px) * Pp + grp * 8), o);
        }
    }
}

// Stacks in FP32 whose 2 x 2 pixel blocks meet at most four bins of a view, with at least five plane groups
// to share a tile's entries and tiles that fill the rounds of two blocks per SM to 5/6; the others run the
// general kernel.  All of 45 drawn sizes on this side are faster than there (1.04 to 1.39 times).  Few groups
// leave large tiles, few of them and their entries to few threads: 100 x 100 x 2 (180 views) takes 461 us here
// and 169 there, 256 x 256 x 17 255 and 241; 200 x 200 x 64, whose 340 tiles are 1.1 rounds, 279 and 202;
// 128 x 128 x 128 (0.84 of a round) 146 and 173.
bool back_quad_path(const BackArgs &a, int arith)
{
    if (!a.proj || a.g.G != 8 || arith == AR_FP64 || a.g.table || a.g.T > 1 || a.g.K > 2 || a.g.KQ > 4 || a.g.NG < 5)
        return false;
    int tx, ty;
    quad_tile(a.g.NG, a.g.KQ <= 3 ? quad_cap<3>() : quad_cap<4>(), tx, ty);
    const long long nt = (long long)((a.g.N + 2 * tx - 1) / (2 * tx)) * ((a.g.N + 2 * ty - 1) / (2 * ty));
    const long long slots = 2LL * sm_count(), rounds = (nt + slots - 1) / slots;
    return 6 * nt >= 5 * rounds * slots;
}

void back_quad_dispatch(const BackArgs &a, int arith, cudaStream_t st)
{
    const int grid = sm_count() * 2;
    if (a.g.KQ <= 3) {
        if (arith == AR_KAHAN) back_quad_kernel<3, AR_KAHAN><<<grid, 256, 0, st>>>(a);
        else back_quad_kernel<3, AR_FP32><<<grid, 256, 0, st>>>(a);
    } else {
        if (arith == AR_KAHAN) back_quad_kernel<4, AR_KAHAN><<<grid, 256, 0, st>>>(a);
        else back_quad_kernel<4, AR_FP32><<<grid, 256, 0, st>>>(a);
    }
}

}  // namespace pet
