// Layout conversions between the C-ABI layouts (plane outermost) and the internal ones
// (planes innermost, padded to the plane group; sinogram views sorted by subset), and the
// input check of the data (counts >= 0, gamma > 0 and finite: Eq. model-Poisson needs
// gamma in R_{++}^p).
#include "kernels.cuh"
#include "profile.cuh"

namespace pet {

// Plane-outermost <-> planes-innermost copies, through a shared tile of 64 positions x up to 32
// planes so that both sides are accessed in runs (element by element, one side touched a 32-byte
// sector per 4-byte value: 29 us for a 256 x 256 x 89 image and 53 us for its sinogram).
// A position j is a pixel, or a sinogram's (row u, entry b); Map::at(j) is its offset within one
// plane of the plane-outermost array.
struct ImageMap {
    __device__ __forceinline__ long long at(long long j) const { return j; }
};
struct SinoMap {               // rows u of NB entries, row u being row v(u) of the outer array
    const int *view_of_slot;   // NULL: v(u) = u
    int slot0, NB;
    __device__ __forceinline__ long long at(long long j) const
    {
        const int u = (int)((unsigned)j / (unsigned)NB), b = (int)(j - (long long)u * NB);   // j < 2^32
        return (long long)(view_of_slot ? __ldg(view_of_slot + slot0 + u) : u) * NB + b;
    }
};
static inline unsigned blocks(long long n) { return (unsigned)((n + 255) / 256); }

constexpr int TR_J = 64, TR_P = 32;

// src [P][plane] -> dst [n][Pp]; pad planes get `pad`
template <typename S, typename D, class Map>
__global__ void __launch_bounds__(256) planes_inward(const S *__restrict__ src, D *__restrict__ dst, const Map m,
                                                     long long n, long long plane, int P, int Pp, D pad)
{
    __shared__ D t[TR_P][TR_J + 1];
    const long long j0 = (long long)blockIdx.x * TR_J;
    const int p0 = (int)blockIdx.y * TR_P, pw = min(TR_P, Pp - p0), jx = threadIdx.x % TR_J;
    if (j0 + jx < n) {
        const S *col = src + m.at(j0 + jx);
        for (int r = threadIdx.x / TR_J; r < pw; r += 256 / TR_J)
            t[r][jx] = p0 + r < P ? (D)col[(long long)(p0 + r) * plane] : pad;
    }
    __syncthreads();
    const int live = (int)min((long long)TR_J, n - j0) * pw;
    for (int i = threadIdx.x; i < live; i += 256) {
        const int j = i / pw, r = i - j * pw;
        dst[(j0 + j) * Pp + p0 + r] = t[r][j];
    }
}

// src [n][Pp] -> dst [P][plane]
template <typename S, typename D, class Map>
__global__ void __launch_bounds__(256) planes_outward(const S *__restrict__ src, D *__restrict__ dst, const Map m,
                                                      long long n, long long plane, int P, int Pp)
{
    __shared__ D t[TR_P][TR_J + 1];
    const long long j0 = (long long)blockIdx.x * TR_J;
    const int p0 = (int)blockIdx.y * TR_P, pw = min(TR_P, P - p0), jx = threadIdx.x % TR_J;
    const int live = (int)min((long long)TR_J, n - j0) * pw;
    for (int i = threadIdx.x; i < live; i += 256) {
        const int j = i / pw, r = i - j * pw;
        t[r][j] = (D)src[(j0 + j) * Pp + p0 + r];
    }
    __syncthreads();
    if (j0 + jx >= n) return;
    D *col = dst + m.at(j0 + jx);
    for (int r = threadIdx.x / TR_J; r < pw; r += 256 / TR_J) col[(long long)(p0 + r) * plane] = t[r][jx];
}

// One plane group (Pp = 8): a position is one 32-byte sector of the inner array, so plain copies touch
// nothing twice, and the tiles would be a few planes high (100 positions x planes per block of 256).
template <typename S, typename D, class Map, bool IN>
__global__ void __launch_bounds__(256) group_copy(const S *__restrict__ src, D *__restrict__ dst, const Map m,
                                                  long long n, long long plane, int P, D pad)
{
    const unsigned t = blockIdx.x * 256u + threadIdx.x;      // n Pp < 2^32 (geometry limits)
    if (IN) {                                                // [P][plane] -> [n][8]
        const unsigned j = t / 8u, p = t & 7u;
        if (j >= n) return;
        dst[t] = (int)p < P ? (D)src[(long long)p * plane + m.at(j)] : pad;
    } else {                                                 // [n][8] -> [P][plane]
        const unsigned p = t / (unsigned)n, j = t - p * (unsigned)n;
        if ((int)p >= P) return;
        dst[(long long)p * plane + m.at(j)] = (D)src[(size_t)j * 8u + p];
    }
}

// one plane: dst[j] = src[at(j)] (in) or dst[at(j)] = src[j] (out)
template <typename S, typename D, class Map, bool IN>
__global__ void __launch_bounds__(256) plane_copy(const S *__restrict__ src, D *__restrict__ dst, const Map m, long long n)
{
    const long long j = (long long)blockIdx.x * 256 + threadIdx.x;
    if (j >= n) return;
    if (IN) dst[j] = (D)src[m.at(j)];
    else dst[m.at(j)] = (D)src[j];
}

template <typename S, typename D, class Map>
static void inward(const void *src, void *dst, const Map &m, long long n, long long plane, int P, int Pp, D pad,
                   cudaStream_t st)
{
    if (Pp == 1) {
        plane_copy<S, D, Map, true><<<blocks(n), 256, 0, st>>>((const S *)src, (D *)dst, m, n);
        return;
    }
    if (Pp == 8) {
        group_copy<S, D, Map, true><<<blocks(8 * n), 256, 0, st>>>((const S *)src, (D *)dst, m, n, plane, P, pad);
        return;
    }
    const dim3 grid((unsigned)((n + TR_J - 1) / TR_J), (unsigned)((Pp + TR_P - 1) / TR_P));
    planes_inward<S, D, Map><<<grid, 256, 0, st>>>((const S *)src, (D *)dst, m, n, plane, P, Pp, pad);
}
template <typename S, typename D, class Map>
static void outward(const void *src, void *dst, const Map &m, long long n, long long plane, int P, int Pp,
                    cudaStream_t st)
{
    if (Pp == 1) {
        plane_copy<S, D, Map, false><<<blocks(n), 256, 0, st>>>((const S *)src, (D *)dst, m, n);
        return;
    }
    if (Pp == 8) {
        group_copy<S, D, Map, false><<<blocks(P * n), 256, 0, st>>>((const S *)src, (D *)dst, m, n, plane, P, D(0));
        return;
    }
    const dim3 grid((unsigned)((n + TR_J - 1) / TR_J), (unsigned)((P + TR_P - 1) / TR_P));
    planes_outward<S, D, Map><<<grid, 256, 0, st>>>((const S *)src, (D *)dst, m, n, plane, P, Pp);
}

// one plane: dst = src (unless they are the same array) and dst_t[x][y] = src[y][x], through a
// 32 x 32 shared tile so that both sides are read and written in whole rows
__global__ void __launch_bounds__(256) plane_transpose(const float *src, float *dst, float *dst_t, int N)
{
    __shared__ float t[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int x = x0 + threadIdx.x, y = y0 + r;
        if (x >= N || y >= N) continue;
        const float v = src[(size_t)y * N + x];
        t[r][threadIdx.x] = v;
        if (dst != src) dst[(size_t)y * N + x] = v;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int x = x0 + r, y = y0 + threadIdx.x;
        if (x < N && y < N) dst_t[(size_t)x * N + y] = t[threadIdx.x][r];
    }
}

// ones in the valid planes, zero in the pad planes
template <typename D>
__global__ void img_ones_internal(D *dst, long long n, int P, int Pp)
{
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= n) return;
    dst[tid] = (int)(tid % Pp) < P ? (D)1 : (D)0;
}

__global__ void check_data(const int *counts, const float *gamma, size_t n, int *flag)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gm = gamma[i];
    if (counts[i] < 0 || !(gm > 0.f) || !isfinite(gm)) atomicOr(flag, 1);
}

__global__ void check_factors(const float *mult, size_t n, int *flag)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float a = mult[i];
    if (!(a >= 0.f) || !isfinite(a)) atomicOr(flag, 1);
}


pet_status to_internal_image(const GeoDev &g, const void *src, void *dst, int sd, int dd,
                             cudaStream_t st)
{
    const long long n = (long long)g.N * g.N;
    LaunchScope ls(PET_K_LAYOUT, st);
    if (!sd && !dd) inward<float, float>(src, dst, ImageMap{}, n, n, g.P, g.Pp, 0.f, st);
    else if (!sd && dd) inward<float, double>(src, dst, ImageMap{}, n, n, g.P, g.Pp, 0.0, st);
    else if (sd && !dd) inward<double, float>(src, dst, ImageMap{}, n, n, g.P, g.Pp, 0.f, st);
    else inward<double, double>(src, dst, ImageMap{}, n, n, g.P, g.Pp, 0.0, st);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "to_internal_image");
}

pet_status plane_with_transpose(const GeoDev &g, const void *src, void *dst, void *dst_t, cudaStream_t st)
{
    LaunchScope ls(PET_K_LAYOUT, st);
    const unsigned b = (unsigned)((g.N + 31) / 32);
    plane_transpose<<<dim3(b, b), dim3(32, 8), 0, st>>>((const float *)src, (float *)dst, (float *)dst_t, g.N);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "plane_transpose");
}

pet_status from_internal_image(const GeoDev &g, const void *src, void *dst, int sd, int dd,
                               cudaStream_t st)
{
    const long long n = (long long)g.N * g.N;
    LaunchScope ls(PET_K_LAYOUT, st);
    if (!sd && !dd) outward<float, float>(src, dst, ImageMap{}, n, n, g.P, g.Pp, st);
    else if (!sd && dd) outward<float, double>(src, dst, ImageMap{}, n, n, g.P, g.Pp, st);
    else if (sd && !dd) outward<double, float>(src, dst, ImageMap{}, n, n, g.P, g.Pp, st);
    else outward<double, double>(src, dst, ImageMap{}, n, n, g.P, g.Pp, st);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "from_internal_image");
}

// full [P][V][SB] (original view order) or subset [P][nviews][SB] -> [nviews][SB][Pp]
pet_status to_internal_sino(const GeoDev &g, const int *d_view_of_slot, int slot0, int nviews,
                            const void *src, void *dst, int elem, int src_is_subset,
                            cudaStream_t st)
{
    const long long n = (long long)nviews * g.SB;           // SB: bins x TOF bins
    if (n == 0) return PET_OK;
    const long long plane = (long long)(src_is_subset ? nviews : g.V) * g.SB;
    const SinoMap m{src_is_subset ? nullptr : d_view_of_slot, slot0, g.SB};
    LaunchScope ls(PET_K_LAYOUT, st);
    // elem: 0 int32 counts (pad 0), 1 float gamma (pad 1), 2 float data (pad 0), 3 double
    // data, 4 float data to double (pad 0)
    if (elem == 4) inward<float, double>(src, dst, m, n, plane, g.P, g.Pp, 0.0, st);
    else if (elem == 0) inward<int, int>(src, dst, m, n, plane, g.P, g.Pp, 0, st);
    else if (elem == 1) inward<float, float>(src, dst, m, n, plane, g.P, g.Pp, 1.f, st);
    else if (elem == 2) inward<float, float>(src, dst, m, n, plane, g.P, g.Pp, 0.f, st);
    else inward<double, double>(src, dst, m, n, plane, g.P, g.Pp, 0.0, st);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "to_internal_sino");
}

// [nviews][SB][Pp] -> [P][nviews][SB], or -> [P][V][SB] in original view order when view_of_slot is
// given (all views, slot0 = 0)
pet_status from_internal_sino(const GeoDev &g, const int *d_view_of_slot, int nviews,
                              const void *src, void *dst, int is_double, cudaStream_t st)
{
    const long long n = (long long)nviews * g.SB;
    if (n == 0) return PET_OK;
    const SinoMap m{d_view_of_slot, 0, g.SB};
    LaunchScope ls(PET_K_LAYOUT, st);
    if (is_double) outward<double, double>(src, dst, m, n, n, g.P, g.Pp, st);
    else outward<float, float>(src, dst, m, n, n, g.P, g.Pp, st);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "from_internal_sino");
}

pet_status fill_internal_ones(const GeoDev &g, void *dst, int is_double, cudaStream_t st,
                              bool transposed)
{
    const long long n = (long long)g.N * g.N * g.Pp * (transposed ? 2 : 1);   // the copy follows
    LaunchScope ls(PET_K_LAYOUT, st);
    if (is_double) img_ones_internal<double><<<blocks(n), 256, 0, st>>>((double *)dst, n, g.P, g.Pp);
    else img_ones_internal<float><<<blocks(n), 256, 0, st>>>((float *)dst, n, g.P, g.Pp);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "img_ones_internal");
}

// Per-bin detection factors: finite and >= 0 (sets *d_flag, which the caller cleared, else).
pet_status validate_factors(const float *mult, size_t n, int *d_flag, cudaStream_t st)
{
    if (n == 0) return PET_OK;
    LaunchScope ls(PET_K_LAYOUT, st);
    check_factors<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mult, n, d_flag);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "check_factors");
}

pet_status validate_data(const GeoDev &g, const int *counts, const float *gamma, size_t n,
                         int *d_flag, cudaStream_t st)
{
    (void)g;
    PET_CUDA(cudaMemsetAsync(d_flag, 0, sizeof(int), st));
    if (n == 0) return PET_OK;
    LaunchScope ls(PET_K_LAYOUT, st);
    check_data<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(counts, gamma, n, d_flag);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PET_OK : cuda_fail(e, "check_data");
}

}  // namespace pet
