// pass_fp64.cu -- the plain Jacobi pass of Smart Laplacian smoothing with
// every step on the FP64 pipe, plus the small auxiliary kernels.
//
// One thread per node (grid-stride).  For a free node i the thread
//   1. sums its neighbours' coordinates in the stored summation order and
//      divides by the degree (Eq. 2, Form A: only pass-q coordinates);
//   2. evaluates alpha of every incident triangle with node i at its pass-q
//      position (q_old) and at the centre (q_new), keeping the minima
//      (Section 3.3.4 and the per-pass refresh of all qualities);
//   3. keeps the centre iff q_new >= q_old (strict: >), writes the node, and
//      contributes its squared move and acceptance to the pass statistics.
// The FP64 pipe of GB300 is narrow, so this kernel is the exact baseline and
// the fallback of the screened kernel, not the fast path.
#include "kernels.h"
#include "node_exact.cuh"

namespace sls {

namespace {

template <int LAYOUT>
__global__ void __launch_bounds__(1024) pass_fp64_kernel(PassArgs a)
{
    if (pass_is_skipped(a.stats, a.q, a.tol_active, a.thr_bits)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.stats[a.q].executed = 1u;

    unsigned long long best = 0ull, nacc = 0ull;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // every node, or (a colour class of Form B) a range of ids
    const int64_t cnt = a.ranged ? a.count : a.n;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < cnt; j += stride) {
        const int64_t i = a.first + j;
        const uint32_t meta = __ldg(a.adj + __ldg(a.node_off + i));
        if (meta & kMetaFixed) {
            if (a.accept) a.accept[i] = 0;
            continue;
        }
        unsigned long long bits;
        bool ok, moved;
        exact_update<LAYOUT>(a, i, bits, ok, moved);
        best = bits > best ? bits : best;
        nacc += ok ? 1ull : 0ull;
    }
    block_reduce_stats(a.stats + a.q, best, nacc, 0ull);
}

__global__ void copy_back_kernel(const double2 *__restrict__ src, double2 *__restrict__ dst,
                                 int64_t n2, const PassStats *stats, int q)
{
    if (stats[q].executed == 0u) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n2; k += stride)
        dst[k] = __ldg(src + k);
}

__device__ __forceinline__ unsigned long long order_key(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Bin of quality q, as the definition has it.
__device__ __forceinline__ int exact_bin(double q, double lo, double width, int nbins)
{
    const double f = floor(__dmul_rn(__ddiv_rn(__dsub_rn(q, lo), width), (double)nbins));
    return f < 0.0 ? 0 : (f >= (double)nbins ? nbins - 1 : (int)f);
}

// 1/s to within a unit in the last place for normal s well inside the range:
// from the hardware's 20-bit estimate x, with e = 1 - s x, the series
// x (1 + e + e^2) is off by e^3.
__device__ __forceinline__ double reciprocal(double s)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(s));
    const double e = __fma_rn(-s, x, 1.0);
    return __fma_rn(x, __fma_rn(e, e, e), x);
}

// The FP64 pipe (2 operations per clock and SM) is what a quality costs.  The
// definition's tree, a correctly rounded division for alpha and another for
// the bin are 46 FP64 instructions a triangle; here the mean takes cross / s
// with fused products and a reciprocal (20 instructions, fewer roundings; the
// factor 2 sqrt(3) once at the end), and the definition's tree is evaluated
// only where it can matter: for a thread's least quality where that can be the
// block's, for one next to a bin's edge (FP32 arithmetic on its leading bits
// says which), and where the edge sum leaves the safe range.  The counters are 32
// bits in shared memory (a 64-bit shared addition is a compare-and-swap loop,
// and most triangles fall in a few bins).  8.4M triangles (2048^2 grid, 20
// bins): 332 us a call against 762; the FP64 pipe alone takes 270 for them.  A
// mesh of equal qualities evaluates every triangle both ways (1024^2: 211 us
// against 250; jittered 113 against 227).
struct HistogramRange {
    double lo, hi;
    float lof, scale;  // bin number about (q - lof) * scale
    float err_q;       // its error: at most err_q + 2^-20 of it
};

template <int LAYOUT>
__global__ void __launch_bounds__(256) histogram_kernel(const double *xy, int64_t n, const int32_t *__restrict__ tri,
                                                        int64_t m, int nbins, HistogramRange hr,
                                                        unsigned long long *counts, unsigned long long *qmin_key,
                                                        double *qsum)
{
    extern __shared__ unsigned s_counts[];
    __shared__ unsigned long long s_min;
    __shared__ int s_least;  // order key of the least of the threads' least qualities
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) s_counts[b] = 0u;
    if (threadIdx.x == 0) {
        s_min = ~0ull;
        s_least = 0x7fffffff;
    }
    __syncthreads();
    const float kTwoSqrt3f = 3.46410161514f;
    const double width = __dsub_rn(hr.hi, hr.lo);
    // twice how far the two trees and the FP32 value can be apart (absolutely
    // so next to alpha = 0)
    auto apart = [](float q) { return fabsf(q) * 3.9e-6f + 1e-14f; };
    float least = __int_as_float(0x7f800000);  // the thread's least quality, of triangle least_t
    int64_t least_t = -1;
    unsigned long long exact_min = ~0ull;  // key of the least quality evaluated by the definition's tree
    double sum = 0.0, rest = 0.0;  // of cross / s, and of qualities taken whole
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += stride) {
        const double2 A = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * t));
        const double2 B = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * t + 1));
        const double2 C = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * t + 2));
        const double e1x = B.x - A.x, e1y = B.y - A.y, e2x = C.x - A.x, e2y = C.y - A.y;
        const double e3x = C.x - B.x, e3y = C.y - B.y;
        const double cross = __fma_rn(e1x, e2y, -(e1y * e2x));
        const double s = __fma_rn(
            e1x, e1x, __fma_rn(e1y, e1y, __fma_rn(e2x, e2x, __fma_rn(e2y, e2y, __fma_rn(e3x, e3x, e3y * e3y)))));
        const unsigned es = (unsigned)(__double_as_longlong(s) >> 52) & 0x7ffu;
        const bool safe = es - 123u < 1800u;  // 2^-900 <= s < 2^900: no product under- or overflows
        const double r = safe ? cross * reciprocal(s) : 0.0;
        // leading bits as a float (zero below 2^-126): |qf - alpha| < 2^-20 |alpha| + 2^-100
        const unsigned long long rb = (unsigned long long)__double_as_longlong(r);
        const unsigned hw = (unsigned)(rb >> 32), lw = (unsigned)rb, er = (hw >> 20) & 0x7ffu;
        const float rf = __uint_as_float((hw & 0x80000000u) | ((er - 896u) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29));
        const float qf = er - 897u <= 253u ? rf * kTwoSqrt3f : 0.0f;
        const float f = (qf - hr.lof) * hr.scale, near = rintf(f);
        // inside a bin by more than the error (also beyond either end)
        const bool inside = fabsf(f - near) > hr.err_q + fabsf(f) * 9.6e-7f;
        int bin = (int)fminf(fmaxf(floorf(f), 0.0f), (float)(nbins - 1));
        bool tie = false;  // too near the thread's least to tell which is less
        if (safe && qf - apart(qf) <= least + apart(least)) {
            tie = qf + apart(qf) >= least - apart(least);
            if (!tie) {
                least = qf;
                least_t = t;
            }
        }
        if (!safe || !inside || tie) {
            const double q = alpha_fp64(A.x, A.y, B.x, B.y, C.x, C.y);
            if (!safe || !inside) bin = exact_bin(q, hr.lo, width, nbins);
            if (!safe) rest = __dadd_rn(rest, q);
            const unsigned long long key = order_key(q);
            exact_min = key < exact_min ? key : exact_min;
        }
        sum = __dadd_rn(sum, r);
        atomicAdd(&s_counts[bin], 1u);
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum = __dadd_rn(sum, __shfl_xor_sync(0xffffffffu, sum, o));
        rest = __dadd_rn(rest, __shfl_xor_sync(0xffffffffu, rest, o));
    }
    if ((threadIdx.x & 31u) == 0) atomicAdd(qsum, __fma_rn(3.4641016151377544, sum, rest));
    const int bits = __float_as_int(least), key = bits < 0 ? bits ^ 0x7fffffff : bits;  // orders like the value
    atomicMin(&s_least, key);
    __syncthreads();
    const float block_least = __int_as_float(s_least < 0 ? s_least ^ 0x7fffffff : s_least);
    if (least_t >= 0 && least - apart(least) <= block_least + apart(block_least)) {
        const double2 A = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * least_t));
        const double2 B = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * least_t + 1));
        const double2 C = Coords<LAYOUT>::get(xy, n, __ldg(tri + 3 * least_t + 2));
        const unsigned long long k = order_key(alpha_fp64(A.x, A.y, B.x, B.y, C.x, C.y));
        exact_min = k < exact_min ? k : exact_min;
    }
    if (exact_min != ~0ull) atomicMin(&s_min, exact_min);
    __syncthreads();
    if (threadIdx.x == 0) atomicMin(qmin_key, s_min);
    for (int b = threadIdx.x; b < nbins; b += blockDim.x)
        if (s_counts[b]) atomicAdd(&counts[b], (unsigned long long)s_counts[b]);
}

__global__ void soa_to_aos_kernel(const double *__restrict__ soa, double *__restrict__ aos, int64_t n, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        store_pair(aos, i, make_double2(__ldg(soa + i), __ldg(soa + n + i)), wide);
}

__global__ void aos_to_soa_kernel(const double *__restrict__ aos, double *__restrict__ soa, int64_t n, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double2 v = load_pair(aos, i, wide);
        soa[i] = v.x;
        soa[n + i] = v.y;
    }
}

}  // namespace

cudaError_t launch_pass_fp64(const PassArgs &a, int layout, int block, int grid, cudaStream_t s)
{
    if (layout == 0) pass_fp64_kernel<0><<<grid, block, 0, s>>>(a);
    else pass_fp64_kernel<1><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

int pass_fp64_occupancy(int layout, int block)
{
    int nb = 0;
    if (layout == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pass_fp64_kernel<0>, block, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pass_fp64_kernel<1>, block, 0);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_copy_back(const double *src, double *dst, int64_t n_doubles,
                             const PassStats *stats, int q, int grid, cudaStream_t s)
{
    copy_back_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<const double2 *>(src),
                                         reinterpret_cast<double2 *>(dst), n_doubles / 2, stats, q);
    return cudaGetLastError();
}

cudaError_t launch_histogram(const double *xy, int layout, int64_t n, const int32_t *tri,
                             int64_t m, int nbins, double lo, double hi,
                             unsigned long long *counts, unsigned long long *qmin_key,
                             double *qsum, int grid, cudaStream_t s)
{
    const size_t smem = sizeof(unsigned) * (size_t)nbins;
    HistogramRange hr{lo, hi, (float)lo, 0.0f, 1e30f};
    // error of the FP32 bin number: the quality's (2^-19 of at most 1.01), lo's
    // rounding, the subtraction's; where it or the scale is out of hand every
    // triangle takes the definition's way
    const double scale = (double)nbins / (hi - lo);
    const double err = scale * (2e-6 + (lo < 0.0 ? -lo : lo) * 2.4e-7);
    if (scale < 1e30 && err < 0.25) {
        hr.scale = (float)scale;
        hr.err_q = (float)(1.01 * err);
    }
    // blocks enough to fill the GPU, and few enough that a block's 32-bit
    // counters cannot overflow
    const int64_t need = (m + 255) / 256;
    if (need < grid) grid = (int)need;
    if (layout == 0)
        histogram_kernel<0><<<grid, 256, smem, s>>>(xy, n, tri, m, nbins, hr, counts, qmin_key, qsum);
    else
        histogram_kernel<1><<<grid, 256, smem, s>>>(xy, n, tri, m, nbins, hr, counts, qmin_key, qsum);
    return cudaGetLastError();
}

namespace {

// Coordinates of the listed nodes out of the current array (ghost exchange
// of a domain-decomposed mesh); an id outside [0, n) sets *bad and is skipped.
template <int LAYOUT>
__global__ void gather_nodes_kernel(const double *__restrict__ xy, int64_t n, const int32_t *__restrict__ idx,
                                    int64_t k, const uint32_t *__restrict__ inv, double *__restrict__ out,
                                    bool wide, unsigned *bad)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k; t += stride) {
        const int32_t i = __ldg(idx + t);
        if (i < 0 || (int64_t)i >= n) {
            atomicOr(bad, 1u);
            continue;
        }
        store_pair(out, t, Coords<LAYOUT>::get(xy, n, inv ? (int64_t)__ldg(inv + i) : (int64_t)i), wide);
    }
}

// The listed nodes' coordinates written into both arrays of the ping-pong.
template <int LAYOUT>
__global__ void scatter_nodes_kernel(double *xy0, double *xy1, int64_t n, const int32_t *__restrict__ idx,
                                     int64_t k, const uint32_t *__restrict__ inv, const double *__restrict__ in,
                                     bool wide, unsigned *bad)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k; t += stride) {
        const int32_t i = __ldg(idx + t);
        if (i < 0 || (int64_t)i >= n) {
            atomicOr(bad, 1u);
            continue;
        }
        const double2 v = load_pair(in, t, wide);
        const int64_t j = inv ? (int64_t)__ldg(inv + i) : (int64_t)i;
        Coords<LAYOUT>::put(xy0, n, j, v);
        Coords<LAYOUT>::put(xy1, n, j, v);
    }
}

}  // namespace

cudaError_t launch_gather_nodes(const double *xy, int layout, int64_t n, const int32_t *idx, int64_t k,
                                const uint32_t *inv, double *out, unsigned *bad, int grid, cudaStream_t s)
{
    if (k <= 0) return cudaSuccess;
    if (layout == 0)
        gather_nodes_kernel<0><<<grid, 256, 0, s>>>(xy, n, idx, k, inv, out, pair_aligned(out), bad);
    else
        gather_nodes_kernel<1><<<grid, 256, 0, s>>>(xy, n, idx, k, inv, out, pair_aligned(out), bad);
    return cudaGetLastError();
}

cudaError_t launch_scatter_nodes(double *xy0, double *xy1, int layout, int64_t n, const int32_t *idx, int64_t k,
                                 const uint32_t *inv, const double *in, unsigned *bad, int grid, cudaStream_t s)
{
    if (k <= 0) return cudaSuccess;
    if (layout == 0)
        scatter_nodes_kernel<0><<<grid, 256, 0, s>>>(xy0, xy1, n, idx, k, inv, in, pair_aligned(in), bad);
    else
        scatter_nodes_kernel<1><<<grid, 256, 0, s>>>(xy0, xy1, n, idx, k, inv, in, pair_aligned(in), bad);
    return cudaGetLastError();
}

namespace {

// Coordinates in a layout and an element type (double or float).
template <class T, int LAYOUT>
struct Pair;
template <class T>
struct Pair<T, 0> {
    static __device__ __forceinline__ void get(const T *p, int64_t, int64_t i, T &x, T &y)
    {
        x = p[2 * i];
        y = p[2 * i + 1];
    }
    static __device__ __forceinline__ void put(T *p, int64_t, int64_t i, T x, T y)
    {
        p[2 * i] = x;
        p[2 * i + 1] = y;
    }
};
template <class T>
struct Pair<T, 1> {
    static __device__ __forceinline__ void get(const T *p, int64_t n, int64_t i, T &x, T &y)
    {
        x = p[i];
        y = p[n + i];
    }
    static __device__ __forceinline__ void put(T *p, int64_t n, int64_t i, T x, T y)
    {
        p[i] = x;
        p[n + i] = y;
    }
};

// dst[k] = src[perm[k]] (same layout and type)
template <class T, int LAYOUT>
__global__ void permute_kernel(const T *__restrict__ src, T *__restrict__ dst, int64_t n,
                               const uint32_t *__restrict__ perm)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        T x, y;
        Pair<T, LAYOUT>::get(src, n, perm[k], x, y);
        Pair<T, LAYOUT>::put(dst, n, k, x, y);
    }
}

// dst (interleaved doubles, the caller's numbering)[perm[k]] = src[k] (exact widening of floats)
template <class T, int LAYOUT>
__global__ void unpermute_to_aos_kernel(const T *__restrict__ src, int64_t n, const uint32_t *__restrict__ perm,
                                        double *__restrict__ dst, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        T x, y;
        Pair<T, LAYOUT>::get(src, n, k, x, y);
        store_pair(dst, perm[k], make_double2((double)x, (double)y), wide);
    }
}

// dst[k] = src (interleaved doubles, the caller's numbering)[perm[k]], rounded to T
template <class T, int LAYOUT>
__global__ void permute_from_aos_kernel(const double *__restrict__ src, int64_t n, const uint32_t *__restrict__ perm,
                                        T *__restrict__ dst, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        const double2 v = load_pair(src, perm[k], wide);
        Pair<T, LAYOUT>::put(dst, n, k, (T)v.x, (T)v.y);
    }
}

__global__ void unpermute_u8_kernel(const uint8_t *__restrict__ src, int64_t n, const uint32_t *__restrict__ perm,
                                    uint8_t *__restrict__ dst)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) dst[perm[k]] = src[k];
}

}  // namespace

cudaError_t launch_permute_coords(const double *src, double *dst, int layout, bool f32, int64_t n,
                                  const uint32_t *perm, int grid, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (f32) {
        const float *fs = reinterpret_cast<const float *>(src);
        float *fd = reinterpret_cast<float *>(dst);
        if (layout == 0) permute_kernel<float, 0><<<grid, 256, 0, s>>>(fs, fd, n, perm);
        else permute_kernel<float, 1><<<grid, 256, 0, s>>>(fs, fd, n, perm);
    } else {
        if (layout == 0) permute_kernel<double, 0><<<grid, 256, 0, s>>>(src, dst, n, perm);
        else permute_kernel<double, 1><<<grid, 256, 0, s>>>(src, dst, n, perm);
    }
    return cudaGetLastError();
}

cudaError_t launch_unpermute_to_aos(const double *src, int layout, bool f32, int64_t n, const uint32_t *perm,
                                    double *dst_aos, int grid, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    double *d = dst_aos;
    const bool w = pair_aligned(d);
    if (f32) {
        const float *f = reinterpret_cast<const float *>(src);
        if (layout == 0) unpermute_to_aos_kernel<float, 0><<<grid, 256, 0, s>>>(f, n, perm, d, w);
        else unpermute_to_aos_kernel<float, 1><<<grid, 256, 0, s>>>(f, n, perm, d, w);
    } else {
        if (layout == 0) unpermute_to_aos_kernel<double, 0><<<grid, 256, 0, s>>>(src, n, perm, d, w);
        else unpermute_to_aos_kernel<double, 1><<<grid, 256, 0, s>>>(src, n, perm, d, w);
    }
    return cudaGetLastError();
}

cudaError_t load_numbering_kernels()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, (const void *)permute_kernel<double, 0>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, (const void *)unpermute_to_aos_kernel<double, 0>);
    return e;
}

cudaError_t launch_permute_from_aos(const double *src_aos, int layout, bool f32, int64_t n, const uint32_t *perm,
                                    double *dst, int grid, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const double *v = src_aos;
    const bool w = pair_aligned(v);
    if (f32) {
        float *f = reinterpret_cast<float *>(dst);
        if (layout == 0) permute_from_aos_kernel<float, 0><<<grid, 256, 0, s>>>(v, n, perm, f, w);
        else permute_from_aos_kernel<float, 1><<<grid, 256, 0, s>>>(v, n, perm, f, w);
    } else {
        if (layout == 0) permute_from_aos_kernel<double, 0><<<grid, 256, 0, s>>>(v, n, perm, dst, w);
        else permute_from_aos_kernel<double, 1><<<grid, 256, 0, s>>>(v, n, perm, dst, w);
    }
    return cudaGetLastError();
}

cudaError_t launch_unpermute_u8(const uint8_t *src, int64_t n, const uint32_t *perm, uint8_t *dst, int grid,
                                cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    unpermute_u8_kernel<<<grid, 256, 0, s>>>(src, n, perm, dst);
    return cudaGetLastError();
}

cudaError_t launch_soa_to_aos(const double *soa, double *aos, int64_t n, int grid, cudaStream_t s)
{
    soa_to_aos_kernel<<<grid, 256, 0, s>>>(soa, aos, n, pair_aligned(aos));
    return cudaGetLastError();
}

cudaError_t launch_aos_to_soa(const double *aos, double *soa, int64_t n, int grid, cudaStream_t s)
{
    aos_to_soa_kernel<<<grid, 256, 0, s>>>(aos, soa, n, pair_aligned(aos));
    return cudaGetLastError();
}

}  // namespace sls
