// mesh_build_gpu.cu -- the adjacency build of sls_mesh_create on the device.
//
// Same records, word for word, as the host build in mesh_build.cpp (Section
// 3.3.2: neighbours and incident triangles; Section 3.3.3: constraints), with
// the work spread over one thread per triangle or per node instead of the
// paper's single GPU thread:
//   1. validate triangles and coordinates;
//   2. count the incidences of every node, exclusive scan;
//   3. scatter (node, triangle) incidences;
//   4. per node: sort its incident triangles, collect the other vertices of
//      each, de-duplicate them while counting how many triangles share each
//      edge (1 = boundary edge, > 2 = non-manifold), order the neighbours for
//      summation (ascending x, y, id) and write the record: meta word,
//      neighbours, triangle codes.  The words are the host build's; only where
//      a record starts differs (node_records_kernel);
//   5. a mesh with a record longer than its place: sized first, an exclusive
//      scan of the lengths, then written (node_pass1_kernel, node_pass2_kernel);
//   6. free-node count with 4, bounding box with 1.
// Nodes with more than kMaxInc incident triangles are left to the host build
// (the whole mesh then takes the host path).
#include <cstring>
#include <vector>

#include "api_common.h"
#include "kernels.h"

namespace sls {

namespace {

constexpr int kMaxInc = 32;  // incident triangles per node handled on the device

enum : unsigned {
    kErrRange = 1u,
    kErrRepeat = 2u,
    kErrFinite = 4u,
    kErrManifold = 8u,
    kErrTooMany = 16u,
    kErrRoom = 32u  // a record longer than its place (node_records_kernel)
};

// Words the build's kernels report to the host through one array of 64-bit
// words (kReport of them).
enum : int {
    kBadTri = 0,    // first bad triangle * 2 (+ 1: repeated vertex)
    kBadCoord = 1,  // first coordinate that is not finite
    kBox = 2,       // okeys of xmin, ymin, xmax, ymax
    kFree = 6,      // free nodes
    kCrossing = 7,  // triangle edges whose ends lie in different 128-id windows
    kFlags = 8,     // kErr* bits
    kReport = 9
};

// Order-preserving 64-bit keys of finite doubles, for min / max with atomics.
__device__ __forceinline__ unsigned long long okey(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__global__ void report_init_kernel(unsigned long long *rep)
{
    const int k = threadIdx.x;
    if (k < kReport) rep[k] = k < kBox + 2 ? ~0ull : 0ull;
}

__global__ void validate_tri_kernel(const int32_t *__restrict__ tri, int64_t m, int64_t n, unsigned long long *rep)
{
    unsigned crossing = 0u;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += stride) {
        const int32_t a = tri[3 * t], b = tri[3 * t + 1], c = tri[3 * t + 2];
        const bool range = a < 0 || b < 0 || c < 0 || a >= n || b >= n || c >= n;
        const bool again = a == b || a == c || b == c;
        if (range || again) {
            atomicOr(rep + kFlags, (unsigned long long)(range ? kErrRange : kErrRepeat));
            // the first bad triangle; at equal index the range error comes first
            atomicMin(rep + kBadTri, (unsigned long long)t * 2ull + (range ? 0ull : 1ull));
        }
        crossing += ((a ^ b) >> 7 ? 1u : 0u) + ((b ^ c) >> 7 ? 1u : 0u) + ((c ^ a) >> 7 ? 1u : 0u);
    }
    crossing = __reduce_add_sync(0xffffffffu, crossing);
    if ((threadIdx.x & 31) == 0 && crossing) atomicAdd(rep + kCrossing, (unsigned long long)crossing);
}

// Finiteness of every coordinate and the bounding box, one pass over them.
__global__ void __launch_bounds__(256) validate_xy_kernel(const double2 *__restrict__ xy, int64_t n,
                                                          unsigned long long *rep)
{
    __shared__ unsigned long long s_key[8][4];
    unsigned long long lo_x = ~0ull, lo_y = ~0ull, hi_x = 0ull, hi_y = 0ull;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double2 p = xy[i];
        const unsigned long long bx = (unsigned long long)__double_as_longlong(p.x);
        const unsigned long long by = (unsigned long long)__double_as_longlong(p.y);
        const bool badx = ((bx >> 52) & 0x7ffull) == 0x7ffull, bady = ((by >> 52) & 0x7ffull) == 0x7ffull;
        if (badx || bady) {
            atomicOr(rep + kFlags, (unsigned long long)kErrFinite);
            atomicMin(rep + kBadCoord, 2ull * (unsigned long long)i + (badx ? 0ull : 1ull));
        }
        const unsigned long long kx = okey(p.x), ky = okey(p.y);
        lo_x = kx < lo_x ? kx : lo_x;
        lo_y = ky < lo_y ? ky : lo_y;
        hi_x = kx > hi_x ? kx : hi_x;
        hi_y = ky > hi_y ? ky : hi_y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long t;
        t = __shfl_xor_sync(0xffffffffu, lo_x, o); lo_x = t < lo_x ? t : lo_x;
        t = __shfl_xor_sync(0xffffffffu, lo_y, o); lo_y = t < lo_y ? t : lo_y;
        t = __shfl_xor_sync(0xffffffffu, hi_x, o); hi_x = t > hi_x ? t : hi_x;
        t = __shfl_xor_sync(0xffffffffu, hi_y, o); hi_y = t > hi_y ? t : hi_y;
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_key[warp][0] = lo_x;
        s_key[warp][1] = lo_y;
        s_key[warp][2] = hi_x;
        s_key[warp][3] = hi_y;
    }
    __syncthreads();
    if (threadIdx.x < 4) {  // one atomic per bound and block
        const int k = threadIdx.x;
        unsigned long long v = s_key[0][k];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            const unsigned long long u = s_key[w][k];
            v = k < 2 ? (u < v ? u : v) : (u > v ? u : v);
        }
        if (k < 2) atomicMin(rep + kBox + k, v);
        else atomicMax(rep + kBox + k, v);
    }
}

// ---- spatial numbering -------------------------------------------------------
// The screened pass stages every window of 128 consecutive ids with its
// neighbours, so ids have to be near each other where nodes are.  A mesh whose
// edges mostly leave their windows (a random numbering: all of them; rows of a
// grid: two thirds; Morton order: a quarter) is renumbered along a Z-order
// curve of square cells holding about half a node each, before its adjacency
// is built; the build's own gathers then fall close together too.  A random
// numbering of a 1009 x 701 grid runs 48 us a pass renumbered and 73 (AoS) or
// 111 (SoA) as it is; its creation takes the same time either way.

struct CellGrid {
    double x0, y0, scale;  // cell = floor((v - v0) * scale), clamped to [0, side)
    unsigned side;         // a power of two
};

__device__ __forceinline__ unsigned spread_bits(unsigned v)
{
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    return (v | (v << 1)) & 0x55555555u;
}

__device__ __forceinline__ unsigned cell_of(double2 p, const CellGrid &g)
{
    const double fx = (p.x - g.x0) * g.scale, fy = (p.y - g.y0) * g.scale, top = (double)(g.side - 1u);
    const unsigned cx = (unsigned)fmin(fmax(fx, 0.0), top), cy = (unsigned)fmin(fmax(fy, 0.0), top);
    return spread_bits(cx) | (spread_bits(cy) << 1);
}

__global__ void remap_ids_kernel(int32_t *ids, int64_t count, const uint32_t *__restrict__ inv);

__global__ void cell_count_kernel(const double2 *__restrict__ xy, int64_t n, CellGrid g, unsigned *cnt)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        atomicAdd(cnt + cell_of(xy[i], g), 1u);
}

// Ids inside a cell come in no particular order (they change nothing but the
// order of work).
__global__ void cell_place_kernel(const double2 *__restrict__ xy, int64_t n, CellGrid g,
                                  const uint32_t *__restrict__ off, unsigned *left, uint32_t *perm, uint32_t *inv,
                                  double2 *__restrict__ xy_out)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double2 p = xy[i];
        const unsigned c = cell_of(p, g);
        const uint32_t k = off[c] + atomicSub(left + c, 1u) - 1u;
        perm[k] = (uint32_t)i;
        inv[i] = k;
        xy_out[k] = p;
    }
}

__global__ void count_kernel(const int32_t *__restrict__ tri, int64_t m3, unsigned *cnt)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m3; k += stride)
        atomicAdd(cnt + tri[k], 1u);
}

__global__ void scatter_kernel(const int32_t *__restrict__ tri, int64_t m3, const unsigned *__restrict__ ptr,
                               unsigned *cursor, int32_t *inc)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m3; k += stride) {
        const int32_t v = tri[k];
        const unsigned slot = atomicAdd(cursor + v, 1u);
        inc[ptr[v] + slot] = (int32_t)(k / 3);
    }
}

// Ascending (x, y, id) with the comparisons of the host build; ids are the
// caller's (perm: of a renumbered mesh).
__device__ __forceinline__ bool canon_less(double xa, double ya, int32_t a, double xb, double yb, int32_t b,
                                           const uint32_t *perm)
{
    if (xa < xb) return true;
    if (xb < xa) return false;
    if (ya < yb) return true;
    if (yb < ya) return false;
    return perm ? perm[a] < perm[b] : a < b;
}

// ---- node records ------------------------------------------------------------
// A closed ring of t triangles has t neighbours, so the record of node i (meta
// word, neighbours, triangle codes) has 2 t + 1 words, and an open fan's one
// more: records are written at 2 (incidences before i) + 2 i, without a scan of
// their lengths.  Only a node with several fans can need more; a mesh with
// such a free node is built again with exact lengths (node_pass1_kernel,
// node_pass2_kernel).

constexpr int kRingFast = 10;  // triangles of a node handled in registers

// The coordinate as canon_less orders it: an unsigned key, -0 as +0.
__device__ __forceinline__ unsigned long long canon_key(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if ((b << 1) == 0ull) b = 0ull;
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// The record of a node of any shape, with sorted lists in local memory.
__device__ __noinline__ void record_any(int64_t i, unsigned s, unsigned nt, const double2 *__restrict__ xy,
                                        const int32_t *__restrict__ tri, const int32_t *__restrict__ inc, int given,
                                        const uint32_t *perm, uint32_t *w, unsigned long long *rep)
{
    int32_t tl[kMaxInc], rec[2 * kMaxInc], uq[2 * kMaxInc];
    double ux[2 * kMaxInc], uy[2 * kMaxInc];
    for (unsigned k = 0; k < nt; ++k) {
        const int32_t t = inc[s + k];
        unsigned j = k;
        while (j > 0 && tl[j - 1] > t) {
            tl[j] = tl[j - 1];
            --j;
        }
        tl[j] = t;
    }
    // the other two vertices of every incident triangle, sorted by id
    unsigned r = 0;
    for (unsigned k = 0; k < nt; ++k) {
        for (int c = 0; c < 3; ++c) {
            const int32_t v = tri[3 * (int64_t)tl[k] + c];
            if (v == (int32_t)i) continue;
            unsigned j = r++;
            while (j > 0 && rec[j - 1] > v) {
                rec[j] = rec[j - 1];
                --j;
            }
            rec[j] = v;
        }
    }
    bool open_edge = r == 0;
    unsigned deg = 0;
    for (unsigned k = 0; k < r;) {
        unsigned f = k;
        while (f < r && rec[f] == rec[k]) ++f;
        const unsigned times = f - k;
        if (times == 1u) open_edge = true;
        if (times > 2u) atomicOr(rep + kFlags, (unsigned long long)kErrManifold);
        // summation order: ascending (x, y, id) of the creation coordinates
        const double2 p = xy[rec[k]];
        const int32_t id = rec[k];
        unsigned j = deg++;
        while (j > 0 && canon_less(p.x, p.y, id, ux[j - 1], uy[j - 1], uq[j - 1], perm)) {
            ux[j] = ux[j - 1];
            uy[j] = uy[j - 1];
            uq[j] = uq[j - 1];
            --j;
        }
        ux[j] = p.x;
        uy[j] = p.y;
        uq[j] = id;
        k = f;
    }
    if (given >= 0 ? (given != 0 || r == 0) : open_edge) {
        w[0] = kMetaFixed;
        return;
    }
    if (1u + deg + nt > 2u * nt + 2u) {
        w[0] = kMetaFixed;
        atomicOr(rep + kFlags, (unsigned long long)kErrRoom);
        return;
    }
    w[0] = (nt << 16) | deg;
    for (unsigned k = 0; k < deg; ++k) w[1 + k] = (uint32_t)uq[k];
    for (unsigned k = 0; k < nt; ++k) {
        uint32_t slot = 0, pos[2] = {0u, 0u}, np = 0;
        for (int c = 0; c < 3; ++c) {
            const int32_t v = tri[3 * (int64_t)tl[k] + c];
            if (v == (int32_t)i) {
                slot = (uint32_t)c;
                continue;
            }
            uint32_t p = 0;
            while (p + 1 < deg && uq[p] != v) ++p;
            pos[np++] = p;
        }
        w[1 + deg + k] = (slot << 30) | (pos[0] << 15) | pos[1];
    }
}

// One thread per node.  What a closed ring whose triangles are all stored the
// same way round needs (every neighbour once as the vertex after the node and
// once as the vertex before it) stays in registers: sorting by comparing all
// pairs; lists in local memory went through L2 (4.2M nodes: 984 us to size the
// records and 359 us to write them, in two kernels with a scan and a wait of
// the host between them, against 526 us; a create + 77 passes + destroy request of such a mesh
// went from 17.6 to 15.1 ms).
__global__ void __launch_bounds__(128) node_records_kernel(int64_t n, const double2 *__restrict__ xy,
                                                           const int32_t *__restrict__ tri,
                                                           const unsigned *__restrict__ ptr,
                                                           const int32_t *__restrict__ inc,
                                                           const uint8_t *__restrict__ boundary,
                                                           const uint32_t *__restrict__ perm, uint32_t *node_off,
                                                           uint32_t *adj, unsigned long long *rep)
{
    unsigned nfree = 0u;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned s = ptr[i], nt = ptr[i + 1] - s;
        const uint32_t off = 2u * s + 2u * (uint32_t)i;
        node_off[i] = off;
        if (i == n - 1) node_off[n] = 2u * ptr[n] + 2u * (uint32_t)n;
        uint32_t *w = adj + off;
        if (nt > (unsigned)kMaxInc) {
            atomicOr(rep + kFlags, (unsigned long long)kErrTooMany);
            w[0] = kMetaFixed;
            continue;
        }
        const int given = boundary ? (boundary[perm ? perm[i] : i] != 0 ? 1 : 0) : -1;
        bool done = false;
        if (nt > 0u && nt <= (unsigned)kRingFast) {
            // incident triangles in ascending order (unused places last)
            int32_t t[kRingFast];
#pragma unroll
            for (int k = 0; k < kRingFast; ++k) t[k] = k < (int)nt ? inc[s + k] : 0x7fffffff;
#pragma unroll
            for (int r = 0; r < kRingFast; ++r) {
#pragma unroll
                for (int k = r & 1; k + 1 < kRingFast; k += 2) {
                    const int32_t lo = min(t[k], t[k + 1]), hi = max(t[k], t[k + 1]);
                    t[k] = lo;
                    t[k + 1] = hi;
                }
            }
            // triangle k is (node, P, Q) in its stored direction
            int32_t P[kRingFast], Q[kRingFast];
            uint32_t slots = 0u;
#pragma unroll
            for (int k = 0; k < kRingFast; ++k) {
                P[k] = -1 - k;  // unlike every id and each other
                Q[k] = -1 - kRingFast - k;
                if (k < (int)nt) {
                    const int32_t *v = tri + 3 * (int64_t)t[k];
                    const int32_t v0 = v[0], v1 = v[1], v2 = v[2];
                    const uint32_t slot = v0 == (int32_t)i ? 0u : (v1 == (int32_t)i ? 1u : 2u);
                    P[k] = slot == 0u ? v1 : (slot == 1u ? v2 : v0);
                    Q[k] = slot == 0u ? v2 : (slot == 1u ? v0 : v1);
                    slots |= slot << (2 * k);
                }
            }
            bool plain = true;
            uint32_t met = 0u;  // triangles whose Q is some triangle's P
#pragma unroll
            for (int k = 0; k < kRingFast; ++k)
#pragma unroll
                for (int j = 0; j < kRingFast; ++j) {
                    if (j < k) plain = plain && P[j] != P[k] && Q[j] != Q[k];
                    if (j != k && Q[k] == P[j]) met |= 1u << k;
                }
            const bool closed = met == (1u << nt) - 1u;
            if (plain && (given == 1 || (given < 0 && !closed))) {
                w[0] = kMetaFixed;
                done = true;
            } else if (plain && closed) {
                unsigned long long kx[kRingFast], ky[kRingFast];
                uint32_t rank[kRingFast];
#pragma unroll
                for (int k = 0; k < kRingFast; ++k) {
                    rank[k] = 0u;
                    kx[k] = ky[k] = 0ull;
                    if (k < (int)nt) {
                        const double2 p = xy[P[k]];
                        kx[k] = canon_key(p.x);
                        ky[k] = canon_key(p.y);
                    }
                }
#pragma unroll
                for (int k = 1; k < kRingFast; ++k) {
                    if (k < (int)nt) {
#pragma unroll
                        for (int j = 0; j < k; ++j) {
                            bool less = kx[j] < kx[k];
                            if (kx[j] == kx[k]) {
                                less = ky[j] < ky[k];
                                if (ky[j] == ky[k]) less = perm ? perm[P[j]] < perm[P[k]] : P[j] < P[k];
                            }
                            rank[k] += less ? 1u : 0u;
                            rank[j] += less ? 0u : 1u;
                        }
                    }
                }
                w[0] = (nt << 16) | nt;
#pragma unroll
                for (int k = 0; k < kRingFast; ++k) {
                    if (k < (int)nt) {
                        w[1 + rank[k]] = (uint32_t)P[k];
                        uint32_t rq = 0u;
#pragma unroll
                        for (int j = 0; j < kRingFast; ++j) rq = Q[k] == P[j] ? rank[j] : rq;
                        const uint32_t slot = (slots >> (2 * k)) & 3u;
                        const uint32_t a = slot == 1u ? rq : rank[k], b = slot == 1u ? rank[k] : rq;
                        w[1 + nt + k] = (slot << 30) | (a << 15) | b;
                    }
                }
                done = true;
            }
        }
        if (!done) record_any(i, s, nt, xy, tri, inc, given, perm, w, rep);
        nfree += (w[0] & kMetaFixed) ? 0u : 1u;
    }
    nfree = __reduce_add_sync(0xffffffffu, nfree);
    if ((threadIdx.x & 31) == 0 && nfree) atomicAdd(rep + kFree, (unsigned long long)nfree);
}

__global__ void node_pass1_kernel(int64_t n, const double2 *__restrict__ xy, const int32_t *__restrict__ tri,
                                  const unsigned *__restrict__ ptr, int32_t *inc, const uint8_t *boundary,
                                  const uint32_t *perm, int32_t *nbtmp, unsigned *words, uint8_t *fixed_out,
                                  unsigned *deg_out, unsigned long long *rep)
{
    unsigned nfree = 0u;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned s = ptr[i], e = ptr[i + 1], nt = e - s;
        if (nt > (unsigned)kMaxInc) {
            atomicOr(rep + kFlags, (unsigned long long)kErrTooMany);
            words[i] = 1u;
            fixed_out[i] = 1;
            deg_out[i] = 0u;
            continue;
        }
        int32_t tl[kMaxInc];
        for (unsigned k = 0; k < nt; ++k) {
            const int32_t t = inc[s + k];
            unsigned j = k;
            while (j > 0 && tl[j - 1] > t) {
                tl[j] = tl[j - 1];
                --j;
            }
            tl[j] = t;
        }
        for (unsigned k = 0; k < nt; ++k) inc[s + k] = tl[k];
        // the other two vertices of every incident triangle, sorted by id
        int32_t rec[2 * kMaxInc];
        unsigned r = 0;
        for (unsigned k = 0; k < nt; ++k) {
            for (int c = 0; c < 3; ++c) {
                const int32_t v = tri[3 * (int64_t)tl[k] + c];
                if (v == (int32_t)i) continue;
                unsigned j = r++;
                while (j > 0 && rec[j - 1] > v) {
                    rec[j] = rec[j - 1];
                    --j;
                }
                rec[j] = v;
            }
        }
        bool open_edge = r == 0;
        unsigned deg = 0;
        int32_t uq[2 * kMaxInc];
        for (unsigned k = 0; k < r;) {
            unsigned f = k;
            while (f < r && rec[f] == rec[k]) ++f;
            const unsigned times = f - k;
            if (times == 1u) open_edge = true;
            if (times > 2u) atomicOr(rep + kFlags, (unsigned long long)kErrManifold);
            uq[deg++] = rec[k];
            k = f;
        }
        // summation order: ascending (x, y, id) of the creation coordinates
        double ux[2 * kMaxInc], uy[2 * kMaxInc];
        for (unsigned k = 0; k < deg; ++k) {
            const double2 p = xy[uq[k]];
            const int32_t id = uq[k];
            unsigned j = k;
            while (j > 0 && canon_less(p.x, p.y, id, ux[j - 1], uy[j - 1], uq[j - 1], perm)) {
                ux[j] = ux[j - 1];
                uy[j] = uy[j - 1];
                uq[j] = uq[j - 1];
                --j;
            }
            ux[j] = p.x;
            uy[j] = p.y;
            uq[j] = id;
        }
        for (unsigned k = 0; k < deg; ++k) nbtmp[2ull * s + k] = uq[k];
        const bool fx = boundary ? (boundary[perm ? perm[i] : i] != 0 || r == 0) : open_edge;
        fixed_out[i] = fx ? 1 : 0;
        deg_out[i] = deg;
        words[i] = fx ? 1u : 1u + deg + nt;
        nfree += fx ? 0u : 1u;
    }
    nfree = __reduce_add_sync(0xffffffffu, nfree);
    if ((threadIdx.x & 31) == 0 && nfree) atomicAdd(rep + kFree, (unsigned long long)nfree);
}

__global__ void node_pass2_kernel(int64_t n, const int32_t *__restrict__ tri, const unsigned *__restrict__ ptr,
                                  const int32_t *__restrict__ inc, const int32_t *__restrict__ nbtmp,
                                  const unsigned *__restrict__ deg_in, const uint8_t *__restrict__ fixed_in,
                                  const uint32_t *__restrict__ node_off, uint32_t *adj)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        uint32_t *w = adj + node_off[i];
        if (fixed_in[i]) {
            w[0] = 0x80000000u;
            continue;
        }
        const unsigned s = ptr[i], nt = ptr[i + 1] - s, deg = deg_in[i];
        w[0] = (nt << 16) | deg;
        const int32_t *list = nbtmp + 2ull * s;
        for (unsigned k = 0; k < deg; ++k) w[1 + k] = (uint32_t)list[k];
        for (unsigned k = 0; k < nt; ++k) {
            const int32_t *v = tri + 3 * (int64_t)inc[s + k];
            uint32_t slot = 0, pos[2] = {0u, 0u}, np = 0;
            for (int c = 0; c < 3; ++c) {
                if (v[c] == (int32_t)i) {
                    slot = (uint32_t)c;
                    continue;
                }
                uint32_t p = 0;
                while (p + 1 < deg && list[p] != v[c]) ++p;
                pos[np++] = p;
            }
            w[1 + deg + k] = (slot << 30) | (pos[0] << 15) | pos[1];
        }
    }
}

// Exclusive scan of cnt[0..len) into out[0..len] (out[len] = total), in three
// steps: per-block sums, a single-block scan of those sums, per-block scans.
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;  // per thread

__global__ void scan_sums_kernel(const unsigned *__restrict__ in, int64_t len, unsigned long long *sums)
{
    __shared__ unsigned long long s[32];
    const int64_t base = (int64_t)blockIdx.x * kScanBlock * kScanItems;
    unsigned long long acc = 0ull;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t j = base + (int64_t)k * kScanBlock + threadIdx.x;
        if (j < len) acc += in[j];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = s[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) sums[blockIdx.x] = acc;
    }
}

// One block: exclusive scan of the block sums, the total after them.
__global__ void __launch_bounds__(1024) scan_offsets_kernel(unsigned long long *sums, int64_t nblocks)
{
    __shared__ unsigned long long s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long carry = 0ull;
    for (int64_t b0 = 0; b0 < nblocks; b0 += 1024) {
        const int64_t b = b0 + threadIdx.x;
        const unsigned long long v = b < nblocks ? sums[b] : 0ull;
        unsigned long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        unsigned long long t = s_warp[lane];  // every warp scans the 32 sums itself
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        const unsigned long long before = warp ? __shfl_sync(0xffffffffu, t, warp - 1) : 0ull;
        if (b < nblocks) sums[b] = carry + before + x - v;
        carry += __shfl_sync(0xffffffffu, t, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nblocks] = carry;
}

__global__ void scan_final_kernel(const unsigned *__restrict__ in, int64_t len,
                                  const unsigned long long *__restrict__ offs, uint32_t *out)
{
    __shared__ unsigned long long warp_tot[32];
    __shared__ unsigned long long carry;
    const int64_t base = (int64_t)blockIdx.x * kScanBlock * kScanItems;
    if (threadIdx.x == 0) carry = offs[blockIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t j = base + (int64_t)k * kScanBlock + threadIdx.x;
        const unsigned long long v = j < len ? in[j] : 0ull;
        unsigned long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[warp] = x;
        __syncthreads();
        if (warp == 0) {
            unsigned long long t = warp_tot[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            warp_tot[lane] = t;  // inclusive over warps
        }
        __syncthreads();
        const unsigned long long before = carry + (warp ? warp_tot[warp - 1] : 0ull) + x - v;
        if (j < len) out[j] = (uint32_t)before;
        __syncthreads();
        if (threadIdx.x == 0) carry += warp_tot[31];
        __syncthreads();
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[len] = (uint32_t)offs[gridDim.x];
}

// A device buffer of the build, from the library's pool on stream s (memory
// comes and goes in stream order, so no call waits for the whole device).
struct DevBuf {
    void *p = nullptr;
    cudaStream_t s = nullptr;
    ~DevBuf() { pool_free(p, s); }
};

struct Alloc {
    cudaStream_t s;
};

cudaError_t raw_alloc(const Alloc &a, void **p, size_t bytes) { return pool_alloc(p, bytes, a.s); }

#define GB_TRY(expr, what)                                  \
    do {                                                    \
        cudaError_t e_ = (expr);                            \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

template <class T>
sls_status dalloc(DevBuf &b, size_t count, T **out, const char *what, const Alloc &a)
{
    b.s = a.s;
    cudaError_t e = raw_alloc(a, &b.p, sizeof(T) * (count > 0 ? count : 1));
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(SLS_ERR_OOM, std::string("device allocation failed: ") + what);
    }
    if (e != cudaSuccess) return cuda_fail(e, what);
    *out = static_cast<T *>(b.p);
    return SLS_OK;
}

// Scan of len uint32 values into len+1 offsets on stream s; total (may be
// NULL) receives the sum once the stream has been synchronised.
sls_status scan_async(const unsigned *in, int64_t len, uint32_t *out, unsigned long long *total, const Alloc &al)
{
    const int64_t per_block = (int64_t)kScanBlock * kScanItems;
    const int64_t nblocks = (len + per_block - 1) / per_block;
    DevBuf sb;
    unsigned long long *sums = nullptr;
    sls_status st = dalloc(sb, (size_t)nblocks + 1, &sums, "scan", al);
    if (st != SLS_OK) return st;
    if (nblocks > 0) {
        scan_sums_kernel<<<(unsigned)nblocks, kScanBlock, 0, al.s>>>(in, len, sums);
        scan_offsets_kernel<<<1, 1024, 0, al.s>>>(sums, nblocks);
        scan_final_kernel<<<(unsigned)nblocks, kScanBlock, 0, al.s>>>(in, len, sums, out);
        GB_TRY(cudaGetLastError(), "scan");
        if (total)
            GB_TRY(cudaMemcpyAsync(total, sums + nblocks, sizeof *total, cudaMemcpyDeviceToHost, al.s), "scan total");
    } else {
        GB_TRY(cudaMemsetAsync(out, 0, sizeof(uint32_t), al.s), "scan");
        if (total) *total = 0ull;
    }
    return SLS_OK;
}

// The same, waiting for the total.
sls_status scan_u32(const unsigned *in, int64_t len, uint32_t *out, unsigned long long *total, cudaStream_t s)
{
    sls_status st = scan_async(in, len, out, total, Alloc{s});
    if (st != SLS_OK) return st;
    GB_TRY(cudaStreamSynchronize(s), "scan");
    return SLS_OK;
}

// One block of kOrderTile threads per tile: the number of free nodes (of
// colour c, when colour is given).
__global__ void __launch_bounds__(kOrderTile) order_count_kernel(const uint32_t *__restrict__ node_off,
                                                                  const uint32_t *__restrict__ adj, int64_t n,
                                                                  const int32_t *__restrict__ colour, int32_t c,
                                                                  unsigned *cnt)
{
    const int64_t i = (int64_t)blockIdx.x * kOrderTile + threadIdx.x;
    const bool fr = i < n && !(adj[node_off[i]] & 0x80000000u) && (!colour || colour[i] == c);
    const int k = __syncthreads_count(fr);
    if (threadIdx.x == 0) cnt[blockIdx.x] = (unsigned)k;
}

// One block of kOrderTile threads per tile: the tile's free nodes of the
// class in id order (a bitonic sort of the members' ids in shared memory,
// non-members sorting last), written at the tile's offset.
__global__ void __launch_bounds__(kOrderTile) order_sort_kernel(const uint32_t *__restrict__ node_off,
                                                                 const uint32_t *__restrict__ adj, int64_t n,
                                                                 const int32_t *__restrict__ colour, int32_t c,
                                                                 const uint32_t *__restrict__ tile_off,
                                                                 uint32_t *order)
{
    __shared__ uint32_t key[kOrderTile];
    const unsigned tid = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * kOrderTile + tid;
    uint32_t k = 0xffffffffu;  // fixed nodes and the tail sort last
    if (i < n) {
        const uint32_t meta = adj[node_off[i]];
        if (!(meta & 0x80000000u) && (!colour || colour[i] == c))
            k = tid;
    }
    key[tid] = k;
    __syncthreads();
    for (unsigned size = 2; size <= (unsigned)kOrderTile; size <<= 1) {
        for (unsigned stride = size >> 1; stride > 0; stride >>= 1) {
            const unsigned j = tid ^ stride;
            if (j > tid) {
                const uint32_t a = key[tid], b = key[j];
                const bool up = (tid & size) == 0;
                if ((a > b) == up) {
                    key[tid] = b;
                    key[j] = a;
                }
            }
            __syncthreads();
        }
    }
    const uint32_t nf = tile_off[blockIdx.x + 1] - tile_off[blockIdx.x];
    if (tid < nf) order[tile_off[blockIdx.x] + tid] = (uint32_t)(blockIdx.x * kOrderTile) + (key[tid] & 1023u);
}

// splitmix64 (Steele, Lea and Flood, OOPSLA 2014): the colouring priorities.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x)
{
    unsigned long long z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Initial colouring state: -2 fixed, -1 free and uncoloured.
__global__ void colour_init_kernel(const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ adj,
                                   int64_t n, int32_t *colour)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        colour[i] = (adj[node_off[i]] & 0x80000000u) ? -2 : -1;
}

// One Jones-Plassmann round.  cur is the state at the start of the round,
// next a copy of it that receives the winners' colours: an uncoloured free
// node wins when its (priority, index) exceeds that of every uncoloured free
// neighbour, and takes the smallest colour no neighbour holds.  Winners are
// never neighbours, so the round's result does not depend on thread order.
__global__ void colour_round_kernel(const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ adj,
                                    int64_t n, unsigned long long seed, const int32_t *__restrict__ cur,
                                    int32_t *next, unsigned long long *left, unsigned *flags)
{
    unsigned long long cnt = 0ull;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        if (cur[i] != -1) continue;
        const uint32_t *w = adj + node_off[i];
        const uint32_t deg = w[0] & 0xffffu;
        const unsigned long long pi = splitmix64(seed + (unsigned long long)i);
        bool win = true;
        unsigned long long used = 0ull;
        for (uint32_t k = 0; k < deg; ++k) {
            const uint32_t j = w[1 + k];
            const int32_t cj = cur[j];
            if (cj == -1) {
                const unsigned long long pj = splitmix64(seed + (unsigned long long)j);
                if (!(pi > pj || (pi == pj && (uint32_t)i > j))) win = false;
            } else if (cj >= 0) {
                if (cj < 64) used |= 1ull << cj;
                else atomicOr(flags, 1u);
            }
        }
        if (win) {
            if (used == ~0ull) atomicOr(flags, 1u);  // would need a colour past 63
            next[i] = __ffsll((long long)~used) - 1;
        } else {
            cnt += 1ull;
        }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(left, cnt);
}

__global__ void colour_max_kernel(const int32_t *__restrict__ colour, int64_t n, int *cmax)
{
    int m = -1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        m = max(m, colour[i]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(cmax, m);
}

// Unchanged-tile skipping: for tile t (nodes 32t .. 32t+31), the tiles that
// hold its nodes and the neighbours of its free nodes, each with the mask of
// those nodes; (kHaloNever, 0) when more than kHaloEntries tiles are involved
// (such a tile is always computed).  *skippable counts the others.  One thread per
// tile.
__global__ void tile_halo_kernel(const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ adj,
                                 int64_t n, int64_t ntiles, uint2 *halo, unsigned *skippable)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntiles) return;
    uint32_t ids[kHaloEntries], masks[kHaloEntries];
    int cnt = 1;
    ids[0] = (uint32_t)t;
    masks[0] = 0xffffffffu;
    bool over = false;
    for (int l = 0; l < 32 && !over; ++l) {
        const int64_t i = t * 32 + l;
        if (i >= n) break;
        const uint32_t off = node_off[i], meta = adj[off];
        if (meta & kMetaFixed) continue;
        const uint32_t deg = meta_degree(meta);
        for (uint32_t k = 0; k < deg; ++k) {
            const uint32_t j = adj[off + 1 + k];
            const uint32_t tj = j >> 5;
            int e = 0;
            while (e < cnt && ids[e] != tj) ++e;
            if (e == cnt) {
                if (cnt == kHaloEntries) {
                    over = true;
                    break;
                }
                ids[cnt] = tj;
                masks[cnt] = 0u;
                ++cnt;
            }
            masks[e] |= 1u << (j & 31);
        }
    }
    if (!over) atomicAdd(skippable, 1u);
    uint2 *h = halo + t * kHaloEntries;
    for (int e = 0; e < kHaloEntries; ++e)
        h[e] = over ? make_uint2(e == 0 ? kHaloNever : 0u, 0u)
                    : (e < cnt ? make_uint2(ids[e], masks[e]) : make_uint2(0u, 0u));
}

}  // namespace

sls_status build_tile_halo(sls_mesh *M, cudaStream_t s)
{
    if (!M->opt.skip_unchanged) return SLS_OK;
    const int64_t nt = (M->n + 31) / 32;
    GB_TRY(pool_alloc((void **)&M->halo, sizeof(uint2) * (size_t)kHaloEntries * (size_t)nt, s), "tile halo");
    for (int k = 0; k < 2; ++k) GB_TRY(pool_alloc((void **)&M->chg[k], sizeof(uint32_t) * (size_t)nt, s), "tile masks");
    GB_TRY(pool_alloc((void **)&M->accm, sizeof(uint32_t) * (size_t)nt, s), "tile masks");
    for (int k = 0; k < 2; ++k) GB_TRY(cudaMemsetAsync(M->chg[k], 0xff, sizeof(uint32_t) * (size_t)nt, s), "tile masks");
    GB_TRY(cudaMemsetAsync(M->accm, 0, sizeof(uint32_t) * (size_t)nt, s), "tile masks");
    DevBuf b_cnt;
    unsigned *cnt = nullptr, skippable = 0u;
    sls_status st = dalloc(b_cnt, 1, &cnt, "tile halo", Alloc{s});
    if (st != SLS_OK) return st;
    GB_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned), s), "tile halo");
    tile_halo_kernel<<<(unsigned)((nt + 127) / 128), 128, 0, s>>>(M->node_off, M->adj, M->n, nt, M->halo, cnt);
    GB_TRY(cudaGetLastError(), "tile halo");
    GB_TRY(cudaMemcpyAsync(&skippable, cnt, sizeof skippable, cudaMemcpyDeviceToHost, s), "tile halo");
    GB_TRY(cudaStreamSynchronize(s), "tile halo");
    if (skippable == 0u) {
        // a numbering so far from local that no tile can ever be skipped: the
        // passes without the masks, which also start early (random ids, 1009 x 701
        // nodes: 66.5 us a pass against 77.1, SoA 84.4 against 98.9)
        for (void *p : {(void *)M->halo, (void *)M->chg[0], (void *)M->chg[1], (void *)M->accm}) pool_free(p, s);
        M->halo = nullptr;
        M->chg[0] = M->chg[1] = M->accm = nullptr;
    }
    return SLS_OK;
}

namespace {

// One segment of the processing order: the free nodes of colour c (all free
// nodes when colour is null), in id order.
sls_status order_segment(sls_mesh *M, const int32_t *colour, int32_t c, uint32_t *dst, int64_t expect,
                         int64_t *count, cudaStream_t s)
{
    const int64_t n = M->n;
    const int64_t tiles = (n + kOrderTile - 1) / kOrderTile;
    DevBuf b_cnt, b_off;
    unsigned *cnt = nullptr;
    uint32_t *off = nullptr;
    sls_status st;
    if ((st = dalloc(b_cnt, (size_t)tiles, &cnt, "order counts", Alloc{s})) != SLS_OK) return st;
    if ((st = dalloc(b_off, (size_t)tiles + 1, &off, "order offsets", Alloc{s})) != SLS_OK) return st;
    order_count_kernel<<<(unsigned)tiles, kOrderTile, 0, s>>>(M->node_off, M->adj, n, colour, c, cnt);
    GB_TRY(cudaGetLastError(), "order count");
    unsigned long long total = 0ull;
    if ((st = scan_u32(cnt, tiles, off, &total, s)) != SLS_OK) return st;
    if (expect >= 0 && (int64_t)total > expect) return fail(SLS_ERR_INVALID, "processing order overflow");
    if (total > 0) {
        order_sort_kernel<<<(unsigned)tiles, kOrderTile, 0, s>>>(M->node_off, M->adj, n, colour, c, off, dst);
        GB_TRY(cudaGetLastError(), "order sort");
    }
    GB_TRY(cudaStreamSynchronize(s), "processing order");
    *count = (int64_t)total;
    return SLS_OK;
}

}  // namespace

namespace {

// ---- renumbering: Form B lists every colour class as a contiguous id range

__global__ void fixed_flag_kernel(const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ adj, int64_t n,
                                  unsigned *flag)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        flag[i] = (__ldg(adj + __ldg(node_off + i)) & kMetaFixed) ? 1u : 0u;
}

// perm[base + scan[i]] = i for the flagged nodes, in id order.
__global__ void compact_kernel(const unsigned *__restrict__ flag, const uint32_t *__restrict__ scan, int64_t n,
                               int64_t base, uint32_t *perm)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        if (flag[i]) perm[base + scan[i]] = (uint32_t)i;
}

__global__ void inverse_kernel(const uint32_t *__restrict__ perm, int64_t n, uint32_t *inv)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) inv[perm[k]] = (uint32_t)k;
}

__global__ void record_len_kernel(const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ perm, int64_t n,
                                  unsigned *len)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        const uint32_t i = perm[k];
        len[k] = node_off[i + 1] - node_off[i];
    }
}

// The record of new node k is the record of old node perm[k] with its
// neighbour ids renumbered; the meta word and the triangle codes (positions
// in the neighbour list, whose order is kept) are copied as they are.
__global__ void remap_adj_kernel(const uint32_t *__restrict__ off_old, const uint32_t *__restrict__ adj_old,
                                 const uint32_t *__restrict__ perm, const uint32_t *__restrict__ inv,
                                 const uint32_t *__restrict__ off_new, int64_t n, uint32_t *__restrict__ adj_new)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        const uint32_t *src = adj_old + off_old[perm[k]];
        uint32_t *dst = adj_new + off_new[k];
        const uint32_t meta = src[0];
        dst[0] = meta;
        if (meta & kMetaFixed) continue;
        const uint32_t deg = meta & 0xffffu, ntri = (meta >> 16) & 0x7fffu;
        for (uint32_t w = 1; w <= deg; ++w) dst[w] = inv[src[w]];
        for (uint32_t w = deg + 1; w <= deg + ntri; ++w) dst[w] = src[w];
    }
}

__global__ void remap_ids_kernel(int32_t *ids, int64_t count, const uint32_t *__restrict__ inv)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += stride)
        ids[t] = (int32_t)inv[ids[t]];
}

}  // namespace

// Renumbers the mesh by M->perm (new id -> caller's id, a permutation of
// [0, n) already on the device): fills M->inv and replaces the adjacency (the
// records in the new order, neighbour ids renumbered, each list's order
// kept, so every pass sums and tests exactly as before), the triangles and
// both coordinate arrays (which hold the creation coordinates).
static sls_status apply_renumbering(sls_mesh *M, cudaStream_t s)
{
    const int64_t n = M->n;
    const int grid = device_sm_count() * 8, block = 256;
    GB_TRY(pool_alloc((void **)&M->inv, sizeof(uint32_t) * (size_t)n, s), "renumbering");
    DevBuf b_len, b_off, b_adj;
    unsigned *len = nullptr;
    uint32_t *off_new = nullptr, *adj_new = nullptr;
    sls_status st;
    if ((st = dalloc(b_len, (size_t)n + 1, &len, "renumbering", Alloc{s})) != SLS_OK) return st;
    inverse_kernel<<<grid, block, 0, s>>>(M->perm, n, M->inv);
    record_len_kernel<<<grid, block, 0, s>>>(M->node_off, M->perm, n, len);
    GB_TRY(cudaGetLastError(), "renumbering");
    if ((st = dalloc(b_off, (size_t)n + 1, &off_new, "renumbering", Alloc{s})) != SLS_OK) return st;
    unsigned long long words = 0ull;
    if ((st = scan_u32(len, n, off_new, &words, s)) != SLS_OK) return st;
    if (words != M->adj_words) return fail(SLS_ERR_INVALID, "adjacency size mismatch in the renumbering");
    if ((st = dalloc(b_adj, (size_t)words, &adj_new, "renumbering", Alloc{s})) != SLS_OK) return st;
    remap_adj_kernel<<<grid, block, 0, s>>>(M->node_off, M->adj, M->perm, M->inv, off_new, n, adj_new);
    remap_ids_kernel<<<grid, block, 0, s>>>(M->tri, 3 * M->m, M->inv);
    GB_TRY(cudaGetLastError(), "renumbering");
    GB_TRY(launch_permute_coords(M->xy[0], M->xy[1], M->opt.layout, M->f32, n, M->perm, grid, s), "renumbering");
    GB_TRY(cudaMemcpyAsync(M->xy[0], M->xy[1], (M->f32 ? sizeof(float) : sizeof(double)) * 2 * (size_t)n,
                           cudaMemcpyDeviceToDevice, s), "renumbering");
    GB_TRY(cudaStreamSynchronize(s), "renumbering");
    pool_free(M->node_off, s);
    pool_free(M->adj, s);
    M->node_off = off_new;
    M->adj = adj_new;
    b_off.p = nullptr;  // now the mesh's
    b_adj.p = nullptr;
    return SLS_OK;
}

// Form B: renumbers the mesh so that every colour class is a contiguous id
// range (the classes in order, each in its old id order, then the fixed
// nodes in id order): a sweep then reads and writes each class's nodes
// contiguously.  The colouring was computed on the caller's numbering, and
// the neighbour lists keep their order (only the ids change), so every pass
// computes what it computed before.  Fills M->perm (new -> caller's id) and
// M->inv; replaces the adjacency, the triangles and both coordinate arrays.
sls_status renumber_classes(sls_mesh *M, cudaStream_t s)
{
    const int64_t n = M->n;
    const int grid = device_sm_count() * 8, block = 256;
    GB_TRY(pool_alloc((void **)&M->perm, sizeof(uint32_t) * (size_t)n, s), "renumbering");
    // the free nodes by class: the processing order already lists them so
    if (M->n_free > 0)
        GB_TRY(cudaMemcpyAsync(M->perm, M->node_order, sizeof(uint32_t) * (size_t)M->n_free,
                               cudaMemcpyDeviceToDevice, s), "renumbering");
    DevBuf b_flag, b_scan;
    unsigned *flag = nullptr;
    uint32_t *scan = nullptr;
    sls_status st;
    if ((st = dalloc(b_flag, (size_t)n + 1, &flag, "renumbering", Alloc{s})) != SLS_OK) return st;
    if ((st = dalloc(b_scan, (size_t)n + 1, &scan, "renumbering", Alloc{s})) != SLS_OK) return st;
    fixed_flag_kernel<<<grid, block, 0, s>>>(M->node_off, M->adj, n, flag);
    GB_TRY(cudaGetLastError(), "renumbering");
    unsigned long long nfixed = 0ull;
    if ((st = scan_u32(flag, n, scan, &nfixed, s)) != SLS_OK) return st;
    if ((int64_t)nfixed + M->n_free != n) return fail(SLS_ERR_INVALID, "node count mismatch in the renumbering");
    compact_kernel<<<grid, block, 0, s>>>(flag, scan, n, M->n_free, M->perm);
    GB_TRY(cudaGetLastError(), "renumbering");
    if ((st = apply_renumbering(M, s)) != SLS_OK) return st;
    pool_free(M->node_order, s);
    M->node_order = nullptr;
    return SLS_OK;
}

sls_status build_node_order(sls_mesh *M, cudaStream_t s)
{
    // Form A visits every node in index order: no list needed
    if (M->opt.form != 1) return SLS_OK;
    GB_TRY(pool_alloc((void **)&M->node_order, sizeof(uint32_t) * (size_t)(M->n_free > 0 ? M->n_free : 1), s),
           "processing order");
    // Form B: Jones-Plassmann colouring, then one order segment per colour
    const int64_t n = M->n;
    DevBuf b_col[2], b_cnt;
    int32_t *col[2] = {nullptr, nullptr};
    unsigned long long *cnt = nullptr;
    sls_status st;
    for (int k = 0; k < 2; ++k)
        if ((st = dalloc(b_col[k], (size_t)n, &col[k], "colours", Alloc{s})) != SLS_OK) return st;
    if ((st = dalloc(b_cnt, 2, &cnt, "colouring counters", Alloc{s})) != SLS_OK) return st;
    const int grid = device_sm_count() * 8, block = 256;
    colour_init_kernel<<<grid, block, 0, s>>>(M->node_off, M->adj, n, col[0]);
    GB_TRY(cudaGetLastError(), "colouring");
    int cur = 0;
    unsigned long long h[2] = {0ull, 0ull};
    for (int round = 0;; ++round) {
        if (round > 100000) return fail(SLS_ERR_INVALID, "colouring did not finish");
        GB_TRY(cudaMemcpyAsync(col[cur ^ 1], col[cur], sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s),
               "colouring");
        GB_TRY(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), s), "colouring");
        colour_round_kernel<<<grid, block, 0, s>>>(M->node_off, M->adj, n, kColourSeed, col[cur], col[cur ^ 1], cnt,
                                                   reinterpret_cast<unsigned *>(cnt + 1));
        GB_TRY(cudaGetLastError(), "colouring round");
        GB_TRY(cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, s), "colouring");
        GB_TRY(cudaStreamSynchronize(s), "colouring");
        cur ^= 1;
        if (h[1]) return fail(SLS_ERR_INVALID, "the coloured form needs more than 64 colours");
        if (h[0] == 0ull) break;
    }
    int *cmax = reinterpret_cast<int *>(cnt);
    GB_TRY(cudaMemsetAsync(cmax, 0xff, sizeof(int), s), "colouring");
    colour_max_kernel<<<grid, block, 0, s>>>(col[cur], n, cmax);
    int hmax = -1;
    GB_TRY(cudaMemcpyAsync(&hmax, cmax, sizeof hmax, cudaMemcpyDeviceToHost, s), "colouring");
    GB_TRY(cudaStreamSynchronize(s), "colouring");
    const int nc = hmax + 1;
    M->colour_off.assign((size_t)nc + 1, 0);
    int64_t at = 0;
    for (int c = 0; c < nc; ++c) {
        int64_t k = 0;
        if ((st = order_segment(M, col[cur], c, M->node_order + at, M->n_free - at, &k, s)) != SLS_OK) return st;
        at += k;
        M->colour_off[(size_t)c + 1] = at;
    }
    if (at != M->n_free) return fail(SLS_ERR_INVALID, "free-node count mismatch in the colouring");
    return renumber_classes(M, s);
}

namespace {

double unkey(unsigned long long k)
{
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    double v;
    std::memcpy(&v, &b, sizeof v);
    return v;
}

// Blocks of `block` threads for `count` items, at most what fills the GPU.
unsigned blocks_for(int64_t count, int block)
{
    const int64_t cap = (int64_t)device_sm_count() * 8, need = (count + block - 1) / block;
    return (unsigned)(need < 1 ? 1 : (need < cap ? need : cap));
}

// Renumbers the triangles and coordinates along the Z-order curve (see
// CellGrid above); perm (new id -> old) and inv are allocated for the caller.
sls_status number_spatially(int64_t n, int64_t m, double *d_xy, int32_t *d_tri, const unsigned long long *box,
                            cudaStream_t s, DevBuf &b_perm, DevBuf &b_inv)
{
    const int block = 256;
    const unsigned grid = blocks_for(n, block);
    const Alloc al{s};
    const double x0 = unkey(box[0]), y0 = unkey(box[1]), w = unkey(box[2]) - x0, h = unkey(box[3]) - y0;
    // square cells over the box's larger side, between one and four per node
    const double big = w > h ? w : h;
    int bits = 1;
    while (bits < 13 && (int64_t(1) << (2 * bits)) <= n) ++bits;
    const CellGrid g{x0, y0, big > 0.0 ? (double)(1u << bits) / big : 0.0, 1u << bits};
    const int64_t ncell = int64_t(1) << (2 * bits);
    DevBuf b_cnt, b_off, b_xy;
    unsigned *cnt = nullptr;
    uint32_t *off = nullptr, *perm = nullptr, *inv = nullptr;
    double2 *xy2 = nullptr;
    sls_status st;
    if ((st = dalloc(b_cnt, (size_t)ncell, &cnt, "numbering", al)) != SLS_OK) return st;
    if ((st = dalloc(b_off, (size_t)ncell + 1, &off, "numbering", al)) != SLS_OK) return st;
    if ((st = dalloc(b_perm, (size_t)n, &perm, "numbering", al)) != SLS_OK) return st;
    if ((st = dalloc(b_inv, (size_t)n, &inv, "numbering", al)) != SLS_OK) return st;
    if ((st = dalloc(b_xy, (size_t)n, &xy2, "numbering", al)) != SLS_OK) return st;
    GB_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned) * (size_t)ncell, s), "numbering");
    const double2 *xy = reinterpret_cast<const double2 *>(d_xy);
    cell_count_kernel<<<grid, block, 0, s>>>(xy, n, g, cnt);
    GB_TRY(cudaGetLastError(), "numbering");
    if ((st = scan_async(cnt, ncell, off, nullptr, al)) != SLS_OK) return st;
    cell_place_kernel<<<grid, block, 0, s>>>(xy, n, g, off, cnt, perm, inv, xy2);
    remap_ids_kernel<<<blocks_for(3 * m, block), block, 0, s>>>(d_tri, 3 * m, inv);
    GB_TRY(cudaGetLastError(), "numbering");
    GB_TRY(cudaMemcpyAsync(d_xy, xy2, sizeof(double2) * (size_t)n, cudaMemcpyDeviceToDevice, s), "numbering");
    return SLS_OK;
}

// Meshes below this keep the caller's numbering (their passes are bound by
// latency, not by what they gather).
constexpr int64_t kSpatialMin = 8192;

}  // namespace

// Builds the adjacency of a mesh whose coordinates (AoS) and triangles are
// already on the device.  With `renumber`, a mesh whose numbering is not local
// is first renumbered (d_xy and d_tri are changed then, and out.perm / out.inv
// set).  On success out holds the node offsets and the adjacency words (the
// caller owns them), the free-node count and D.  Returns SLS_ERR_NOT_FOUND
// (with nothing allocated, but perhaps d_xy and d_tri renumbered) when a node
// has more incident triangles than the device build handles, so the caller can
// use the host build instead.  Synchronises only stream s.
sls_status build_device_adjacency(int64_t n, int64_t m, double *d_xy, int32_t *d_tri, const uint8_t *h_boundary,
                                  bool renumber, cudaStream_t s, DeviceAdjacency &out)
{
    out = DeviceAdjacency{};
    if (3 * m >= (int64_t(1) << 32)) return SLS_ERR_NOT_FOUND;
    const int block = 256;
    const unsigned ngrid = blocks_for(n, block), tgrid = blocks_for(m, block), cgrid = blocks_for(3 * m, block);
    const Alloc al{s};

    DevBuf b_rep, b_cnt, b_ptr, b_inc, b_nbtmp, b_words, b_fixed, b_deg, b_bnd, b_off, b_adj, b_perm, b_inv;
    unsigned *cnt = nullptr, *words = nullptr, *deg = nullptr;
    uint32_t *ptr = nullptr;
    int32_t *inc = nullptr, *nbtmp = nullptr;
    uint8_t *fixed = nullptr, *bnd = nullptr;
    unsigned long long *rep = nullptr, h[kReport];
    sls_status st;
    if ((st = dalloc(b_rep, kReport, &rep, "build report", al)) != SLS_OK) return st;
    const double2 *xy2 = reinterpret_cast<const double2 *>(d_xy);
    report_init_kernel<<<1, 32, 0, s>>>(rep);
    validate_xy_kernel<<<ngrid, block, 0, s>>>(xy2, n, rep);
    validate_tri_kernel<<<tgrid, block, 0, s>>>(d_tri, m, n, rep);
    GB_TRY(cudaGetLastError(), "validate");
    GB_TRY(cudaMemcpyAsync(h, rep, sizeof h, cudaMemcpyDeviceToHost, s), "validate");
    GB_TRY(cudaStreamSynchronize(s), "validate");
    if (h[kFlags] & kErrFinite)
        return fail(SLS_ERR_INVALID, "coordinate " + std::to_string(h[kBadCoord]) + " is not finite");
    if (h[kFlags] & (kErrRange | kErrRepeat)) {
        const unsigned long long t = h[kBadTri] >> 1;
        return fail(SLS_ERR_INVALID, "triangle " + std::to_string(t) +
                                         ((h[kBadTri] & 1ull) ? " repeats a vertex" : " has a vertex id out of range"));
    }
    const double xmin = unkey(h[kBox]), ymin = unkey(h[kBox + 1]), xmax = unkey(h[kBox + 2]), ymax = unkey(h[kBox + 3]);
    out.diag = bbox_diagonal(xmin, xmax, ymin, ymax);
    // 45%: Morton order has a quarter of its edges across windows, the rows of
    // a grid two thirds
    renumber = renumber && n >= kSpatialMin && (double)h[kCrossing] > 0.45 * 3.0 * (double)m;
    if (renumber && (st = number_spatially(n, m, d_xy, d_tri, h + kBox, s, b_perm, b_inv)) != SLS_OK) return st;
    const uint32_t *perm = static_cast<const uint32_t *>(b_perm.p);

    if ((st = dalloc(b_cnt, (size_t)n + 1, &cnt, "incidence counts", al)) != SLS_OK) return st;
    if ((st = dalloc(b_ptr, (size_t)n + 1, &ptr, "incidence offsets", al)) != SLS_OK) return st;
    if ((st = dalloc(b_inc, (size_t)(3 * m), &inc, "incidences", al)) != SLS_OK) return st;
    GB_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned) * (n + 1), s), "build");
    count_kernel<<<cgrid, block, 0, s>>>(d_tri, 3 * m, cnt);
    GB_TRY(cudaGetLastError(), "count");
    if ((st = scan_async(cnt, n, ptr, nullptr, al)) != SLS_OK) return st;
    GB_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned) * (n + 1), s), "build");
    scatter_kernel<<<cgrid, block, 0, s>>>(d_tri, 3 * m, ptr, cnt, inc);
    GB_TRY(cudaGetLastError(), "scatter");

    if (h_boundary) {
        if ((st = dalloc(b_bnd, (size_t)n, &bnd, "boundary flags", al)) != SLS_OK) return st;
        GB_TRY(cudaMemcpyAsync(bnd, h_boundary, (size_t)n, cudaMemcpyHostToDevice, s), "upload flags");
    }
    uint32_t *node_off = nullptr, *adj = nullptr;
    if ((st = dalloc(b_off, (size_t)n + 1, &node_off, "node offsets", al)) != SLS_OK) return st;
    unsigned long long wtotal = 6ull * (unsigned long long)m + 2ull * (unsigned long long)n;
    bool exact = wtotal >= (1ull << 32);  // (exact lengths may still fit)
    if (!exact) {
        if ((st = dalloc(b_adj, (size_t)wtotal, &adj, "adjacency", al)) != SLS_OK) return st;
        node_records_kernel<<<blocks_for(n, 128), 128, 0, s>>>(n, xy2, d_tri, ptr, inc, bnd, perm, node_off, adj, rep);
        GB_TRY(cudaGetLastError(), "node records");
        GB_TRY(cudaMemcpyAsync(h, rep, sizeof h, cudaMemcpyDeviceToHost, s), "build");
        GB_TRY(cudaStreamSynchronize(s), "node records");
        exact = (h[kFlags] & kErrRoom) != 0u && !(h[kFlags] & (kErrManifold | kErrTooMany));
        if (exact) {
            pool_free(adj, s);
            b_adj.p = nullptr;
            GB_TRY(cudaMemsetAsync(rep + kFree, 0, sizeof(unsigned long long), s), "build");
        }
    }
    if (exact) {
        if ((st = dalloc(b_nbtmp, (size_t)(6 * m), &nbtmp, "neighbour scratch", al)) != SLS_OK) return st;
        if ((st = dalloc(b_words, (size_t)n + 1, &words, "word counts", al)) != SLS_OK) return st;
        if ((st = dalloc(b_fixed, (size_t)n, &fixed, "fixed flags", al)) != SLS_OK) return st;
        if ((st = dalloc(b_deg, (size_t)n, &deg, "degrees", al)) != SLS_OK) return st;
        node_pass1_kernel<<<ngrid, block, 0, s>>>(n, xy2, d_tri, ptr, inc, bnd, perm, nbtmp, words, fixed, deg, rep);
        GB_TRY(cudaGetLastError(), "node pass 1");
        if ((st = scan_async(words, n, node_off, &wtotal, al)) != SLS_OK) return st;
        GB_TRY(cudaMemcpyAsync(h, rep, sizeof h, cudaMemcpyDeviceToHost, s), "build");
        GB_TRY(cudaStreamSynchronize(s), "node pass 1");
    }
    if (h[kFlags] & kErrManifold) return fail(SLS_ERR_NONMANIFOLD, "an edge is shared by more than two triangles");
    if (h[kFlags] & kErrTooMany) return SLS_ERR_NOT_FOUND;
    if (exact) {
        if (wtotal >= (1ull << 32)) return fail(SLS_ERR_INVALID, "adjacency exceeds 2^32 words");
        if ((st = dalloc(b_adj, (size_t)wtotal, &adj, "adjacency", al)) != SLS_OK) return st;
        node_pass2_kernel<<<ngrid, block, 0, s>>>(n, d_tri, ptr, inc, nbtmp, deg, fixed, node_off, adj);
        GB_TRY(cudaGetLastError(), "node pass 2");
    }
    out.n_free = (int64_t)h[kFree];
    out.adj_words = wtotal;
    out.node_off = node_off;
    out.adj = adj;
    out.perm = static_cast<uint32_t *>(b_perm.p);
    out.inv = static_cast<uint32_t *>(b_inv.p);
    b_off.p = b_adj.p = b_perm.p = b_inv.p = nullptr;  // handed to the caller
    return SLS_OK;
}

sls_status build_device_mesh(sls_mesh *M, double *d_xy, int32_t *d_tri, const uint8_t *h_boundary, cudaStream_t s)
{
    DeviceAdjacency da;
    sls_status st = build_device_adjacency(M->n, M->m, d_xy, d_tri, h_boundary, numbers_spatially(M->opt), s, da);
    if (st != SLS_OK) return st;
    M->node_off = da.node_off;
    M->adj = da.adj;
    M->adj_words = da.adj_words;
    M->n_free = da.n_free;
    M->diag = da.diag;
    M->perm = da.perm;
    M->inv = da.inv;
    return SLS_OK;
}

}  // namespace sls
