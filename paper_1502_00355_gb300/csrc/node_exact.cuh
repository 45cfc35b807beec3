// node_exact.cuh -- the FP64 node update (Eq. 2 with the accept test of
// Section 3.3.4), as the plain FP64 kernel runs it.
#pragma once

#include "device.cuh"

namespace sls {

// Coordinates of node i; COHERENT: read from L2, for kernels in which other
// blocks write them.
template <int LAYOUT, bool COHERENT>
__device__ __forceinline__ double2 read_node(const double *p, int64_t n, int64_t i)
{
    if (!COHERENT) return Coords<LAYOUT>::get(p, n, i);
    if (LAYOUT == 0) return __ldcg(reinterpret_cast<const double2 *>(p) + i);
    return make_double2(__ldcg(p + i), __ldcg(p + n + i));
}

// alpha of incident triangle `code` of node i with node i placed at (x, y).
template <int LAYOUT>
__device__ __forceinline__ double alpha_with(const PassArgs &a, const uint32_t *nb, uint32_t code,
                                             double x, double y)
{
    const double2 A = Coords<LAYOUT>::get(a.in, a.n, __ldg(nb + code_first(code)));
    const double2 B = Coords<LAYOUT>::get(a.in, a.n, __ldg(nb + code_second(code)));
    return alpha_at_slot(code_slot(code), x, y, A.x, A.y, B.x, B.y);
}

// Decides the update of node i from its qualities and writes the node and its
// decision; returns the squared move bits (0 if not accepted), whether it was
// accepted and whether its coordinates changed.
template <int LAYOUT>
__device__ __forceinline__ void finish_exact(const PassArgs &a, int64_t i, double2 p, double2 c, double q_old,
                                             double q_new, unsigned long long &d2_bits, bool &accepted, bool &moved)
{
    const bool ok = a.strict ? (q_new > q_old) : (q_new >= q_old);
    double2 o = p;
    d2_bits = 0ull;
    moved = ok && (__double_as_longlong(c.x) != __double_as_longlong(p.x) ||
                   __double_as_longlong(c.y) != __double_as_longlong(p.y));
    if (ok) {
        const double dx = __dsub_rn(c.x, p.x), dy = __dsub_rn(c.y, p.y);
        const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
        d2_bits = (unsigned long long)__double_as_longlong(d2);
        o = c;
    }
    Coords<LAYOUT>::put(a.out, a.n, i, o);
    if (a.accept) a.accept[i] = ok ? 1 : 0;
    accepted = ok;
}

// Exact update of free node i, one thread: the neighbour sum in stored order,
// IEEE division, both qualities of every incident triangle.
template <int LAYOUT>
__device__ __forceinline__ void exact_update(const PassArgs &a, int64_t i, unsigned long long &d2_bits,
                                             bool &accepted, bool &moved)
{
    const uint32_t off = __ldg(a.node_off + i);
    const uint32_t meta = __ldg(a.adj + off);
    const uint32_t deg = meta_degree(meta), ntri = meta_ntri(meta);
    const uint32_t *nb = a.adj + off + 1;
    const double2 p = Coords<LAYOUT>::get(a.in, a.n, i);
    double2 s = Coords<LAYOUT>::get(a.in, a.n, __ldg(nb));
    for (uint32_t k = 1; k < deg; ++k) {
        const double2 v = Coords<LAYOUT>::get(a.in, a.n, __ldg(nb + k));
        s.x = __dadd_rn(s.x, v.x);
        s.y = __dadd_rn(s.y, v.y);
    }
    const double fd = (double)deg;
    const double2 c = make_double2(__ddiv_rn(s.x, fd), __ddiv_rn(s.y, fd));
    double q_old = 0.0, q_new = 0.0;
    for (uint32_t t = 0; t < ntri; ++t) {
        const uint32_t code = __ldg(nb + deg + t);
        const double qo = alpha_with<LAYOUT>(a, nb, code, p.x, p.y);
        const double qn = alpha_with<LAYOUT>(a, nb, code, c.x, c.y);
        if (t == 0 || qo < q_old) q_old = qo;
        if (t == 0 || qn < q_new) q_new = qn;
    }
    finish_exact<LAYOUT>(a, i, p, c, q_old, q_new, d2_bits, accepted, moved);
}

// The same update by a whole warp (every lane calls it with the same node):
// the neighbours are loaded 32 at a time and added in the stored order by
// every lane, the triangles are shared out over the lanes.  For nodes with
// long rings, whose one-thread update is a chain of dependent loads and FP64
// divisions (the few 14-rings of a 100,000-point Delaunay mesh held up its
// whole pass: 58 us).  Only lane 0's results count.
template <int LAYOUT, bool COHERENT>
__device__ __forceinline__ void exact_update_warp(const PassArgs &a, int64_t i, unsigned long long &d2_bits,
                                                  bool &accepted, bool &moved)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t off = __ldg(a.node_off + i);
    const double2 p = read_node<LAYOUT, COHERENT>(a.in, a.n, i);
    const uint32_t meta = __ldg(a.adj + off);
    const uint32_t deg = meta_degree(meta), ntri = meta_ntri(meta);
    const uint32_t *nb = a.adj + off + 1;
    const uint32_t code0 = lane < ntri ? __ldg(nb + deg + lane) : 0u;
    double2 v = make_double2(0.0, 0.0);  // the lane's neighbour of the last 32
    double2 s = make_double2(-0.0, -0.0);  // -0 + x == x
    for (uint32_t k0 = 0; k0 < deg; k0 += 32) {
        if (k0 + lane < deg) v = read_node<LAYOUT, COHERENT>(a.in, a.n, __ldg(nb + k0 + lane));
        const uint32_t m = deg - k0 < 32u ? deg - k0 : 32u;
        for (uint32_t k = 0; k < m; ++k) {
            s.x = __dadd_rn(s.x, __shfl_sync(0xffffffffu, v.x, (int)k));
            s.y = __dadd_rn(s.y, __shfl_sync(0xffffffffu, v.y, (int)k));
        }
    }
    const double fd = (double)deg;
    const double2 c = make_double2(__ddiv_rn(s.x, fd), __ddiv_rn(s.y, fd));
    // the minimum as exact_update's loop finds it: a later quality replaces the
    // current one when it is smaller, so a NaN is kept only from triangle 0
    const double inf = __longlong_as_double(0x7ff0000000000000ll);
    double q_old = inf, q_new = inf;
    bool nan_old = false, nan_new = false;
    for (uint32_t t0 = 0; t0 < ntri; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t code = t0 == 0u ? code0 : (t < ntri ? __ldg(nb + deg + t) : 0u);
        double2 A, B;
        if (deg <= 32u) {  // the lanes hold the neighbours
            A.x = __shfl_sync(0xffffffffu, v.x, (int)code_first(code));
            A.y = __shfl_sync(0xffffffffu, v.y, (int)code_first(code));
            B.x = __shfl_sync(0xffffffffu, v.x, (int)code_second(code));
            B.y = __shfl_sync(0xffffffffu, v.y, (int)code_second(code));
        } else {
            A = read_node<LAYOUT, COHERENT>(a.in, a.n, __ldg(nb + code_first(code)));
            B = read_node<LAYOUT, COHERENT>(a.in, a.n, __ldg(nb + code_second(code)));
        }
        if (t < ntri) {
            const double qo = alpha_at_slot(code_slot(code), p.x, p.y, A.x, A.y, B.x, B.y);
            const double qn = alpha_at_slot(code_slot(code), c.x, c.y, A.x, A.y, B.x, B.y);
            if (qo < q_old) q_old = qo;
            if (qn < q_new) q_new = qn;
            if (t == 0u) {
                nan_old = qo != qo;
                nan_new = qn != qn;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double uo = __shfl_xor_sync(0xffffffffu, q_old, o), un = __shfl_xor_sync(0xffffffffu, q_new, o);
        if (uo < q_old) q_old = uo;
        if (un < q_new) q_new = un;
    }
    d2_bits = 0ull;
    accepted = moved = false;
    if (lane == 0u) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        finish_exact<LAYOUT>(a, i, p, c, nan_old ? nan : q_old, nan_new ? nan : q_new, d2_bits, accepted, moved);
    }
}

}  // namespace sls
