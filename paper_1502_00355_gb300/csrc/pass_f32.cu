// pass_f32.cu -- Smart Laplacian passes in binary32, the paper's precision
// (Section 4).
//
// The coordinates are stored as floats and every step is one binary32
// round-to-nearest operation in the order of the FP64 definition: the
// neighbour sum of Eq. 2 in the stored order, the division by the neighbour
// count, alpha of Section 3.3.1 with the same expression tree, the accept test
// of Section 3.3.4, the squared move.  Nothing here needs screening: the
// exact binary32 evaluation is itself cheap on the FP32 pipe, so one thread
// takes one node from start to end.
#include <cfloat>

#include "api_common.h"
#include "kernels.h"
#include "screen.cuh"
#include "window_pipe.cuh"

namespace sls {

namespace {

// RN(1/N), N up to the longest ring of the window lists.
__constant__ const float c_recip32[16] = {0.0f,        1.0f,        1.0f / 2.0f,  1.0f / 3.0f,  1.0f / 4.0f, 1.0f / 5.0f,
                                          1.0f / 6.0f, 1.0f / 7.0f, 1.0f / 8.0f,  1.0f / 9.0f,  1.0f / 10.0f, 1.0f / 11.0f,
                                          1.0f / 12.0f, 1.0f / 13.0f, 1.0f / 14.0f, 1.0f / 15.0f};

template <int LAYOUT>
struct Coords32;

template <>
struct Coords32<0> {  // AoS: one float2 per node
    static __device__ __forceinline__ float2 get(const float *p, int64_t, int64_t i)
    {
        return __ldcg(reinterpret_cast<const float2 *>(p) + i);
    }
    static __device__ __forceinline__ void put(float *p, int64_t, int64_t i, float2 v)
    {
        reinterpret_cast<float2 *>(p)[i] = v;
    }
};

template <>
struct Coords32<1> {  // SoA: x[n] then y[n]
    static __device__ __forceinline__ float2 get(const float *p, int64_t n, int64_t i)
    {
        return make_float2(__ldcg(p + i), __ldcg(p + n + i));
    }
    static __device__ __forceinline__ void put(float *p, int64_t n, int64_t i, float2 v)
    {
        p[i] = v.x;
        p[n + i] = v.y;
    }
};

// alpha of the triangle (a, b, c) in stored order, in binary32, with the
// tree of the FP64 definition; every operation an explicit round-to-nearest
// intrinsic (no contraction).  K is the float nearest to 2 sqrt(3).
__device__ __forceinline__ float alpha_f32(float ax, float ay, float bx, float by, float cx, float cy)
{
    const float kTwoSqrt3 = 3.46410161514f;
    const float e1x = __fsub_rn(bx, ax), e1y = __fsub_rn(by, ay);
    const float e2x = __fsub_rn(cx, ax), e2y = __fsub_rn(cy, ay);
    const float e3x = __fsub_rn(cx, bx), e3y = __fsub_rn(cy, by);
    const float cross = __fsub_rn(__fmul_rn(e1x, e2y), __fmul_rn(e1y, e2x));
    const float l1 = __fadd_rn(__fmul_rn(e1x, e1x), __fmul_rn(e1y, e1y));
    const float l2 = __fadd_rn(__fmul_rn(e2x, e2x), __fmul_rn(e2y, e2y));
    const float l3 = __fadd_rn(__fmul_rn(e3x, e3x), __fmul_rn(e3y, e3y));
    const float s = __fadd_rn(__fadd_rn(l1, l2), l3);
    return s > 0.0f ? __fdiv_rn(__fmul_rn(kTwoSqrt3, cross), s) : 0.0f;
}

// alpha of an incident triangle with the node at x, from its two other
// vertices in ring order P -> Q (window.cuh): slot is the node's place in the
// stored triangle, rev whether the step runs against the stored direction.
// With dP = x - P, dQ = x - Q, E = Q - P and base = Q for slot 1, else P (the
// other way round with rev), alpha_f32's tree on the stored order is
//   slot 0:     cross = dP x dQ,        s = (|dP|^2 + |dQ|^2) + |E|^2
//   slots 1, 2: cross = -(dbase x E),   s = (|dbase|^2 + |E|^2) + |dother|^2
// with the cross product negated for rev: every edge of the stored order is
// one of these or its negative, negation commutes with rounding, and so do the
// operands of a product or of the first sum.
__device__ __forceinline__ float alpha_ring(uint32_t slot, bool rev, float2 x, float2 P, float2 Q)
{
    const float2 dP = make_float2(__fsub_rn(x.x, P.x), __fsub_rn(x.y, P.y));
    const float2 dQ = make_float2(__fsub_rn(x.x, Q.x), __fsub_rn(x.y, Q.y));
    const float2 E = make_float2(__fsub_rn(Q.x, P.x), __fsub_rn(Q.y, P.y));
    const float lP = __fadd_rn(__fmul_rn(dP.x, dP.x), __fmul_rn(dP.y, dP.y));
    const float lQ = __fadd_rn(__fmul_rn(dQ.x, dQ.x), __fmul_rn(dQ.y, dQ.y));
    const float lE = __fadd_rn(__fmul_rn(E.x, E.x), __fmul_rn(E.y, E.y));
    const bool zero = slot == 0u, first = zero || (slot == 1u) == rev;  // the base (slot 0: d1) is P
    const float2 d = first ? dP : dQ, z = zero ? dQ : E;
    float cross = __fsub_rn(__fmul_rn(d.x, z.y), __fmul_rn(d.y, z.x));
    cross = zero == rev ? -cross : cross;
    const float l1 = first ? lP : lQ, other = first ? lQ : lP;
    const float s = __fadd_rn(__fadd_rn(l1, zero ? other : lE), zero ? lE : other);
    return s > 0.0f ? __fdiv_rn(__fmul_rn(3.46410161514f, cross), s) : 0.0f;
}

template <int LAYOUT>
__device__ __forceinline__ float alpha_at(const float *in, int64_t n, const uint32_t *nb, uint32_t code, float2 x)
{
    const float2 A = Coords32<LAYOUT>::get(in, n, __ldg(nb + code_first(code)));
    const float2 B = Coords32<LAYOUT>::get(in, n, __ldg(nb + code_second(code)));
    switch (code_slot(code)) {
    case 0: return alpha_f32(x.x, x.y, A.x, A.y, B.x, B.y);
    case 1: return alpha_f32(A.x, A.y, x.x, x.y, B.x, B.y);
    default: return alpha_f32(A.x, A.y, B.x, B.y, x.x, x.y);
    }
}

// One node from its adjacency record, one thread: rings that are not in the
// window lists, and values outside the range in which the pass's quick
// quotients are understood.  Returns (bits of the squared move, 1) when it
// moved to its centre, else (0, 0).
template <int LAYOUT>
__device__ __noinline__ uint2 update_by_record(const PassArgs &a, const float *in, float *out, int64_t i)
{
    const uint32_t off = __ldg(a.node_off + i);
    const uint32_t meta = __ldg(a.adj + off);
    const uint32_t deg = meta_degree(meta), ntri = meta_ntri(meta);
    const uint32_t *nb = a.adj + off + 1;
    const float2 p = Coords32<LAYOUT>::get(in, a.n, i);
    float2 s = Coords32<LAYOUT>::get(in, a.n, __ldg(nb));
    for (uint32_t k = 1; k < deg; ++k) {
        const float2 v = Coords32<LAYOUT>::get(in, a.n, __ldg(nb + k));
        s.x = __fadd_rn(s.x, v.x);
        s.y = __fadd_rn(s.y, v.y);
    }
    const float fd = (float)deg;
    const float2 c = make_float2(__fdiv_rn(s.x, fd), __fdiv_rn(s.y, fd));
    // a tie (the centre is the node itself) means q_new == q_old
    bool ok = !a.strict;
    if (__float_as_uint(c.x) != __float_as_uint(p.x) || __float_as_uint(c.y) != __float_as_uint(p.y)) {
        float q_old = 0.0f, q_new = 0.0f;
        for (uint32_t t = 0; t < ntri; ++t) {
            const uint32_t code = __ldg(nb + deg + t);
            const float qo = alpha_at<LAYOUT>(in, a.n, nb, code, p);
            const float qn = alpha_at<LAYOUT>(in, a.n, nb, code, c);
            q_old = (t == 0u || qo < q_old) ? qo : q_old;  // first wins, as in the definition
            q_new = (t == 0u || qn < q_new) ? qn : q_new;
        }
        ok = a.strict ? (q_new > q_old) : (q_new >= q_old);
    }
    Coords32<LAYOUT>::put(out, a.n, i, ok ? c : p);
    if (a.accept) a.accept[i] = ok ? 1 : 0;
    const float dx = __fsub_rn(c.x, p.x), dy = __fsub_rn(c.y, p.y);
    return ok ? make_uint2(__float_as_uint(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy))), 1u) : make_uint2(0u, 0u);
}

// ---- the pass ------------------------------------------------------------------
// Windows of nodes staged in shared memory and rings walked once, as in
// pass_screened.cu, here with 8-byte entries and no splits.  Every step of
// alpha's tree is the definition's operation (before and after the move in
// the halves of packed pairs); only its last, the division, is replaced by a
// product with the approximate reciprocal, within 3 units in the last place
// (or of 2^-149, below the normal range).  The minima of the approximate
// qualities differ from the exact ones by no more, so a difference above 16
// units, and above 1e-36, decides the test; what is left (about a
// node in a thousand) is evaluated with IEEE divisions, a lane per triangle
// and side.
//
// Bound by instruction issue (70% of slots; 815 warp instructions per 32
// nodes, 118 of them the selections that the stored order asks for, against
// 1,072 with a thread gathering its own ring).  2048^2 jittered grid: 126 us a
// pass against 164.

constexpr int kBlock32 = 128;
constexpr int kBlocks32 = 9;  // per SM; 126.3 us a pass on 2048^2 (6: 130.4, 8: 127.2, 10: 128.1, 12: 130.8)

struct Block32 {
    Ahead *ahead;
    uint32_t *ids, *rows;
    char *xy;
    uint32_t ids_words, rows_words, stage;  // buffer sizes: words, words, bytes; the last two 0 where there is one
};

size_t smem_f32(const WindowShape &s)
{
    return sizeof(Ahead) + 2 * 4 * (size_t)ids_words_of(s) +
           (size_t)s.buffers32 * (128 * (size_t)(s.hot + win::kColdRows) + 8 * (size_t)(s.entries + 1));
}

__device__ __forceinline__ float2 entry32(const char *xy, uint32_t off)
{
    return *reinterpret_cast<const float2 *>(xy + off);
}

// s / N by Markstein's correction: with y = RN(1/N) and q0 = RN(s y), the
// remainder s - q0 N is exact and RN(q0 + remainder y) is the rounded quotient
// (checked over every significand for N = 2 .. 15).  Outside the range where
// nothing under- or overflows: the division.
__device__ __forceinline__ float div_degree(float s, float fn, float y)
{
    const float q0 = __fmul_rn(s, y);
    const float q = __fmaf_rn(__fmaf_rn(-q0, fn, s), y, q0);
    const float m = fabsf(s);
    return (m > 1e-30f && m < 1e30f) ? q : __fdiv_rn(s, fn);
}

// x - vertex before | after the move, and the squared lengths.
struct Vertex32 {
    float x, y;
    uint64_t dx, dy, l;
};

__device__ __forceinline__ Vertex32 vertex32(const char *xy, uint32_t off, float2 p, float2 c)
{
    const float2 v = entry32(xy, off);
    Vertex32 r;
    r.x = v.x;
    r.y = v.y;
    r.dx = pair(__fsub_rn(p.x, v.x), __fsub_rn(c.x, v.x));
    r.dy = pair(__fsub_rn(p.y, v.y), __fsub_rn(c.y, v.y));
    r.l = add2(mul2(r.dx, r.dx), mul2(r.dy, r.dy));
    return r;
}

struct Minima32 {
    float o, n, smin, smax;
};

// alpha_ring before and after the move, with a quick quotient.
template <bool IRREGULAR>
__device__ __forceinline__ void step32(Minima32 &m, const Vertex32 &P, const Vertex32 &Q, uint32_t slot, bool rev)
{
    if (IRREGULAR && slot == 3u) return;
    const float ex = __fsub_rn(Q.x, P.x), ey = __fsub_rn(Q.y, P.y);
    const float le = __fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey));
    const bool r = IRREGULAR && rev;
    const bool zero = slot == 0u, first = zero || (slot == 1u) == r;
    const uint64_t ex2 = pair(ex, ex), ey2 = pair(ey, ey), le2 = pair(le, le), minus = pair(-1.0f, -1.0f);
    const uint64_t dx = first ? P.dx : Q.dx, dy = first ? P.dy : Q.dy;
    const uint64_t zx = zero ? Q.dx : ex2, zy = zero ? Q.dy : ey2;
    // a * b - c * d with both products rounded: RN(c d) times -1 is exact
    const uint64_t cross = fma2(mul2(dy, zx), minus, mul2(dx, zy));
    const uint64_t l1 = first ? P.l : Q.l, other = first ? Q.l : P.l;
    const uint64_t s2 = add2(add2(l1, zero ? other : le2), zero ? le2 : other);
    float so, sn, ko, kn;
    halves(s2, so, sn);
    const float k = zero == r ? -3.46410161514f : 3.46410161514f;
    halves(mul2(cross, pair(k, k)), ko, kn);
    m.o = fminf(m.o, ko * scr::rcp_ring(so));
    m.n = fminf(m.n, kn * scr::rcp_ring(sn));
    m.smin = fminf(m.smin, fminf(so, sn));
    m.smax = max_nan(m.smax, max_nan(so, sn));
}

// To the subtile's largest step number l, two steps at a time.  Lists of
// closed rings go on around the ring, so a lane past its own steps meets its
// first triangles again; irregular subtiles look at each lane's steps.
template <bool IRREGULAR, int BITS>
__device__ __forceinline__ Minima32 walk32(const char *xy, uint32_t l, uint32_t steps, const uint32_t *list, float2 p,
                                           float2 c, uint32_t slots, uint32_t rev)
{
    using L = List<BITS, 3>;
    Minima32 m;
    m.o = m.n = m.smin = FLT_MAX;
    m.smax = 0.0f;
    uint32_t word = list[0];
    Vertex32 A = vertex32(xy, L::in_word(word, 0), p, c);
    for (uint32_t t = 0;; t += L::kPer) {
#pragma unroll
        for (uint32_t j = 0; j < L::kPer; j += 2) {
            const uint32_t e1 = L::in_word(word, j + 1);
            if (j + 2 == L::kPer) {
                list += 32;
                word = *list;
            }
            const uint32_t e2 = L::in_word(word, (j + 2) % L::kPer);
            const Vertex32 B = vertex32(xy, e1, p, c);
            const Vertex32 C = vertex32(xy, e2, p, c);
            const uint32_t t1 = t + j, t2 = t + j + 1u;
            if (!IRREGULAR || t1 < steps) step32<IRREGULAR>(m, A, B, (slots >> (2u * t1)) & 3u, (rev >> t1) & 1u);
            if (!IRREGULAR || t2 < steps) step32<IRREGULAR>(m, B, C, (slots >> (2u * t2)) & 3u, (rev >> t2) & 1u);
            A = C;
            if (t2 + 1u >= l) return m;
        }
    }
}

// Works subtile `sub` of a staged window; best: bits of the largest squared
// move (non-negative floats order as integers).
template <int LAYOUT, int BITS>
__device__ __forceinline__ void work32(const PassArgs &a, const float *in, float *out, const char *xy,
                                       const uint32_t *h, const uint32_t *rows, int sub, unsigned &best,
                                       unsigned &nacc)
{
    using L = List<BITS, 3>;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t d = (h[3] >> (8 * sub)) & 15u, l = (h[3] >> (8 * sub + 4)) & 15u;
    const uint32_t *at = rows + ((h[4] >> (8 * sub)) & 0xffu) * 32u + lane;
    const uint32_t *cold = rows + (h[5] + 2u * sub) * 32u + lane;
    const uint32_t meta = *at;
    const int64_t node = (int64_t)h[1] + win::meta_place(meta);
    const bool have = (meta & win::kNode) != 0u, free = (meta & win::kFree) != 0u;
    if (have && !(meta & (win::kFree | win::kBig)) && a.accept) a.accept[node] = 0;
    bool record = have && (meta & win::kBig);
    if (d > 0u) {
        const uint32_t deg = win::meta_deg(meta), steps = win::meta_steps(meta);
        const uint32_t *list = at + 32;
        uint32_t word = *list;
        float2 s = entry32(xy, L::in_word(word, 0));
        for (uint32_t k = 0;;) {  // Eq. 2 in the stored order; padding adds -0
#pragma unroll
            for (uint32_t j = 0; j < L::kPer; ++j) {
                if (j == 0u && k == 0u) continue;
                const float2 v = entry32(xy, L::in_word(word, j));
                s.x = __fadd_rn(s.x, v.x);
                s.y = __fadd_rn(s.y, v.y);
            }
            k += L::kPer;
            list += 32;
            if (k >= d) break;
            word = *list;
        }
        list = at + 32u * (1u + win::list_rows(d, BITS));
        const float2 p = entry32(xy, (win::meta_place(meta) + 1u) * 8u);
        float2 c = p;
        if (free) {
            const float fn = (float)deg, y = c_recip32[deg];
            c = make_float2(div_degree(s.x, fn, y), div_degree(s.y, fn, y));
        }
        // a tie (the centre is the node itself) means q_new == q_old
        bool act = __float_as_uint(c.x) != __float_as_uint(p.x) || __float_as_uint(c.y) != __float_as_uint(p.y);
        int verdict = free && !act ? (a.strict ? -1 : 1) : 0;
        if (__any_sync(0xffffffffu, act)) {
            const uint32_t slots = *cold, rev = cold[32];
            const bool irregular = win::hdr_irregular(h[2], (uint32_t)sub);
            const Minima32 m = irregular ? walk32<true, BITS>(xy, l, steps, list, p, c, slots, rev)
                                         : walk32<false, BITS>(xy, l, steps, list, p, c, slots, 0u);
            // normal sums and finite points: the quick quotients are within 3 units
            // (an infinite or NaN coordinate among the node's, the centre's and the
            // neighbours' makes some sum infinite or NaN, and smax with it: the
            // definition's quality is 0 there, the quick one has no value)
            const float far = fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fmaxf(fabsf(c.x), fabsf(c.y)));
            const bool fine = m.smin > 1e-30f && m.smax > 1e-30f && m.smax < 1e30f && far < 1e30f;
            if (act && !fine) record = true;
            act = act && fine;
            // (a quality below the normal range is a whole number of units of 2^-149,
            // and a quick one off by about a unit: the absolute part of the margin)
            const float gap = m.n - m.o;
            if (act && fabsf(gap) > fmaf(2e-6f, fmaxf(fabsf(m.o), fabsf(m.n)), 1e-36f)) verdict = gap > 0.0f ? 1 : -1;
            // the others: lane t takes step t before the move, lane 16 + t after it
            for (unsigned open = __ballot_sync(0xffffffffu, act && verdict == 0); open; open &= open - 1u) {
                const uint32_t src = (uint32_t)__ffs((int)open) - 1u, t = lane & 15u;
                const uint32_t st = __shfl_sync(0xffffffffu, steps, src), sl = __shfl_sync(0xffffffffu, slots, src);
                const uint32_t rv = __shfl_sync(0xffffffffu, irregular ? rev : 0u, src);
                const float2 ps = make_float2(__shfl_sync(0xffffffffu, p.x, src), __shfl_sync(0xffffffffu, p.y, src));
                const float2 cs = make_float2(__shfl_sync(0xffffffffu, c.x, src), __shfl_sync(0xffffffffu, c.y, src));
                const uint32_t *ring = list + (int)src - (int)lane;
                const uint32_t slot = (sl >> (2u * t)) & 3u;
                float q = FLT_MAX;
                if (t < st && slot != 3u)
                    q = alpha_ring(slot, ((rv >> t) & 1u) != 0u, lane < 16u ? ps : cs, entry32(xy, L::at(ring, t)),
                                   entry32(xy, L::at(ring, t + 1u)));
                for (int w = 8; w > 0; w >>= 1) q = fminf(q, __shfl_xor_sync(0xffffffffu, q, w));
                const float q_old = __shfl_sync(0xffffffffu, q, 0), q_new = __shfl_sync(0xffffffffu, q, 16);
                if (lane == src) verdict = (a.strict ? q_new > q_old : q_new >= q_old) ? 1 : -1;
            }
        }
        if (verdict != 0) {
            if (verdict > 0) {
                const float dx = __fsub_rn(c.x, p.x), dy = __fsub_rn(c.y, p.y);
                best = max(best, __float_as_uint(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy))));
                nacc += 1u;
            }
            Coords32<LAYOUT>::put(out, a.n, node, verdict > 0 ? c : p);
            if (a.accept) a.accept[node] = verdict > 0 ? 1 : 0;
        }
    }
    if (record) {
        const uint2 r = update_by_record<LAYOUT>(a, in, out, node);
        best = max(best, r.x);
        nacc += r.y;
    }
    __syncwarp();
}

// One pass over a mesh's windows, or over those of one colour class of Form B
// (in place).  a.in / a.out hold floats.  TWO: shape.buffers32 is 2.
template <int LAYOUT, int BITS, bool TWO>
__global__ void __launch_bounds__(kBlock32, kBlocks32)
    pass_f32_kernel(const __grid_constant__ PassArgs a, const __grid_constant__ WindowShape shape)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const float *in = reinterpret_cast<const float *>(a.in);
    float *out = reinterpret_cast<float *>(a.out);
    const int tid = threadIdx.x, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
    Block32 b;
    b.ahead = reinterpret_cast<Ahead *>(smem);
    b.ids = reinterpret_cast<uint32_t *>(smem + sizeof(Ahead));
    b.ids_words = ids_words_of(shape);
    b.rows = b.ids + 2 * b.ids_words;
    b.rows_words = 32u * (uint32_t)(shape.hot + (int)win::kColdRows);
    b.xy = reinterpret_cast<char *>(b.rows + (TWO ? 2 : 1) * b.rows_words);
    b.stage = TWO ? (uint32_t)(shape.entries + 1) * 8u : 0u;
    if (!TWO) b.rows_words = 0u;
    if (tid < 2) *reinterpret_cast<float2 *>(b.xy + tid * b.stage) = make_float2(-0.0f, -0.0f);  // the padding entries

    // windows blockIdx.x, + gridDim.x, ...: headers three ahead, halo ids two,
    // rows and coordinates one (see run_windows in pass_screened.cu)
    const int64_t w0 = a.win_first + blockIdx.x;
    const int n = (int64_t)blockIdx.x < a.win_count ? (int)((a.win_count - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
    Ahead *ah = b.ahead;
    auto fetch_header = [&](int i) {
        if (i < n && tid < 2)
            copy16(&ah->hdr[i & 3][4 * tid],
                   a.win_hdr + (w0 + (int64_t)i * gridDim.x) * win::kHeaderWords + 4 * tid);
    };
    auto fetch_ids = [&](int i) {
        if (i >= n) return;
        const uint32_t *h = ah->hdr[i & 3];
        const uint32_t *src = a.win_rows + (size_t)h[0] * 32u;
        uint32_t *dst = b.ids + (i & 1) * b.ids_words;
        for (uint32_t k = 4 * tid; k < win::hdr_halo(h[2]); k += 4 * nthr) copy16(dst + k, src + k);
    };
    auto fetch_data = [&](int i) {
        if (i >= n) return;
        const uint32_t *h = ah->hdr[i & 3];
        const uint32_t count = win::hdr_count(h[2]), nhalo = win::hdr_halo(h[2]);
        const uint32_t *src = a.win_rows + ((size_t)h[0] + win::halo_rows(nhalo)) * 32u;
        uint32_t *rows = b.rows + (i & 1) * b.rows_words;
        for (uint32_t k = 4 * tid; k < 32u * (h[5] + win::kColdRows); k += 4 * nthr) copy16(rows + k, src + k);
        const uint32_t *ids = b.ids + (i & 1) * b.ids_words;
        char *xy = b.xy + (i & 1) * b.stage + 8;
        for (uint32_t e = tid; e < count + nhalo; e += nthr) {
            const int64_t id = e < count ? (int64_t)h[1] + e : (int64_t)ids[e - count];
            if (LAYOUT == 0) {
                copy8(xy + e * 8u, in + 2 * id);
            } else {
                copy4(xy + e * 8u, in + id);
                copy4(xy + e * 8u + 4u, in + a.n + id);
            }
        }
    };
    fetch_header(0);
    fetch_header(1);
    fetch_header(2);
    copies_done();
    __syncthreads();
    fetch_ids(0);
    fetch_ids(1);
    copies_done();
    __syncthreads();
    after_previous();
    if (pass_is_skipped(a.stats, a.q, a.tol_active, a.thr_bits)) return;
    if (blockIdx.x == 0 && tid == 0) a.stats[a.q].executed = 1u;
    if (TWO) fetch_data(0);
    unsigned best = 0u, nacc = 0u;
    for (int i = 0; i < n; ++i) {
        copies_done();
        __syncthreads();
        if (TWO) {
            fetch_data(i + 1);
        } else {  // window i - 1 is finished
            fetch_data(i);
            copies_done();
            __syncthreads();
        }
        fetch_ids(i + 2);
        fetch_header(i + 3);
        for (int sub = warp; sub < 4; sub += nwarps)
            work32<LAYOUT, BITS>(a, in, out, b.xy + (i & 1) * b.stage, ah->hdr[i & 3],
                                 b.rows + (i & 1) * b.rows_words, sub, best, nacc);
    }
    // widened exactly to double, so the pass records compare like FP64 ones
    const unsigned long long b64 = (unsigned long long)__double_as_longlong((double)__uint_as_float(best));
    block_reduce_stats(a.stats + a.q, b64, nacc, 0ull);
}

__global__ void copy_back_f32_kernel(const float *__restrict__ src, float *__restrict__ dst, int64_t count,
                                     const PassStats *stats, int q)
{
    if (stats[q].executed == 0u) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += stride)
        dst[k] = __ldg(src + k);
}

// interleaved doubles -> floats in the mesh's layout (round to nearest)
__global__ void narrow_kernel(const double *__restrict__ aos, float *dst, int64_t n, int layout, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double2 v = load_pair(aos, i, wide);
        const float x = __double2float_rn(v.x), y = __double2float_rn(v.y);
        if (layout == 0) {
            reinterpret_cast<float2 *>(dst)[i] = make_float2(x, y);
        } else {
            dst[i] = x;
            dst[n + i] = y;
        }
    }
}

// floats in the mesh's layout -> interleaved doubles (exact)
__global__ void widen_kernel(const float *__restrict__ src, double *aos, int64_t n, int layout, bool wide)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float x, y;
        if (layout == 0) {
            const float2 v = __ldg(reinterpret_cast<const float2 *>(src) + i);
            x = v.x;
            y = v.y;
        } else {
            x = __ldg(src + i);
            y = __ldg(src + n + i);
        }
        store_pair(aos, i, make_double2((double)x, (double)y), wide);
    }
}

}  // namespace

namespace {

template <int LAYOUT>
const void *kernel32_of(const WindowShape &s)
{
    if (s.bits == 8) return (const void *)pass_f32_kernel<LAYOUT, 8, true>;  // (at most 255 entries)
    return s.buffers32 == 2 ? (const void *)pass_f32_kernel<LAYOUT, 16, true>
                            : (const void *)pass_f32_kernel<LAYOUT, 16, false>;
}
// Wide windows of separate x and y arrays take two 4-byte copies a coordinate, which
// go through L1: with all the blocks an SM could hold, shared memory leaves little
// of it.  1009 x 701 nodes, us a pass with 9 (8 in Form B), 6, 5, 4, 3 blocks: random
// ids kept 48.2, 47.8, 59.6, 54.1, 70.2; Form B, random ids 124.8, 84.6, 90.0, 81.8,
// 97.4, Morton order 61.1, 60.7, 62.7, 60.5, 69.8.
constexpr int kWideSoaBlocks = 6;
bool wide_soa(int layout, const WindowShape &s) { return layout == 1 && s.bits == 16 && s.buffers32 == 1; }
const void *kernel32(int layout, const WindowShape &s) { return layout == 0 ? kernel32_of<0>(s) : kernel32_of<1>(s); }

}  // namespace

cudaError_t launch_pass_f32(const PassArgs &a, int layout, int block, int grid, const WindowShape &shape,
                            cudaStream_t s)
{
    if (a.win_count < grid) grid = a.win_count > 0 ? (int)a.win_count : 1;
    void *args[] = {const_cast<PassArgs *>(&a), const_cast<WindowShape *>(&shape)};
    return launch_early(kernel32(layout, shape), grid, block, args, smem_f32(shape), s, false,
                        wide_soa(layout, shape) ? kWideSoaBlocks : 0);
}

// Also allows the kernel the shared memory that the shape takes; a launch in
// another context would need it again, and meshes belong to their context.
int pass_f32_occupancy(int layout, int block, const WindowShape &shape)
{
    const void *f = kernel32(layout, shape);
    int nb = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
        cudaGetLastError();
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, block, smem_f32(shape));
    if (wide_soa(layout, shape) && nb > kWideSoaBlocks) nb = kWideSoaBlocks;
    return nb > 0 ? nb : 1;
}

// A second buffer, into which the next window is copied while one is worked on,
// costs blocks where windows are wide: 1009 x 701 nodes, us a pass with one and with
// two buffers, random ids kept (about 900 entries a window) 37.3 and 49.4, SoA 49.0
// and 75.9; Form B (colour classes, about 510) 58.8 and 64.1; rows of the grid
// kept (about 390) 29.2 and 28.9.  With about a window a block it has nothing to do
// either, but fewer blocks an SM then spread the windows evenly, where early
// launches would fill some SMs first: 100,000 Delaunay points, random ids kept (782
// windows) 25.8 with one, 19.9 with two.
void choose_buffers32(int layout, int block, int64_t windows, WindowShape &shape)
{
    constexpr int kTwoBuffers = 448;
    shape.buffers32 = 2;
    if (shape.entries > kTwoBuffers &&
        windows > 2 * (int64_t)device_sm_count() * pass_f32_occupancy(layout, block, shape))
        shape.buffers32 = 1;
}

cudaError_t launch_copy_back_f32(const float *src, float *dst, int64_t count, const PassStats *stats, int q,
                                 int grid, cudaStream_t s)
{
    copy_back_f32_kernel<<<grid, 256, 0, s>>>(src, dst, count, stats, q);
    return cudaGetLastError();
}

cudaError_t launch_narrow(const double *aos, float *dst, int64_t n, int layout, int grid, cudaStream_t s)
{
    narrow_kernel<<<grid, 256, 0, s>>>(aos, dst, n, layout, pair_aligned(aos));
    return cudaGetLastError();
}

cudaError_t launch_widen(const float *src, double *aos, int64_t n, int layout, int grid, cudaStream_t s)
{
    widen_kernel<<<grid, 256, 0, s>>>(src, aos, n, layout, pair_aligned(aos));
    return cudaGetLastError();
}

}  // namespace sls
