// pass_screened.cu -- the fast exact Jacobi pass of Smart Laplacian smoothing.
//
// Same results, bit for bit, as the FP64 pass (Eq. 2 with the accept test of
// Section 3.3.4); what changes is which pipe does which work.  GB300 issues
// about two FP64 operations per SM per clock against ~128 FP32/INT32, so the
// FP64 pipe does only what decides the result's bits, and the rest moves to
// the FP32 and integer pipes.  Per window of 128 nodes (window.cuh), one
// block:
//
//  1. The window's nodes and their neighbours outside it are staged in shared
//     memory, as FP64 bit patterns and as float head/tail splits (integer
//     operations only).
//  2. The neighbour sums (Eq. 2) are the FP64 additions themselves, in the
//     stored summation order.
//  3. The division by the degree is one FP64 multiplication by RN(1/N) and an
//     exact integer remainder that picks the correctly rounded quotient
//     (div_small.cuh), instead of a full division.
//  4. If the centre equals the node's position bit for bit, q_new == q_old
//     exactly and no quality needs evaluating.
//  5. Otherwise alpha of every incident triangle, before and after the move, is
//     evaluated in FP32 in a frame centred on the node, around the node's ring,
//     with a rigorous bound on its distance to the exact alpha of the FP64
//     inputs, wide enough to also cover the FP64 evaluation's own rounding.
//     When the intervals of q_new and q_old are disjoint the FP64 decision is
//     known.
//  6. If one triangle alone attains both minima, a second screen takes the
//     sign of alpha(centre) - alpha(node) from a formula in the move itself
//     (no cancellation) and decides all but rounding-level ties.
//  7. What is left goes to the block's queue: one item per quality to be
//     evaluated in FP64, with the coordinates it needs, so that full warps
//     evaluate independent items side by side on the narrow FP64 pipe.  A warp
//     most of whose nodes are left, or that finds the queue full, looks closer
//     and evaluates its items itself, 32 at a time.
//
// Coordinates are moved as 64-bit patterns, never held in FP64 registers
// unless they take part in FP64 arithmetic: the compiler copies FP64
// registers with FP64-pipe instructions.
//
// What bounds it: instruction issue (65% of slots in an early pass of a 2048^2
// grid), the FP64 pipe (58% there; half of the time over a 4096^2 run to the
// tolerance) and the latency of shared-memory loads together; HBM stands at about
// a sixth of the measured copy rate.  Gathering and splitting a coordinate once
// per window (1.4 times a node) instead of once per neighbour visit (6.5 times)
// took 1,653 warp instructions per 32 nodes to 1,148 and 23.5 FP64 instructions to
// 13.8.  Measured, to the tolerance, against one thread per node gathering for
// itself: 2048^2 jittered grid 293.7 -> 200.8 us a pass, 1024^2 96.9 -> 59.2,
// 4096^2 942 -> 630..700 (by GPU; clustered about fewer centres 1058 -> 741).
#include <atomic>
#include <cfloat>
#include <mutex>

#include "api_common.h"
#include "div_small.cuh"
#include "kernels.h"
#include "node_exact.cuh"
#include "screen.cuh"
#include "window_pipe.cuh"

namespace sls {

namespace {

constexpr int kRingMax = win::kRingMax;
__constant__ double c_recip[kRingMax + 1];  // RN(1/N)
__constant__ double c_degree[kRingMax + 1]; // N as a double

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ double bitsd(unsigned long long b) { return __longlong_as_double((long long)b); }

using namespace scr;

// ---- shared memory of a block ----------------------------------------------

constexpr int kBlockMax = 128;
constexpr int kItems = 112;       // qualities waiting for their FP64 evaluation
constexpr int kPending = 64;      // nodes they belong to
constexpr int kItemsFull = 72;    // the queue is worked off once it holds this many items
constexpr int kPendingFull = 44;  // or nodes
constexpr uint32_t kNoItem = 0xffffffffu;

struct __align__(16) Queue {
    ulonglong2 p[kPending], c[kPending];                    // the node, its centre
    double px[kItems], py[kItems], qx[kItems], qy[kItems];  // the step's vertices in ring order; then px: quality
    uint32_t item[kItems];      // pending node | side << 8 (1: after the move) | step << 9
    int32_t node[kPending];     // -1: no entry
    uint32_t range[kPending];   // first item | items << 8 | lane << 16
    uint32_t cold[kPending];    // row of the lane's slots and, next to it, directions
    uint32_t nitems, npending;  // claimed (may exceed the capacity)
    unsigned int nacc, nexact;  // accepted and exactly decided nodes (flush)
    unsigned long long best;    // bits of the block's largest squared move
    float best_low;             // at most that (-1: none yet)
};

struct Block {
    Queue *q;
    Ahead *ahead;
    uint32_t *ids;            // halo ids, window i's in buffer i & 1
    uint32_t *rows;           // hot rows
    char *xy;                 // staged entries: coordinates, then head/tail splits
    uint32_t ids_words, rows_words, half, stage;  // buffer sizes: words, words, bytes of one array, bytes
                                                  // from one buffer to the other (0: there is one, of the
                                                  // rows too)
};

// Buffers of staged entries: one where two would leave an SM with few blocks.
// Colour classes (about 510 entries a window) run 233 us a sweep with one and
// 281 with two (1500 x 1100 grid), a random numbering kept as it is (900
// entries) 111 against 144 us a pass; local numberings (at most 255) gain 8%
// from the second.  The lists' rows, fetched with the entries, have as many
// buffers: with one instead of two, 38 sweeps of that grid take 7.06 instead
// of 7.33 ms.  (Shared memory by colour class, 37 to 51 KB, made each class's
// kernel faster by itself, 38 against 44 us, but the sweeps slower, 7.46
// against 7.14 ms: launches of unlike sizes overlap less.)
constexpr int kTwoBufferEntries = 320;
static_assert(kTwoBufferEntries >= 255, "8-bit lists");
__host__ __device__ inline int buffers_for(const WindowShape &s) { return s.entries <= kTwoBufferEntries ? 2 : 1; }
size_t smem_for(const WindowShape &s)
{
    return sizeof(Queue) + sizeof(Ahead) + 2 * 4 * (size_t)ids_words_of(s) +
           (size_t)buffers_for(s) * (128 * (size_t)s.hot + 32 * (size_t)(s.entries + 1));
}

struct Tally {
    unsigned int nacc, nexact;
};

__device__ __forceinline__ void reset(Queue *q)
{
    q->nitems = q->npending = q->nacc = q->nexact = 0u;
    q->best = 0ull;
    q->best_low = -1.0f;
}

// The block's statistics into a pass record; the queue starts afresh.  All
// threads call it; nothing may be pushed before the next barrier.
__device__ __forceinline__ void flush(Queue *q, PassStats *st, const Tally &tally)
{
    const unsigned acc = __reduce_add_sync(0xffffffffu, tally.nacc), ex = __reduce_add_sync(0xffffffffu, tally.nexact);
    if ((threadIdx.x & 31) == 0) {
        if (acc) atomicAdd(&q->nacc, acc);
        if (ex) atomicAdd(&q->nexact, ex);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (q->best) atomicMax(&st->maxd2_bits, q->best);
        if (q->nacc) atomicAdd(&st->nacc, (unsigned long long)q->nacc);
        if (q->nexact) atomicAdd(&st->fallbacks, (unsigned long long)q->nexact);
        reset(q);
    }
}

// A squared move (FP64 bits) towards the block's largest.
__device__ __forceinline__ void note_move(Queue *q, unsigned long long b2)
{
    if (b2 <= *const_cast<volatile unsigned long long *>(&q->best)) return;
    atomicMax(&q->best, b2);
    atomicMax(reinterpret_cast<int *>(&q->best_low), __float_as_int(__double2float_rd(bitsd(b2))));
}

template <bool TWO>
__device__ __forceinline__ Block block_memory(unsigned char *smem, const WindowShape &s)
{
    Block b;
    b.q = reinterpret_cast<Queue *>(smem);
    b.ahead = reinterpret_cast<Ahead *>(smem + sizeof(Queue));
    b.ids = reinterpret_cast<uint32_t *>(smem + sizeof(Queue) + sizeof(Ahead));
    b.ids_words = ids_words_of(s);
    b.rows = b.ids + 2 * b.ids_words;
    b.xy = reinterpret_cast<char *>(b.rows + (TWO ? 2 : buffers_for(s)) * 32 * s.hot);
    b.rows_words = 32u * (uint32_t)s.hot;
    b.half = (uint32_t)(s.entries + 1) * 16u;
    b.stage = buffers_for(s) == 2 ? 2u * b.half : 0u;
    // the padding entries: -0 for the sums, NaN for the rings
    const float nan = __int_as_float(0x7fffffff);
    for (uint32_t k = threadIdx.x; k < (uint32_t)buffers_for(s); k += blockDim.x) {
        *reinterpret_cast<ulonglong2 *>(b.xy + k * b.stage) =
            make_ulonglong2(0x8000000000000000ull, 0x8000000000000000ull);
        *reinterpret_cast<float4 *>(b.xy + k * b.stage + b.half) = make_float4(nan, nan, nan, nan);
    }
    if (threadIdx.x == 0) reset(b.q);
    return b;
}

// ---- the FP64 queue ---------------------------------------------------------

// FP64 quality of step t (P -> Q) of a ring with the node at x.  The step runs
// in the triangle's stored direction unless `rev`; the stored order of P and Q
// is P, Q for slots 0 and 2 and Q, P for slot 1.
__device__ __forceinline__ double step_quality(ulonglong2 x, unsigned long long px, unsigned long long py,
                                               unsigned long long qx, unsigned long long qy, uint32_t slots,
                                               uint32_t rev, uint32_t t)
{
    const uint32_t slot = (slots >> (2u * t)) & 3u;
    const bool swap = (((rev >> t) & 1u) != 0u) != (slot == 1u);
    return alpha_at_slot(slot, bitsd(x.x), bitsd(x.y), bitsd(swap ? qx : px), bitsd(swap ? qy : py),
                         bitsd(swap ? px : qx), bitsd(swap ? py : qy));
}

// Evaluates every waiting item and finishes the nodes they belong to.  All
// threads of the block call it, with no push in flight.
template <int LAYOUT, bool HALO>
__device__ __noinline__ Tally drain(const PassArgs &a, Queue *q, Tally tally)
{
    const uint32_t ni = q->nitems < (uint32_t)kItems ? q->nitems : (uint32_t)kItems;
    for (uint32_t k = threadIdx.x; k < ni; k += blockDim.x) {
        const uint32_t it = q->item[k];
        if (it == kNoItem) continue;
        const uint32_t e = it & 0xffu;
        const uint32_t *row = a.win_rows + (size_t)q->cold[e] * 32u + (q->range[e] >> 16);
        const ulonglong2 x = (it & 0x100u) ? q->c[e] : q->p[e];
        q->px[k] = step_quality(x, dbits(q->px[k]), dbits(q->py[k]), dbits(q->qx[k]), dbits(q->qy[k]), __ldg(row),
                                __ldg(row + 32), it >> 9);
    }
    __syncthreads();
    const uint32_t np = q->npending < (uint32_t)kPending ? q->npending : (uint32_t)kPending;
    for (uint32_t e = threadIdx.x; e < np; e += blockDim.x) {
        const int32_t node = q->node[e];
        if (node < 0) continue;
        const uint32_t i0 = q->range[e] & 0xffu, cnt = (q->range[e] >> 8) & 0xffu;
        double q_old = bitsd(0x7ff0000000000000ull), q_new = q_old;
#pragma unroll 4
        for (uint32_t k = i0; k < i0 + cnt; ++k) {
            const double v = q->px[k];
            if (q->item[k] & 0x100u) {
                if (v < q_new) q_new = v;
            } else {
                if (v < q_old) q_old = v;
            }
        }
        unsigned long long b2;
        bool acc, moved;
        const ulonglong2 p = q->p[e], c = q->c[e];
        finish_exact<LAYOUT>(a, node, make_double2(bitsd(p.x), bitsd(p.y)), make_double2(bitsd(c.x), bitsd(c.y)),
                             q_old, q_new, b2, acc, moved);
        note_move(q, b2);
        tally.nacc += acc ? 1u : 0u;
        if (HALO) {  // the node's bits in its tile's masks (written with the tile's other nodes)
            const uint32_t bit = 1u << (node & 31);
            if (moved) atomicOr(a.chg_cur + (node >> 5), bit);
            if (acc) atomicOr(a.accm + (node >> 5), bit);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) q->nitems = q->npending = 0u;
    __syncthreads();
    return tally;
}

// ---- one subtile --------------------------------------------------------------

// ---- the ring walk: screen.cuh's ring form, both sides of the move in the
// halves of packed FP32 pairs.

// What the walk knows of the node.
struct RingWalk {
    const char *split;         // staged head/tail splits
    float phx, plx, phy, ply;  // the node's splits
    float Cx, Cy;              // the centre's offset
    uint32_t slots, rev;       // irregular subtiles only

    __device__ __forceinline__ RingVertex vertex(uint32_t off) const
    {
        const float4 h = *reinterpret_cast<const float4 *>(split + off);
        return ring_vertex(h.x, h.y, h.z, h.w, phx, plx, phy, ply, Cx, Cy);
    }
};

// ring_vertex's values before | after the move; TURNED: y and yc negated.
// Steps go from plain to turned vertices and back, so that their cross
// products need no negation.
struct PairVertex {
    float x, y;
    uint64_t xx, yy, nn;
};

template <bool TURNED>
__device__ __forceinline__ PairVertex pair_vertex(const RingWalk &w, uint32_t off)
{
    const float4 h = *reinterpret_cast<const float4 *>(w.split + off);
    PairVertex v;
    v.x = (h.x - w.phx) + (h.y - w.plx);
    v.y = TURNED ? (w.phy - h.z) + (w.ply - h.w) : (h.z - w.phy) + (h.w - w.ply);
    v.xx = pair(v.x, v.x - w.Cx);
    v.yy = pair(v.y, TURNED ? v.y + w.Cy : v.y - w.Cy);
    v.nn = fma2(v.xx, v.xx, mul2(v.yy, v.yy));
    return v;
}

struct Minima {
    float m1o, m2o, m1n, m2n;  // smallest and second smallest value before and after the move
    float smin, rn;            // smallest edge sum, largest local coordinate
};

// ring_values of the step P -> Q (FROM_PLAIN: P is the plain one), packed with
// its number; NaN for a step that has no triangle.
template <bool IRREGULAR, bool FROM_PLAIN>
__device__ __forceinline__ void ring_step(const RingWalk &w, Minima &m, const PairVertex &P, const PairVertex &Q,
                                          uint32_t t, float &vo, float &vn)
{
    m.rn = fmaxf(m.rn, fmaxf(fabsf(Q.x), fabsf(Q.y)));
    const float bx = Q.x - P.x, by = Q.y + P.y;
    const float b2 = fmaf(bx, bx, by * by);
    float so, sn, co, cn;
    halves(add2(add2(P.nn, Q.nn), pair(b2, b2)), so, sn);
    halves(fma2(P.xx, Q.yy, mul2(P.yy, Q.xx)), co, cn);  // the cross product, negated from a plain vertex
    vo = (FROM_PLAIN ? -co : co) * rcp_ring(so);
    vn = (FROM_PLAIN ? -cn : cn) * rcp_ring(sn);
    if (IRREGULAR) {
        if ((w.rev >> t) & 1u) {
            vo = -vo;
            vn = -vn;
        }
        if (((w.slots >> (2u * t)) & 3u) == 3u) vo = vn = so = sn = __int_as_float(0x7fffffff);
    }
    vo = with_step(vo, t);
    vn = with_step(vn, t);
    m.smin = fminf(m.smin, fminf(so, sn));
}

// Two values into the smallest two.  Values of padding steps are NaN and
// change nothing.
__device__ __forceinline__ void two_least(float &m1, float &m2, float v1, float v2)
{
    const float lo = fminf(v1, v2);
    m2 = fminf(m2, fminf(max_nan(m1, lo), max_nan(v1, v2)));
    m1 = fminf(m1, lo);
}

// Walks the rings of a warp's lanes to the subtile's largest step number l,
// two steps between branches (so that the loads of one overlap the other's
// arithmetic).
template <bool IRREGULAR, int BITS>
__device__ __forceinline__ Minima walk_ring(RingWalk w, uint32_t l, const uint32_t *list)
{
    using L = List<BITS>;
    Minima m;
    m.m1o = m.m2o = m.m1n = m.m2n = m.smin = FLT_MAX;
    uint32_t word = list[0];
    PairVertex A = pair_vertex<false>(w, L::in_word(word, 0));
    m.rn = fmaxf(fabsf(A.x), fabsf(A.y));
    for (uint32_t t = 0;; t += L::kPer) {  // a word's entries per trip; A is entry t
#pragma unroll
        for (uint32_t j = 0; j < L::kPer; j += 2) {
            const uint32_t e1 = L::in_word(word, j + 1);
            if (j + 2 == L::kPer) {
                list += 32;
                word = *list;
            }
            const uint32_t e2 = L::in_word(word, (j + 2) % L::kPer);
            const PairVertex B = pair_vertex<true>(w, e1);
            const PairVertex C = pair_vertex<false>(w, e2);
            float vo1, vn1, vo2, vn2;
            ring_step<IRREGULAR, true>(w, m, A, B, t + j, vo1, vn1);
            ring_step<IRREGULAR, false>(w, m, B, C, t + j + 1u, vo2, vn2);
            two_least(m.m1o, m.m2o, vo1, vo2);
            two_least(m.m1n, m.m2n, vn1, vn2);
            A = C;
            if (t + j + 2u >= l) return m;
        }
    }
}

// (kept out of line: it would cost the regular walk registers)
template <int BITS>
__device__ __noinline__ Minima walk_irregular(RingWalk w, uint32_t l, const uint32_t *list)
{
    return walk_ring<true, BITS>(w, l, list);
}

// Writes a node that a screen has decided; the centre differs from it.
template <int LAYOUT>
__device__ __forceinline__ void finish_screened(const PassArgs &a, Queue *q, int32_t node, bool accept, ulonglong2 p,
                                                ulonglong2 c, float Cx, float Cy)
{
    if (accept) {
        // the exact squared move is needed only where it can be the block's
        // largest: the screen's offset gives it to within a few units of 2^-24
        const float about = fmaf(Cx, Cx, Cy * Cy) * 1.000001f + 1e-37f;
        if (about >= *const_cast<volatile float *>(&q->best_low)) {
            const double dx = __dsub_rn(bitsd(c.x), bitsd(p.x)), dy = __dsub_rn(bitsd(c.y), bitsd(p.y));
            note_move(q, dbits(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))));
        }
    }
    CoordBits<LAYOUT>::put(a.out, a.n, node, accept ? c : p);
    if (a.accept) a.accept[node] = accept ? 1 : 0;
}

// Position of bit number k (from 0) of the set bits of m.
__device__ __forceinline__ uint32_t set_bit(unsigned m, uint32_t k)
{
    uint32_t at = 0u;
#pragma unroll
    for (uint32_t w = 16u; w > 0u; w >>= 1) {
        const uint32_t below = __popc(m & ((1u << w) - 1u));
        if (k >= below) {
            k -= below;
            m >>= w;
            at += w;
        }
    }
    return at;
}

// A quality as a signed integer of the same order (-0 below +0, which no
// comparison of the minima sees: they are compared as doubles).
__device__ __forceinline__ long long quality_key(double q)
{
    const long long b = __double_as_longlong(q);
    return b < 0 ? b ^ 0x7fffffffffffffffll : b;
}
__device__ __forceinline__ double key_quality(long long k)
{
    return __longlong_as_double(k < 0 ? k ^ 0x7fffffffffffffffll : k);
}

// FP32 offset of the centre from the node (relative error below 2^-23).  With
// equal sign and exponent field the difference is a whole number of units in
// the last place; otherwise one FP64 subtraction.
__device__ __forceinline__ void offset_of(ulonglong2 c, ulonglong2 p, float &Cx, float &Cy)
{
    const uint32_t hx = (uint32_t)(p.x >> 32), hy = (uint32_t)(p.y >> 32);
    const uint32_t ex = (hx >> 20) & 0x7ffu, ey = (hy >> 20) & 0x7ffu;
    const uint32_t other = ((uint32_t)((c.x ^ p.x) >> 32) | (uint32_t)((c.y ^ p.y) >> 32)) & 0xfff00000u;
    if (other == 0u && ex - 949u <= 200u && ey - 949u <= 200u) {
        // unit in the last place, with the sign of the coordinate
        const float ux = __uint_as_float((hx & 0x80000000u) | ((ex - 948u) << 23));
        const float uy = __uint_as_float((hy & 0x80000000u) | ((ey - 948u) << 23));
        Cx = __ll2float_rn((long long)(c.x - p.x)) * ux;
        Cy = __ll2float_rn((long long)(c.y - p.y)) * uy;
    } else {
        Cx = trunc_float(dbits(__dsub_rn(bitsd(c.x), bitsd(p.x))));
        Cy = trunc_float(dbits(__dsub_rn(bitsd(c.y), bitsd(p.y))));
    }
}

// Decides the open nodes of a warp (mask) without the queue: those for which it
// has no room, or all of a warp with many.  For each node, lane t looks at step t
// before the move and lane 16 + t after it.  First the screen again, closer: each
// side with its own radius, edge sums and largest quality (the walk has one bound
// for both sides and all qualities), and without the steps' numbers.  A node still
// open has the steps that can attain a side's minimum evaluated in FP64, 32 at a
// time from as many nodes as it takes: a node by itself would leave most lanes of
// the narrow FP64 pipe idle.  Returns per lane 1 accepted, 2 moved.
//
// What bounds it: the FP64 pipe (46 operations an item).  Meshes most of whose
// nodes are open, 1009 x 701 nodes, us a pass: flattened to 1e-3 of their height
// 237, to 1e-5 921, 1e5 away from the origin 907, rows graded by 1e6 335; a node
// at a time and without the closer screen 689, 1706, 1683, 662; one thread per node
// gathering for itself 319, 1274, 1159, 470.
//
// It holds little and finds again what it can (offsets, a node that has to wait
// for the next 32 items; one register for the lane's counts): the pass's own loop
// has to do without the registers that it takes, and spills (2% of every mesh's
// pass when it kept them).
template <int LAYOUT, int BITS>
__device__ __noinline__ uint32_t settle_open(const PassArgs &a, Queue *q, const char *xy, uint32_t half,
                                             const uint32_t *list, uint32_t cold, bool irregular, int32_t node,
                                             ulonglong2 c, uint32_t meta0, unsigned mask)
{
    const uint32_t lane = threadIdx.x & 31u;
    // the lane's state: bits 0..4 and 5..9 its item's node (by lane) and step (bit 9:
    // after the move); of its own node among the items held: 10..14 the first, 15..19
    // how many, 20..23 of those before the move; 24 accepted, 25 moved
    uint32_t state = 0u;
    uint32_t fill = 0u;  // items held
    do {
        bool evaluate = mask == 0u;
        if (mask) {
            const uint32_t src = (uint32_t)__ffs((int)mask) - 1u, t = lane & 15u;
            const bool after = lane >= 16u;
            const uint32_t meta = __shfl_sync(0xffffffffu, meta0, src), own = (win::meta_place(meta) + 1u) * 16u;
            float Cx, Cy;
            {
                ulonglong2 cs;
                cs.x = __shfl_sync(0xffffffffu, c.x, src);
                cs.y = __shfl_sync(0xffffffffu, c.y, src);
                offset_of(cs, *reinterpret_cast<const ulonglong2 *>(xy + own), Cx, Cy);
            }
            const float4 h = *reinterpret_cast<const float4 *>(xy + half + own);
            bool step = false;
            float v = FLT_MAX, s = FLT_MAX;  // cross / s and s of the lane's step and side
            float rn = 0.0f, sgn = 1.0f;
            RingVertex P, Q;
            P.x = P.y = Q.x = Q.y = 0.0f;
            if (t < win::meta_steps(meta)) {
                const uint32_t *ring = list + (int)src - (int)lane;
                const float4 hP = *reinterpret_cast<const float4 *>(xy + half + List<BITS>::at(ring, t));
                const float4 hQ = *reinterpret_cast<const float4 *>(xy + half + List<BITS>::at(ring, t + 1u));
                P = ring_vertex(hP.x, hP.y, hP.z, hP.w, h.x, h.y, h.z, h.w, Cx, Cy);
                Q = ring_vertex(hQ.x, hQ.y, hQ.z, hQ.w, h.x, h.y, h.z, h.w, Cx, Cy);
                rn = fmaxf(fmaxf(fabsf(P.x), fabsf(P.y)), fmaxf(fabsf(Q.x), fabsf(Q.y)));
                step = true;
                if (irregular) {
                    const uint32_t *row = a.win_rows + (size_t)cold * 32u + src;
                    step = ((__ldg(row) >> (2u * t)) & 3u) != 3u;
                    if ((__ldg(row + 32) >> t) & 1u) sgn = -1.0f;
                }
                if (step) {
                    float vo, vn, so, sn;
                    ring_values(P, Q, vo, vn, so, sn);
                    v = sgn * (after ? vn : vo);
                    s = after ? sn : so;
                }
            }
            float least = v, most = step ? fabsf(v) : 0.0f, smin = s;  // of the side's 16 lanes
#pragma unroll
            for (int w = 8; w > 0; w >>= 1) {
                least = fminf(least, __shfl_xor_sync(0xffffffffu, least, w));
                most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, w));
                smin = fminf(smin, __shfl_xor_sync(0xffffffffu, smin, w));
                rn = fmaxf(rn, __shfl_xor_sync(0xffffffffu, rn, w));
            }
            const float rN = fmaxf(rn, fmaxf(fabsf(Cx), fabsf(Cy)));
            const float M = fmaxf(fabsf(h.x), fabsf(h.z)) * 1.0001f + rN;
            const float g = side_g(after ? rN : rn, smin), amax = kTwoSqrt3f * most;
            const bool ok = frame_ok(rn, rN, M) & bound_ok(smin, g, amax);
            const float b = side_bound(amax, g), up = kTwoSqrt3f * least + b, lo = kTwoSqrt3f * least - b;
            const unsigned cands = __ballot_sync(0xffffffffu, step && !(ok && kTwoSqrt3f * v - b > up));
            const bool both = __all_sync(0xffffffffu, ok);
            const bool above = __shfl_sync(0xffffffffu, lo, 16) > __shfl_sync(0xffffffffu, up, 0);
            const bool below = __shfl_sync(0xffffffffu, up, 16) < __shfl_sync(0xffffffffu, lo, 0);
            int verdict = both ? (above ? 1 : (below ? -1 : 0)) : 0;
            const unsigned first = cands & 0xffffu;
            if (both && verdict == 0 && first == cands >> 16 && (first & (first - 1u)) == 0u) {
                verdict = diff_screen(P.x, P.y, Q.x, Q.y, Cx, Cy, sgn, M * M);
                verdict = __shfl_sync(0xffffffffu, verdict, __ffs((int)first) - 1);
            }
            const uint32_t cnt = __popc(cands);
            if (verdict != 0) {
                mask &= mask - 1u;
                if (lane == src) {
                    finish_screened<LAYOUT>(a, q, node, verdict > 0,
                                            *reinterpret_cast<const ulonglong2 *>(xy + own), c, Cx, Cy);
                    if (verdict > 0) state |= 3u << 24;
                }
            } else if (fill + cnt <= 32u) {
                mask &= mask - 1u;
                if (lane >= fill && lane < fill + cnt)
                    state = (state & ~0x3ffu) | src | (set_bit(cands, lane - fill) << 5);
                if (lane == src) state |= (fill << 10) | (cnt << 15) | (__popc(first) << 20);
                fill += cnt;
            } else {  // it comes again once there is room
                evaluate = true;
            }
        }
        if (evaluate && fill > 0u) {
            const uint32_t of = state & 31u, ts = (state >> 5) & 15u;
            const uint32_t own = (win::meta_place(__shfl_sync(0xffffffffu, meta0, of)) + 1u) * 16u;
            long long key;
            {
                ulonglong2 x;
                x.x = __shfl_sync(0xffffffffu, c.x, of);
                x.y = __shfl_sync(0xffffffffu, c.y, of);
                const uint32_t *row = a.win_rows + (size_t)cold * 32u + of;
                key = quality_key(bitsd(0x7ff0000000000000ull));
                if (lane < fill) {
                    if (!(state & 0x200u)) x = *reinterpret_cast<const ulonglong2 *>(xy + own);
                    const uint32_t *ring = list + (int)of - (int)lane;
                    const ulonglong2 A = *reinterpret_cast<const ulonglong2 *>(xy + List<BITS>::at(ring, ts));
                    const ulonglong2 B = *reinterpret_cast<const ulonglong2 *>(xy + List<BITS>::at(ring, ts + 1u));
                    key = quality_key(step_quality(x, A.x, A.y, B.x, B.y, __ldg(row), __ldg(row + 32), ts));
                }
            }
            const uint32_t i0 = (state >> 10) & 31u, n = (state >> 15) & 31u, n_old = (state >> 20) & 15u;
            const uint32_t most = __reduce_max_sync(0xffffffffu, n);
            long long k_old = quality_key(bitsd(0x7ff0000000000000ull)), k_new = k_old;
            for (uint32_t k = 0; k < most; ++k) {
                const long long u = __shfl_sync(0xffffffffu, key, (int)((i0 + k) & 31u));
                if (k < n_old) k_old = u < k_old ? u : k_old;
                else if (k < n) k_new = u < k_new ? u : k_new;
            }
            if (n) {
                unsigned long long b2;
                bool acc, moved;
                const ulonglong2 p =
                    *reinterpret_cast<const ulonglong2 *>(xy + (win::meta_place(meta0) + 1u) * 16u);
                finish_exact<LAYOUT>(a, node, make_double2(bitsd(p.x), bitsd(p.y)), make_double2(bitsd(c.x), bitsd(c.y)),
                                     key_quality(k_old), key_quality(k_new), b2, acc, moved);
                note_move(q, b2);
                state |= ((acc ? 1u : 0u) | (moved ? 2u : 0u)) << 24;
            }
            state &= ~0xfffc00u;
            fill = 0u;
        }
    } while (mask | fill);
    return state >> 24;
}

// What a lane knows of a node that its screen left open.
struct Open {
    float Cx, Cy;        // the centre's offset
    float b, up_o, up_n; // a step is a candidate unless its value less b lies above the side's up
    uint32_t own, steps;
    uint32_t meta;       // the lane's meta word
};

// Open nodes of a warp from which it settles them itself (settle_open): its items
// then fill the FP64 pipe's lanes without the block's queue, and the closer screen
// decides a part.  A mesh flattened to 1e-3 (15 of 32 nodes open) takes 264 us a
// pass without this, 237 with 16, 217 with 12; 100,000 Delaunay points, few of whose
// warps have as many, take 1.36 ms a call with 16, 1.37 with 12 and 1.41 with 8.
constexpr int kManyOpen = 16;

// The nodes of a warp that its screen left open (mask): for each, lane t looks
// at step t before the move and lane 16 + t after it; the steps that can
// attain a side's minimum go into the queue.  The others: settle_open.  list: a
// lane's ring; cold: the subtile's slots row.  Returns per lane 1 accepted, 2
// moved (decided here), 8 queue full enough to be worked off.
template <int LAYOUT, int BITS>
__device__ __noinline__ uint32_t work_open(const PassArgs &a, Queue *q, const char *xy, uint32_t half,
                                           const uint32_t *list, uint32_t cold, bool irregular, int32_t node,
                                           ulonglong2 c, Open o, unsigned mask)
{
    const uint32_t lane = threadIdx.x & 31u, t = lane & 15u;
    const bool after = lane >= 16u;
    uint32_t out = 0u;
    unsigned left = 0u;
    if (__popc(mask) >= kManyOpen) {
        left = mask;
        mask = 0u;
    }
    for (; mask; mask &= mask - 1u) {
        const uint32_t src = (uint32_t)__ffs((int)mask) - 1u;
        const uint32_t own = __shfl_sync(0xffffffffu, o.own, src), steps = __shfl_sync(0xffffffffu, o.steps, src);
        const float Cx = __shfl_sync(0xffffffffu, o.Cx, src), Cy = __shfl_sync(0xffffffffu, o.Cy, src);
        const float b = __shfl_sync(0xffffffffu, o.b, src);
        const float up_o = __shfl_sync(0xffffffffu, o.up_o, src), up_n = __shfl_sync(0xffffffffu, o.up_n, src);
        const uint32_t *ring = list + (int)src - (int)lane;
        const uint32_t *row = a.win_rows + (size_t)cold * 32u + src;
        uint32_t eP = 0u, eQ = 0u;
        bool cand = false;
        if (t < steps) {
            eP = List<BITS>::at(ring, t);
            eQ = List<BITS>::at(ring, t + 1u);
            const float4 h = *reinterpret_cast<const float4 *>(xy + half + own);
            const float4 hP = *reinterpret_cast<const float4 *>(xy + half + eP);
            const float4 hQ = *reinterpret_cast<const float4 *>(xy + half + eQ);
            const RingVertex P = ring_vertex(hP.x, hP.y, hP.z, hP.w, h.x, h.y, h.z, h.w, Cx, Cy);
            const RingVertex Q = ring_vertex(hQ.x, hQ.y, hQ.z, hQ.w, h.x, h.y, h.z, h.w, Cx, Cy);
            float vo, vn, so, sn;
            ring_values(P, Q, vo, vn, so, sn);
            float v = after ? vn : vo;
            cand = true;
            if (irregular) {
                cand = ((__ldg(row) >> (2u * t)) & 3u) != 3u;
                if ((__ldg(row + 32) >> t) & 1u) v = -v;
            }
            cand = cand && !(kTwoSqrt3f * with_step(v, t) - b > (after ? up_n : up_o));
        }
        const unsigned cands = __ballot_sync(0xffffffffu, cand);
        const uint32_t cnt = __popc(cands), place = __popc(cands & ((1u << lane) - 1u));
        uint32_t e = 0u, i0 = 0u;
        if (lane == 0u) {
            e = atomicAdd(&q->npending, 1u);
            i0 = atomicAdd(&q->nitems, cnt);
        }
        e = __shfl_sync(0xffffffffu, e, 0);
        i0 = __shfl_sync(0xffffffffu, i0, 0);
        if (e + 1u >= (uint32_t)kPendingFull || i0 + cnt >= (uint32_t)kItemsFull) out |= 8u;
        const ulonglong2 P = *reinterpret_cast<const ulonglong2 *>(xy + eP);
        const ulonglong2 Q = *reinterpret_cast<const ulonglong2 *>(xy + eQ);
        if (e < (uint32_t)kPending && i0 + cnt <= (uint32_t)kItems) {
            if (cand) {
                const uint32_t at = i0 + place;
                q->px[at] = bitsd(P.x);
                q->py[at] = bitsd(P.y);
                q->qx[at] = bitsd(Q.x);
                q->qy[at] = bitsd(Q.y);
                q->item[at] = e | (after ? 0x100u : 0u) | (t << 9);
            }
            if (lane == src) {
                q->p[e] = *reinterpret_cast<const ulonglong2 *>(xy + own);
                q->c[e] = c;
                q->node[e] = node;
                q->cold[e] = cold;
                q->range[e] = i0 | (cnt << 8) | (lane << 16);
            }
            continue;
        }
        // no room: what was claimed stays empty
        if (i0 + lane < (uint32_t)kItems && lane < cnt) q->item[i0 + lane] = kNoItem;
        if (lane == 0u && e < (uint32_t)kPending) q->node[e] = -1;
        left |= 1u << src;
    }
    if (left) out |= settle_open<LAYOUT, BITS>(a, q, xy, half, list, cold, irregular, node, c, o.meta, left);
    return out;
}

// A subtile's rows, for one lane.
struct Rows {
    const uint32_t *at;    // the lane's word of the first row (shared memory)
    uint32_t cold;         // its slots row of the stream; its directions row is the next
    uint32_t d, l;         // the subtile's largest degree and step number
    uint32_t meta;
    bool irregular;
};

// Updates the free node a lane holds (Eq. 2 and the accept test of Section
// 3.3.4).  res: bit 0 accepted, bit 1 coordinates changed.  Returns true when
// the node's record has to decide (a coordinate outside the splits' range).
template <int LAYOUT, int BITS>
__device__ __forceinline__ bool update_lane(const PassArgs &a, Queue *q, const char *xy, uint32_t half, const Rows &r,
                                            int32_t node, Tally &tally, uint32_t &res, bool &full)
{
    using L = List<BITS>;
    const uint32_t deg = win::meta_deg(r.meta), steps = win::meta_steps(r.meta);
    const uint32_t own = (win::meta_place(r.meta) + 1u) * 16u;
    // the sums, to the subtile's largest degree: lists are padded with the
    // entry that holds (-0, -0)
    const uint32_t *list = r.at + 32;
    uint32_t word = *list;
    double sx = 0.0, sy = 0.0;
    for (uint32_t k = 0;;) {  // four neighbours' loads go out together
        ulonglong2 v[4];
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
            if (j > 0u && j % L::kPer == 0u) word = list[32u * (j / L::kPer)];
            v[j] = *reinterpret_cast<const ulonglong2 *>(xy + L::in_word(word, j % L::kPer));
        }
        // branches out, not conditions: an addition that is not due must not
        // occupy the FP64 pipe
        if (k == 0u) {
            sx = bitsd(v[0].x);
            sy = bitsd(v[0].y);
        } else {
            sx = __dadd_rn(sx, bitsd(v[0].x));
            sy = __dadd_rn(sy, bitsd(v[0].y));
        }
        if (++k >= r.d) break;
        sx = __dadd_rn(sx, bitsd(v[1].x));
        sy = __dadd_rn(sy, bitsd(v[1].y));
        if (++k >= r.d) break;
        sx = __dadd_rn(sx, bitsd(v[2].x));
        sy = __dadd_rn(sy, bitsd(v[2].y));
        if (++k >= r.d) break;
        sx = __dadd_rn(sx, bitsd(v[3].x));
        sy = __dadd_rn(sy, bitsd(v[3].y));
        if (++k >= r.d) break;
        list += 32u * (4u / L::kPer);
        word = *list;
    }
    list = r.at + 32u * (1u + win::list_rows(r.d, BITS));  // the ring
    res = 0u;
    const bool free = (r.meta & win::kFree) != 0u;
    const ulonglong2 pb = *reinterpret_cast<const ulonglong2 *>(xy + own);
    ulonglong2 cb = pb;
    if (free) {
        const double y = c_recip[deg];
        bool okx, oky;
        cb.x = divs::div_small_fast(dbits(sx), deg, y, okx);
        cb.y = divs::div_small_fast(dbits(sy), deg, y, oky);
        if (!(okx & oky)) {
            const double fd = c_degree[deg];
            cb.x = dbits(__ddiv_rn(sx, fd));
            cb.y = dbits(__ddiv_rn(sy, fd));
        }
    }
    bool act = cb.x != pb.x || cb.y != pb.y;
    if (free && !act) {
        // the centre is the node itself: q_new == q_old exactly
        const bool acc = !a.strict;
        CoordBits<LAYOUT>::put(a.out, a.n, node, pb);
        if (a.accept) a.accept[node] = acc ? 1 : 0;
        tally.nacc += acc ? 1u : 0u;
        res = acc ? 1u : 0u;
    }
    bool record = false;
    if (__any_sync(0xffffffffu, act)) {
        int verdict = 0;
        RingWalk w;
        w.split = xy + half;
        {
            const float4 h = *reinterpret_cast<const float4 *>(xy + half + own);
            w.phx = h.x;
            w.plx = h.y;
            w.phy = h.z;
            w.ply = h.w;
        }
        w.Cx = w.Cy = 0.0f;
        if (act) offset_of(cb, pb, w.Cx, w.Cy);
        w.slots = w.rev = 0u;
        Minima m;
        if (r.irregular) {
            const uint32_t *row = a.win_rows + (size_t)r.cold * 32u + (threadIdx.x & 31u);
            w.slots = __ldg(row);
            w.rev = __ldg(row + 32);
            m = walk_irregular<BITS>(w, r.l, list);
        } else {
            m = walk_ring<false, BITS>(w, r.l, list);
        }
        // a coordinate of the node or of a neighbour outside the splits' range
        record = act && !(fmaxf(m.rn, fmaxf(fabsf(w.phx), fabsf(w.phy))) < FLT_MAX);
        act = act && !record;
        const float rN = fmaxf(m.rn, fmaxf(fabsf(w.Cx), fabsf(w.Cy)));
        const float M = fmaxf(fabsf(w.phx), fabsf(w.phy)) * 1.0001f + rN;
        const float g = side_g(rN, m.smin);
        const bool bok = frame_ok(m.rn, rN, M) & ring_ok(m.smin, g);
        Open o;
        o.b = ring_bound(g);
        // per side: q (FP64) lies in [amin - b, amin + b]; the minimum is attained
        // by one triangle alone when every other value lies above amin + b + b
        const float amin_o = kTwoSqrt3f * m.m1o, amin_n = kTwoSqrt3f * m.m1n;
        o.up_o = amin_o + o.b;
        o.up_n = amin_n + o.b;
        if (act && bok) verdict = amin_n - o.b > o.up_o ? 1 : (o.up_n < amin_o - o.b ? -1 : 0);
        const uint32_t to = step_of(m.m1o);
        if (act && verdict == 0 && bok && to == step_of(m.m1n) && kTwoSqrt3f * m.m2o - o.b > o.up_o &&
            kTwoSqrt3f * m.m2n - o.b > o.up_n) {
            const RingVertex P = w.vertex(L::at(list, to)), Q = w.vertex(L::at(list, to + 1u));
            verdict = diff_screen(P.x, P.y, Q.x, Q.y, w.Cx, w.Cy, ((w.rev >> to) & 1u) ? -1.0f : 1.0f, M * M);
        }
        const unsigned open = __ballot_sync(0xffffffffu, act && verdict == 0);
        if (act && verdict > 0) {
            // the exact squared move is needed only where it can be the block's
            // largest: the screen's offset gives it to within a few units of 2^-24
            const float about = fmaf(w.Cx, w.Cx, w.Cy * w.Cy) * 1.000001f + 1e-37f;
            if (about >= *const_cast<volatile float *>(&q->best_low)) {
                const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(xy + own);
                const double dx = __dsub_rn(bitsd(cb.x), bitsd(p.x)), dy = __dsub_rn(bitsd(cb.y), bitsd(p.y));
                note_move(q, dbits(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))));
            }
            tally.nacc += 1u;
            res = 3u;  // the centre differs from the node (equal centres are done above)
        }
        if (verdict != 0) {
            if (verdict < 0) cb = *reinterpret_cast<const ulonglong2 *>(xy + own);
            CoordBits<LAYOUT>::put(a.out, a.n, node, cb);
            if (a.accept) a.accept[node] = verdict > 0 ? 1 : 0;
        }
        if (open) {
            if (act && verdict == 0) tally.nexact += 1u;
            if (!bok) {  // every step is a candidate
                o.b = 0.0f;
                o.up_o = o.up_n = __int_as_float(0x7f800000);
            }
            o.Cx = w.Cx;
            o.Cy = w.Cy;
            o.own = own;
            o.steps = steps;
            o.meta = r.meta;
            const uint32_t done =
                work_open<LAYOUT, BITS>(a, q, xy, half, list, r.cold, r.irregular, node, cb, o, open);
            full = full || (done & 8u);
            if (done & 3u) res = done & 3u;
            tally.nacc += done & 1u;
        }
    }
    return record;
}

// ---- a block's windows ----------------------------------------------------------

// Nodes of a subtile that their records decide, a warp each.  Coordinates come
// from L2: all kernels but those with masks (HALO) start early or run several
// passes, so they may be resident while the coordinates that they will read
// are still being written, and the read-only path (__ldg) is for data that
// nobody writes while the kernel lives.
template <int LAYOUT, bool HALO>
__device__ __noinline__ Tally by_record(const PassArgs &a, Queue *q, int32_t node, unsigned left, Tally tally)
{
    while (left) {
        const int src = __ffs((int)left) - 1;
        left &= left - 1u;
        const int32_t nd = __shfl_sync(0xffffffffu, node, src);
        unsigned long long b2;
        bool acc, moved;
        exact_update_warp<LAYOUT, !HALO>(a, nd, b2, acc, moved);
        if ((threadIdx.x & 31) == 0) {
            note_move(q, b2);
            tally.nacc += acc ? 1u : 0u;
            tally.nexact += 1u;
            if (HALO) {
                const uint32_t bit = 1u << (nd & 31);
                if (moved) atomicOr(a.chg_cur + (nd >> 5), bit);
                if (acc) atomicOr(a.accm + (nd >> 5), bit);
            }
        }
    }
    return tally;
}

// Splits the staged entries a thread copied itself (first, first + step, ...).
__device__ __forceinline__ void split_staged(char *xy, uint32_t half, uint32_t staged, uint32_t first, uint32_t step)
{
    for (uint32_t e = first; e < staged; e += step) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(xy + (e + 1u) * 16u);
        float4 s;
        const bool okx = head_tail(v.x, s.x, s.y), oky = head_tail(v.y, s.z, s.w);
        // no split: the rings it is on then fail their range check
        if (!(okx & oky)) s = make_float4(__int_as_float(0x7f800000), 0.f, __int_as_float(0x7f800000), 0.f);
        *reinterpret_cast<float4 *>(xy + half + (e + 1u) * 16u) = s;
    }
}

// Updates the nodes of subtile `sub` of a staged window (h: its header, rows:
// its hot rows in shared memory).
template <int LAYOUT, int BITS, bool HALO>
__device__ __forceinline__ void work_subtile(const PassArgs &a, Queue *q, const char *xy, uint32_t half,
                                             const uint32_t *h, const uint32_t *rows, int sub, Tally &tally,
                                             bool &full)
{
    const int lane = threadIdx.x & 31;
    Rows r;
    r.d = (h[3] >> (8 * sub)) & 15u;
    r.l = (h[3] >> (8 * sub + 4)) & 15u;
    r.at = rows + ((h[4] >> (8 * sub)) & 0xffu) * 32u + lane;
    r.cold = h[0] + win::halo_rows(win::hdr_halo(h[2])) + h[5] + 2u * sub;
    r.meta = *r.at;
    r.irregular = win::hdr_irregular(h[2], (uint32_t)sub);
    const int32_t node = (int32_t)(h[1] + win::meta_place(r.meta));
    const bool have = (r.meta & win::kNode) != 0u;
    if (have && !(r.meta & (win::kFree | win::kBig)) && a.accept) a.accept[node] = 0;
    uint32_t res = 0u;
    bool record = have && (r.meta & win::kBig);
    if (r.d > 0u) record |= update_lane<LAYOUT, BITS>(a, q, xy, half, r, node, tally, res, full);
    __syncwarp();
    if (HALO) {  // before any other write to the tile's masks
        const int64_t wt = (int64_t)(h[1] >> 5) + sub;
        const unsigned cb = __ballot_sync(0xffffffffu, (res & 2u) != 0u);
        const unsigned ab = __ballot_sync(0xffffffffu, (res & 1u) != 0u);
        if (lane == 0 && wt * 32 < (int64_t)h[1] + win::hdr_count(h[2])) {
            a.chg_cur[wt] = cb;
            a.accm[wt] = ab;
        }
    }
    const unsigned left = __ballot_sync(0xffffffffu, record);
    if (left) tally = by_record<LAYOUT, HALO>(a, q, node, left, tally);
}

// Works windows w0, w0 + stride, ... (n of them).  Every thread of the block
// calls it; `full` is this thread's note that the queue should be worked off,
// which happens at the next window's barrier.
//
// Window i's data was copied in while window i - 1 was worked on; one barrier
// per window says that it is there and that window i - 1, whose buffer the
// next copies overwrite, is finished.  (With one buffer of staged entries the
// copies wait for that barrier, and a second one says that they are there.)
//
// EARLY: the kernel may have started before the one in front of it ended
// (after_previous); whether the pass is to run is known only then.
// TWO: there are two buffers whatever the windows (8-bit lists: at most 255
// entries).
template <int LAYOUT, int BITS, bool HALO, bool EARLY, bool TWO>
__device__ __forceinline__ void run_windows(const PassArgs &a, const Block &blk, int64_t w0, int n, int64_t stride,
                                            Tally &tally, unsigned &nskip, bool &full)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
    Ahead *ah = blk.ahead;
    const bool two = blk.stage != 0u;

    auto fetch_header = [&](int i) {
        if (i < n && tid < 2)
            copy16(&ah->hdr[i & 3][4 * tid], a.win_hdr + (w0 + i * stride) * win::kHeaderWords + 4 * tid);
    };
    auto fetch_ids = [&](int i) {
        if (i >= n) return;
        const uint32_t *h = ah->hdr[i & 3];
        const uint32_t *src = a.win_rows + (size_t)h[0] * 32u;
        uint32_t *dst = blk.ids + (i & 1) * blk.ids_words;
        for (uint32_t k = 4 * tid; k < win::hdr_halo(h[2]); k += 4 * nthr) copy16(dst + k, src + k);
    };
    auto all_idle = [&](int i) {
        return HALO && a.skip && *reinterpret_cast<const uint32_t *>(ah->idle[i & 3]) == 0x01010101u;
    };
    auto fetch_data = [&](int i) {
        if (i >= n || all_idle(i)) return;
        const uint32_t *h = ah->hdr[i & 3];
        const uint32_t count = win::hdr_count(h[2]), nhalo = win::hdr_halo(h[2]);
        const uint32_t *src = a.win_rows + ((size_t)h[0] + win::halo_rows(nhalo)) * 32u;
        uint32_t *rows = blk.rows + (TWO || two ? i & 1 : 0) * blk.rows_words;
        for (uint32_t k = 4 * tid; k < 32u * h[5]; k += 4 * nthr) copy16(rows + k, src + k);
        const uint32_t *ids = blk.ids + (i & 1) * blk.ids_words;
        char *xy = blk.xy + (i & 1) * blk.stage + 16;
        for (uint32_t e = tid; e < count + nhalo; e += nthr) {
            const int64_t id = e < count ? (int64_t)h[1] + e : (int64_t)ids[e - count];
            if (LAYOUT == 0) {
                copy16(xy + e * 16u, a.in + 2 * id);
            } else {
                copy8(xy + e * 16u, a.in + id);
                copy8(xy + e * 16u + 8u, a.in + a.n + id);
            }
        }
    };
    // skip_unchanged: whether the subtiles of window i have only unchanged
    // inputs; such a tile's results are those of the previous pass, which
    // `out` and the masks already hold
    auto check_idle = [&](int i) {
        if (!HALO || !a.skip || i >= n) return;
        const uint32_t *h = ah->hdr[i & 3];
        for (int sub = warp; sub < 4; sub += nwarps) {
            const int64_t wt = (int64_t)(h[1] >> 5) + sub;
            bool idle = true;
            if (wt * 32 < (int64_t)h[1] + win::hdr_count(h[2])) {
                // the tile's inputs: its own nodes and every neighbour, by tile
                const uint2 e = lane < kHaloEntries ? __ldg(a.halo + wt * kHaloEntries + lane) : make_uint2(0u, 0u);
                const bool never = __shfl_sync(0xffffffffu, e.x, 0) == kHaloNever;
                const uint32_t c = e.y != 0u && !never ? __ldg(a.chg_prev + e.x) & e.y : 0u;
                idle = !__any_sync(0xffffffffu, c != 0u) && !never;
                if (idle && lane == 0) {
                    a.chg_cur[wt] = 0u;
                    tally.nacc += (unsigned)__popc(a.accm[wt]);
                    nskip += (unsigned)(a.n - wt * 32 < 32 ? a.n - wt * 32 : 32);
                }
            }
            if (lane == 0) ah->idle[i & 3][sub] = idle ? 1 : 0;
        }
    };

    __syncthreads();  // whatever was worked on before is finished
    fetch_header(0);
    fetch_header(1);
    fetch_header(2);
    copies_done();
    __syncthreads();
    fetch_ids(0);
    fetch_ids(1);
    if (!EARLY) {
        check_idle(0);
        check_idle(1);
    }
    copies_done();
    __syncthreads();
    if (EARLY) {
        after_previous();
        if (pass_is_skipped(a.stats, a.q, a.tol_active, a.thr_bits)) return;
        if (blockIdx.x == 0 && tid == 0) a.stats[a.q].executed = 1u;
    }
    if (two) fetch_data(0);
    for (int i = 0; i < n; ++i) {
        if (!two) {  // one buffer: window i - 1 has to be finished first
            copies_done();
            __syncthreads();
            fetch_data(i);
        }
        copies_done();
        char *xy = blk.xy + (i & 1) * blk.stage;
        const uint32_t *h = ah->hdr[i & 3];
        const bool rest = all_idle(i);
        if (!rest) {
            split_staged(xy, blk.half, win::hdr_count(h[2]) + win::hdr_halo(h[2]), tid, nthr);
        }
        if (__syncthreads_or(full)) {
            tally = drain<LAYOUT, HALO>(a, blk.q, tally);
            full = false;
        }
        if (two) fetch_data(i + 1);
        fetch_ids(i + 2);
        fetch_header(i + 3);
        check_idle(i + 2);
        if (rest) continue;
        for (int sub = warp; sub < 4; sub += nwarps) {
            if (HALO && a.skip && ah->idle[i & 3][sub]) continue;
            work_subtile<LAYOUT, BITS, HALO>(a, blk.q, xy, blk.half, h,
                                             blk.rows + (TWO || two ? i & 1 : 0) * blk.rows_words, sub, tally,
                                                    full);
        }
    }
}

// The kernels are compiled for 7 blocks of 128 threads per SM (72 registers):
// 2048^2 ran 201 us a pass with 7, 207 with 6 and 218 with 8, whose 64
// registers spill, when this was chosen (174 now).
constexpr int kBlocksPerSm = 7;

// HALO: the mesh keeps the masks of skip_unchanged (apart: their code costs
// other meshes registers, 217 against 202 us a pass on 2048^2 at the time).
template <int LAYOUT, int BITS, bool HALO>
__global__ void __launch_bounds__(kBlockMax, kBlocksPerSm)
    pass_screened_kernel(const __grid_constant__ PassArgs a, const __grid_constant__ WindowShape shape)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // (the masks of skip_unchanged are read where a window's header is: no early start)
    if (HALO || a.win_count == 0) {  // the launch over an empty list has no window to start with
        if (!HALO) after_previous();
        if (pass_is_skipped(a.stats, a.q, a.tol_active, a.thr_bits)) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) a.stats[a.q].executed = 1u;
    }
    const Block blk = block_memory<BITS == 8>(smem_raw, shape);
    Tally tally{0u, 0u};
    unsigned nskip = 0u;  // node updates this warp left as they were (lane 0)
    bool full = false;
    if ((int64_t)blockIdx.x < a.win_count)
        run_windows<LAYOUT, BITS, HALO, !HALO, BITS == 8>(
            a, blk, a.win_first + blockIdx.x, (int)((a.win_count - blockIdx.x + gridDim.x - 1) / gridDim.x), gridDim.x,
            tally, nskip, full);
    __syncthreads();
    if (blk.q->npending) tally = drain<LAYOUT, HALO>(a, blk.q, tally);
    if (nskip) atomicAdd(&a.stats[a.q].nodes_skipped, nskip);
    flush(blk.q, a.stats + a.q, tally);
}

// ---- all passes of a small mesh in one launch -----------------------------------
// A mesh with at most one window per resident block: every block keeps its
// window's lists in shared memory and runs pass after pass, with a grid-wide
// barrier between passes instead of a launch.  What is left of a pass is its
// own chain of dependent steps (coordinates from L2, the sums, the ring walk,
// the queue, the barrier).  A 64^2 mesh runs 9.3 us a pass against 13.5 with an
// ordinary launch each, 100,000 Delaunay points 16 to 19 against 23; past one window per
// resident block (about 136,000 nodes) the blocks would have to fetch their
// lists again every pass, as separate launches do.

struct __align__(8) GridBarrier {
    unsigned int arrived;  // blocks that arrived, over all passes of the launch
    unsigned int lost;     // a wait ran out: nobody waits or computes any more, in this launch or in a
                           // later one of the call (the call's end reads it)
};

__device__ __forceinline__ unsigned long long barrier_words(GridBarrier *b)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(b) : "memory");
    return v;  // arrived, lost << 32
}

// All threads call it; false when some block's wait ran out (after `limit`
// polls).  Writes to global memory before it are visible after it to reads
// from L2.
__device__ __forceinline__ bool grid_barrier(GridBarrier *b, unsigned target, unsigned limit)
{
    __shared__ bool s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&b->arrived, 1u);
        unsigned long long seen = 0ull;
        unsigned polls = 0u;
        do {
            seen = barrier_words(b);
        } while ((unsigned)seen < target && (seen >> 32) == 0ull && ++polls < limit);
        s_ok = (unsigned)seen >= target && (seen >> 32) == 0ull;
        if (!s_ok) atomicExch(&b->lost, 1u);
    }
    __syncthreads();
    return s_ok;
}

template <int LAYOUT, int BITS>
__global__ void __launch_bounds__(kBlockMax, kBlocksPerSm)
    resident_kernel(const __grid_constant__ PassArgs a0, const __grid_constant__ WindowShape shape, int passes,
                    GridBarrier *barrier, unsigned poll_limit)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ PassArgs s_args;
    __shared__ bool s_stop;
    const int tid = threadIdx.x, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
    const Block blk = block_memory<BITS == 8>(smem_raw, shape);
    if (tid == 0) {
        s_args = a0;
        s_stop = pass_is_skipped(a0.stats, a0.q, a0.tol_active, a0.thr_bits) || (barrier_words(barrier) >> 32) != 0ull;
    }
    // the window's header, halo ids and lists, once
    uint32_t *h = blk.ahead->hdr[0];
    if (tid < 2) copy16(h + 4 * tid, a0.win_hdr + (size_t)blockIdx.x * win::kHeaderWords + 4 * tid);
    copies_done();
    __syncthreads();
    if (s_stop) return;
    const uint32_t count = win::hdr_count(h[2]), nhalo = win::hdr_halo(h[2]), staged = count + nhalo;
    const uint32_t *src = a0.win_rows + (size_t)h[0] * 32u;
    for (uint32_t k = 4 * tid; k < nhalo; k += 4 * nthr) copy16(blk.ids + k, src + k);
    src += win::halo_rows(nhalo) * 32u;
    for (uint32_t k = 4 * tid; k < 32u * h[5]; k += 4 * nthr) copy16(blk.rows + k, src + k);
    copies_done();
    __syncthreads();
    const PassArgs &a = s_args;
    const double *in = a0.in;
    for (int done = 1;; ++done) {
        for (uint32_t e = tid; e < staged; e += nthr) {  // from L2: other blocks wrote them
            const int64_t id = e < count ? (int64_t)h[1] + e : (int64_t)blk.ids[e - count];
            char *dst = blk.xy + (e + 1u) * 16u;
            if (LAYOUT == 0) {
                copy16(dst, in + 2 * id);
            } else {
                *reinterpret_cast<double2 *>(dst) = make_double2(__ldcg(in + id), __ldcg(in + a0.n + id));
            }
        }
        if (tid == 0 && done > 1 && a0.tol_active) {  // the pass before met the tolerance
            unsigned long long moved;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(moved) : "l"(&a0.stats[a.q - 1].maxd2_bits));
            s_stop = moved < a0.thr_bits;
        }
        copies_done();
        split_staged(blk.xy, blk.half, staged, tid, nthr);
        __syncthreads();
        if (s_stop) return;
        if (blockIdx.x == 0 && tid == 0) a.stats[a.q].executed = 1u;
        Tally tally{0u, 0u};
        bool full = false;  // (one window: the queue is worked off after it)
        for (int sub = warp; sub < 4; sub += nwarps)
            work_subtile<LAYOUT, BITS, false>(a, blk.q, blk.xy, blk.half, h, blk.rows, sub, tally, full);
        __syncthreads();
        if (blk.q->npending) tally = drain<LAYOUT, false>(a, blk.q, tally);
        flush(blk.q, a.stats + a.q, tally);
        if (done == passes) return;
        in = (done & 1) ? a0.out : a0.in;
        if (tid == 0) {
            s_args.in = in;
            s_args.out = (done & 1) ? const_cast<double *>(a0.in) : a0.out;
            s_args.q += 1;
        }
        if (!grid_barrier(barrier, (unsigned)done * gridDim.x, poll_limit)) return;
    }
}

// ---- batched / served form: many meshes, one launch per round -----------
// Work is a list of window tasks.  With chunk > 0 the blocks take chunks of
// `chunk` consecutive tasks in a grid stride (block b: chunks b, b + B,
// b + 2B, ...); with chunk < 0 they claim chunks of -chunk tasks in list order
// from the round's counter (*claim, zero at the launch); chunk = 0 gives each
// block one contiguous share of the list.  A job takes part in round r as its
// pass q = r - base_round while q < max_iter and its tolerance is not met.
// The queue is worked off and the statistics flushed whenever the block moves
// to another job, so every record gets exactly its own job's counts.
// WIDE: some job's lists may have 16-bit entries.
// (The tables may be written by the kernel in front, so they are not
// __restrict__: a load known never to change could move above after_previous.)
template <int LAYOUT, bool WIDE>
__global__ void __launch_bounds__(kBlockMax, kBlocksPerSm)
    batch_pass_kernel(const JobDesc *jobs, const WindowTask *tasks, int64_t ntasks,
                      int round, int64_t chunk, unsigned long long *claim, const __grid_constant__ WindowShape shape)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ PassArgs s_args;
    __shared__ int64_t s_claim;
    __shared__ int s_active, s_wide, s_windows;
    const Block blk = block_memory<!WIDE>(smem_raw, shape);
    const bool dynamic = chunk < 0;
    const int64_t nblocks = gridDim.x;
    const int64_t per = chunk > 0 ? chunk : (dynamic ? -chunk : (ntasks + nblocks - 1) / nblocks);
    const int64_t cstride = chunk > 0 ? nblocks * chunk : ntasks;  // one share per block when chunk == 0
    auto claim_next = [&]() -> int64_t {
        __syncthreads();
        if (threadIdx.x == 0) s_claim = (int64_t)atomicAdd(claim, (unsigned long long)per);
        __syncthreads();
        return s_claim;
    };
    int64_t c0 = dynamic ? claim_next() : (int64_t)blockIdx.x * per;  // first task of the current chunk
    after_previous();  // (a round has its own claim counter)
    int64_t t = c0;
    int cur_job = -1;
    Tally tally{0u, 0u};
    unsigned nskip = 0u;
    bool full = false, active = false;
    for (;;) {
        if (t >= c0 + per || t >= ntasks) {  // next chunk of this block
            c0 = dynamic ? (c0 < ntasks ? claim_next() : c0) : c0 + cstride;
            t = c0;
        }
        const bool more = t < ntasks && c0 < ntasks;
        const int job = more ? tasks[t].job : -2;
        if (job != cur_job) {
            __syncthreads();
            if (cur_job >= 0 && active) {
                if (blk.q->npending) tally = drain<LAYOUT, false>(s_args, blk.q, tally);
                flush(blk.q, s_args.stats + s_args.q, tally);
                __syncthreads();
            }
            tally = Tally{0u, 0u};
            full = false;
            cur_job = job;
            if (job < 0) break;
            if (threadIdx.x == 0) {
                const JobDesc *J = jobs + job;
                const int q = round - J->base_round;
                PassArgs &a = s_args;
                a = PassArgs{};
                const bool odd = ((J->cur0 + q) & 1) != 0;
                a.in = odd ? J->xy[1] : J->xy[0];
                a.out = odd ? J->xy[0] : J->xy[1];
                a.node_off = J->node_off;
                a.adj = J->adj;
                a.n = J->n;
                a.win_hdr = J->win_hdr;
                a.win_rows = J->win_rows;
                a.stats = J->stats;
                a.q = q;
                a.strict = J->strict;
                a.tol_active = J->tol_active;
                a.thr_bits = J->thr_bits;
                a.accept = J->accept;
                s_wide = J->bits != 8;
                s_windows = J->windows;
                s_active = q >= 0 && q < J->max_iter && !pass_is_skipped(J->stats, q, J->tol_active, J->thr_bits);
            }
            __syncthreads();
            active = s_active != 0;
        }
        // the job's windows up to the end of the chunk
        const int window = tasks[t].window;
        int64_t run = s_windows - window;
        if (run > c0 + per - t) run = c0 + per - t;
        if (run > ntasks - t) run = ntasks - t;
        t += run;
        if (!active) continue;
        if (window == 0 && threadIdx.x == 0) s_args.stats[s_args.q].executed = 1u;
        if (WIDE && s_wide)
            run_windows<LAYOUT, 16, false, false, false>(s_args, blk, window, (int)run, 1, tally, nskip, full);
        else
            run_windows<LAYOUT, 8, false, false, !WIDE>(s_args, blk, window, (int)run, 1, tally, nskip, full);
    }
}

template <bool HALO>
const void *kernel_of(int layout, int bits)
{
    if (layout == 0)
        return bits == 8 ? (const void *)pass_screened_kernel<0, 8, HALO>
                         : (const void *)pass_screened_kernel<0, 16, HALO>;
    return bits == 8 ? (const void *)pass_screened_kernel<1, 8, HALO> : (const void *)pass_screened_kernel<1, 16, HALO>;
}

const void *resident_kernel_of(int layout, int bits)
{
    if (layout == 0) return bits == 8 ? (const void *)resident_kernel<0, 8> : (const void *)resident_kernel<0, 16>;
    return bits == 8 ? (const void *)resident_kernel<1, 8> : (const void *)resident_kernel<1, 16>;
}

const void *batch_kernel_of(int layout, int bits)
{
    if (layout == 0)
        return bits == 8 ? (const void *)batch_pass_kernel<0, false> : (const void *)batch_pass_kernel<0, true>;
    return bits == 8 ? (const void *)batch_pass_kernel<1, false> : (const void *)batch_pass_kernel<1, true>;
}

// Constant memory and function attributes belong to a context: they are set
// up once per device and context, with that device current (a context made
// after cudaDeviceReset is set up again).
constexpr int kMaxDevices = 64;
std::atomic<unsigned long long> g_consts_ctx[kMaxDevices] = {};
std::mutex g_consts_mu;

cudaError_t ensure_constants()
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const unsigned long long id = current_context_id();
    const unsigned long long key = id ? id : ~0ull;  // ~0: the context is not known yet
    if (g_consts_ctx[dev].load(std::memory_order_acquire) == key) return cudaSuccess;
    std::lock_guard<std::mutex> lock(g_consts_mu);
    if (g_consts_ctx[dev].load(std::memory_order_relaxed) == key) return cudaSuccess;
    double r[kRingMax + 1];
    double dg[kRingMax + 1];
    r[0] = 0.0;
    dg[0] = 0.0;
    for (int k = 1; k <= kRingMax; ++k) {
        r[k] = 1.0 / (double)k;
        dg[k] = (double)k;
    }
    e = cudaMemcpyToSymbol(c_recip, r, sizeof r);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_degree, dg, sizeof dg);
    if (e != cudaSuccess) return e;
    const int forms[4][2] = {{0, 8}, {0, 16}, {1, 8}, {1, 16}};
    for (const auto &f : forms)
        for (const void *k : {kernel_of<false>(f[0], f[1]), kernel_of<true>(f[0], f[1]), batch_kernel_of(f[0], f[1]),
                              resident_kernel_of(f[0], f[1])}) {
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            if (e != cudaSuccess) return e;
        }
    g_consts_ctx[dev].store(key, std::memory_order_release);
    return cudaSuccess;
}

int occupancy(const void *f, int block, const WindowShape &shape)
{
    if (ensure_constants() != cudaSuccess) return 1;
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, block, smem_for(shape));
    return nb > 0 ? nb : 1;
}

}  // namespace

cudaError_t launch_pass_screened(const PassArgs &a, int layout, int block, int grid, const WindowShape &shape,
                                 cudaStream_t s)
{
    cudaError_t e = ensure_constants();
    if (e != cudaSuccess) return e;
    if (a.win_count < grid) grid = a.win_count > 0 ? (int)a.win_count : 1;
    void *args[] = {const_cast<PassArgs *>(&a), const_cast<WindowShape *>(&shape)};
    if (a.halo) return cudaLaunchKernel(kernel_of<true>(layout, shape.bits), dim3(grid), dim3(block), args, smem_for(shape), s);
    return launch_early(kernel_of<false>(layout, shape.bits), grid, block, args, smem_for(shape), s);
}

bool resident_fits(const PassArgs &a, int layout, int block, const WindowShape &shape)
{
    return a.win_count > 0 &&
           a.win_count <= (int64_t)device_sm_count() * occupancy(resident_kernel_of(layout, shape.bits), block, shape);
}

cudaError_t launch_resident(const PassArgs &a, int layout, int block, const WindowShape &shape, int passes,
                            unsigned *barrier, unsigned poll_limit, cudaStream_t s)
{
    static_assert(sizeof(GridBarrier) == kBarrierWords * sizeof(unsigned), "barrier words");
    cudaError_t e = ensure_constants();
    if (e != cudaSuccess) return e;
    GridBarrier *b = reinterpret_cast<GridBarrier *>(barrier);
    void *args[] = {const_cast<PassArgs *>(&a), const_cast<WindowShape *>(&shape), &passes, &b, &poll_limit};
    return cudaLaunchCooperativeKernel(resident_kernel_of(layout, shape.bits), dim3((unsigned)a.win_count), dim3(block),
                                       args, smem_for(shape), s);
}

cudaError_t launch_batch_pass(const JobDesc *jobs, const WindowTask *tasks, int64_t ntasks, int round, int layout,
                              int block, int grid, const WindowShape &shape, cudaStream_t s, int64_t chunk,
                              unsigned long long *claim, bool own_graph)
{
    cudaError_t e = ensure_constants();
    if (e != cudaSuccess) return e;
    if (ntasks <= 0) return cudaSuccess;
    if (chunk < 0 && !claim) return cudaErrorInvalidValue;
    if (ntasks < grid) grid = (int)ntasks;
    void *args[] = {&jobs, &tasks, &ntasks, &round, &chunk, &claim, const_cast<WindowShape *>(&shape)};
    return launch_early(batch_kernel_of(layout, shape.bits), grid, block, args, smem_for(shape), s, own_graph);
}

namespace {

// `out` is page-locked host memory: the records arrive without a copy behind
// the kernel.
__global__ void gather_round_kernel(const JobDesc *jobs, int na, int round, PassStats *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    after_previous();
    if (j >= na) return;
    const JobDesc &J = jobs[j];
    int q = round - J.base_round;
    const int last = J.max_iter > 1 ? J.max_iter - 1 : 0;
    q = q < last ? q : last;
    out[j] = J.stats[q];
}

// The window tasks of na jobs: job j's at task_off[j] onwards.
__global__ void expand_tasks_kernel(const JobDesc *__restrict__ jobs, const int64_t *__restrict__ task_off, int na,
                                    WindowTask *__restrict__ tasks)
{
    for (int j = blockIdx.x; j < na; j += gridDim.x) {
        const int64_t t0 = task_off[j];
        for (int k = threadIdx.x; k < jobs[j].windows; k += blockDim.x) tasks[t0 + k] = WindowTask{j, k};
    }
}

}  // namespace

cudaError_t launch_expand_tasks(const JobDesc *jobs, const int64_t *task_off, int na, WindowTask *tasks,
                                cudaStream_t s)
{
    if (na <= 0) return cudaSuccess;
    expand_tasks_kernel<<<na < 4096 ? na : 4096, 256, 0, s>>>(jobs, task_off, na, tasks);
    return cudaGetLastError();
}

cudaError_t launch_gather_round(const JobDesc *jobs, int na, int round, PassStats *out, cudaStream_t s)
{
    if (na <= 0) return cudaSuccess;
    void *args[] = {&jobs, &na, &round, &out};
    return launch_early((const void *)gather_round_kernel, (na + 127) / 128, 128, args, 0, s);
}

int batch_pass_occupancy(int layout, int block, const WindowShape &shape)
{
    return occupancy(batch_kernel_of(layout, shape.bits), block, shape);
}

int pass_screened_occupancy(int layout, int block, const WindowShape &shape)
{
    return occupancy(kernel_of<false>(layout, shape.bits), block, shape);
}

}  // namespace sls
