// window.cuh -- the window stream the screened pass reads instead of the
// per-node adjacency records.
//
// The nodes of a mesh (of a colour class in Form B) are taken in windows of
// kWindow consecutive ids, one window per thread block and step.  A window's
// nodes and their neighbours outside it (its halo) are staged in shared
// memory once, so a coordinate is gathered and split once per window instead
// of once per neighbour visit, and every visit after that is a shared-memory
// load.  Each node has two lists of staged entries: its neighbours in summation order (Eq. 2), and its ring,
// the same neighbours in the order in which its triangles follow one another,
// so that the screen computes every ring vertex once for both triangles that
// share it.
//
// Staged entries: 0 holds (-0, -0), the padding of the summation lists
// (x + (-0) == x for every double); 1 .. count the window's nodes in id
// order; then the halo.  Lists hold entry numbers, in 8 bits where no window
// of the mesh has more than 255 entries (meshes numbered with any locality),
// else in 16.
//
// A window is four subtiles of 32 lanes.  Inside the window the nodes are
// dealt to the lanes by ring length (fixed nodes last), so that the lanes of
// a warp run loops of similar length; nothing is renumbered.
//
// Stream rows are 32 words (one per lane, 128 bytes, coalesced).  A window's
// rows: its halo's ids; the rows a pass always reads ("hot"), per subtile
//   1            meta word per lane
//   d entries    summation list (d: the subtile's largest degree)
//   l + 1        ring list (l: its largest step number, rounded up to an even
//                one), both in whole words; unused entries are 0, which the
//                ring walk reads as NaN
// (the meta row alone where a subtile has no node to update); then per subtile
// two rows that only open or irregular nodes need
//   1            the steps' slots: 2 bits a step, the node's slot in the
//                stored triangle, 3 = no triangle between the two
//   1            bit t: step t's triangle is stored against the ring's
//                direction (zero in a regular subtile)
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SLS_WN_HD __host__ __device__ __forceinline__
#else
#define SLS_WN_HD static inline
#endif

namespace sls {
namespace win {

constexpr int kWindow = 128;   // nodes per window (64 where a halo would not fit)
constexpr int kRingMax = 15;   // degree and step limit; a node past it is marked kBig
constexpr int kEntryMax = 1024;  // staged entries of a window, without the padding entry

// Window header: 8 words, of which 6 are used.
//   w0 first row, w1 first id, w2 count | halo << 8 | irregular subtiles << 24,
//   w3 byte per subtile: d | l << 4, w4 byte per subtile: first row, from the
//   first hot row, w5 hot rows
constexpr int kHeaderWords = 8;
SLS_WN_HD uint32_t hdr_count(uint32_t w2) { return w2 & 0xffu; }
SLS_WN_HD uint32_t hdr_halo(uint32_t w2) { return (w2 >> 8) & 0xffffu; }
SLS_WN_HD bool hdr_irregular(uint32_t w2, uint32_t sub) { return ((w2 >> (24u + sub)) & 1u) != 0u; }
SLS_WN_HD uint32_t halo_rows(uint32_t halo) { return (halo + 31u) >> 5; }
constexpr uint32_t kColdRows = 8;  // slots and directions of four subtiles

// Meta word: bits 0..6 the node's place in the window, 8..11 degree,
// 12..15 ring steps, then flags.
constexpr uint32_t kNode = 0x10000u;  // the lane holds a node
constexpr uint32_t kFree = 0x20000u;  // it is free and in the lists
constexpr uint32_t kBig = 0x40000u;   // it is free and not in the lists: its record decides
SLS_WN_HD uint32_t meta_word(uint32_t place, uint32_t deg, uint32_t steps, uint32_t flags)
{
    return place | (deg << 8) | (steps << 12) | flags;
}
SLS_WN_HD uint32_t meta_place(uint32_t m) { return m & 0x7fu; }
SLS_WN_HD uint32_t meta_deg(uint32_t m) { return (m >> 8) & 15u; }
SLS_WN_HD uint32_t meta_steps(uint32_t m) { return (m >> 12) & 15u; }

// Rows of `entries` list entries of `bits` bits per lane.
SLS_WN_HD uint32_t list_rows(uint32_t entries, uint32_t bits)
{
    return bits == 8u ? (entries + 3u) >> 2 : (entries + 1u) >> 1;
}
// Entries of a ring list: the walk takes two steps at a time.
SLS_WN_HD uint32_t ring_entries(uint32_t l) { return ((l + 1u) & ~1u) + 1u; }
// Hot rows of a subtile whose largest degree and step number are d and l.
SLS_WN_HD uint32_t subtile_rows(uint32_t d, uint32_t l, uint32_t bits)
{
    return d == 0u ? 1u : 1u + list_rows(d, bits) + list_rows(ring_entries(l), bits);
}

// A node's ring.
struct Ring {
    uint64_t seq;    // nibble t: position (in the neighbour list) of ring entry t, t = 0 .. steps
    uint32_t steps;  // steps t from entry t to entry t + 1
    uint32_t slots;  // 2 bits per step
    uint32_t rev;    // bit per step
    bool regular;    // one closed ring, every triangle in the ring's direction
    bool ok;         // fits
};

SLS_WN_HD uint32_t nib(uint64_t v, uint32_t k) { return (uint32_t)(v >> (4u * k)) & 15u; }

// Orders the ntri <= 15 triangles around a node of degree deg <= 15 (codes as
// in the adjacency record: slot, positions of the other two vertices in
// stored order).  The link of the node is a set of paths and closed rings (an
// edge belongs to at most two triangles); they are listed one after another,
// paths first, with a step without a triangle (slot 3) from the end of one to
// the start of the next.
SLS_WN_HD Ring order_ring(const uint32_t *codes, uint32_t deg, uint32_t ntri)
{
    Ring r;
    r.seq = 0;
    r.steps = 0;
    r.slots = 0;
    r.rev = 0;
    r.regular = false;
    r.ok = false;
    if (deg > (uint32_t)kRingMax || ntri > (uint32_t)kRingMax || ntri == 0u) return r;
    uint64_t from = 0, to = 0;  // nibble k: triangle k goes from -> to in its stored direction
    uint64_t out = ~0ull;       // nibble p: the triangle leaving position p (15: none)
    uint32_t nslots = 0, outs = 0, ins = 0;
    bool single = ntri == deg;
    for (uint32_t k = 0; k < ntri; ++k) {
        const uint32_t c = codes[k], slot = c >> 30, a = (c >> 15) & 0x7fffu, b = c & 0x7fffu;
        const uint32_t p = slot == 1u ? b : a, q = slot == 1u ? a : b;
        from |= (uint64_t)p << (4u * k);
        to |= (uint64_t)q << (4u * k);
        nslots |= slot << (2u * k);
        if (((outs >> p) & 1u) || ((ins >> q) & 1u)) single = false;
        outs |= 1u << p;
        ins |= 1u << q;
        out = (out & ~(15ull << (4u * p))) | ((uint64_t)k << (4u * p));
    }
    if (single) {
        uint32_t at = nib(from, 0), t = 0;
        const uint32_t start = at;
        do {
            const uint32_t k = nib(out, at);
            r.seq |= (uint64_t)at << (4u * t);
            r.slots |= ((nslots >> (2u * k)) & 3u) << (2u * t);
            at = nib(to, k);
            ++t;
        } while (at != start && t < ntri);
        if (at == start && t == ntri) {
            r.seq |= (uint64_t)start << (4u * t);
            r.steps = ntri;
            r.regular = true;
            r.ok = true;
            return r;
        }
        r.seq = 0;
        r.slots = 0;
    }
    uint32_t left = (1u << ntri) - 1u, t = 0;  // unused triangles; next entry
    while (left) {
        // start: a position with one unused triangle, else the first triangle's own
        uint32_t once = 0, twice = 0;
        for (uint32_t k = 0; k < ntri; ++k)
            if ((left >> k) & 1u) {
                const uint32_t p = 1u << nib(from, k), q = 1u << nib(to, k);
                twice |= (once & p) | (once & q);
                once |= p | q;
            }
        const uint32_t ends = once & ~twice;
        uint32_t at = 0;
        if (ends) {
            while (!((ends >> at) & 1u)) ++at;
        } else {
            uint32_t k = 0;
            while (!((left >> k) & 1u)) ++k;
            at = nib(from, k);
        }
        if (t > 0) {  // no triangle between the last entry and this one
            if (t > (uint32_t)kRingMax) return r;
            r.slots |= 3u << (2u * (t - 1u));
        }
        if (t > (uint32_t)kRingMax) return r;
        r.seq |= (uint64_t)at << (4u * t);
        ++t;
        for (;;) {
            uint32_t k = 0;
            while (k < ntri && !(((left >> k) & 1u) && (nib(from, k) == at || nib(to, k) == at))) ++k;
            if (k == ntri) break;
            if (t > (uint32_t)kRingMax) return r;
            left &= ~(1u << k);
            const bool rev = nib(from, k) != at;
            at = rev ? nib(from, k) : nib(to, k);
            r.slots |= ((nslots >> (2u * k)) & 3u) << (2u * (t - 1u));
            if (rev) r.rev |= 1u << (t - 1u);
            r.seq |= (uint64_t)at << (4u * t);
            ++t;
        }
    }
    r.steps = t - 1u;
    r.ok = true;
    return r;
}

}  // namespace win
}  // namespace sls
