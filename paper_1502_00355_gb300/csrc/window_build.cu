// window_build.cu -- the window stream (window.cuh) of a mesh, made on the
// device from its adjacency records.
//
// One block of kWindow threads per window, a thread per node.  The halo is
// collected in a hash table in shared memory, whose slots also give every
// neighbour its staged entry.  The kernel runs twice: the first time it sizes
// every window and claims its rows from a counter (where a window's rows lie
// does not matter), the second time, with the stream allocated, it writes
// them.
#include <string>

#include "api_common.h"
#include "device.cuh"
#include "window.cuh"

namespace sls {
namespace {

constexpr uint32_t kNoId = 0xffffffffu;
constexpr int kHash = 2048;  // slots; a window has at most kWindow * kRingMax = 1920 neighbours

struct BuildTotals {
    unsigned long long rows;
    unsigned int entries;   // most staged entries of a window
    unsigned int halo, hot; // most halo nodes and hot rows
    unsigned int too_large; // windows with more than kEntryMax
};

__device__ __forceinline__ uint32_t hash_of(uint32_t id) { return (id * 2654435761u) >> 21; }

// WRITE = false: hdr and totals; WRITE = true: the rows.
// cyclic: the ring lists (and slots) of closed rings go on around the ring up to
// their row's end (the binary32 walk), else unused entries are 0.
// Windows are `width` ids wide; window w of segment s (win_off[s] <= w) starts
// at seg_off[s] + (w - win_off[s]) * width.
template <bool WRITE>
__global__ void __launch_bounds__(win::kWindow) window_build_kernel(
    const uint32_t *__restrict__ node_off, const uint32_t *__restrict__ adj, const int64_t *__restrict__ seg_off,
    const int64_t *__restrict__ win_off, int nseg, int64_t nwin, int width, int bits, int group, int cyclic, uint32_t *hdr,
    uint32_t *rows, BuildTotals *totals)
{
    __shared__ uint32_t s_key[kHash];
    __shared__ uint16_t s_val[kHash];
    __shared__ uint32_t s_place[16][4];   // first lane of a (key, warp) group
    __shared__ uint32_t s_deg[4], s_steps[4], s_irr, s_halo;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int64_t w = blockIdx.x; w < nwin; w += gridDim.x) {
        int seg = 0;
        while (seg + 1 < nseg && win_off[seg + 1] <= w) ++seg;
        const int64_t first = seg_off[seg] + (w - win_off[seg]) * width;
        const int64_t end = seg_off[seg + 1];
        const int count = end - first < width ? (int)(end - first) : width;
        for (int k = t; k < kHash; k += win::kWindow) s_key[k] = kNoId;
        if (t < 4) s_deg[t] = s_steps[t] = 0u;
        if (t == 0) {
            s_irr = 0u;
            s_halo = 0u;
        }
        __syncthreads();

        // the node's record
        const bool have = t < count;
        uint32_t meta = kMetaFixed;
        const uint32_t *nb = adj;
        if (have) {
            const uint32_t off = node_off[first + t];
            meta = adj[off];
            nb = adj + off + 1;
        }
        const bool fixed = (meta & kMetaFixed) != 0u;
        const uint32_t deg = fixed ? 0u : meta_degree(meta), ntri = fixed ? 0u : meta_ntri(meta);
        win::Ring ring;
        ring.ok = false;
        ring.steps = 0u;
        ring.regular = false;
        if (!fixed && deg <= (uint32_t)win::kRingMax && ntri <= (uint32_t)win::kRingMax)
            ring = win::order_ring(nb + deg, deg, ntri);
        const bool listed = have && !fixed && ring.ok;
        // the halo
        if (listed)
            for (uint32_t k = 0; k < deg; ++k) {
                const uint32_t id = nb[k];
                if ((int64_t)id >= first && (int64_t)id < first + count) continue;
                uint32_t h = hash_of(id);
                for (int probe = 0; probe < kHash; ++probe, h = (h + 1u) & (kHash - 1)) {
                    const uint32_t old = atomicCAS(s_key + h, kNoId, id);
                    if (old == kNoId) s_val[h] = (uint16_t)atomicAdd(&s_halo, 1u);
                    if (old == kNoId || old == id) break;
                }
            }
        // the node's lane: by ring length inside the window, the others last
        const uint32_t key = listed ? (deg > ring.steps ? deg : ring.steps) : 15u;
        uint32_t place = (uint32_t)t;
        if (group) {
            if (t < 64) s_place[t >> 2][t & 3] = 0u;
            __syncthreads();
            const uint32_t same = __match_any_sync(0xffffffffu, have ? key : 16u);
            const uint32_t before = __popc(same & ((1u << lane) - 1u));
            if (have && before == 0u) s_place[key][warp] = __popc(same);
            __syncthreads();
            if (warp == 0) {  // exclusive sums over (key, warp), two values a lane
                const uint32_t a = s_place[lane >> 1][(lane & 1) * 2], b = s_place[lane >> 1][(lane & 1) * 2 + 1];
                uint32_t x = a + b;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                s_place[lane >> 1][(lane & 1) * 2] = x - a - b;
                s_place[lane >> 1][(lane & 1) * 2 + 1] = x - b;
            }
            __syncthreads();
            place = have ? s_place[key][warp] + before : (uint32_t)t;
        }
        const uint32_t sub = place >> 5;
        if (listed) {  // the subtile's largest degree and step number
            atomicMax(&s_deg[sub], deg);
            atomicMax(&s_steps[sub], ring.steps);
            if (!ring.regular) atomicOr(&s_irr, 1u << sub);
        }
        __syncthreads();
        const uint32_t halo = s_halo;
        uint32_t starts = 0u, dls = 0u, hot = 0u;
        for (int k = 0; k < 4; ++k) {
            dls |= (s_deg[k] | (s_steps[k] << 4)) << (8 * k);
            starts |= hot << (8 * k);
            hot += win::subtile_rows(s_deg[k], s_steps[k], (uint32_t)bits);
        }
        if (!WRITE) {
            if (t == 0) {
                const uint32_t all = halo + (uint32_t)count;
                uint32_t *h = hdr + w * win::kHeaderWords;
                const unsigned long long r0 =
                    atomicAdd(&totals->rows, (unsigned long long)(win::halo_rows(halo) + hot + win::kColdRows));
                h[0] = (uint32_t)r0;
                h[1] = (uint32_t)first;
                h[2] = (uint32_t)count | (halo << 8) | (s_irr << 24);
                h[3] = dls;
                h[4] = starts;
                h[5] = hot;
                atomicMax(&totals->entries, all);
                atomicMax(&totals->halo, halo);
                atomicMax(&totals->hot, hot);
                if (all > (uint32_t)(bits == 8 ? 255 : win::kEntryMax)) atomicAdd(&totals->too_large, 1u);
            }
        } else {
            uint32_t *base = rows + (size_t)hdr[w * win::kHeaderWords] * 32u;
            for (int k = t; k < kHash; k += win::kWindow)
                if (s_key[k] != kNoId) base[s_val[k]] = s_key[k];
            const uint32_t d = (dls >> (8 * sub)) & 15u, l = (dls >> (8 * sub + 4)) & 15u;
            const uint32_t lane_at = place & 31u;
            uint32_t *hot_base = base + win::halo_rows(halo) * 32u;
            uint32_t *row = hot_base + ((starts >> (8 * sub)) & 0xffu) * 32u + lane_at;
            uint32_t *cold = hot_base + (hot + 2u * sub) * 32u + lane_at;
            row[0] = have ? win::meta_word((uint32_t)t, listed ? deg : 0u, listed ? ring.steps : 0u,
                                           win::kNode | (listed ? win::kFree : (fixed ? 0u : win::kBig)))
                          : 0u;
            uint32_t slots = listed ? ring.slots : 0u;
            if (cyclic && listed && ring.regular)
                for (uint32_t k = ring.steps; k < 16u; ++k) slots |= ((slots >> (2u * (k - ring.steps))) & 3u) << (2u * k);
            cold[0] = slots;
            cold[32] = listed ? ring.rev : 0u;
            if (d > 0u) {
                uint16_t entry[win::kRingMax];
                const uint32_t ndeg = listed ? deg : 0u, nring = listed ? ring.steps + 1u : 0u;
                for (uint32_t k = 0; k < ndeg; ++k) {
                    const uint32_t id = nb[k];
                    if ((int64_t)id >= first && (int64_t)id < first + count) {
                        entry[k] = (uint16_t)(1u + (id - (uint32_t)first));
                    } else {
                        uint32_t h = hash_of(id);
                        while (s_key[h] != id) h = (h + 1u) & (kHash - 1);
                        entry[k] = (uint16_t)(1u + (uint32_t)count + s_val[h]);
                    }
                }
                const uint32_t per = 32u / (uint32_t)bits;
                uint32_t *o = row + 32;
                for (uint32_t k = 0; k < win::list_rows(d, (uint32_t)bits); ++k, o += 32) {
                    uint32_t word = 0u;
                    for (uint32_t j = 0; j < per; ++j)
                        if (k * per + j < ndeg) word |= (uint32_t)entry[k * per + j] << (j * (uint32_t)bits);
                    *o = word;
                }
                for (uint32_t k = 0; k < win::list_rows(win::ring_entries(l), (uint32_t)bits); ++k, o += 32) {
                    uint32_t word = 0u;
                    for (uint32_t j = 0; j < per; ++j)
                        if (k * per + j < nring || (cyclic && listed && ring.regular))
                            word |= (uint32_t)entry[win::nib(ring.seq, k * per + j < nring ? k * per + j
                                                                                            : (k * per + j) % ring.steps)]
                                    << (j * (uint32_t)bits);
                    *o = word;
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace

sls_status build_windows(int64_t n, const std::vector<int64_t> &segments, const uint32_t *node_off,
                         const uint32_t *adj, bool group, bool cyclic, cudaStream_t s, WindowStream &out)
{
    out.release(s);
    std::vector<int64_t> segs = segments;
    if (segs.empty()) segs = {0, n};
    const int nseg = (int)segs.size() - 1;
    int64_t *d_offs = nullptr;
    BuildTotals *d_tot = nullptr;
    BuildTotals h{};
    cudaError_t e = cudaSuccess;
    auto done = [&](cudaError_t err, const char *what) {
        pool_free(d_offs, s);
        pool_free(d_tot, s);
        if (err == cudaSuccess) return SLS_OK;
        out.release(s);
        if (err == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            return fail(SLS_ERR_OOM, std::string("device allocation failed: ") + what);
        }
        return cuda_fail(err, what);
    };
    // 8-bit lists of 128-node windows first; a mesh whose numbering is not
    // local, or a colour class, whose neighbours are all outside it, takes 16
    // bits, and halves of windows where even those would not fit
    int bits = segments.empty() ? 8 : 16, width = win::kWindow;
    for (;;) {
        std::vector<int64_t> offs(2 * segs.size(), 0);  // segment starts, then each segment's first window
        for (int c = 0; c <= nseg; ++c) {
            offs[c] = segs[c];
            if (c > 0) offs[nseg + 1 + c] = offs[nseg + c] + (segs[c] - segs[c - 1] + width - 1) / width;
        }
        out.first_window.assign(offs.begin() + nseg + 1, offs.end());
        out.width = width;
        out.count = offs[2 * nseg + 1];
        if (out.count == 0) return done(cudaSuccess, "windows");
        if (!d_offs) e = pool_alloc((void **)&d_offs, sizeof(int64_t) * offs.size(), s);
        if (e == cudaSuccess && !d_tot) e = pool_alloc((void **)&d_tot, sizeof(BuildTotals), s);
        if (e == cudaSuccess)
            e = pool_alloc((void **)&out.hdr, sizeof(uint32_t) * win::kHeaderWords * (size_t)out.count, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(d_offs, offs.data(), sizeof(int64_t) * offs.size(), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(d_tot, 0, sizeof(BuildTotals), s);
        if (e != cudaSuccess) return done(e, "windows");
        const int64_t cap = (int64_t)device_sm_count() * 12;
        const unsigned grid = (unsigned)(out.count < cap ? out.count : cap);
        window_build_kernel<false><<<grid, win::kWindow, 0, s>>>(node_off, adj, d_offs, d_offs + nseg + 1, nseg,
                                                                 out.count, width, bits, group ? 1 : 0, cyclic ? 1 : 0, out.hdr, nullptr,
                                                                 d_tot);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d_tot, sizeof h, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // also: offs has been read
        if (e != cudaSuccess) return done(e, "windows");
        if (h.too_large == 0u) {
            if (h.rows >= (1ull << 32)) return done(cudaErrorMemoryAllocation, "window stream");
            out.shape.entries = (int)h.entries;
            out.shape.halo = (int)h.halo;
            out.shape.hot = (int)h.hot;
            out.shape.bits = bits;
            out.rows_bytes = (size_t)h.rows * 128u;
            e = pool_alloc((void **)&out.rows, out.rows_bytes, s);
            if (e != cudaSuccess) return done(e, "window stream");
            window_build_kernel<true><<<grid, win::kWindow, 0, s>>>(node_off, adj, d_offs, d_offs + nseg + 1, nseg,
                                                                    out.count, width, bits, group ? 1 : 0, cyclic ? 1 : 0, out.hdr,
                                                                    out.rows, nullptr);
            return done(cudaGetLastError(), "windows");
        }
        if (bits == 8) {
            bits = 16;
        } else {
            // 64 nodes and their halo of at most 64 * 15 always fit
            if (width < win::kWindow) return done(cudaErrorUnknown, "windows");
            width = win::kWindow / 2;
        }
        pool_free(out.hdr, s);
        out.hdr = nullptr;
    }
}

void WindowStream::release(cudaStream_t s)
{
    pool_free(hdr, s);
    pool_free(rows, s);
    *this = WindowStream{};
}

}  // namespace sls
