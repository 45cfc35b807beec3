// api_common.h -- the mesh handle and the helpers behind the C ABI.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"

namespace sls {

// The window stream of a mesh's screened pass (window.cuh), in device memory
// from the library's pool.
struct WindowStream {
    uint32_t *hdr = nullptr, *rows = nullptr;
    int64_t count = 0;                  // windows
    int width = 0;                      // nodes per window
    WindowShape shape;
    size_t rows_bytes = 0;
    std::vector<int64_t> first_window;  // of every segment, and the end
    void release(cudaStream_t s);
};

// What a mesh handle needs besides device memory and is slow to make: a
// non-blocking stream and kHostStats page-locked records (take_kit).
constexpr int kHostStats = 512;
struct HandleKit {
    cudaStream_t stream = nullptr;
    PassStats *host = nullptr;
    int device = -1;
    unsigned long long ctx = 0;
};

}  // namespace sls

struct sls_mesh {
    sls_options opt{};
    int64_t n = 0, m = 0, n_free = 0;
    double diag = 0.0;            // bounding-box diagonal of the creation coordinates
    int device = 0;
    cudaStream_t stream = nullptr;  // the caller's or the kit's
    sls::HandleKit kit;
    double *xy[2] = {nullptr, nullptr};  // the two coordinate arrays (2n doubles each, 2n floats when f32)
    bool f32 = false;             // binary32 coordinates and arithmetic
    int cur = 0;                  // which of the two holds the current coordinates
    uint32_t *node_off = nullptr; // n+1
    uint32_t *adj = nullptr;      // node_off[n] words
    uint64_t adj_words = 0;
    uint32_t *node_order = nullptr;  // n_free: processing order of the free nodes (Form A: none)
    sls::WindowStream windows;    // what the screened pass reads
    uint32_t *perm = nullptr;     // renumbered mesh (Form B: colour classes contiguous; Form A:
                                  // along a Z-order curve): internal id -> the caller's id
    uint32_t *inv = nullptr;      // the caller's id -> internal id
    std::vector<int64_t> colour_off; // segments of node_order: one per colour (Form B), else one
    int32_t *tri = nullptr;       // 3m, for the histogram
    sls::PassStats *stats = nullptr;  // one record per pass of a call; the record before the first
                                      // holds the blocks' barrier of the resident form
    int stats_cap = 0;
    sls::PassStats *h_stats = nullptr;  // page-locked, kHostStats records
    uint8_t *accept = nullptr;    // n, when record_accept
    uint2 *halo = nullptr;        // skip_unchanged: kHaloEntries (tile, mask) pairs per 32-node tile
    uint32_t *chg[2] = {nullptr, nullptr};  // per tile: nodes changed by the last two passes
    uint32_t *accm = nullptr;     // per tile: nodes accepted when the tile was last computed
    size_t l2_persist = 0;        // l2_window: persisting L2 bytes set aside for this context
    size_t l2_win_max = 0;        //            largest access-policy window the device accepts
    unsigned *xfer_bad = nullptr; // gather/scatter: set when an id was out of range
    int block = 256, grid = 0;
    bool resident = false;        // all passes of a call in one launch (pass_screened.cu)
    unsigned next_polls = 0u;     // poll limit of the next such launch; 0 = kPollLimit (sls_test_resident)
    bool screened = true;         // screened kernel (else the plain FP64 kernel)
    sls_info last{};
};

namespace sls {

sls_status cuda_fail(cudaError_t e, const char *what);
int device_sm_count();
// Unique id of the calling thread's current CUDA context, 0 when there is
// none.  Per-device set-up (constant memory, symbol addresses) is keyed on it,
// so a context created after cudaDeviceReset is set up again.
unsigned long long current_context_id();
// Loads the allocation-free entry point's scratch array on the current
// device (noalloc.cu); sls_mesh_create calls it, so sls_smooth_noalloc on a
// mesh never loads code or data itself (a renumbered mesh's creation loads the
// kernels of its numbering too, load_numbering_kernels).
sls_status noalloc_prepare();
sls_options resolve_options(const sls_options *opt);
sls_status check_options(const sls_options &o);

sls_status mesh_upload(sls_mesh *M, const HostMesh &hm, const double *xy, const int32_t *tri,
                       const sls_options &o);
// Uploads coordinates and triangles and builds the adjacency on the device
// (host build as a fallback for very high-valence nodes).
sls_status mesh_create_on_device(sls_mesh *M, const double *xy, int64_t n, const int32_t *tri, int64_t m,
                                 const uint8_t *boundary, const sls_options &o);
// Adjacency built on the device (mesh_build_gpu.cu).
struct DeviceAdjacency {
    uint32_t *node_off = nullptr;  // n+1
    uint32_t *adj = nullptr;       // adj_words
    uint64_t adj_words = 0;
    uint32_t *perm = nullptr, *inv = nullptr;  // spatially renumbered: new id -> the caller's, and back
    int64_t n_free = 0;
    double diag = 0.0;
};
// Validates the mesh and builds its adjacency from device copies of the
// coordinates (AoS) and triangles, with stream-ordered allocations on s (the
// caller frees the outputs).  renumber: a mesh whose numbering is not local
// may be renumbered first, d_xy and d_tri with it.
// SLS_ERR_NOT_FOUND = a node is in too many triangles: use the host build.
sls_status build_device_adjacency(int64_t n, int64_t m, double *d_xy, int32_t *d_tri, const uint8_t *h_boundary,
                                  bool renumber, cudaStream_t s, DeviceAdjacency &out);
// Whether options o let the build renumber a mesh: Form-A passes that read a
// window stream (Form B's colouring follows the caller's numbering,
// skip_unchanged's tiles are the caller's) unless the caller's numbering is to
// be kept.
inline bool numbers_spatially(const sls_options &o)
{
    return o.form == 0 && (o.precision == 32 || o.kernel != SLS_KERNEL_FP64) && !o.skip_unchanged && o.numbering != 1;
}
// Device memory of the handles (memory.cu): stream-ordered allocations from
// the library's pool on the current device, which keeps freed memory for
// later handles (sls_trim_memory returns it).  Allocate and free on the
// stream that uses the buffer; pool_free ignores NULL.
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s);
// A handle's stream and page-locked records, from a small cache on the current
// device (memory.cu); give back a kit whose stream is idle (keep = false: not
// for reuse).  sls_trim_memory empties the current device's cache.
cudaError_t take_kit(HandleKit *kit);
void give_kit(const HandleKit &kit, bool keep);
void pool_free(void *p, cudaStream_t s);
// The window stream of a built adjacency (window_build.cu); segments: the id
// ranges to cover one after another (Form B: the colour classes' bounds),
// empty = one segment of all n nodes.  group: nodes dealt to the lanes by ring
// length inside a window.  cyclic: ring lists padded for the binary32 walk.
// Waits for s between its two kernels; the second one, which writes the rows, may
// still run when it returns.
sls_status build_windows(int64_t n, const std::vector<int64_t> &segments, const uint32_t *node_off,
                         const uint32_t *adj, bool group, bool cyclic, cudaStream_t s, WindowStream &out);
// Whether options o deal a window's nodes to the lanes by ring length: not
// where the caller's order is asked for, nor with skip_unchanged, whose
// 32-node tiles are the subtiles.
inline bool groups_lanes(const sls_options &o) { return !o.skip_unchanged && o.numbering != 1; }
// Device adjacency build of a mesh handle; SLS_ERR_NOT_FOUND = use the host build.
sls_status build_device_mesh(sls_mesh *M, double *d_xy, int32_t *d_tri, const uint8_t *h_boundary, cudaStream_t s);
// The processing order of the free nodes, from the adjacency on the device
// (mesh_build_gpu.cu): fills M->node_order.
sls_status build_node_order(sls_mesh *M, cudaStream_t s);
// The tile lists and masks of unchanged-tile skipping (mesh_build_gpu.cu),
// when opt.skip_unchanged is set and some tile can be skipped at all.
sls_status build_tile_halo(sls_mesh *M, cudaStream_t s);
void mesh_release(sls_mesh *M);
sls_status mesh_run(sls_mesh *M, int32_t max_iter, double tol_rel, sls_info &info);
sls_status mesh_download(const sls_mesh *M, double *xy_out, bool dst_is_device);
sls_status mesh_set_coords(sls_mesh *M, const double *xy, bool src_is_device);
// Device gather (scatter = false: buf <- current coordinates of the listed
// nodes) or scatter (buf -> both coordinate arrays) of k nodes; returns when done.
sls_status mesh_transfer_nodes(sls_mesh *M, const int32_t *idx, int64_t k, double *buf, bool scatter);
sls_status mesh_histogram(const sls_mesh *M, int nbins, double lo, double hi, int64_t *counts,
                          double *qmin, double *qmean);

// (tol * D)^2 with the tolerance stop's exact rounding.
inline double tolerance_threshold(double tol_rel, double diag)
{
    double a = tol_rel * diag;
    return a * a;
}

}  // namespace sls
