// Host-side launchers of the stage kernels (one per translation unit).
#pragma once

#include "pt_common.cuh"

namespace ptk {

// Brackets the kernel launches of its scope with two CUDA events on the
// stream while kernel timing is enabled (pt_kernel_timing); does nothing
// otherwise or while the stream is being captured.
class KernelTimer {
  public:
    KernelTimer(const char *name, cudaStream_t s);
    ~KernelTimer();
    KernelTimer(const KernelTimer &) = delete;
    KernelTimer &operator=(const KernelTimer &) = delete;

  private:
    const char *name_;
    cudaStream_t s_;
    cudaEvent_t a_;
};

// Launch with programmatic stream serialisation: the grid is set up while the
// kernel before it on the stream drains, which its pdl_enter() waits for.  A
// chain of ~25 short kernels spends much of its time between them: 177 -> 125
// us from the first to the last for a 50-helix event, 238 -> 193 us for a
// PU50 event, 571 -> 526 us for a PU200 event, and a percent off the batches.
// (Letting the next grid's blocks be placed from the start of a kernel,
// griddepcontrol.launch_dependents, gained no more on the small events and
// cost the batches 2 to 6%: waiting blocks hold what running ones could use.)
template <typename... P, typename... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// Size of a persistent grid: `resident` blocks per SM (what the kernel's
// registers and shared memory let an SM hold), or what the tuning's factor
// allows when that is smaller: `per` blocks for each unit of it, a unit being 256 threads
// (128 in the Fishbone's two-warp teams and in the adjoint), so that a caller who
// lowers the factor to leave room on the SMs gets that from every kernel.  More
// blocks than are resident only start, find the queue
// or the range used up, and end: 5-10 us of empty waves per kernel in the
// smallest events with a grid of 24 blocks per SM whatever the kernel.
struct Grid {
    int sms, factor;
    int blocks(int resident, int per = 1) const { return sms * (factor * per < resident ? factor * per : resident); }
};

void launch_scan(int32_t *a, int64_t n, int32_t *part, cudaStream_t s);
void launch_binning(const Params &p, const Grid &g, cudaStream_t s);
void launch_doublets(const Params &p, int lanes, const Grid &g, cudaStream_t s);
void launch_fishbone(const Params &p, float unit_thr, float du, const Grid &g, cudaStream_t s);
void launch_connect(const Params &p, const Grid &g, cudaStream_t s);
void launch_ntuplets(const Params &p, const Grid &g, cudaStream_t s);
void launch_select(const Params &p, cudaStream_t s);
void launch_fit(const Params &p, const Grid &g, cudaStream_t s);
void launch_fit_grad(const Params &p, const float *gpar, const float *gchi, float *gx, float *gy, float *gz,
                     const Grid &g, cudaStream_t s);
void launch_ambiguities(const int32_t *hits, const int32_t *cells, const uint8_t *n, const int32_t *track_tuple,
                        int32_t n_tracks, const float *chi2, const float *tip, int32_t tip_stride, int32_t n_cells,
                        int32_t n_hits, uint32_t *scratch, uint8_t *keep, int grid, cudaStream_t s);
void launch_align(int n, const float *x, const float *y, const float *z, const int32_t *module, const float *centre,
                  const float *shift, const float *rot, float *xo, float *yo, float *zo, int grid, cudaStream_t s);
void launch_align_grad(int n, const float *x, const float *y, const float *z, const int32_t *module,
                       const float *centre, const float *rot, const float *gxa, const float *gya, const float *gza,
                       float *gx, float *gy, float *gz, float *gshift, float *grot, int grid, cudaStream_t s);
size_t vertex_scratch_bytes(int32_t n_tracks, int32_t n_events);
pt_status launch_vertices(const pt_vertex_tracks &in, int32_t n_tracks, int32_t n_events,
                          const pt_vertex_cuts &cuts, int32_t max_vertices, void *scratch, const pt_vertices &out,
                          int grid, cudaStream_t s);
void launch_track_summary(int32_t n_tracks, const int32_t *hits, const uint8_t *tn, const float *params,
                          const float *cov, const int32_t *tuple, const int32_t *ev_off, int32_t n_events, float bz,
                          int32_t *ev, float *z0, float *ez0, float *pt, uint8_t *nhits, int grid, cudaStream_t s);

}  // namespace ptk
