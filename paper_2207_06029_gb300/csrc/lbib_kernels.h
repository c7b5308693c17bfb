// Host-side launchers of the liblbib kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbib_device.cuh"

namespace lbib {

// Launches a kernel of the step chain with programmatic stream
// serialization: its blocks may be scheduled while the previous kernel in
// the stream ends, and wait in chain_wait() for that kernel's results
// (this hides the launch gap between the short kernels of the IB stage).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr int kNodeThreads = 64;            // threads per block of the support-box kernels (spread over the SMs)
// The one-lattice MLS kernel: four lanes per point, 32 points a block, for few
// points, else a thread per point.  Four lanes shorten a point's chain of
// operations but add to their number; in FP64, of which an SM quarter issues
// a warp instruction per 64 cycles, they pay up to about a warp per quarter
// (8 points x 608), in FP32 until the warps fill the GPU.  Us a step, four
// lanes / one, sphere and capsule at 48^3: FP32 3202 points 19.5 / 21.7 and
// 17.0 / 18.3, 10 242 21.7 / 22.3 and 18.1 / 19.3, 12 802 22.7 / 22.3 and 18.4 /
// 19.3, 20 482 27.3 / 24.5 and 22.5 / 19.9; FP64 3202 79.2 / 95.1 and 78.4 / 93.0,
// 5122 82.9 / 96.1 and 85.9 / 92.1, 7682 98.5 / 95.4 and 96.7 / 103.7, 12 802 111.8 /
// 107.1 and 124.1 / 119.2.
inline bool mls_quads(int prec, const BodyView &B) { return B.nm + 2 * B.nt <= (prec == 0 ? 6000 : 20000); }
// points per block; a thread per point, FP64 takes blocks of one warp, which
// spread over more SMs
constexpr int mls_threads(int prec) { return prec == 0 ? 32 : 64; }
inline int mls_points(int prec, const BodyView &B) { return mls_quads(prec, B) ? 32 : mls_threads(prec); }

// sweep.cu
// part: 0 the whole lattice, 1 the nodes outside box, 2 the nodes inside box
// stamp == nullptr: no IB force is read; step points to the device step counter
// sr: the lattice's two-word rounding-seed counter, parity: the step's parity;
// box_nodes: about the nodes of the box (part 2)
cudaError_t launch_sweep(int prec, const void *fin, void *fout, void *force, const uint32_t *stamp,
                         const uint32_t *step, const Lattice &L, void *fields, int part, const int *box,
                         uint32_t *sr, int parity, int nsm, int box_nodes, cudaStream_t s);
// blocks of `threads` for a grid-stride loop over about `nodes` nodes
inline int node_blocks(int nodes, int threads, int nsm) {
    const long long g = ((long long)nodes + threads - 1) / threads;
    return (int)(g < 1 ? 1 : g > 8LL * nsm ? 8LL * nsm : g);
}
cudaError_t prepare_sweep_kernels();
// global mass and momentum (FP64): part holds totals_scratch_doubles() doubles,
// count one word that starts (and is left) at zero, out 4 doubles
cudaError_t launch_totals(int prec, const void *fin, const Lattice &L, double *part, unsigned int *count,
                          double *out, cudaStream_t s);
int totals_scratch_doubles();
// divergence watchdog: part and count as for launch_totals (shared with it,
// same stream), w 2 doubles (reference mass, last mass), err the context's
// error word
cudaError_t launch_watch(int prec, const void *fin, const Lattice &L, double *part, unsigned int *count, double *w,
                         double tol, int *err, cudaStream_t s);
// rho and u null: density 1 and u_x = shear_lo + (shear_hi - shear_lo) z / (nz - 1)
cudaError_t launch_init_equilibrium(int prec, void *fout, const Lattice &L, const double *rho, const double *u,
                                    void *fields, cudaStream_t s, double shear_lo = 0.0, double shear_hi = 0.0);
cudaError_t launch_pop_to_aos(int prec, const void *fin, const Lattice &L, double *out, cudaStream_t s);
cudaError_t launch_aos_to_pop(int prec, const double *in, const Lattice &L, void *fout, cudaStream_t s);
// err_out (mapped host memory) receives the error word err
cudaError_t launch_fields_out(int prec, const void *fields, const Lattice &L, double *rho, double *u, const int *err,
                              int *err_out, cudaStream_t s);

// ib.cu
constexpr int kBatchMlsThreads = 128;       // MLS points per block of the batched kernel
constexpr int kPersistThreads = 256;        // threads per block of the persistent batched kernel
constexpr int kMarkersPerBlock = 32;        // markers per block of 256 threads (batched structure kernels)
// blocks of `threads` MLS points (markers and probes) of a body
int mls_blocks(const BodyView &B, int threads);
// whether the MLS partials of blocks of `threads` points are added up by a
// launch of their own
bool needs_body_sums(const BodyView &B, int threads);
// step_inc: device step counter incremented at the start of the step (first
// body only), or nullptr.  grid_cap > 0: the MLS, structure and spreading
// kernels launch at most grid_cap blocks, each taking its share of their
// blocks' work in turn (0: their full grids)
cudaError_t launch_ib_front(int prec, const void *fin, const Lattice &L, const BodyView &B, void *mom, int nsm,
                            int box_nodes, int *err, uint32_t *step_inc, int grid_cap, cudaStream_t s);
// structure update and spreading; chained: programmatically behind the
// previous kernel of the stream
cudaError_t launch_structure(int prec, const Lattice &L, const BodyView &B, void *force, uint32_t *stamp,
                             const uint32_t *step, int nsm, int grid_cap, bool chained, cudaStream_t s);

// batches (sweep.cu and ib.cu); grid sizes are the totals of the prefix tables
struct BatchGrid {
    int sweep, mom, mls, sums, memb, rm, cen;
};
// chained: the previous kernel of the stream is the batched sweep of the step
// before, in the same capture
cudaError_t launch_batch_ib(int prec, const BatchTables &T, const BatchGrid &G, int phase, bool chained,
                            cudaStream_t s);
cudaError_t launch_batch_sweep(int prec, const BatchTables &T, const BatchGrid &G, int phase, int store_fields,
                               cudaStream_t s);
// persistent batched step (ib.cu): P.nsteps steps of every lattice in one
// launch of `grid` blocks of 256 threads; the counters P.ticket, P.abort and
// P.done must be zero at launch
cudaError_t launch_batch_persistent(int prec, const BatchTables &T, const PersistTables &P, int grid, cudaStream_t s);
// resident blocks per SM of the persistent kernel
int batch_persistent_blocks_per_sm(int prec, bool off32);

}  // namespace lbib
