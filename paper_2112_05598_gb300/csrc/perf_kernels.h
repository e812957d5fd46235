// perf_kernels.h -- host launchers of the libperf kernels (internal).
#pragma once
#include <cuda_runtime.h>
#include "perf_device.cuh"

namespace perf {

// One scene of a batch: its geometry and where its parameters, rays and
// tiles start in the batch's concatenated vectors / work queue.
struct BatchItem {
    DevScene sc;
    long long x_off;      // first parameter (floats; multiple of 4)
    long long r_off;      // first ray
    long long tile_off;   // first tile in the work queue
};

// Batched ray marches over many scenes in one persistent launch: warps take
// tiles from the work queue `counter` (zeroed here); `start[n]` are the
// scenes' first tiles.  Forward: mode 0 image into res, 1 residual
// (+F[scene]), 2 F[scene] only,
// scenes with active[s] == 0 skipped (active may be null).  Scatter: mode 1
// A p (+ p^T A p into pap[scene * pap_stride]), 2 diag (+ grad with v = r).
cudaError_t launch_forward_batch(const BatchItem* items, const long long* start, int n,
                                 long long total, unsigned long long* counter, const float* x,
                                 const float* target, float* res, double* F, const int* active,
                                 int mode, int cap_per_sm, cudaStream_t st, bool copy = false);
struct PcgScalars;
// pcg (may be null): per-scene Algorithm 2 state; scenes whose solve has
// exited (done) are skipped.
// coef / tile_off (mode 2, may be null): also store the per-sample
// coefficients, tile_off indexed by the global tile list.
cudaError_t launch_scatter_batch(const BatchItem* items, const long long* start, int n,
                                 long long total, unsigned long long* counter, const float* x,
                                 const float* p, const float* v, float* out, float* out2,
                                 double* pap, int pap_stride, int mode, int cap_per_sm,
                                 cudaStream_t st, const PcgScalars* pcg = nullptr,
                                 float* coef = nullptr, const long long* tile_off = nullptr,
                                 bool brick = false, bool copy = false);
// copy (here and above): every scene's items[i].sc holds the gather copies of
// the launch's x (and p).  launch_gather_copy_batch makes those of x (sig: and
// the opacity records) in the places items[i].sc.xcopy and .sigma8, chunks as
// in the segmented vector kernels, active (may be null) as in
// launch_forward_batch.
cudaError_t launch_gather_copy_batch(const BatchItem* items, const int4* chunks, long long n_chunks,
                                     const float* x, bool sig, const int* active, cudaStream_t st);
// Coefficient-cached A p over a batch, and the rows of every tile of the
// global tile list (see launch_tile_rows).  brick: p and A p of each scene
// are in the block order of its items[i].sc layout (else all canonical).
cudaError_t launch_apply_coef_batch(const BatchItem* items, const long long* start, int n,
                                    long long total, unsigned long long* counter, const float* p,
                                    const float* coef, const long long* tile_off, float* out,
                                    double* pap, int pap_stride, int cap_per_sm, cudaStream_t st,
                                    const PcgScalars* pcg, bool brick = false, bool copy = false);
cudaError_t launch_tile_rows_batch(const BatchItem* items, const long long* start, int n,
                                   long long total, int* rows, cudaStream_t st);

// Device scalars of Algorithm 2 and the line search (FP64).
struct PcgScalars {
    double rz;        // r_k^T z_k
    double R0;        // r_0^T r_0
    double R_prev;    // r_{k}^T r_{k} of the previous iteration
    double R;         // latest r^T r
    double pAp;       // accumulator: p^T A p
    double acc_R;     // accumulator: r_{k+1}^T r_{k+1}
    double acc_rz;    // accumulator: r_{k+1}^T z_{k+1}
    double beta;
    double F;         // accumulator: objective
    int iter;
    int done;
    int exit_reason;
    int max_iter;
    int fixed;
    int pad;
    double eps_rel;
    double stall;
    double* hist;     // null, or R after iteration k written to hist[k - 1] (k <= hist_cap)
    long long hist_cap;
};

// DevScene::spread of marches over this many pixel tiles together.  The lane
// order and the spread of the scatter's classes raise the throughput of the L1
// and of the atomics; a march that leaves most of the GPU's warp slots empty
// waits for its loads' latency instead, and keeps the plain order, whose
// sums of neighbouring rays arrive next to each other.  Plain / spread, 64^3, 128^2
// images: A p 189 / 179 us at 1024 tiles, 283 / 237 at 2048, 474 / 404 at 4096,
// 1621 / 1314 at 16384; Gauss-Newton step 999 / 990 us, 1303 / 1166, 2139 /
// 1889, 6565 / 5072.
inline int spread_of(long long tiles) { return tiles >= 152 * 10 ? 3 : 0; }

// The same for a march that scatters.  A parameter that very many rays see is a
// long chain of binary32 additions, and what it rounds to follows the order of
// the chain, run after run.  Either order is as exact (A p at 2^3, 92 k rays:
// 5.8 to 7.9e-6 off plain, 6.9 to 8.5e-6 spread), but a Gauss-Newton step of a
// small system turns the difference into its objective, so scenes with more
// than 32 residuals a parameter keep the plain order, the one that small
// launches have too.  F after a step, relative difference of the two orders (of
// two runs of one: 1e-6): 1 to 8e-5 at 25^3 to 36^3 with 50 to 110 residuals a
// parameter, at most 6e-6 up to 32 (1e-7 at 128^3, 100 x 800^2: 19).
inline int scatter_spread_of(long long tiles, long long rays, long long params) {
    return 3 * rays > 32 * params ? 0 : spread_of(tiles);
}

// Sets the parameter-vector block order of d (see LayoutKey): s = 0 the
// canonical order, s > 0 bricks of 2^s voxels per edge.  Returns false (and
// leaves d canonical) when G is not a multiple of the brick edge.
inline bool set_layout(DevScene& d, int s) {
    const long long G = d.G;
    if (s <= 0 || G % (1ll << s) != 0) {
        d.lay_s = 0;
        d.lay_ys = (int)G;
        d.lay_zs = (int)(G * G);
        return s <= 0;
    }
    const long long B = 1ll << s, nb = G / B;
    d.lay_s = s;
    d.lay_ys = (int)(nb * B * B * B);
    d.lay_zs = (int)(nb * nb * B * B * B);
    return true;
}

// Kernels launched by this library since load (instrumentation).
extern unsigned long long g_launches;
inline void count_launch(unsigned long long k = 1) { __atomic_fetch_add(&g_launches, k, __ATOMIC_RELAXED); }

// Launches of at most this many tiles (warps) gather from the grid itself,
// several samples of a ray at once (kAheadForward and its neighbours in
// k_march.cu): a copy costs a launch, 4-5 us, and pays where the gathers bound the
// march, not their latency.  us a call, copies / groups: image 32^3, 12 x 64^2
// (1536 tiles) 31 / 26 and 16 x 64^2 (2048 tiles) 32 / 37, so 12 tiles an SM
// (168 registers a thread keep them resident); forward marches then take
// groups of two up to 28 an SM: 16 x 64^2 32 / 30; residual 107^3, 64 x 45 x 42
// (4224 tiles) 223 / 137; the other way round 128^3, 300^2 (2888 tiles) 109 /
// 119.  J^T v and the diagonal, bound by their reductions, up to the spread
// lane order: J^T v 32^3, 12 x 64^2 (1536 tiles) 75 / 88, 30^3, 103 x 417 (1365)
// 67 / 60.
constexpr long long kFewTiles = 152 * 12, kMidTiles = 152 * 28, kFewScatterTiles = 152 * 10 - 1;
// The diagonal's groups of two leave 8 warps an SM room (255 registers): 90^3, 283
// x 166 (1512 tiles) 220 / 284 us, 204^3 BF16, 231 x 179 (1305) 602 / 791; up to 8
// an SM 5% the other way.
constexpr long long kFewDiagTiles = 152 * 8;
// The marches of a batch gather from copies when its scenes have at least this
// many samples per voxel together (a single scene's: kCopyRule in perf_api.cu).
constexpr double kCopyRatio = 0.3;
// Gather copies of the n_vox grid voxels of x (and of p, if given) and x's
// opacity records (sig, may be null): see GatherKey (gather_size(G) voxels per
// copy, 8 floats per voxel of sig).
cudaError_t launch_gather_copy(long long n_vox, int G, int dtype, const void* x, float4* copy,
                               float* sig, cudaStream_t st, int p_dtype = 0,
                               const void* p = nullptr, float4* pcopy = nullptr);

// The diagonal of n_blocks blocks from the packed sums a COPY diagonal march
// (mode 2 of launch_scatter / launch_scatter_batch with sc.xcopy) adds to
// sc.diag2, zeroed by the caller, in the same block order.
cudaError_t launch_expand_diag(long long n_blocks, const float2* diag2, float* diag, cudaStream_t st);

// Where a PCG kernel also writes the direction p of one system for the A p's
// gathers: the gather copy of its grid.
struct GatherDst {
    float4* copy;          // null: not written
    long long first;       // first parameter block of the system
    long long nv;          // its grid voxels
    int G;
};

// While it lives, this thread's allocations are allowed beside a capture on
// another stream (which they would otherwise end): a march that is not captured
// may make its workspace at any time.
struct BesideCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    BesideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~BesideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    BesideCapture(const BesideCapture&) = delete;
    BesideCapture& operator=(const BesideCapture&) = delete;
};

// Total grid samples and shell hits over all rays (one march of the scene).
cudaError_t launch_count_samples(const DevScene& sc, unsigned long long* out, cudaStream_t st);

// mode: 0 render (out = float rgb, T_out), 1 residual (out = r, F), 2 F only.
// target and the residual are in the scene's storage type (float / bf16).
// cut (mode 0): the rendering opacity threshold (see composite in k_march.cu).
cudaError_t launch_forward(const DevScene& sc, int dtype, const void* x, const void* target,
                           void* out, float* T_out, double* F, int mode, cudaStream_t st,
                           float cut = 0.0f);
cudaError_t launch_jvp(const DevScene& sc, int dtype, const void* x, const void* p, int p_dtype,
                       float* out, cudaStream_t st);
// mode: 0 J^T v (v float32), 1 A p (+p^T A p), 2 diag(J^T J) (+ J^T r when v = r,
// in the scene's storage type, and out2 given).
// out3 (mode 2, may be null): per grid voxel the cross entries (colour k,
// opacity) of the 4x4 diagonal block of J^T J.
// coef / tile_off (mode 2, may be null): also store the per-sample
// coefficients (w_i, dH/dsigma_i) of the coefficient-cached A p.
cudaError_t launch_scatter(const DevScene& sc, int dtype, int mode, const void* x, const void* p,
                           int p_dtype, const void* v, float* out, float* out2, double* pap,
                           cudaStream_t st, float* out3 = nullptr, float* coef = nullptr,
                           const long long* tile_off = nullptr);
// Coefficient-cached A p (k_march.cu): rows[t] = rows of pixel tile t in the
// coefficient store (its largest grid sample count + shells); A p (+p^T A p)
// from p (p_dtype: 0 float, 1 bf16) and the stored coefficients.
cudaError_t launch_tile_rows(const DevScene& sc, int* rows, cudaStream_t st);
// sums[0] += sum of keff[ray], sums[1] += sum of K over the rays of tiles
// [tile_lo, n_tiles) of sc
cudaError_t launch_coef_prefix(const DevScene& sc, const int* keff, unsigned long long* sums,
                               cudaStream_t st);
cudaError_t launch_apply_coef(const DevScene& sc, const void* p, int p_dtype, const float* coef,
                              const long long* tile_off, float* out, double* pap, cudaStream_t st);
// Shell-hit table of a scene (k_march.cu): n_rays x S float4 entries (first
// texel index, fu, fv, column step) for the shells each ray hits, equirect
// texel coordinates in FP64; a march reads it when sc.shell_tab is set.
cudaError_t launch_shell_table(const DevScene& sc, float4* tab, cudaStream_t st);

// Algorithm 2 vector work (k_pcg.cu).  Delta, rho, p: FP32 (p is also the
// array the ray march gathers); p16 (may be null): its BF16 copy for BF16
// scenes; Ap: FP32 scatter target, zeroed by begin and update; dst: GatherDst.
cudaError_t launch_pcg_begin(long long n, const float* grad, const float* diag, float* delta,
                             float* rho, float* p, __nv_bfloat16* p16, float* Ap, PcgScalars* s,
                             int max_iter, int fixed, double eps_rel, double stall,
                             const float* blocks, long long n_block, cudaStream_t st,
                             double* hist = nullptr, long long hist_cap = 0,
                             GatherDst dst = GatherDst{});
cudaError_t launch_pcg_update(long long n, float* delta, float* rho, const float* p, float* Ap,
                              const float* diag, const float* blocks, long long n_block,
                              PcgScalars* s, cudaStream_t st);
// One thread: the exit test of Algorithm 2 and beta (after launch_pcg_update).
cudaError_t launch_pcg_finish(PcgScalars* s, cudaStream_t st);
cudaError_t launch_pcg_dir(long long n, const float* rho, const float* diag, const float* blocks,
                           long long n_block, float* p, __nv_bfloat16* p16, PcgScalars* s,
                           cudaStream_t st, GatherDst dst = GatherDst{});
// x_out = P(x + gamma delta) (project: sigma >= 0, 0 <= c <= 1), formed in FP64;
// optional float32 and bf16 outputs.  delta is in the block order lay
// (x = G, y = brick shift s, z = ys, w = zs of the LayoutKey; y = 0:
// canonical, the default), x and the outputs are canonical.
cudaError_t launch_trial(long long n, const float* x, const float* delta, double gamma,
                         int project, float* x_out, __nv_bfloat16* x16_out, cudaStream_t st,
                         int4 lay = int4{0, 0, 0, 0});
// The int4 block order of d for launch_trial.
inline int4 layout_of(const DevScene& d) { return int4{d.G, d.lay_s, d.lay_ys, d.lay_zs}; }
cudaError_t launch_to_bf16(long long n, const float* x, __nv_bfloat16* y, cudaStream_t st);
// One Adam step with projection (k_pcg.cu); c1, c2 the bias corrections.
cudaError_t launch_adam(long long n, float* x, const float* g, float* m, float* v, float b1,
                        float b2, float lr, float eps, float c1, float c2, int project,
                        cudaStream_t st);

// Segmented forms (a batch of independent systems, scalars s[y] for system
// y < n_seg): chunks (device, n_chunks int4) assigns CTA b the parameter
// blocks [chunks[b].y, chunks[b].z) of system chunks[b].x; null = one system.
cudaError_t launch_pcg_begin_seg(long long n, int n_seg, const int4* chunks, long long n_chunks,
                                 const float* grad, const float* diag, float* delta, float* rho,
                                 float* p, __nv_bfloat16* p16, float* Ap, PcgScalars* s,
                                 int max_iter, int fixed, double eps_rel, double stall,
                                 const float* blocks, long long n_block, cudaStream_t st,
                                 const GatherDst* dsts = nullptr);
cudaError_t launch_pcg_update_seg(long long n, int n_seg, const int4* chunks, long long n_chunks,
                                  float* delta, float* rho, const float* p, float* Ap,
                                  const float* diag, const float* blocks, long long n_block,
                                  PcgScalars* s, cudaStream_t st);
cudaError_t launch_pcg_finish_seg(PcgScalars* s, int n_seg, cudaStream_t st);
cudaError_t launch_pcg_dir_seg(long long n, int n_seg, const int4* chunks, long long n_chunks,
                               const float* rho, const float* diag, const float* blocks,
                               long long n_block, float* p, __nv_bfloat16* p16, PcgScalars* s,
                               cudaStream_t st, const GatherDst* dsts = nullptr);
// Segment y: x_out = P(x + gamma[y] Delta) where mask[y] (or every segment).
// lay / base (device, n_seg entries each, may be null): segment y's Delta is
// in the block order lay[y] (see launch_trial) from its first block base[y].
cudaError_t launch_trial_seg(long long n, int n_seg, const int4* chunks, long long n_chunks,
                             const float* x, const float* delta, const double* gamma,
                             const int* mask, int project, float* x_out, cudaStream_t st,
                             const int4* lay = nullptr, const long long* base = nullptr);

// Level change of the hierarchical formulation (k_hier.cu): y (level 2G,
// maps 2He x 2We) from x (level G, maps He x We).
cudaError_t launch_upsample(const float* x, int G, int S, int He, int We, int cube, float* y,
                            cudaStream_t st);

}  // namespace perf
