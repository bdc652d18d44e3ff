// fr_internal.h -- types shared by the kernels and the host runtime of libfr.
//
// Accumulator layout in HBM.  Folding puts every insertion point at q_x >= 0,
// so a voxel with x < -floor(a) is never touched; the context stores only
// x in [xa0, S/2] with xa0 = -floor(a).  Six float planes, each
// [z][y][x - xa0] (x fastest), hold a double-float (hi + lo) running sum of
// V.re, V.im and W:  plane p at acc + p * plane_elems, order
// {Vre_hi, Vim_hi, W_hi, Vre_lo, Vim_lo, W_lo}.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace fr {

// blob weights: table staged in shared memory (precomputed), Abramowitz &
// Stegun Bessel approximations evaluated per pixel, or a Chebyshev polynomial
// in r^2 held in registers (both on the fly)
enum WeightMode { W_LUT = 0, W_OTF = 1, W_POLY = 2 };
constexpr int POLY_N = 12;  // coefficients of the degree-11 weight polynomial
enum Algo { ALGO_GATHER = 0, ALGO_SCATTER = 1, ALGO_GATHER2 = 2 };

struct Geom {
  int S;      // image side (even)
  int H;      // S / 2
  int NX;     // stored columns per row, S / 2 + 1
  int D;      // volume side, S + 1
  int xa0;    // first stored accumulator x coordinate, -floor(a)
  int NXa;    // stored accumulator x extent, H - xa0 + 1
  float a;    // blob radius
  float a2;   // a * a
  float alpha;
  int KB;     // candidate box width per axis: floor(2a) + 1 rounded up to 4 or 6
};

// Per-launch arguments of the insertion kernels.
struct InsertArgs {
  Geom g;
  const void *images;   // [n][S][NX] complex, FP32 (float2) or FP16 (half2)
  int f16;              // 1 if images are FP16
  const float *rot;     // [n][9]
  int n;                // images in this launch
  float *acc;           // 6 planes (see above)
  size_t plane;         // elements per plane
  const float2 *lut;    // blob table: (value at node i, value[i+1] - value[i]), lut_n entries
  int lut_n;
  float lut_scale;      // (lut_n - 1) / a^2
  float inv_i0a;        // 1 / I0(alpha) (on-the-fly weights)
  float inv_pa;         // 1 / (A&S 9.8.2 polynomial at 3.75 / alpha) (on-the-fly weights)
  float poly[POLY_N];   // b as a polynomial in x = 2 r^2 / a^2 - 1, power basis (W_POLY)
  float2 poly2[POLY_N]; // the same coefficients as pairs (c_k, c_k) for packed FP32x2 FMAs
  int *err;             // device error word
  // gather geometry
  int nbx, nby, nbz;    // bricks per axis
  int chunk;            // capacity of a warp's image list
  // work units: (brick x, y, z, split | nsplit << 16); direct-drain gather: (brick x |
  // y << 10 | z << 20, slab, 0, split | nsplit << 16)
  const int4 *units;
  int nunits;
  // direct-drain gather: units of the fold columns, computed in the same launch.
  // units == null (no list in device memory): each of nunits / nfold is one of
  // unit_most splits of a brick, which uses as many as its load over unit_share
  const int4 *fold;
  int nfold;
  float unit_share;
  int unit_most;
  // correct the projections for a rotation that FP32 rounding left short of
  // orthonormal.  fr_insert_noalloc does, whose scatter places every sample to
  // FP32 accuracy.  fr_insert keeps the plain R^T c: the correction would cost 1 % and
  // cut the error at S = 128 from 1.6e-6 to 3.8e-7, but it moves single voxels by up to
  // 2.3e-4 of the RMS at S = 156, more at 256, and the performance cases (perf/cases.py)
  // take results that differ by up to 3e-4 for the same
  int ortho;
  int any_split;        // 1 if some unit shares its brick with other units
  unsigned long long *phase;  // optional per-phase cycle and item counters (PH_*), or null
  // scatter
  float4 *scratch;      // [z][y][x - xa0] (re, im, w, 0)
  // direct-drain gather: slabs of the split units' partial sums (SLAB_BLOCK), the
  // state of each footprint whose unit may fold its sums more than once (0: no sums, 1:
  // FP32 sums, 2: FP32 pairs) at its first block, and the planes of a slab (3, or 6 if
  // there are such units).  null:
  // split units add to scratch
  float *slab;
  int *slab_state;
  int slab_planes;
};

// Per-phase counters of the gather kernel (diagnostics, enabled by
// fr_options.debug bit 1): SM clock cycles spent by warps in each phase and
// item counts.
enum PhaseCounter {
  PH_CULL = 0, PH_QUEUE, PH_DRAIN_FAST, PH_DRAIN_EDGE, PH_DRAIN_CAREFUL, PH_FLUSH,
  PH_ITEMS_FAST, PH_ITEMS_EDGE, PH_ITEMS_CAREFUL, PH_LIST_IMAGES, PH_WARP_CYCLES, PH_ROUNDS,
  PH_DRAIN_FOLD, PH_ITEMS_FOLD,
  PH_COUNT = 16
};

// Error bits written to the device error word.
enum DevErr { DERR_RANGE = 1, DERR_TIMEOUT = 2 };

struct KernelInfo {
  const void *fn;       // __global__ function pointer
  int threads;          // block size
  size_t smem;          // dynamic shared memory for the launch
};

// ---- gather family: template parameters of one instantiation
struct GatherShape {
  int bx, by, zc;       // brick: bx x by columns of zc voxels (one column per thread)
};

// Private partial sums of the direct-drain gather's split units.  A unit's slab number
// counts blocks of SLAB_BLOCK voxels; its footprints follow one another, each of
// footprint voxels / SLAB_BLOCK blocks and slab_planes planes (re, im, w, and their
// low parts), a plane in the order of the warp's partial sums: (y, x, z).
constexpr int SLAB_BLOCK = 256;
// Whether a unit of one of ns splits of n images folds its sums at most once (a list
// of 128 images or fewer is folded with the last)
__host__ __device__ constexpr bool slab_once(int n, int ns) { return (n + ns - 1) / ns <= 128; }
// What the merge of an insert's slabs reads: split bricks (brick x | y << 10 | z << 20,
// first slab, splits, 1 if they have states), first nmain of the main shape, then nfold of
// the fold columns
struct SlabMerge {
  const int4 *list;
  int nmain, nfold;
  GatherShape main, fold;
};
// warp footprints (fw x 8 x 8 voxels) of a brick
__host__ __device__ constexpr int gather2_footprints(const GatherShape &sh, int fw) {
  return sh.bx / fw * (sh.by / 8) * (sh.zc / 8);
}
// the slab memory of a launch: blocks of SLAB_BLOCK voxels, planes a block
struct SlabNeed {
  int blocks = 0, planes = 3;
  size_t state_bytes() const { return ((size_t)blocks * sizeof(int) + 255) & ~(size_t)255; }
  size_t bytes() const { return state_bytes() + (size_t)blocks * SLAB_BLOCK * planes * sizeof(float); }
};
cudaError_t launch_merge_slabs(const InsertArgs &a, const SlabMerge &m, cudaStream_t st);

// launchers implemented in the .cu files
cudaError_t launch_gather(int shape_id, int wmode, const InsertArgs &a, cudaStream_t st,
                          int query_only, KernelInfo *info);
// direct-drain gather (fr_gather2.cuh): brick shape id of gather2_shape()
int num_gather2_shapes();
GatherShape gather2_shape(int id);
cudaError_t launch_gather2(int shape_id, const InsertArgs &a, cudaStream_t st,
                           int query_only, KernelInfo *info);
size_t gather2_smem_bytes(const GatherShape &sh, int chunk);
// allow a kernel `smem` bytes of dynamic shared memory on the current device
// (and, if carveout >= 0, set its preferred shared-memory carveout in percent);
// remembered per device and kernel; thread-safe
cudaError_t allow_dynamic_smem(const void *fn, size_t smem, int carveout = -1);
// load a kernel's code on the current device if that has not happened yet (remembered
// per device and kernel; thread-safe): lazily, its first launch would
cudaError_t load_kernel(const void *fn);
cudaError_t load_merge_kernels();
// SM count of the current device (cached per device; thread-safe)
int device_sm_count();
// resident CTAs per SM of kernel fn with `threads` threads and `smem` bytes
// of dynamic shared memory on the current device (cached per device, kernel
// and size; thread-safe); 0 if it cannot run
int resident_ctas(const void *fn, int threads, size_t smem);
cudaError_t launch_scatter(int threads, int wmode, const InsertArgs &a, cudaStream_t st,
                           int query_only, KernelInfo *info);
cudaError_t launch_merge_scratch(const InsertArgs &a, cudaStream_t st);
// 1 / (A&S 9.8.2 polynomial at 3.75 / alpha): the constant of the on-the-fly weights
float otf_inv_pa(double alpha);
// coefficients (power basis in x = 2 r^2 / a^2 - 1) of the weight polynomial
void weight_polynomial(double alpha, float *poly);
// the weighting and inverse transform of fr_reconstruct; spec: S * S * S / 2 float2
bool fft_volume_here(int S);
cudaError_t fft_volume(const Geom &g, const float *acc, size_t plane, float w_clip, float2 *spec,
                       float *out, cudaStream_t st);
// images' transforms by this library's kernels (fr_fft.cu): whether there are any
// for this size, and the transforms of m real images into out (float2 or half2
// spectra), by way of spec (m S (S/2 + 1) float2; may be out itself for float2)
bool fft_images_here(int S);
cudaError_t fft_images(int S, const float *real, float2 *spec, int m, int center, void *out,
                       int f16, cudaStream_t st);
// Waits for set-up work on the legacy stream (a memset, a copy from pageable memory, which
// may return before it has reached the device): launches on non-blocking streams are not
// ordered behind it.
inline cudaError_t setup_done() { return cudaStreamSynchronize(cudaStreamLegacy); }
// record a CUDA error for fr_last_cuda_error
void fr_note_cuda_error(int e);
cudaError_t launch_finalize(const Geom &g, const float *acc, size_t plane, float2 *V, float *W,
                            cudaStream_t st);
cudaError_t launch_count(const Geom &g, const float *rot, int n, unsigned long long *out,
                         cudaStream_t st);
cudaError_t launch_debug_fold(const float *r, const int *k, int m, int *out, cudaStream_t st);
cudaError_t launch_debug_blob(const InsertArgs &a, const float *r2, int m, int mode, float *out,
                              cudaStream_t st);

// number of gather shapes and their geometry
int num_gather_shapes();
GatherShape gather_shape(int id);
// bricks of the direct-drain gather's fold-column units (|x| <= floor(a)), one
// footprint wide: 4 columns (8 for KB = 6) x 32 x 8
GatherShape fold_shape(int kb);
// dynamic shared memory a gather launch needs
size_t gather_smem_bytes(const GatherShape &sh, int wmode, int lut_n, int chunk);
size_t gather_persistent_smem_bytes(const GatherShape &sh, int chunk);

// One persistent gather launch over the work items of several batches.
struct PersistentLaunch {
  const InsertArgs *descs;  // device, one per batch
  const int4 *items;        // device, {bx | by << 10 | bz << 20, split word, batch, 0}, one per unit
  int nitems;
  int chunk;                // image-list capacity per warp, common to all batches
  unsigned *counter;        // device, zero at launch
};
cudaError_t launch_gather_persistent(int shape_id, int kb, int f16, const PersistentLaunch &p,
                                     cudaStream_t st);

// One launch over the work items of several batches, one CTA per warp footprint
// of an item (the hardware block scheduler hands them out, heaviest first).  The
// batches of one launch share S, blob, dtype and configuration: what they
// share stays in the kernel parameters (base), the rest is read per batch.
constexpr int MULTI_MAX = 64;  // batches per multi-batch launch
struct MultiLaunch {
  InsertArgs base;           // common arguments: geometry, weights, list capacity
  const InsertArgs *descs;   // device, one per batch (images, rot, n, acc, slab, err)
  // device, {bx | by << 10 | bz << 20, split word, batch | slot << 24, slab}: nfold items
  // of the fold columns, then nitems of the rest
  const int4 *items;
  int nfold;
  int nitems;
  const void *images[MULTI_MAX];  // images of the launch's batches, by slot (read in the inner loop)
};
// the direct-drain gather, FP32 or FP16 images
cudaError_t launch_gather2_multi(int shape_id, int f16, const MultiLaunch &p, cudaStream_t st);

// MLP kernels
cudaError_t mlp_forward(const float *params, const float *x, int m, float *y, cudaStream_t st);
cudaError_t mlp_backward(const float *params, const float *x, const float *t, int m, float *grad,
                         float *loss, float *work, cudaStream_t st);
cudaError_t mlp_adam(float *params, const float *grad, float *m1, float *m2, int t, float lr,
                     float b1, float b2, float eps, cudaStream_t st);
size_t mlp_work_floats(int m);

constexpr int MLP_IN = 16, MLP_H = 64;
constexpr int MLP_NPARAM = MLP_IN * MLP_H + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1;

}  // namespace fr
