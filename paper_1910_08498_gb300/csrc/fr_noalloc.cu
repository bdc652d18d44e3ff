// fr_noalloc.cu -- fr_insert_noalloc: the insertion with its scratch volume in a
// fixed array of static device memory, for callers that must not enter the
// device allocator (they may be sharing the device with latency-bound streams
// that a cudaMalloc/cudaFree would synchronise, or hold all device memory in
// their own pool allocator).  The direct-drain gather runs without a unit list
// (its CTAs work theirs out), every unit adding to the scratch; the atomic
// scatter stays where the gather cannot decide as exactly or has no box (see
// gather_here).  Nothing here allocates:
// no cudaMalloc, no cudaFree, no allocating library routine; the scratch
// address is looked up and every kernel loaded in the device's first call.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "fr_ctx.h"
#include "fr_device.cuh"
#include "fr_internal.h"
#include "fr_noalloc.h"

// One float4 {w re, w im, w, 0} per accumulator voxel of the largest volume:
// D x D x NXa with D = 65 and NXa = S/2 + floor(a) + 1 <= 35 (a < 3); 2.37 MB.
static constexpr size_t NOALLOC_CELLS = (size_t)(FR_NOALLOC_MAX_S + 1) *
                                        (FR_NOALLOC_MAX_S + 1) * (FR_NOALLOC_MAX_S / 2 + 3);
static __device__ __align__(256) float4 g_noalloc_scratch[NOALLOC_CELLS];

namespace fr {
namespace {

constexpr int NOALLOC_SUB = 1024;  // images per scatter launch (span of one FP32 atomic sum)
constexpr int MAX_DEVICES = 64;

struct DeviceSlot {
  bool ready = false;
  float4 *scratch = nullptr;
};
std::mutex g_mu;
DeviceSlot g_slots[MAX_DEVICES];

// Add the scratch sums to V and W (full (S+1)^3 grid) and clear the cells read.
__global__ void noalloc_add_kernel(const Geom g, float4 *__restrict__ scratch,
                                   float2 *__restrict__ V, float *__restrict__ W) {
  const size_t cells = (size_t)g.D * g.D * g.NXa;
  for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < cells;
       v += (size_t)gridDim.x * blockDim.x) {
    const float4 s = scratch[v];
    if (s.x != 0.f || s.y != 0.f || s.z != 0.f) {
      const size_t zy = v / g.NXa;
      const int x = (int)(v - zy * g.NXa) + g.xa0;  // >= -floor(a) > -S/2
      const size_t o = zy * g.D + (size_t)(x + g.H);
      float2 cur = V[o];
      cur.x += s.x;
      cur.y += s.y;
      V[o] = cur;
      W[o] += s.z;
      scratch[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

// The scatter decides r <= a as the real numbers do for every candidate; the
// gather does only in the fold columns for a >= 2.  A candidate that rounding puts on
// the wrong side of the edge costs its weight b(a) = 1 / I0(alpha): at alpha = 0 a
// whole pixel, at alpha = 15 2.9e-6 of one.  At most eight pixels of an image lie at
// one distance < 3 from a voxel (four below 1.58), and the voxel that all n images meet
// holds W > 1.1 n (n), so with b(a) <= 3e-6 even all of them wrong at once, in every
// image, make 2e-5 of the largest W.  Larger b(a) keep the scatter (a = sqrt(3.6),
// rotations by the 3-4-5 angle: by the gather, V is off by 0.17 of its largest value at
// alpha = 0, 1.2e-3 at 8).  So do a^2 within 1e-4 of an integer, where whole lattices of
// candidates can sit on the edge (the DC pixel against the axes' voxels for every
// rotation), and alpha > 16, where the weight polynomial is less accurate than the
// scatter's Bessel approximations (2e-7).
// For the rest by size: the scatter's time goes with the pixels and a^3, the gather's
// with the pixels, hardly with a (the 5 x 5 and 6 x 6 boxes from a = 2 on aside),
// and with the footprints' halo, which weighs more on a small volume.  Gather over
// scatter at 2.5e5 / 5.5e5 / 1.2e6 pixels a launch, S = 64: a = 1.3 1.24 / 1.10 /
// 0.92, 1.6 1.12 / 0.96 / 0.79, 1.75 0.95 / 0.79 / 0.68, 1.9 0.89 / 0.77 / 0.65, 2.1
// 1.24 / 0.85 / 0.65, 2.5 1.01 / 0.74 / 0.58, 2.9 0.84 / 0.67 / 0.56; S = 48: a = 1.6 1.25 /
// 1.05 / 0.97, 1.75 1.06 / 0.91 / 0.83, 1.9 0.99 / 0.86 / 0.79, 2.1 1.38 / 0.99 / 0.80, 2.5
// 1.17 / 0.82 / 0.73; S = 32 and 40 (5.5e5): 0.96 to 1.6.  FP16 images alike.
constexpr float EDGE_WEIGHT_MAX = 3e-6f;  // alpha >= 14.99
bool gather_here(const Geom &g, float edge_weight, int n) {
  const double a2 = (double)g.a * (double)g.a, pixels = (double)n * g.S * g.NX;
  const double enough = g.a < 1.25f  ? 1e30
                        : g.a < 1.5f ? 2e6
                        : g.a < 1.7f ? 1.25e6
                        : g.a < 1.85f ? 5.5e5
                        : g.a < 2.0f ? (g.S >= 60 ? 2.5e5 : 4e5)
                        : g.a < 2.3f ? 1e6
                                     : 6e5;
  return std::fabs(a2 - std::round(a2)) > 1e-4 * a2 && edge_weight <= EDGE_WEIGHT_MAX && g.alpha <= 16.0f &&
         g.S >= 44 && pixels >= enough;
}

// weight polynomial of the last alpha asked for (12 numbers; no allocation)
void cached_polynomial(float alpha, float *poly) {
  static std::mutex mu;
  static float last = -1.0f, c[POLY_N];
  std::lock_guard<std::mutex> lk(mu);
  if (alpha != last) {
    weight_polynomial((double)alpha, c);
    last = alpha;
  }
  std::copy(c, c + POLY_N, poly);
}

// Expected images over all bricks of shape sh that tile x in [x0, x1], for a
// batch of n; *bricks: how many they are.
double brick_images(const Geom &g, const GatherShape &sh, int x0, int x1, int n, int *bricks) {
  const int nbx = (x1 - x0 + sh.bx) / sh.bx, nby = (g.D + sh.by - 1) / sh.by,
            nbz = (g.D + sh.zc - 1) / sh.zc;
  const double hx = 0.5 * (sh.bx - 1), hy = 0.5 * (sh.by - 1), hz = 0.5 * (sh.zc - 1);
  const double r = g.a + std::sqrt(hx * hx + hy * hy + hz * hz);
  double total = 0;
  for (int b = 0; b < nbx * nby * nbz; ++b) {
    const double cx = x0 + b % nbx * sh.bx + hx, cy = -g.H + b / nbx % nby * sh.by + hy,
                 cz = -g.H + b / (nbx * nby) * sh.zc + hz;
    const double d = std::sqrt(cx * cx + cy * cy + cz * cz);
    total += n * ((d <= r ? 1.0 : r / d) + 0.02);
  }
  *bricks = nbx * nby * nbz;
  return total;
}

constexpr int GATHER_SHAPE = 1;  // 16 x 8 x 8 bricks
constexpr int GATHER_CHUNK = 64;
constexpr int UNITS_PER_SM = 96;  // finer than fr_insert's, which have slabs to merge

// Everything a later call would otherwise set up on its way: the code of each kernel
// that some call can launch (cudaFuncGetAttributes loads it), the gather's shared
// memory attribute and the host-side caches behind both.  Once per device, under
// g_mu.
cudaError_t setup_device(DeviceSlot &slot) {
  void *p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  cudaFuncAttributes fa{};
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, noalloc_add_kernel);
  for (float a : {1.9f, 2.25f, 2.75f}) {  // 4 x 4, 5 x 5 and 6 x 6 boxes
    InsertArgs q{};
    q.g.a = a;
    q.g.KB = a < 2.0f ? 4 : 6;
    q.chunk = GATHER_CHUNK;
    KernelInfo info{};
    for (q.f16 = 0; q.f16 < 2 && e == cudaSuccess; ++q.f16) {
      e = launch_gather2(GATHER_SHAPE, q, nullptr, 1, &info);
      if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, info.fn);
    }
    if (e == cudaSuccess) e = launch_scatter(256, W_OTF, q, nullptr, 1, &info);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, info.fn);
  }
  if (e != cudaSuccess) return e;
  device_sm_count();
  slot.scratch = static_cast<float4 *>(p);
  slot.ready = true;
  return cudaSuccess;
}

int cuda_status(cudaError_t e) {
  fr_note_cuda_error((int)e);
  return FR_ERR_CUDA;
}

}  // namespace
}  // namespace fr

extern "C" int fr_insert_noalloc(int S, float a, float alpha, const void *images, fr_dtype dtype,
                                 const float *rotations, int n, void *V, float *W, void *stream) {
  using namespace fr;
  if (S < 8) return FR_ERR_INVALID_ARG;
  if (S & 1) return FR_ERR_UNSUPPORTED;
  if (S > FR_NOALLOC_MAX_S) return FR_ERR_NOALLOC_LIMIT;
  if (!(a > 0.f) || !(alpha >= 0.f && alpha <= 40.f)) return FR_ERR_INVALID_ARG;
  if (!(a < 3.f)) return FR_ERR_UNSUPPORTED;
  if (n < 0 || n > (1 << 24) || (dtype != FR_F32 && dtype != FR_F16)) return FR_ERR_INVALID_ARG;
  if (!V || !W) return FR_ERR_INVALID_ARG;
  if (n == 0) return FR_OK;
  if (!images || !rotations || ((uintptr_t)images & 15)) return FR_ERR_INVALID_ARG;

  // one-time setup per device, with that device current
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_status(e);
  if (dev < 0 || dev >= MAX_DEVICES) return FR_ERR_INVALID_ARG;
  float4 *scratch = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceSlot &slot = g_slots[dev];
    if (!slot.ready) {
      e = setup_device(slot);
      if (e != cudaSuccess) return cuda_status(e);
    }
    scratch = slot.scratch;
  }

  Geom g{};
  g.S = S;
  g.H = S / 2;
  g.NX = S / 2 + 1;
  g.D = S + 1;
  g.a = a;
  g.a2 = a * a;
  g.alpha = alpha;
  g.xa0 = -(int)std::floor(a);
  g.NXa = g.H - g.xa0 + 1;
  g.KB = a < 2.0f ? 4 : 6;
  const size_t cells = (size_t)g.D * g.D * g.NXa;  // <= NOALLOC_CELLS by the checks above
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  InsertArgs args{};
  args.g = g;
  args.f16 = dtype == FR_F16 ? 1 : 0;
  args.inv_i0a = (float)(1.0 / std::cyl_bessel_i(0.0, (double)alpha));
  args.inv_pa = otf_inv_pa((double)alpha);
  args.err = nullptr;
  args.scratch = scratch;

  e = cudaMemsetAsync(scratch, 0, cells * sizeof(float4), st);
  if (e != cudaSuccess) return cuda_status(e);
  const size_t img_bytes = (size_t)S * g.NX * (dtype == FR_F16 ? 4 : 8);
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_status(e);
  const int add_threads = 256;
  const int add_blocks = (int)std::min<size_t>((cells + add_threads - 1) / add_threads,
                                               (size_t)sms * 8);
  const bool gather_any = gather_here(g, args.inv_i0a, std::min(n, NOALLOC_SUB));
  if (gather_any) {
    cached_polynomial(alpha, args.poly);
    for (int k = 0; k < POLY_N; ++k) args.poly2[k] = make_float2(args.poly[k], args.poly[k]);
    args.chunk = GATHER_CHUNK;
    args.any_split = 1;
    args.ortho = 1;
  }
  for (int i0 = 0; i0 < n; i0 += NOALLOC_SUB) {
    args.n = std::min(NOALLOC_SUB, n - i0);
    args.images = static_cast<const unsigned char *>(images) + (size_t)i0 * img_bytes;
    args.rot = rotations + (size_t)i0 * 9;
    if (gather_any && gather_here(g, args.inv_i0a, args.n)) {
      int bricks = 0, fold_bricks = 0;
      const double total = brick_images(g, gather2_shape(GATHER_SHAPE), 1 - g.xa0, g.H, args.n, &bricks);
      brick_images(g, fold_shape(g.KB), g.xa0, -g.xa0, args.n, &fold_bricks);
      args.unit_share = (float)unit_share(total, sms, UNITS_PER_SM, true);
      // splits of a central brick, which every image crosses
      args.unit_most = std::max(1, std::min({64, args.n / 2, (int)std::ceil(1.02 * args.n / args.unit_share)}));
      args.nunits = bricks * args.unit_most;
      args.nfold = fold_bricks * args.unit_most;
      e = launch_gather2(GATHER_SHAPE, args, st, 0, nullptr);
    } else {
      e = launch_scatter(256, W_OTF, args, st, 0, nullptr);
    }
    if (e != cudaSuccess) return cuda_status(e);
    noalloc_add_kernel<<<add_blocks, add_threads, 0, st>>>(g, scratch, static_cast<float2 *>(V), W);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e);
  }
  return FR_OK;
}
