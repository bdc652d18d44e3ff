// fr_ctx.h -- the context object behind the opaque fr_ctx handle.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "../../include/fr.h"
#include "fr_internal.h"
#include "fr_tuner.h"

struct fr_ctx {
  int S = 0;
  fr_blob blob{};
  fr::Geom g{};
  int device = 0;
  float *acc = nullptr;
  size_t plane = 0;
  float2 *lut = nullptr;
  int lut_n = 0;
  float lut_scale = 0.f;
  float inv_i0a = 0.f, inv_pa = 0.f;
  float poly[fr::POLY_N] = {};
  double poly_err = 1.0;  // max |poly - b| measured on the host (FP32)
  float4 *scratch = nullptr;
  // slabs of the direct-drain gather's split units; replaced smaller buffers
  void *slabs = nullptr;
  size_t slabs_bytes = 0;
  std::vector<void *> slabs_old;
  int *d_err = nullptr;
  unsigned long long *d_count = nullptr;
  fr_options opt{};
  cudaStream_t last_stream = nullptr;
  unsigned long long images = 0;
  int launches = 0;
  int alloc_countdown = 0;  // fault injection: allocations left before the injected failure
  fr::Tuner tuner;
  // gather work-unit lists, keyed by (brick shape, n); most recent first
  struct Units {
    int shape = -1, n = -1, count = 0, any_split = 0, algo = 0;
    int4 *dev = nullptr;
    // direct-drain gather: the units of its fold columns (|x| <= floor(a)), then the
    // merge's list, stored after the main units in dev; the slabs they need
    int fold_count = 0;
    const int4 *fold = nullptr;
    fr::SlabMerge merge{};
    fr::SlabNeed need{};
  };
  Units units[8];
  unsigned long long *d_phase = nullptr;  // gather phase counters (debug bit 1)
  // cost model
  float *d_mlp = nullptr;
  bool mlp_trained = false;
  // reconstruction (Algorithm 1's last step): weighted half spectrum and the
  // inverse-FFT plan, created on first use
  float2 *spec = nullptr;
  int fft_plan = -1;
  // image transforms: batched R2C plans (full chunk, tail) and the FP16 staging buffer
  int prep_plan[2] = {-1, -1};
  int prep_batch[2] = {0, 0};
  float2 *prep_ws = nullptr;
};


namespace fr {
int key_bucket(int n);
InsertArgs base_args(const fr_ctx *c);
// allocate the context's float4 scratch volume if it has none yet
int ensure_scratch(fr_ctx *c);
// configuration id as this context runs it (see the other form)
Config effective_config(const fr_ctx *c, int id);
// gather work unit with its expected load (images it scans)
struct UnitLoad {
  double load;
  int4 unit;  // brick x, y, z; split | nsplit << 16
};
// have slabs for `need` in the context, and put them into a (a smaller buffer of an
// earlier call lives on: plans and captured graphs hold it)
int ensure_slabs(fr_ctx *c, const SlabNeed &need, InsertArgs &a);
// Give the split units among `units` (all of them if `all`) their slabs from block
// need.blocks on, pack the units as InsertArgs::units of the direct-drain gather says,
// and list their bricks for the merge.  fw: width of the shape's warp footprints.
void assign_slabs(std::vector<UnitLoad> &units, const GatherShape &sh, int fw, int n, bool all,
                  SlabNeed &need, std::vector<int4> &merge);
double gather_unit_loads(const fr_ctx *c, int shape, int n, double target,
                         std::vector<UnitLoad> &out, int &any_split);
// Expected images of one work unit, given the total over all bricks.
// Per-voxel gather: the total over per_sm units per SM, at least 16.  Direct-drain
// gather (direct = true): the same, but at least 8 images (a unit's fixed cost, its
// partial sums cleared and written back, is about one image's work per 512
// voxels), or fewer, down to 2, while the units would not fill 8 per SM.
// Measured on GB300 (insert time before the slabs; floors of 16 / 8 / 4 / 2 images):
// S = 32, 64 images 57 / 45 / 36 / 30 us; S = 64, 200 images 112 / 86 / 85 / 85 us;
// S = 96, 500 images at 18 images a unit 242 us, at 6 images 255.
double unit_share(double total, int sms, int per_sm, bool direct);
// work units of bricks of shape sh tiling x in [x0, x1] (all y, z), split so
// that no unit exceeds `target` expected images (target <= 0: unit_share of the
// total), into at most 64 units per brick of at least 2 images (per-voxel
// gather: 8), unsplit below 16 images; returns the total expected load.
// Units per SM of the direct-drain gather's main bricks (16 / 24 / 32 / 64 / 96
// measured at S = 128, n = 1000: 623 / 607 / 591 / 603 / 617 us; S = 96, n = 777, a =
// 2.5: 589 / 580 / 591 / 613 / 615; S = 256, n = 5000: 8.43 / 8.40 / 8.39 / 8.66 / 8.38
// ms; more units fill the SMs better, and have more slabs to merge) and of its fold
// columns (the fold bricks are few and every plane crosses the central ones: fine
// splits keep their serial path inside the launch's time; 4 to 12 measured alike).
constexpr int MAIN_UNITS_PER_SM = 32;
constexpr int FOLD_UNITS_PER_SM = 8;
double brick_unit_loads(const fr_ctx *c, const GatherShape &sh, int x0, int x1, int n,
                        double target, int per_sm, bool direct, std::vector<UnitLoad> &out,
                        int &any_split);
// drop cached batched-insertion plans that refer to c (called by fr_destroy)
void batched_forget(const fr_ctx *c);
// release the reconstruction buffers of c (called by fr_destroy)
void reconstruct_release(fr_ctx *c);
int do_insert_ctx(fr_ctx *c, const void *images, fr_dtype dtype, const float *rot, int n,
                  cudaStream_t st);
}  // namespace fr
