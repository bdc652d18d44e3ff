// fr_gather_fold.cu -- the direct-drain gather instantiated for the fold
// columns |x| <= floor(a) (FOLD): bricks one footprint wide, 4 columns (8 for
// 2 <= a < 3) x 32 x 8, four warp footprints stacked in y, the fold predicate
// tested per pixel, polynomial weights.  Launched
// beside the main direct-drain launch, which covers x >= floor(a) + 1: for one
// batch, or for the work items of several batches in one launch.
#include "fr_gather2.cuh"

namespace fr {

namespace {
constexpr int FBY = 32, FZC = 8;
constexpr int FOLD_MINW = 16;  // resident warps per SM the registers allow
// three fold columns for a < 2 (a footprint 4 wide), five for 2 <= a < 3
template <int KB>
constexpr int fold_width() { return KB == 4 ? 4 : 8; }
}  // namespace

GatherShape fold_shape(int kb) { return GatherShape{kb == 4 ? fold_width<4>() : fold_width<6>(), FBY, FZC}; }

template <int F16, int KB>
static cudaError_t launch_fold(const InsertArgs &a, cudaStream_t st) {
  constexpr int FW = fold_width<KB>();
  auto fn = gather2_kernel<FW, FBY, FZC, F16, FOLD_MINW, KB, FW, 1>;
  const size_t smem = gather2_warp_smem<FW, KB, 1>(a.chunk);
  cudaError_t e = allow_dynamic_smem((const void *)fn, smem);
  if (e != cudaSuccess) return e;
  if (a.nunits <= 0) return cudaSuccess;
  fn<<<a.nunits * g2_warps<FW, FBY, FZC, FW>(), 32, smem, st>>>(a);
  return cudaGetLastError();
}

template <int F16, int KB>
static cudaError_t launch_fold_multi(const MultiLaunch &p, cudaStream_t st) {
  constexpr int FW = fold_width<KB>();
  auto fn = gather2_multi_kernel<FW, FBY, FZC, F16, FOLD_MINW, KB, FW, 1>;
  const size_t smem = gather2_warp_smem<FW, KB, 1>(p.base.chunk);
  cudaError_t e = allow_dynamic_smem((const void *)fn, smem);
  if (e != cudaSuccess) return e;
  if (p.nitems <= 0) return cudaSuccess;
  return launch_multi((const void *)fn, p, g2_warps<FW, FBY, FZC, FW>(), 32, smem, st);
}

cudaError_t launch_gather_fold_multi(int f16, const MultiLaunch &p, cudaStream_t st) {
  if (p.base.chunk > 128) return cudaErrorInvalidValue;
  if (p.base.g.KB == 4) return f16 ? launch_fold_multi<1, 4>(p, st) : launch_fold_multi<0, 4>(p, st);
  return f16 ? launch_fold_multi<1, 6>(p, st) : launch_fold_multi<0, 6>(p, st);
}

cudaError_t launch_gather_fold(const InsertArgs &a, cudaStream_t st) {
  if (a.chunk > 128) return cudaErrorInvalidValue;
  if (reinterpret_cast<uintptr_t>(a.images) & 15u) return cudaErrorInvalidValue;
  if (a.g.KB == 4) return a.f16 ? launch_fold<1, 4>(a, st) : launch_fold<0, 4>(a, st);
  return a.f16 ? launch_fold<1, 6>(a, st) : launch_fold<0, 6>(a, st);
}

}  // namespace fr
