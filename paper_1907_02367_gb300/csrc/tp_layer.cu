// Instantiations and launchers of the tent kernel for one space dimension, one
// kind of sweep and meshes with or without Neumann facets.  Compiled once per
// dimension (-DTP_DIM=1, 2 or 3), kind (-DTP_KIND=0 forward binary64, 1 forward
// mixed, 2 adjoint binary64, 3 forward mixed on the tensor cores) and
// -DTP_NEU=0 or 1, so that the translation units build in parallel.
#include <algorithm>
#include <utility>

#include "tp_kernel.cuh"

#if !defined(TP_DIM) || !defined(TP_KIND) || !defined(TP_NEU)
#error "compile with -DTP_DIM=1, 2 or 3, -DTP_KIND=0, 1, 2 or 3 and -DTP_NEU=0 or 1"
#endif

#define TP_CAT2(a, b, c, d, e) a##b##c##d##e
#define TP_CAT(a, b, c, d, e) TP_CAT2(a, b, c, d, e)
#define TP_NAME(a) TP_CAT(a, TP_DIM, TP_KIND, _n, TP_NEU)

namespace tp {

namespace {

constexpr bool kMixed = TP_KIND == 1 || TP_KIND == 3, kAdj = TP_KIND == 2, kTc = TP_KIND == 3;

using Kernel = void (*)(const KArgs, const int);

// the variant for (dataflow, split right-hand sides, wide CTAs); launches per
// level have narrow CTAs, the tensor cores take split right-hand sides in wide
// CTAs
constexpr int kVariants = 8;
template <int I>
Kernel variant() {
  constexpr bool PERSIST = I & 4, SPLIT = I & 2, WIDE = I & 1;
  if constexpr (kTc ? !(SPLIT && WIDE) : (WIDE && !PERSIST)) return nullptr;
  else return k_layer<TP_DIM, kMixed, kAdj, PERSIST, TP_NEU != 0, SPLIT, kTc, WIDE>;
}
template <int... I>
Kernel pick_of(int i, std::integer_sequence<int, I...>) {
  static const Kernel k[kVariants] = {variant<I>()...};
  return k[i];
}
Kernel pick(int i) { return pick_of(i, std::make_integer_sequence<int, kVariants>()); }
Kernel pick(bool persistent, bool split, bool wide) {
  return pick((persistent ? 4 : 0) + (split ? 2 : 0) + (wide ? 1 : 0));
}

cudaLaunchConfig_t config(int n_cluster, int cs, size_t smem, cudaStream_t st, bool wide, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_cluster * cs));
  cfg.blockDim = dim3(wide ? kThreadsWide : kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// largest static shared memory of the instantiations (bytes), and the dynamic limit set on each
cudaError_t TP_NAME(layer_static_smem_d)(size_t* bytes) {
  *bytes = 0;
  for (int i = 0; i < kVariants; ++i)
    if (Kernel k = pick(i)) {
      cudaFuncAttributes fa;
      const cudaError_t e = cudaFuncGetAttributes(&fa, (const void*)k);
      if (e != cudaSuccess) return e;
      *bytes = std::max(*bytes, fa.sharedSizeBytes);
    }
  return cudaSuccess;
}
cudaError_t TP_NAME(layer_attrs_d)(size_t smem) {
  for (int i = 0; i < kVariants; ++i)
    if (Kernel k = pick(i)) {
      const cudaError_t e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}
cudaError_t TP_NAME(launch_layer_d)(const KArgs& a, int n_cluster, int cs, int t0, size_t smem, cudaStream_t st,
                                    bool persistent, bool wide) {
  cudaLaunchAttribute attr[1];
  if (!kTc && !persistent) wide = false;
  const cudaLaunchConfig_t cfg = config(n_cluster, cs, smem, st, wide, attr);
  return cudaLaunchKernelEx(&cfg, pick(persistent, a.rsplit != 0, wide), a, t0);
}
cudaError_t TP_NAME(max_clusters_d)(int cs, size_t smem, bool split, bool wide, int* n) {
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = config(1, cs, smem, nullptr, wide, attr);
  return cudaOccupancyMaxActiveClusters(n, pick(true, split, wide), &cfg);
}

}  // namespace tp
