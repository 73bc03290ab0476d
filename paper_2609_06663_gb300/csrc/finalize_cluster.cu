// Launches of the cluster finalisation (finalize_cluster.cuh): a thread-block
// cluster per unit.

#include <atomic>

#include "finalize_cluster.cuh"

namespace ecokv {
namespace {

template <int kMode, int kSh, bool kVar>
__global__ void __launch_bounds__(kCThreads, Shape<kSh>::kMinCtas) finalize_cluster_kernel(FinalArgs f) {
  extern __shared__ __align__(16) uint8_t fc_smem[];
  ClusterSmem<kSh>& sm = *reinterpret_cast<ClusterSmem<kSh>*>(fc_smem);
  cg::cluster_group cl = cg::this_cluster();
  // The peers must have started before the first store into their shared
  // memory: this arrival is waited for just before it.
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // Launched as a programmatic dependent of the streaming pass: let the gather
  // be scheduled behind this grid, and wait for the previous grid's results
  // (a no-op when launched plainly).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int C = (int)cl.num_blocks();
  cluster_unit<kMode, kSh, kVar, false>(f, sm, cl, blockIdx.x / C, (int)cl.block_rank(), C);
}

template <int kSh>
cudaError_t set_attrs(bool nonportable) {
  const int bytes = (int)sizeof(ClusterSmem<kSh>);
  const void* kernels[5] = {(const void*)finalize_cluster_kernel<0, kSh, false>,
                            (const void*)finalize_cluster_kernel<1, kSh, false>,
                            (const void*)finalize_cluster_kernel<0, kSh, true>,
                            (const void*)finalize_cluster_kernel<1, kSh, true>,
                            (const void*)finalize_cluster_kernel<2, kSh, false>};
  for (const void* k : kernels) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && nonportable) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int kSh>
cudaError_t launch_shape(const FinalArgs& f, int U, int C, bool select_only, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(U * C), 1, 1);
  cfg.blockDim = dim3(kCThreads, 1, 1);
  cfg.dynamicSmemBytes = sizeof(ClusterSmem<kSh>);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const bool var = f.vnorm != nullptr || f.wlo != nullptr || f.mad != nullptr;
  if (select_only) return cudaLaunchKernelEx(&cfg, finalize_cluster_kernel<2, kSh, false>, f);
  if (f.idx == nullptr)
    return var ? cudaLaunchKernelEx(&cfg, finalize_cluster_kernel<0, kSh, true>, f)
               : cudaLaunchKernelEx(&cfg, finalize_cluster_kernel<0, kSh, false>, f);
  return var ? cudaLaunchKernelEx(&cfg, finalize_cluster_kernel<1, kSh, true>, f)
             : cudaLaunchKernelEx(&cfg, finalize_cluster_kernel<1, kSh, false>, f);
}

// Per device: the attributes set, and whether clusters of 16 CTAs of the
// longest shape can be resident (cudaOccupancyMaxActiveClusters > 0).
std::atomic<int> g_setup[64];  // 0 = not yet, 1 = set, clusters of 16 unavailable, 2 = set and available
std::atomic<int> g_sms[64];    // SMs, set before g_setup

int device_setup() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  int st = g_setup[dev].load();
  if (st != 0) return st;
  if (set_attrs<0>(false) != cudaSuccess || set_attrs<1>(false) != cudaSuccess || set_attrs<2>(false) != cudaSuccess ||
      set_attrs<3>(false) != cudaSuccess)
    return -1;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return -1;
  g_sms[dev].store(sms);
  st = 1;
  if (set_attrs<0>(true) == cudaSuccess && set_attrs<3>(true) == cudaSuccess) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(16u * 16u, 1, 1);
    cfg.blockDim = dim3(kCThreads, 1, 1);
    cfg.dynamicSmemBytes = sizeof(ClusterSmem<3>);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 16;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (const void*)finalize_cluster_kernel<1, 3, false>, &cfg) == cudaSuccess &&
        n > 0)
      st = 2;
  }
  cudaGetLastError();  // an unavailable configuration leaves no error behind
  g_setup[dev].store(st);
  return st;
}

// Shape and cluster size for U units of Tv candidates; shape -1 when none takes
// them.  The fewest candidates a thread whose CTAs are all resident at once;
// failing that (many units) the fewest in clusters of at most four.  One layer
// of 4 heads x 32768 keys: 16 CTAs of 8 a thread 15 us, 4 of 32 a thread 25 us;
// 28 layers x 4 heads of that length: 3 waves of the former, one of the latter.
void pick_shape(int Tv, long long U, int long_ok, int sms, int& sh, int& C) {
  const int t = Tv > 0 ? Tv : 1;
  const int cap[4] = {Shape<0>::kCap, Shape<1>::kCap, Shape<2>::kCap, Shape<3>::kCap};
  const int most[4] = {long_ok ? Shape<0>::kMaxCluster : 8, Shape<1>::kMaxCluster, Shape<2>::kMaxCluster,
                       long_ok ? Shape<3>::kMaxCluster : 8};
  const int resident[4] = {Shape<0>::kMinCtas, Shape<1>::kMinCtas, Shape<2>::kMinCtas, Shape<3>::kMinCtas};
  for (sh = 0; sh < 4; ++sh) {
    C = (t + cap[sh] - 1) / cap[sh];
    if (C <= most[sh] && U * C <= (long long)resident[sh] * sms) return;
  }
  for (sh = 0; sh < 4; ++sh) {
    C = (t + cap[sh] - 1) / cap[sh];
    if (C <= (sh < 3 ? 4 : most[3])) return;
  }
  sh = -1;
  C = 0;
}

int current_sms() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? g_sms[dev].load() : 0;
}

}  // namespace

bool cluster_finalize_fits(int Tv) {
  const int st = device_setup();
  if (st < 0) return false;
  int sh, C;
  pick_shape(Tv, 1, st == 2, current_sms(), sh, C);
  return sh >= 0;
}

cudaError_t launch_finalize_cluster(const FinalArgs& f, int U, bool select_only, cudaStream_t s) {
  const int st = device_setup();
  if (st < 0) return cudaErrorUnknown;
  int sh, C;
  pick_shape(f.Tv, U, st == 2, current_sms(), sh, C);
  switch (sh) {
    case 0: return launch_shape<0>(f, U, C, select_only, s);
    case 1: return launch_shape<1>(f, U, C, select_only, s);
    case 2: return launch_shape<2>(f, U, C, select_only, s);
    case 3: return launch_shape<3>(f, U, C, select_only, s);
  }
  return cudaErrorNotSupported;
}

}  // namespace ecokv
