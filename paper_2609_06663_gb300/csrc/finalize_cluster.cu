// Launches of the cluster finalisation (finalize_cluster.cuh): a thread-block
// cluster per unit.

#include <atomic>

#include "finalize_cluster.cuh"

namespace ecokv {
namespace {

template <int kMode, int kSh, bool kVar>
__global__ void __launch_bounds__(Shape<kSh>::kThreads, Shape<kSh>::kMinCtas) finalize_cluster_kernel(FinalArgs f) {
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

// Shared memory a CTA asks for: what it uses, or so much that an SM takes two
// (spread 1) or one (spread 2).  A cluster is placed as soon as one GPC has
// room for it, while the streaming pass still runs on the other SMs; with what
// it uses alone its CTAs then share the two or four SMs that are free first, and
// each runs at a fraction of its speed.  One layer, us a call as used / two /
// one an SM: 4 heads x 32768 keys (16 CTAs each) 59.5 / 53.3 / 50.0, 8 x 65536
// (8 CTAs of 32 candidates a thread) 112 / 99.5 / 90.9, 8 x 8192 38.1 / 35.8 /
// 35.8; but 8 x 131072, whose clusters of 16 are not all resident at one an SM,
// 149 / 142 / 158.  For its few microseconds nothing that needs shared memory
// runs beside it on those SMs; a caller with two streams does not notice: two
// streams of such calls, as used / so, 42.1 / 42.4 us a call at 4 x 32768 and 95.0
// / 86.7 at 8 x 65536, and four 1024 x 1024 matrix products in the second stream
// take 28 / 26 and 45 / 30 us longer with a call beside them.
template <int kSh>
constexpr int smem_bytes(int spread) {
  const int used = (int)sizeof(ClusterSmem<kSh>), wide = spread == 2 ? 200 * 1024 : (spread == 1 ? 110 * 1024 : 0);
  return used > wide ? used : wide;
}

template <int kSh>
cudaError_t set_attrs(bool nonportable) {
  const int bytes = smem_bytes<kSh>(2);
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
cudaError_t launch_shape(const FinalArgs& f, int U, int C, int spread, bool select_only, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(U * C), 1, 1);
  cfg.blockDim = dim3(Shape<kSh>::kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes<kSh>(spread);
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
// Clusters of C CTAs of shapes 0-3 resident at once plus one, at [shape][spread][C - 1]; 0 = not asked yet.
std::atomic<int> g_fit[64][4][3][16];
std::atomic<int> g_sms[64];  // SMs, set before g_setup

// Clusters of C CTAs that the current device holds at once (the occupancy
// query's answer, asked once; a racing thread asks again).
template <int kSh>
int clusters_fit(int dev, int C, int spread) {
  int n = g_fit[dev][kSh][spread][C - 1].load();
  if (n > 0) return n - 1;
  n = 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)C * 1024u, 1, 1);
  cfg.blockDim = dim3(Shape<kSh>::kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes<kSh>(spread);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, (const void*)finalize_cluster_kernel<1, kSh, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();  // an unavailable configuration leaves no error behind
    n = 0;
  }
  g_fit[dev][kSh][spread][C - 1].store(n + 1);
  return n;
}

int clusters_fit(int dev, int sh, int C, int spread) {
  switch (sh) {
    case 0: return clusters_fit<0>(dev, C, spread);
    case 1: return clusters_fit<1>(dev, C, spread);
    case 2: return clusters_fit<2>(dev, C, spread);
  }
  return clusters_fit<3>(dev, C, spread);
}

int device_setup() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  int st = g_setup[dev].load();
  if (st != 0) return st;
  if (set_attrs<0>(false) != cudaSuccess || set_attrs<1>(false) != cudaSuccess || set_attrs<2>(false) != cudaSuccess ||
      set_attrs<3>(false) != cudaSuccess || set_attrs<5>(false) != cudaSuccess)
    return -1;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return -1;
  g_sms[dev].store(sms);
  const bool wide = set_attrs<0>(true) == cudaSuccess && set_attrs<3>(true) == cudaSuccess;
  st = wide && clusters_fit<3>(dev, 16, 0) > 0 ? 2 : 1;
  cudaGetLastError();  // an unavailable configuration leaves no error behind
  g_setup[dev].store(st);
  return st;
}

// Shape and cluster size for U units of Tv candidates; shape -1 when none takes
// them.  The fewest candidates a thread whose clusters are all resident at once
// (one layer of 4 heads x 32768 keys: 16 CTAs of 8 a thread 15 us, 4 of 32 a
// thread 25 us; 28 layers x 4 heads of that length: 3 waves of the former, one
// of the latter), and where they are at most one an SM in number, spread so
// (smem_bytes; two an SM asked of 224 CTAs, 28 x 4 heads of 14500 keys, cost 2
// us).  Failing that (many units) clusters of at most four: of 128-thread CTAs
// up to 8192 candidates, seven to an SM (32 x 32 heads of 2048 keys: 21 us against 27 in CTAs of 256 threads, 608 at once; 20 x 32 of 6000
// keys 42 against 53), else the fewest candidates a thread.  The 128-thread
// CTAs in clusters of more than four, resident at once, lost to 32 candidates a
// thread (28 x 4 heads of 16411 keys, nine CTAs each: 234 against 218 us a
// call).  What is resident is the occupancy query's answer: by the SM count
// alone, 112 clusters of four at three CTAs an SM would fit, but the SMs of a
// GPC hold whole clusters only (28 x 4 heads of 14500 keys: 202 us a call in
// two waves of those, 194 in one of 32 candidates a thread).
void pick_shape(int Tv, long long U, int dev, bool long_ok, int& sh, int& C, int& spread) {
  spread = 0;
  const int t = Tv > 0 ? Tv : 1;
  const int cap[4] = {Shape<0>::kCap, Shape<1>::kCap, Shape<2>::kCap, Shape<3>::kCap};
  const int most[4] = {long_ok ? Shape<0>::kMaxCluster : 8, Shape<1>::kMaxCluster, Shape<2>::kMaxCluster,
                       long_ok ? Shape<3>::kMaxCluster : 8};
  for (sh = 0; sh < 4; ++sh) {
    C = (t + cap[sh] - 1) / cap[sh];
    if (C <= most[sh] && U <= clusters_fit(dev, sh, C, 0)) {
      while (U * C <= g_sms[dev].load() && spread < 2 && U <= clusters_fit(dev, sh, C, spread + 1)) ++spread;
      return;
    }
  }
  sh = 5;
  C = (t + Shape<5>::kCap - 1) / Shape<5>::kCap;
  if (C <= Shape<5>::kMaxCluster) return;
  for (sh = 1; sh < 4; ++sh) {
    C = (t + cap[sh] - 1) / cap[sh];
    if (C <= most[sh]) return;
  }
  sh = -1;
  C = 0;
}

int current_device() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? dev : 0;
}

}  // namespace

bool cluster_finalize_fits(int Tv) {
  const int st = device_setup();
  if (st < 0) return false;
  int sh, C, spread;
  pick_shape(Tv, 1, current_device(), st == 2, sh, C, spread);
  return sh >= 0;
}

cudaError_t launch_finalize_cluster(const FinalArgs& f, int U, bool select_only, cudaStream_t s) {
  const int st = device_setup();
  if (st < 0) return cudaErrorUnknown;
  int sh, C, spread;
  pick_shape(f.Tv, U, current_device(), st == 2, sh, C, spread);
  switch (sh) {
    case 0: return launch_shape<0>(f, U, C, spread, select_only, s);
    case 1: return launch_shape<1>(f, U, C, spread, select_only, s);
    case 2: return launch_shape<2>(f, U, C, spread, select_only, s);
    case 3: return launch_shape<3>(f, U, C, spread, select_only, s);
    case 5: return launch_shape<5>(f, U, C, spread, select_only, s);
  }
  return cudaErrorNotSupported;
}

}  // namespace ecokv
