// Many steps of a small lattice in one launch: the populations live in the shared memory of one
// thread-block cluster (up to 16 blocks), and a cluster barrier takes the place of the launch
// boundary between steps.
//
// A small box is bound by the chain of a step, not by its work: launch by launch (pair_kernel, with
// dependent launches) D2Q9 64^2 takes 1.73 us a step on the GPU, of which the arithmetic of its one warp
// per scheduler is a third, and the host needs 1.64 us to enqueue one. Here a step is the reads and writes
// of distributed shared memory, the collision and one barrier, and the noise of the next step is
// formed between arriving at the barrier and waiting for it.
//
// Block r of the cluster holds the sites [r chunk, (r + 1) chunk) of every population,
// stage[q][site], and a thread one of them: where latency is what counts, half a pair's chain is
// better than half as many threads (D3Q27 16^3 1.97 against 3.1 us). From an even step count it reads
// and writes its own slots; from an odd one it reads slot opposite(i) of x - c_i and writes slot i of
// x + c_i, in whichever block holds them. The place that velocity i is written to is the one that
// opposite(i) is read from, so one table of addresses per thread, formed once, serves both. Within a
// step no two threads touch the same slot (the AA pattern), so one barrier per step suffices.
// The arithmetic is that of the pair kernels, bit for bit.
//
// Only 16 SMs work, so the rule (cluster_applies) ends where the whole GPU is faster.
#include <map>
#include <mutex>
#include <utility>

#include "step_kernels.cuh"

namespace flbm {
namespace {

constexpr int kClusterMax = 16;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of `local` (this block's shared memory) in the block of rank r.
__device__ __forceinline__ uint32_t cluster_address(uint32_t local, uint32_t r) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(r));
  return a;
}
__device__ __forceinline__ float cluster_load(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_store(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <int LAT, bool NOISE, int SCHEME, bool ISO>
__global__ void __launch_bounds__(512) cluster_kernel(const StepArgs a, uint32_t chunk, int nsteps) {
  constexpr int Q = Lat<LAT>::Q;
  extern __shared__ float stage[];  // [Q][chunk]
  const uint32_t first = cluster_rank() * chunk, own = threadIdx.x;
  float *f = static_cast<float *>(a.f);
  const uint32_t n_sites = (uint32_t)a.plane;
  const uint32_t mine = first >= n_sites ? 0u : (n_sites - first < chunk ? n_sites - first : chunk);
  const bool active = own < mine;
  wait_prerequisites();
  if (active) {
#pragma unroll
    for (int q = 0; q < Q; ++q) stage[q * chunk + own] = f[q * n_sites + first + own];
  }
  // Byte addresses of slot opposite(i) of x - c_i (a thread without a site computes site 0's and uses
  // none of them).
  uint32_t at[Q];
  const uint32_t base = shared_address(stage), site = active ? first + own : 0u;
  {
    const int x = (int)(site % (uint32_t)a.nx), y = (int)(site / (uint32_t)a.nx % (uint32_t)a.ny);
    const int z = (int)(site / ((uint32_t)a.nx * (uint32_t)a.ny));
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      int xx = x - Lat<LAT>::cx(i), yy = y - Lat<LAT>::cy(i), zz = z - Lat<LAT>::cz(i);
      xx = xx < 0 ? xx + a.nx : (xx >= a.nx ? xx - a.nx : xx);
      yy = yy < 0 ? yy + a.ny : (yy >= a.ny ? yy - a.ny : yy);
      zz = zz < 0 ? zz + a.nz : (zz >= a.nz ? zz - a.nz : zz);
      const uint32_t s = ((uint32_t)zz * (uint32_t)a.ny + (uint32_t)yy) * (uint32_t)a.nx + (uint32_t)xx;
      const uint32_t r = s / chunk;
      at[i] = cluster_address(base + 4u * ((uint32_t)opposite<LAT>(i) * chunk + (s - r * chunk)), r);
    }
  }

  unsigned long long step = (unsigned long long)a.step_lo | (unsigned long long)a.step_hi << 32;
  float n[Noisy<LAT>::count];
  const auto noise = [&]() {
    if (NOISE && active)
      site_noise<LAT, float, SCHEME, ISO, 0, Noisy<LAT>::blocks>(n, a, site, 0u, (uint32_t)step, (uint32_t)(step >> 32));
  };
  cluster_arrive();
  noise();
  for (int s = 0; s < nsteps; ++s) {
    cluster_wait();  // every block's writes of the step before
    if (active) {
      float F[LAT == 19 ? 19 : 27];
      auto &tile = reinterpret_cast<float(&)[3][3][3]>(F);
      const auto pop = [&](int i) -> float & {
        return LAT == 19 ? F[i] : tile[Lat<LAT>::cz(i) + 1][Lat<LAT>::cy(i) + 1][Lat<LAT>::cx(i) + 1];
      };
      const bool odd = step & 1u;
#pragma unroll
      for (int i = 0; i < Q; ++i) pop(i) = odd ? cluster_load(at[i]) : stage[i * chunk + own];
      if constexpr (LAT == 19)
        collide_site<LAT, NOISE, SCHEME, ISO>(F, a, n);
      else
        collide_site<LAT, NOISE, SCHEME, ISO>(tile, a, n);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        if (odd)
          cluster_store(at[opposite<LAT>(i)], pop(i));
        else
          stage[opposite<LAT>(i) * chunk + own] = pop(i);
      }
    }
    cluster_arrive();
    ++step;
    if (s + 1 < nsteps) noise();
  }
  cluster_wait();
  launch_dependents();
  if (active) {
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q * n_sites + first + own] = stage[q * chunk + own];
  }
}

template <int LAT, bool NOISE, int SCHEME, bool ISO>
cudaError_t launch(const StepArgs &a, int nsteps, cudaStream_t s) {
  auto kernel = cluster_kernel<LAT, NOISE, SCHEME, ISO>;
  // As many blocks as give each at least a warp of sites.
  int blocks = 1;
  while (blocks < kClusterMax && blocks * 32 < a.plane) blocks *= 2;
  const uint32_t chunk = uint32_t((a.plane + blocks - 1) / blocks);
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = unsigned(blocks);
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(blocks));
  cfg.blockDim = dim3((chunk + 31) / 32 * 32);
  cfg.dynamicSmemBytes = size_t(Lat<LAT>::Q) * chunk * sizeof(float);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  {
    // More than eight blocks need the kernel's permission, and a device (or a partition of one) may
    // have no group of SMs that holds them all: asked once per device and number of blocks.
    static std::mutex mu;
    static std::map<std::pair<int, int>, bool> fits;
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    const auto known = fits.find({dev, blocks});
    bool ok = known != fits.end() && known->second;
    if (known == fits.end()) {
      int clusters = 0;
      ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
           cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0;
      fits[{dev, blocks}] = ok;
    }
    if (!ok) return cudaErrorNotSupported;
  }
  return cudaLaunchKernelEx(&cfg, kernel, a, chunk, nsteps);
}

template <int LAT, int SCHEME, bool ISO>
cudaError_t launch_noise(bool noise, const StepArgs &a, int nsteps, cudaStream_t s) {
  return noise ? launch<LAT, true, SCHEME, ISO>(a, nsteps, s) : launch<LAT, false, SCHEME, ISO>(a, nsteps, s);
}

}  // namespace

// Up to 512 threads a block in 2-D, 256 in 3-D (27 populations of 256 sites: 27 KB of shared memory).
// us per step over 100 steps, cluster against pair kernel: D2Q9 64^2 0.86 / 1.84, 90^2 1.26 / 1.88; D3Q27
// 8^3 1.35 / 2.75, 16^3 1.99 / 2.92, 18^3 2.92 / 3.03; D3Q19 16^3 1.49 / 2.40. Setting up the cluster takes
// some 10 us: over 6 steps D2Q9 90^2 2.7 / 2.8, D3Q27 16^3 3.9 / 3.8, over 10 steps 2.1 / 2.5 and 3.0 / 3.5.
bool cluster_applies(int lattice, int storage, long long sites, long long nsteps) {
  return storage == 0 && sites <= (lattice == 0 ? 8192 : 4096) && nsteps >= (lattice == 0 ? 6 : 10);
}

cudaError_t launch_step_cluster(int lattice, bool raw, bool noise, bool shear, const StepArgs &a, int nsteps,
                                cudaStream_t s) {
  if (raw) return lattice == 0 ? launch_noise<2, kRaw, false>(noise, a, nsteps, s) : launch_noise<3, kRaw, false>(noise, a, nsteps, s);
  if (lattice == 0)
    return shear ? launch_noise<2, kShear, false>(noise, a, nsteps, s) : launch_noise<2, kGeneral, false>(noise, a, nsteps, s);
  if (lattice == 1)
    return shear ? launch_noise<3, kShear, false>(noise, a, nsteps, s) : launch_noise<3, kGeneral, false>(noise, a, nsteps, s);
  if (lattice == 2)
    return shear ? launch_noise<3, kShear, true>(noise, a, nsteps, s) : launch_noise<3, kGeneral, true>(noise, a, nsteps, s);
  return shear ? launch_noise<19, kShear, false>(noise, a, nsteps, s) : launch_noise<19, kGeneral, false>(noise, a, nsteps, s);
}

}  // namespace flbm
