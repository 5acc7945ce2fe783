// Statistics reduction over one lattice state: the diagnostics of Sec. III (spatial
// means <u_a>, <u_a u_b> for the equipartition tests, Eq. for <u_a^2> = kBT/rho0) and
// the central-moment means and covariances whose equilibrium form is C^eq (Sec. II-B,
// "Structural properties"), plus mass and momentum for the conservation checks.
//
// Every one of these sums is an entry of the Gram matrix G of the per-site columns
// (gram.cuh: staging layout, BF16 hi/lo products on the tcgen05 tensor cores with a TMEM
// accumulator, output record; k_0 = rho and the central moments k_1..k_D, which vanish
// identically, are rebuilt or set to zero by the host, api.cu). Persistent blocks of
// kStatsBlock threads walk tiles of kStatsBlock site pairs, the flat pairs of the step kernels
// (pair.cuh): each thread computes the columns of two sites with the packed FP32x2 algebra of
// the step (cm.cuh) and writes their BF16 hi/lo words into its warp's operand rows; one thread
// per block multiplies the tile.
// What bounds it: three warps per scheduler (168 registers with the next pair's populations in
// flight) on long chains of packed operations and conversions, 50 % of issue slots, DRAM half busy;
// on small lattices the chain of set-up, one tile, accumulator read and block sums.
// us per sample, before -> now: D3Q27 256^3 421 -> 369 (even step count), 433 -> 406 (odd), 255^3 568 ->
// 422 / 454, 64^3 21.9 -> 20.0; D3Q19 256^3 410 -> 360; D2Q9 4096^2 165 -> 143, 64^2 9.0 -> 6.6. The
// planes' addresses as kernel arguments and one division per pair gave the large ones, no clearing
// launch and the set-up before the wait the small ones.
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <utility>

#include "cm.cuh"
#include "d3q19.cuh"
#include "gram.cuh"
#include "internal.h"
#include "pair.cuh"

namespace flbm {

int stats_nacc(int Q) { return Q == 9 ? StatsPlan<2>::NREC : StatsPlan<3>::NREC; }

namespace {

// The populations of a thread's site pair, as loaded for one tile and consumed by the
// next: F19 for D3Q19 (lattice code 19), the 3x3x3 tile otherwise.
template <int D>
struct PairPops {
  float2 F[3][3][3];
  bool v0, v1;  // the lanes' sites exist
};
template <>
struct PairPops<19> {
  float2 F[19];
  bool v0, v1;
};

// Loads the pair of slot k (the slots of the step kernels, pair.cuh, of the sites the statistics
// cover); zeros for a lane without a site of its own.
template <int LAT, typename S, int PARITY, bool ALIGNED>
__device__ __forceinline__ void load_pair(const StepArgs &a, uint32_t k, PairPops<LAT> &P) {
  constexpr int NP = LAT == 2 ? 27 : Lat<LAT>::Q;  // D2Q9 uses the middle plane of its tile
  float2 *F = reinterpret_cast<float2 *>(&P.F);
  P.v0 = k < a.slots[PARITY];
  P.v1 = false;
  if (P.v0) {
    PairAccess<LAT, S, PARITY, ALIGNED, false, uint64_t, false, 1> p;
    if (PARITY == 0) {
      p.init_flat(PlaneTable{a.pop}, a.first, a.count, k);
    } else {
      int x0, y, z;
      slot_xyz<!ALIGNED>(k, a.nx, a.ny, a.m_hp, a.p_hp, a.m_ny, a.p_ny, x0, y, z);
      p.init_row(PlaneTable{a.pop}, x0, y, z + a.z_lo, a.nx, a.ny, a.nz);
    }
    if constexpr (LAT == 19)
      p.load_list(nullptr, P.F);
    else
      p.load_tile(nullptr, P.F);
    P.v1 = p.two;
    if (!ALIGNED && !p.two) {
#pragma unroll
      for (int q = 0; q < NP; ++q) F[q].y = 0.0f;
    }
  } else {
#pragma unroll
    for (int q = 0; q < NP; ++q) F[q] = make_float2(0.0f, 0.0f);
  }
}

// The columns of the pair from its populations. D3Q19: [1, rho - rho0, j, u, k_4 .. k_18,
// 0 ...] (d3q19.cuh); D2Q9 / D3Q27: gram::moment_columns.
template <int D, bool ISO>
__device__ __forceinline__ void pair_columns(PairPops<D> &P, float rho0, bool v0, bool v1,
                                             float2 (&col)[StatsPlan<D>::NC], unsigned &nonfinite) {
  if constexpr (D == 19) {
    const D3Q19Raw<float2> r(P.F);
    const float2 rho = vadd(splat<float2>(rho0), r.drho), inv_rho = rcp_fast_lanes(rho);
    float2 u[3], k[15];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      u[a] = vmul(r.j[a], inv_rho);
      col[2 + a] = vmul(rho, u[a]);
      col[5 + a] = u[a];
    }
    d3q19_central(r, rho, u, k);
    col[0] = make_float2(v0 ? 1.0f : 0.0f, v1 ? 1.0f : 0.0f);
    col[1] = r.drho;
#pragma unroll
    for (int v = 4; v < 19; ++v) col[8 + v - 4] = k[v - 4];
#pragma unroll
    for (int c = 8 + 15; c < StatsPlan<D>::NC; ++c) col[c] = make_float2(0.0f, 0.0f);
    float2 sum = col[1];
#pragma unroll
    for (int c = 2; c < 8 + 15; ++c) sum = vadd(sum, col[c]);
    const bool valid[2] = {v0, v1};
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      if (valid[l] && !isfinite(lane(sum, l))) {
        ++nonfinite;
#pragma unroll
        for (int c = 0; c < 8 + 15; ++c) set_lane(col[c], l, 0.0f);
      }
    }
  } else {
    float2 drho, rho, ux, uy, uz;
    site_central_moments<D>(P.F, rho0, drho, rho, ux, uy, uz);
    gram::moment_columns<D, ISO>(P.F, drho, rho, ux, uy, uz, v0, v1, col, nonfinite);
  }
}

// One block walks tiles of kStatsBlock pairs: every thread transforms its site pair
// (loaded during the previous tile) and stages the split columns; each warp then arrives
// once on the pipeline's "staged" mbarrier and thread 0 multiplies the tile (gram.cuh,
// Pipeline). Before a thread overwrites the staging rows it waits for the MMAs that read
// them (one phase of each mbarrier per tile; every wait bounded), so the loads and
// arithmetic of the next tile proceed while the tensor cores work.
// The set-up (TMEM, barriers, tables) runs before the wait for the launch before this one
// (programmatic dependent launch). The blocks' sums meet in `work`, which is zero between
// launches: the last block to finish moves them to the record `out` and clears them, so that a
// sample is one launch with no clearing before it. Without `work` they are added to `out`, cleared
// by the caller.
template <int LAT, typename S, int PARITY, bool ALIGNED, bool ISO>
__global__ void __launch_bounds__(kStatsBlock, gram::blocks_per_sm<LAT>())
    stats_kernel(const StepArgs a, uint32_t tiles, double *work, unsigned int *ticket, double *out) {
  constexpr int NC = StatsPlan<LAT>::NC;
  extern __shared__ unsigned char smem_raw[];
  __shared__ unsigned int flags[2];  // non-finite count of the block, failure flag
  gram::Pipeline<LAT> pl;
  pl.init(smem_raw, flags);
  wait_prerequisites();

  unsigned nonfinite = 0u;
  // Software pipelining: the populations of the thread's pair in the next tile are loaded
  // as soon as the current ones are consumed, so the loads are in flight while the thread
  // splits and stages its columns and waits for the tensor cores.
  PairPops<LAT> pp;
  load_pair<LAT, S, PARITY, ALIGNED>(a, blockIdx.x * (uint32_t)kStatsBlock + threadIdx.x, pp);
  for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    float2 col[NC];
    pair_columns<LAT, ISO>(pp, a.rho0, pp.v0, pp.v1, col, nonfinite);
    if (t + gridDim.x < tiles)
      load_pair<LAT, S, PARITY, ALIGNED>(a, (t + gridDim.x) * (uint32_t)kStatsBlock + threadIdx.x, pp);
    pl.tile(col);
  }
  // Only now: blocks of the next step that wait beside a long reduction take its L1 cache
  // (256^3 sample between steps 0.52 against 0.39 ms).
  launch_dependents();
  pl.end(nonfinite, flags, work ? work : out);
  if (work == nullptr) return;
  __threadfence();  // this block's sums before its ticket
  __syncthreads();
  if (threadIdx.x == 0) flags[0] = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
  __syncthreads();
  if (flags[0] == 0u) return;
  __threadfence();
  for (int e = threadIdx.x; e <= StatsPlan<LAT>::NREC; e += kStatsBlock) {
    out[e] = __ldcg(work + e);
    work[e] = 0.0;
  }
  if (threadIdx.x == 0) *ticket = 0u;
}

template <int D, typename S>
size_t stats_smem() {
  return gram::Plan<D>::SMEM;
}

// Persistent grid: `per_sm` blocks per SM, the residency the kernel is built for (its
// launch bounds, 52 KB of shared memory and 128 of the SM's 512 TMEM columns per block),
// at most one block per tile. The attribute that allows more than 48 KB of dynamic shared
// memory is set once per kernel and device.
template <typename K>
cudaError_t stats_grid(K kernel, size_t smem, long long tiles, int per_sm, int *grid) {
  static std::mutex mu;
  static std::map<std::pair<int, const void *>, bool> ready;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lock(mu);
    bool &done = ready[std::make_pair(dev, (const void *)kernel)];
    if (!done) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      done = true;
    }
  }
  const long long cap = (long long)(sms > 0 ? sms : 1) * per_sm;
  *grid = (int)(tiles < cap ? tiles : cap);
  return cudaSuccess;
}

template <int LAT, typename S, int PARITY, bool ALIGNED, bool ISO>
cudaError_t launch_one(const StepArgs &a, double *work, unsigned int *ticket, double *out, cudaStream_t s) {
  auto kernel = stats_kernel<LAT, S, PARITY, ALIGNED, ISO>;
  const size_t smem = stats_smem<LAT, S>();
  const uint32_t tiles = (uint32_t)(((uint64_t)a.slots[PARITY] + kStatsBlock - 1) / kStatsBlock);
  if (tiles == 0) return cudaSuccess;
  int grid = 0;
  const cudaError_t e = stats_grid(kernel, smem, tiles, gram::blocks_per_sm<LAT>(), &grid);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kStatsBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  // Blocks that arrive beside a draining step find the SM's memory split as that kernel left it and
  // may not all fit; where each block has many tiles that costs more than the early start gives
  // (D3Q27 256^3, 144 tiles a block, sample between steps 0.48 against 0.39 ms; 128^3, 18 tiles,
  // 61.8 against 61.4 us; 64^3, 2 tiles, 20.1 against 21.4).
  cfg.numAttrs = tiles > 8u * (uint32_t)grid ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, a, tiles, work, ticket, out);
}

template <int LAT, typename S, bool ISO>
cudaError_t launch_typed(int parity, const StepArgs &a, double *work, unsigned int *ticket, double *out, cudaStream_t s) {
  if (parity == 0)
    return a.aligned[0] ? launch_one<LAT, S, 0, true, ISO>(a, work, ticket, out, s)
                        : launch_one<LAT, S, 0, false, ISO>(a, work, ticket, out, s);
  return a.aligned[1] ? launch_one<LAT, S, 1, true, ISO>(a, work, ticket, out, s)
                      : launch_one<LAT, S, 1, false, ISO>(a, work, ticket, out, s);
}

template <int LAT, bool ISO>
cudaError_t launch_storage(int storage, int parity, const StepArgs &a, double *work, unsigned int *ticket, double *out,
                           cudaStream_t s) {
  if (storage == 0) return launch_typed<LAT, float, ISO>(parity, a, work, ticket, out, s);
  if (storage == 1) return launch_typed<LAT, __nv_bfloat16, ISO>(parity, a, work, ticket, out, s);
  return launch_typed<LAT, __half, ISO>(parity, a, work, ticket, out, s);
}

}  // namespace

cudaError_t launch_stats(int D, int storage, bool iso, int parity, const StepArgs &a, double *work,
                         unsigned int *ticket, double *out, cudaStream_t s) {
  if (D == 19) return launch_storage<19, false>(storage, parity, a, work, ticket, out, s);
  if (D == 2) return launch_storage<2, false>(storage, parity, a, work, ticket, out, s);
  return iso ? launch_storage<3, true>(storage, parity, a, work, ticket, out, s)
             : launch_storage<3, false>(storage, parity, a, work, ticket, out, s);
}

}  // namespace flbm
