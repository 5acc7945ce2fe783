// Batched ensembles: many independent periodic lattices (mixed D2Q9 / D3Q27, own size,
// rates, kBT and noise seed) advanced together, each by exactly the fused update of a
// single context (the collision of collide.cuh, packed FP32x2, the AA pattern of step.cu)
// with its own parameters.
//
// The host lays every lattice's populations out in one allocation and cuts all lattices
// into tiles of equal pair-slot count (one slot of two sites per thread, pair.cuh; a
// tile may span rows, never lattices). Two launch structures (BatchForm):
//
// Per-step forms (the default): per step one plain launch per lattice type, block b on
// tile tile0 + b, the hardware block scheduler balancing the load; the n launches of a
// call are captured once into a CUDA graph and replayed. The kernel is the single lattice's
// (pair_kernel, step_kernels.cuh): reads staged by cp.async while the noise is formed, the next
// launch's blocks starting as this one drains. It is bound like it by the FMA pipe; what a batch
// adds is the addressing (a lattice's array and plane are not kernel arguments of their own).
// us per step, before -> now, in the shape the autotuner picks: 32 D3Q27 64^3 321 -> 277, one
// 256^3 634 -> 564, 233 of 33^3 368 -> 338, 512 of 16^3 86 -> 72, 256 D2Q9 256^2 201 -> 185, 256 of
// 255^2 228 -> 210; 256 mixed lattices (10.7 M sites) 392 -> 355.
//
// Persistent form: one cooperative launch runs n steps; block b takes the work items
// (step s, tile b + j G) in step-major order. There is no grid-wide barrier between
// steps. Lattices are independent, so a tile of lattice L at step s only has to wait
// until every tile of L has finished step s - 1 (in-place AA streaming reads and writes
// neighbour slots across tile boundaries). Each lattice has a completion counter; a block
// announces a finished tile with a release (fence, then atomic add) and checks the
// counter of the next tile's lattice with an acquire before starting it. Progress is
// guaranteed: all blocks are resident (cooperative launch), each walks its items in
// order, and the lowest pending item only depends on items of the step before it, which
// are all complete. Every wait is bounded: a block that polls longer than wait_polls times
// (or sees another block's failure) sets the status word and leaves; the host reports
// FLBM_ETIMEOUT.
//
// The per-lattice parameters travel by value in the kernel arguments (constant bank; at
// most kBatchMaxLattices lattices). A tile's lattice is found by a binary search over the
// lattices' first-tile indices in that table, from the block's own counters only, so the
// lattice's parameters stay block-uniform values (uniform registers) instead of occupying
// every thread's registers. All lattices share the step counter in device memory, read
// by every launch, so that one captured graph serves every call with the same n (and,
// for the per-step forms, the same starting parity).
#include <cuda_runtime.h>

#include "collide.cuh"
#include "internal.h"
#include "pair.cuh"

namespace flbm {
namespace {


// The pair slots of lattice L (pair.cuh): rows of ceil(nx / 2) slots, numbered row-major, so a
// tile spans rows and a warp's accesses stay contiguous for every nx. From an even step count
// slot k is the flat sites 2k and 2k + 1 instead, and the last slots of odd rows stay empty.
__device__ __forceinline__ uint32_t pair_slots(const BatchLattice &L) {
  return (((uint32_t)L.nx + 1u) >> 1) * (uint32_t)L.ny * (uint32_t)L.nz;
}
template <int PARITY>
__device__ __forceinline__ bool pairs_aligned(const BatchLattice &L) {
  return PARITY == 0 ? (L.plane & 1u) == 0u : (L.nx & 1) == 0;
}

// The pair of slot `slot` of lattice L.
template <int D, int PARITY, bool ALIGNED, bool STAGE, typename O, int THREADS, typename Base>
__device__ __forceinline__ auto pair_of(const BatchLattice &L, const Base &planes, uint32_t slot) {
  PairAccess<D, float, PARITY, ALIGNED, false, O, STAGE, THREADS, Base> p;
  if (PARITY == 0) {
    p.init_flat(planes, 0u, L.plane, slot);
  } else {
    int x0, y, z;
    slot_xyz<!ALIGNED && sizeof(O) == 8>(slot, L.nx, L.ny, L.m_hp, L.p_hp(), L.m_ny, L.p_ny(), x0, y, z);
    p.init_row(planes, x0, y, z, L.nx, L.ny, L.nz);
  }
  return p;
}

// The noise and the collision with lattice L's parameters: its three shear-structure numbers
// (SHEAR) or its per-mode arrays; round keys are formed from its key.
template <int D, bool SHEAR, int B0, int B1>
__device__ __forceinline__ void lattice_noise(float2 (&n)[Noisy<D>::count], const BatchLattice &L, const float *rates,
                                              uint32_t s0, uint32_t dsite, unsigned long long step) {
  const KeyBase keys{L.key0, L.key1};
  const uint32_t lo = (uint32_t)step, hi = (uint32_t)(step >> 32);
  if (SHEAR)
    noise_modes<D, float, true, false, B0, B1>(n, ShearRates<D>{L.sqrt_kbt, L.om_shear, L.amp_shear}, s0, lo, hi, keys, dsite);
  else
    noise_modes<D, float, false, false, B0, B1>(n, ArrayRates{rates, rates + 27, nullptr, 0.0f}, s0, lo, hi, keys, dsite);
}
template <int D, bool SHEAR>
__device__ __forceinline__ void lattice_collide(float2 (&F)[3][3][3], const BatchLattice &L, const float *rates,
                                                const float2 (&n)[Noisy<D>::count]) {
  if (SHEAR)
    collide_rates<D, true, float2, true>(F, L.rho0, ShearRates<D>{L.sqrt_kbt, L.om_shear, L.amp_shear}, n);
  else
    collide_rates<D, true, float2, false>(F, L.rho0, ArrayRates{rates, rates + 27, nullptr, 0.0f}, n);
}

// One pair of lattice L in a per-step launch: as pair_kernel (step_kernels.cuh), `early` likewise.
// Only the reads and writes are compiled for both alignments; `stage` (STAGE) holds the pair in
// the same layout for both.
template <int D, int PARITY, bool SHEAR, typename O, bool STAGE, int THREADS, typename Base>
__device__ __forceinline__ void batch_pair(const BatchLattice &L, const Base &planes, const float *rates, uint32_t slot,
                                           unsigned long long step, bool early, float2 *stage) {
  const bool aligned = pairs_aligned<PARITY>(L);
  if (PARITY == 0 && 2ull * slot >= L.plane) return;
  constexpr int B = Noisy<D>::blocks;
  float2 n[Noisy<D>::count], F[3][3][3];
  uint32_t s0, dsite;
  const auto begin = [&](bool read) {
    if (read) wait_prerequisites();
    if (aligned) {
      const auto p = pair_of<D, PARITY, true, STAGE, O, THREADS>(L, planes, slot);
      s0 = p.site0;
      dsite = p.dsite;
      if (read && STAGE) p.fetch(shared_address(stage));
    } else {
      const auto p = pair_of<D, PARITY, false, STAGE, O, THREADS>(L, planes, slot);
      s0 = p.site0;
      dsite = p.dsite;
      if (read && STAGE) p.fetch(shared_address(stage));
    }
  };
  begin(early);
  lattice_noise<D, SHEAR, 0, B>(n, L, rates, s0, dsite, step);
  if (!early) begin(true);
  if (STAGE) cp_async_wait_all();
  if (STAGE || aligned)
    pair_of<D, PARITY, true, STAGE, O, THREADS>(L, planes, slot).load_tile(stage, F);
  else
    pair_of<D, PARITY, false, STAGE, O, THREADS>(L, planes, slot).load_tile(stage, F);
  lattice_collide<D, SHEAR>(F, L, rates, n);
  // The slot is hidden so that the stores' addresses are formed anew instead of staying in
  // registers across the collision.
  uint32_t sl = slot;
  asm volatile("" : "+r"(sl));
  if (aligned)
    pair_of<D, PARITY, true, STAGE, O, THREADS>(L, planes, sl).store_tile(F);
  else
    pair_of<D, PARITY, false, STAGE, O, THREADS>(L, planes, sl).store_tile(F);
}

// Pair slot first + threadIdx.x of tile [first, end) of lattice L (persistent form).
template <int PARITY, bool SHEAR>
__device__ __forceinline__ void batch_tile(const BatchLattice &L, char *pool, const float *rates, uint32_t first,
                                           uint32_t end, unsigned long long step) {
  const uint32_t slot = first + threadIdx.x;
  if (slot >= end) return;
  const PlaneStride planes{pool + 256ull * L.f256, 4ull * L.plane};
  if (L.D() == 3)
    batch_pair<3, PARITY, SHEAR, uint64_t, false, 1>(L, planes, rates, slot, step, true, nullptr);
  else
    batch_pair<2, PARITY, SHEAR, uint64_t, false, 1>(L, planes, rates, slot, step, true, nullptr);
}

// Thread 0: waits until lattice `lat` has finished `target` tiles in this launch.
__device__ __forceinline__ bool wait_done(const int *done, int target, int *status, uint32_t polls) {
  const volatile int *d = done;
  for (uint32_t it = 0; it < polls; ++it) {
    if (*d >= target) return true;
    if (*(volatile int *)status != 0) return false;
    __nanosleep(32);
  }
  atomicCAS(status, 0, 2);
  return false;
}

// Lattice of tile t among table entries [lo, hi): the last whose first tile is <= t
// (binary search over the kernel-argument table). Everything here derives from kernel
// arguments and the block's own counters, so the lattice's parameters stay block-uniform
// values rather than occupying every thread's registers.
__device__ __forceinline__ int lattice_of(const BatchArgs &a, int t, int lo, int hi) {
  --hi;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.lats[mid].tile0 <= t)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ int tiles_of(const BatchArgs &a, int lat) {
  return (lat + 1 < a.nlat ? a.lats[lat + 1].tile0 : a.ntiles) - a.lats[lat].tile0;
}

template <bool SHEAR>
__global__ void __launch_bounds__(kBatchMaxThreads, 2) batch_kernel(const BatchArgs a) {
  __shared__ int s_ok;
  const long long step0 = *a.step_counter;
  int s = 0, t = blockIdx.x;
  while (s < a.nsteps && t < a.ntiles) {
    const int lat = lattice_of(a, t, 0, a.nlat);
    const BatchLattice &L = a.lats[lat];
    if (threadIdx.x == 0) {
      int ok = 1;
      if (s > 0) ok = wait_done(&a.done[lat], s * tiles_of(a, lat) + a.target_bias, a.status, a.wait_polls);
      __threadfence();  // acquire: the lattice's step s - 1 writes are visible
      s_ok = ok;
    }
    __syncthreads();
    if (!s_ok) break;
    const uint32_t per = (uint32_t)a.tile_slots[L.D() == 3 ? 1 : 0];
    const uint32_t first = (uint32_t)(t - L.tile0) * per;
    const uint32_t slots = pair_slots(L);
    const uint32_t end = first + per < slots ? first + per : slots;
    const unsigned long long step = (unsigned long long)(step0 + s);
    if (step & 1)
      batch_tile<1, SHEAR>(L, a.pool, a.rates + 54 * lat, first, end, step);
    else
      batch_tile<0, SHEAR>(L, a.pool, a.rates + 54 * lat, first, end, step);
    __syncthreads();  // every thread's writes of this tile are issued
    if (threadIdx.x == 0) {
      __threadfence();  // release
      atomicAdd(&a.done[lat], 1);
    }
    t += gridDim.x;
    if (t >= a.ntiles) {
      t = blockIdx.x;
      ++s;
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(a.exits, 1u) == gridDim.x - 1 && *(volatile int *)a.status == 0)
      *a.step_counter = step0 + a.nsteps;
  }
}

// One step of the lattices of one type D, table entries [lat_lo, lat_hi), whose tiles
// are tile_base, tile_base + 1, ...: block b takes tile tile_base + b (a plain launch;
// the hardware block scheduler balances the load). One kernel per lattice type keeps
// the D2Q9 blocks at the register count (and occupancy) of D2Q9 alone. The step number
// is read from the device counter plus `k`, so that a captured graph of n such launches
// serves every call with the same n and the same starting parity; PARITY is fixed per
// launch. Every launch of a call but its first starts while the one before it drains
// (programmatic dependent launch); the counter is only written after a call's last launch has
// ended and before the next call's first one starts, so it may be read before the wait.
// THREADS: 64 or 128, reads staged in shared memory, or 256, reads direct (two blocks of 256
// stages would not fit beside each other).
template <int D, bool SHEAR, int PARITY, typename O, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB)
    batch_step_kernel(const __grid_constant__ BatchArgs a, int k, int lat_lo, int lat_hi, int tile_base, bool early) {
  constexpr bool STAGE = THREADS < 256;
  __shared__ float2 stage[STAGE ? Lat<D>::Q * THREADS : 1];
  launch_dependents();
  const int t = tile_base + (int)blockIdx.x;
  const int lat = lattice_of(a, t, lat_lo, lat_hi);
  const BatchLattice &L = a.lats[lat];
  const uint32_t per = (uint32_t)a.tile_slots[D == 3 ? 1 : 0];
  const uint32_t first = (uint32_t)(t - L.tile0) * per;
  const uint32_t slots = pair_slots(L);
  const uint32_t end = first + per < slots ? first + per : slots;
  const uint32_t slot = first + threadIdx.x;
  if (slot >= end) return;
  const unsigned long long step = (unsigned long long)(*(volatile const long long *)a.step_counter + k);
  batch_pair<D, PARITY, SHEAR, O, STAGE, THREADS>(L, PlaneStride{a.pool + 256ull * L.f256, 4ull * L.plane}, a.rates + 54 * lat,
                                                  slot, step, early, stage + threadIdx.x);
}

// Advances the shared step counter after the n step launches of one call.
__global__ void batch_advance_kernel(long long *step_counter, int n) { *step_counter += n; }

}  // namespace

cudaError_t batch_max_blocks(bool shear, int threads, int *blocks_per_sm) {
  return shear ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, batch_kernel<true>, threads, 0)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, batch_kernel<false>, threads, 0);
}

// Launch shapes of the per-step form (BatchForm): blocks of 128 threads per SM (as many threads in
// other block sizes) that the kernel is compiled for, i.e. its register cap.
template <int D>
constexpr int batch_blocks(bool occ) {
  return D == 2 ? (occ ? 10 : 8) : (occ ? 5 : 4);
}

template <int D, bool SHEAR, int PARITY, typename O>
cudaError_t launch_group(int form, const BatchArgs &a, int k, const BatchGroup &g, int threads, bool dependent,
                         cudaStream_t s) {
  if (g.ntiles <= 0) return cudaSuccess;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(g.ntiles);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = dependent ? 1 : 0;
  const bool early = (uint64_t)g.ntiles * (uint64_t)threads > kEarlySlots;
  constexpr int B0 = batch_blocks<D>(false), B1 = batch_blocks<D>(true);
  const auto launch = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, a, k, g.lat_lo, g.lat_hi, g.tile0, early);
  };
  if (threads == 256) return launch(batch_step_kernel<D, SHEAR, PARITY, O, 256, D == 2 ? 4 : 2>);
  if (threads == 64)
    return form == kBatchStepOcc ? launch(batch_step_kernel<D, SHEAR, PARITY, O, 64, 2 * B1>)
                                 : launch(batch_step_kernel<D, SHEAR, PARITY, O, 64, 2 * B0>);
  return form == kBatchStepOcc ? launch(batch_step_kernel<D, SHEAR, PARITY, O, 128, B1>)
                               : launch(batch_step_kernel<D, SHEAR, PARITY, O, 128, B0>);
}

template <int D, bool SHEAR>
cudaError_t launch_group_parity(int form, int parity, const BatchArgs &a, int k, const BatchGroup &g, int threads,
                                bool dependent, cudaStream_t s) {
  if (g.wide)
    return parity ? launch_group<D, SHEAR, 1, uint64_t>(form, a, k, g, threads, dependent, s)
                  : launch_group<D, SHEAR, 0, uint64_t>(form, a, k, g, threads, dependent, s);
  return parity ? launch_group<D, SHEAR, 1, uint32_t>(form, a, k, g, threads, dependent, s)
                : launch_group<D, SHEAR, 0, uint32_t>(form, a, k, g, threads, dependent, s);
}

template <int D>
cudaError_t launch_group_any(int form, bool shear, int parity, const BatchArgs &a, int k, const BatchGroup &g,
                             int threads, bool dependent, cudaStream_t s) {
  return shear ? launch_group_parity<D, true>(form, parity, a, k, g, threads, dependent, s)
               : launch_group_parity<D, false>(form, parity, a, k, g, threads, dependent, s);
}

cudaError_t launch_batch_steps(int form3, int threads3, int form2, int threads2, bool shear, int parity0,
                               const BatchArgs &a, const BatchGroup &g3, const BatchGroup &g2, int n,
                               cudaStream_t s) {
  for (int k = 0; k < n; ++k) {
    const int parity = (parity0 + k) & 1;
    cudaError_t e = launch_group_any<3>(form3, shear, parity, a, k, g3, threads3, k > 0, s);
    if (e == cudaSuccess)
      e = launch_group_any<2>(form2, shear, parity, a, k, g2, threads2, k > 0 || g3.ntiles > 0, s);
    if (e != cudaSuccess) return e;
  }
  batch_advance_kernel<<<1, 1, 0, s>>>(a.step_counter, n);
  return cudaGetLastError();
}

cudaError_t launch_batch(bool shear, const BatchArgs &a, int grid, int threads, cudaStream_t s) {
  void *args[] = {const_cast<BatchArgs *>(&a)};
  const void *fn = shear ? (const void *)batch_kernel<true> : (const void *)batch_kernel<false>;
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, 0, s);
}

}  // namespace flbm
