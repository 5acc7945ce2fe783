// Kernel templates of the fused step (documented in step.cu), shared by the translation
// units that instantiate them: step.cu (FP32 storage and the dispatch), step_16.cu
// (BF16 and FP16 storage), step_iso.cu (the isotropic D3Q27 variant), step19.cu (D3Q19) and
// step_raw.cu (the raw-moment collision).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "collide.cuh"
#include "d3q19.cuh"
#include "internal.h"
#include "pair.cuh"

namespace flbm {
namespace {

// The collision a kernel is compiled for.
enum Scheme { kGeneral = 0, kShear = 1, kRaw = 2 };

template <int LAT>
__device__ __forceinline__ ArrayRates rates_of(const StepArgs &a) {
  return LAT == 19 ? ArrayRates{a.om, a.phc, a.amp, a.sqrt_kbt} : ArrayRates{a.om_t, a.phc_t, a.amp, a.sqrt_kbt};
}
template <int LAT, typename S, int SCHEME, bool ISO, int B0, int B1, typename T>
__device__ __forceinline__ void site_noise(T (&n)[Noisy<LAT>::count], const StepArgs &a, uint32_t site, uint32_t dsite,
                                           uint32_t step_lo, uint32_t step_hi) {
  noise_modes<LAT, S, SCHEME == kShear, ISO, B0, B1>(n, rates_of<LAT>(a), site + a.site_base, step_lo, step_hi,
                                                  KeyTable{a.ks0, a.ks1}, dsite);
}
template <int LAT, bool NOISE, int SCHEME, bool ISO, typename T, typename F>
__device__ __forceinline__ void collide_site(F &pops, const StepArgs &a, const T (&n)[Noisy<LAT>::count]) {
  if constexpr (LAT == 19)
    collide19<NOISE, T, SCHEME == kShear>(pops, a.rho0, rates_of<LAT>(a), n);
  else if constexpr (SCHEME == kRaw)
    collide_raw<LAT, NOISE, T>(pops, a.rho0, rates_of<LAT>(a), n);
  else
    collide_rates<LAT, NOISE, T, SCHEME == kShear, ISO>(pops, a.rho0, rates_of<LAT>(a), n);
}

template <int LAT, typename S, int PARITY, bool NOISE, int SCHEME, bool ISO>
__global__ void __launch_bounds__(kStepBlock) step_kernel(const StepArgs a) {
  const int x = blockIdx.x * kStepBlock + threadIdx.x;
  if (x >= a.nx) return;
  const int y = blockIdx.y, z = blockIdx.z + a.z_lo;
  const Neighbourhood nb = neighbourhood(x, y, z, a.nx, a.ny, a.nz);
  S *__restrict__ f = static_cast<S *>(a.f);
  const uint32_t site = (uint32_t)(x + (long long)a.nx * (y + (long long)a.ny * z));
  float n[Noisy<LAT>::count];
  if (NOISE) site_noise<LAT, S, SCHEME, ISO, 0, Noisy<LAT>::blocks>(n, a, site, 0u, a.step_lo, a.step_hi);
  if constexpr (LAT == 19) {
    float F[19];
    load19<S, PARITY>(f, a.plane, nb, F);
    collide_site<LAT, NOISE, SCHEME, ISO>(F, a, n);
    store19<S, PARITY>(f, a.plane, nb, F);
  } else {
    float F[3][3][3];
    load_logical<LAT, S, PARITY>(f, a.plane, nb, F);
    collide_site<LAT, NOISE, SCHEME, ISO>(F, a, n);
    store_streamed<LAT, S, PARITY>(f, a.plane, nb, F);
  }
}

template <int LAT, typename S, int PARITY, bool NOISE, int SCHEME, bool ISO, bool ALIGNED, bool ROWS, typename O, int MINB>
__global__ void __launch_bounds__(kStepBlock, MINB) pair_kernel(const StepArgs a) {
  using Access = PairAccess<LAT, S, PARITY, ALIGNED, ROWS, O, NOISE, kStepBlock>;
  __shared__ typename Access::Word stage[Access::STAGED ? Access::WORDS * kStepBlock : 1];
  launch_dependents();
  Access p;
  if (ROWS) {
    int x0;
    if (!row_slot(blockIdx.x * (uint32_t)kStepBlock + threadIdx.x, a.nx, x0)) return;
    p.init_row(PlaneTable{a.pop}, x0, blockIdx.y, blockIdx.z + a.z_lo, a.nx, a.ny, a.nz);
  } else {
    const uint32_t slot = blockIdx.x * (uint32_t)kStepBlock + threadIdx.x;
    if (slot >= a.slots[PARITY]) return;
    if (PARITY == 0) {
      p.init_flat(PlaneTable{a.pop}, a.first, a.count, slot);
    } else {
      int x0, y, z;
      slot_xyz<false>(slot, a.nx, a.ny, a.m_hp, a.p_hp, a.m_ny, a.p_ny, x0, y, z);
      p.init_row(PlaneTable{a.pop}, x0, y, z + a.z_lo, a.nx, a.ny, a.nz);
    }
  }
  // Large launches: the reads first, the noise while the populations travel. Small ones: the noise
  // before the wait for the step before, so that it fills the drain of that launch.
  constexpr int B = Noisy<LAT>::blocks;
  float2 n[Noisy<LAT>::count];
  const uint32_t st = shared_address(stage + threadIdx.x);
  if (a.early) {
    wait_prerequisites();
    p.fetch(st);
  }
  if (NOISE) site_noise<LAT, S, SCHEME, ISO, 0, B>(n, a, p.site0, p.dsite, a.step_lo, a.step_hi);
  if (!a.early) {
    wait_prerequisites();
    p.fetch(st);
  }
  if (Access::STAGED) cp_async_wait_all();
  if constexpr (LAT == 19) {
    float2 F[19];
    p.load_list(stage + threadIdx.x, F);
    p.forget();
    collide_site<LAT, NOISE, SCHEME, ISO>(F, a, n);
    p.store_list(F);
  } else {
    float2 F[3][3][3];
    p.load_tile(stage + threadIdx.x, F);
    p.forget();
    collide_site<LAT, NOISE, SCHEME, ISO>(F, a, n);
    p.store_tile(F);
  }
}

// Blocks of 128 threads per SM that a pair kernel is compiled for (its register cap), where the launch
// does not choose by size (launch_kernel): at 256^3 (FP32 D3Q27, ms per step at 3 / 4 / 5 blocks)
// 64-bit offsets, staged reads, the paper's rates .563 / .551 / .548; direct reads without noise .551 /
// .523 / .554, of unaligned elements (255^3) .534 / .559 / .711. The general rates keep the tile and the
// noise together (BGK 96^3 at 4 / 5: 33.8 / 35.1 us).
template <int LAT, int SCHEME, bool DIRECT, bool ALIGNED>
constexpr int pair_blocks() {
  return LAT == 2 ? 8 : DIRECT ? (ALIGNED ? 4 : 3) : SCHEME == kShear ? 5 : 4;
}

template <int N>
using Blocks = std::integral_constant<int, N>;

template <int LAT, typename S, int PARITY, bool NOISE, int SCHEME, bool ISO, bool ALIGNED, typename O, int MINB>
cudaError_t launch_pair(cudaLaunchConfig_t &cfg, const StepArgs &a) {
  if constexpr (PARITY == 1 && ALIGNED) {
    const int per_row = (a.nx / 2 + kStepBlock - 1) / kStepBlock;
    if (per_row * kStepBlock <= a.nx / 2 + a.nx / 16) {
      cfg.gridDim = dim3(per_row, a.ny, a.nz_grid);
      return cudaLaunchKernelEx(&cfg, pair_kernel<LAT, S, PARITY, NOISE, SCHEME, ISO, true, true, O, MINB>, a);
    }
  }
  return cudaLaunchKernelEx(&cfg, pair_kernel<LAT, S, PARITY, NOISE, SCHEME, ISO, ALIGNED, false, O, MINB>, a);
}

template <int LAT, typename S, int PARITY, bool NOISE, int SCHEME, bool ISO>
cudaError_t launch_kernel(int variant, const StepArgs &a, cudaStream_t s) {
  if (variant == kStepOneSite || (a.wide && !a.aligned[PARITY])) {
    const dim3 grid((a.nx + kStepBlock - 1) / kStepBlock, a.ny, a.nz_grid);
    step_kernel<LAT, S, PARITY, NOISE, SCHEME, ISO><<<grid, kStepBlock, 0, s>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((a.slots[PARITY] + kStepBlock - 1) / kStepBlock);
  cfg.blockDim = dim3(kStepBlock);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const bool narrow = !a.wide && (variant == kStepPairOcc || variant == kStepPairRolledOcc || variant == kStepPairOccRows);
  // With noise, more registers let a warp keep several Philox streams and Box-Muller chains going,
  // and a launch of few blocks has no use for room for more of them. us per step (FP32, the paper's
  // rates; blocks per SM):
  //   D3Q27, 32-bit offsets (3 / 4 / 5): 33^3 4.4 / 5.0 / 5.7, 48^3 4.4 / 4.9 / 6.0; 25x50x100 6.4 / 5.4 / 6.9,
  //   64^3 9.4 / 8.9 / 9.9, 80^3 17.6 / 16.6 / 17.4, 192^3 - / 233 / 240, FP16 256^3 515 / 512 / 518;
  //   unaligned (rows of odd length) 63^3 10.6 / 10.2 / 11.3, 127^3 85 / 87 / 89, 255^3 658 / 673 / 689;
  //   general rates 48^3 4.7 / 5.1, BGK 4.5 / 5.0, but 25x50x100 6.2 / 5.6;
  //   D3Q19 unaligned (4 / 5): 25x50x100 4.4 / 5.1, 255^3 467 / 463; aligned 64^3 6.8 / 6.6;
  //   D2Q9 (5 / 8): 512^2 3.30 / 3.41, 4096^2 181 / 180, 4095^2 213 / 215.
  const bool few = a.slots[PARITY] <= kFewSlots;
  constexpr bool SHEAR = SCHEME == kShear, DIRECT = !NOISE || sizeof(S) == 2;
  constexpr int MA = pair_blocks<LAT, SCHEME, !NOISE, true>(), MU = pair_blocks<LAT, SCHEME, DIRECT, false>();
  const auto launch = [&](auto aligned, auto offset, auto blocks) {
    return launch_pair<LAT, S, PARITY, NOISE, SCHEME, ISO, decltype(aligned)::value, decltype(offset),
                       decltype(blocks)::value>(cfg, a);
  };
  using Yes = std::true_type;
  using No = std::false_type;
  if (!a.aligned[PARITY]) {
    if constexpr (!DIRECT && LAT == 3) {
      if (few || (SHEAR && a.early)) return launch(No{}, uint32_t{}, Blocks<3>{});
      return launch(No{}, uint32_t{}, Blocks<4>{});
    } else if constexpr (!DIRECT && SHEAR && LAT == 19) {
      return a.early ? launch(No{}, uint32_t{}, Blocks<5>{}) : launch(No{}, uint32_t{}, Blocks<4>{});
    } else {
      return launch(No{}, uint32_t{}, Blocks<!DIRECT && SHEAR && LAT == 2 ? 5 : MU>{});
    }
  }
  if (narrow) {
    if constexpr (NOISE && LAT == 3)
      return few ? launch(Yes{}, uint32_t{}, Blocks<3>{}) : launch(Yes{}, uint32_t{}, Blocks<4>{});
    else if constexpr (NOISE && SHEAR && LAT == 2)
      return a.early ? launch(Yes{}, uint32_t{}, Blocks<MA>{}) : launch(Yes{}, uint32_t{}, Blocks<5>{});
    else
      return launch(Yes{}, uint32_t{}, Blocks<MA>{});
  }
  return launch(Yes{}, uint64_t{}, Blocks<MA>{});
}

template <int LAT, typename S, bool ISO, int SCHEME>
cudaError_t launch_typed(int variant, int parity, bool noise, const StepArgs &a, cudaStream_t s) {
  if (parity == 0)
    return noise ? launch_kernel<LAT, S, 0, true, SCHEME, ISO>(variant, a, s)
                 : launch_kernel<LAT, S, 0, false, SCHEME, ISO>(variant, a, s);
  return noise ? launch_kernel<LAT, S, 1, true, SCHEME, ISO>(variant, a, s)
               : launch_kernel<LAT, S, 1, false, SCHEME, ISO>(variant, a, s);
}

template <int LAT, typename S, bool ISO>
cudaError_t launch_rates(int variant, int parity, bool noise, bool shear, const StepArgs &a, cudaStream_t s) {
  return shear ? launch_typed<LAT, S, ISO, kShear>(variant, parity, noise, a, s)
               : launch_typed<LAT, S, ISO, kGeneral>(variant, parity, noise, a, s);
}

}  // namespace
}  // namespace flbm
