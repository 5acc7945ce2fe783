// Fused fluctuating central-moment collide-and-stream step (one lattice update).
//
// Per site, in the order of the paper's "Algorithm of computation" (Sec. II-B):
//   load the Q populations arriving at the site, rho and u (Eq. macro),
//   k = T(u) f (Sec. II-B / II-C, factorised, see cm.cuh),
//   k*_v = (1 - L_v) k_v + L_v k^eq_v + I~_v phi_v eta_v (Eq. cm_collision) with
//   k^eq = (rho, 0, ..., 0) and phi_v = sqrt(rho) * sqrt(kBT L_v (2-L_v) b_v / cs^2)
//   (Eq. phi_general), normals from Philox4x32-10 + Box-Muller (philox.cuh),
//   f* = T(u)^{-1} k*, and streaming f_i(x + c_i, t+1) = f*_i(x, t) (Eq. streaming).
//
// Streaming is in place with the AA pattern (one population array): on even steps a
// site reads its own slots i and writes its post-collision values to its own slots
// opposite(i); on odd steps it reads the slot opposite(i) of its neighbour x - c_i and
// writes slot i of its neighbour x + c_i. Each step touches exactly the slots it
// reads, so no two threads race and no second lattice is needed. Logical populations:
// even state f_i(x) = A[i][x]; odd state f_i(x) = A[opposite(i)][x - c_i].
//
// Layout: structure of arrays A[q][z][y][x], x fastest. Kernels (step_kernels.cuh):
//   step_kernel - one site per thread, blocks of 128 consecutive x, grid
//                 (ceil(nx/128), ny, nz); where variant 1 is asked for, and for unaligned rows
//                 of planes of 4 GB or more;
//   pair_kernel - two sites per thread, every floating-point step as packed FP32x2; pairs are
//                 taken flat over the rows (pair.cuh), so short and odd rows fill the warps,
//                 and move as one 8-byte (FP32) or 4-byte (16-bit) word where alignment allows.
// What bounds the pair kernel with noise is the FMA pipe: 40 % of its cycles are Philox's
// 32 x 32 -> 64-bit multiplies (about 4 cycles per warp and scheduler; a packed FP32x2 operation
// takes 2 to 3.3, by its distinct register operands), the rest the packed algebra. So what
// helped is what took operations off that pipe or filled it:
//  - the noise needs no population, only sqrt(rho) at the end (noise_modes): it is formed
//    while the populations travel by cp.async through shared memory, which holds no registers;
//  - amplitudes folded into the logarithm's constants, a cubic instead of a quartic series,
//    exact uniforms by one funnel shift (philox.cuh);
//  - the planes' bases as kernel arguments (forming f + i * plane per access cost 130 ALU and
//    multiply operations a pair: 256^3 FP32 0.575 -> 0.549 ms) and one offset per row;
//  - programmatic dependent launch: on short launches the next step's blocks form their noise
//    while this step drains (half of it before the wait and half while the populations travel was
//    slower: D2Q9 512^2 4.2 against 3.4 us, D3Q27 32^3 4.3 against 3.3).
//  - register caps by size (launch_kernel): more chains in flight per warp, 64^3 9.6 -> 8.8.
// Measured (us per step, before -> now): D2Q9 64^2 4.1 -> 1.8 (and 0.86 in calls of many steps,
// step_cluster.cu), 200^2 5.0 -> 1.9, 512^2 6.2 -> 3.3, 4096^2 BF16 176 -> 160; D3Q27 25x50x100 13.5 ->
// 5.3, 64^3 20 -> 8.8 (13.3 in its best launch shape), 96^3 BGK 62 -> 30, 256^3 FP32 580 -> 548 (6.6
// TB/s, 0.99 of the measured copy), FP16 571 -> 512; D3Q19 256^3 478 -> 388 (with d3q19.cuh).
// Tried and slower: scalar FMAs in place of the packed ones (256^3 FP16 0.615
// against 0.591 ms), six blocks per SM (spills: 0.586 against 0.550 ms).
#include "step_kernels.cuh"

namespace flbm {

cudaError_t launch_step(int lattice, int storage, int variant, int parity, bool noise, bool shear,
                        const StepArgs &a, cudaStream_t s) {
  if (lattice == 2) return launch_step_iso(storage, variant, parity, noise, shear, a, s);
  if (lattice == 3) return launch_step_d3q19(storage, variant, parity, noise, shear, a, s);
  const int D = lattice == 0 ? 2 : 3;
  if (storage != 0) return launch_step_16(D, storage, variant, parity, noise, shear, a, s);
  return D == 3 ? launch_rates<3, float, false>(variant, parity, noise, shear, a, s)
                : launch_rates<2, float, false>(variant, parity, noise, shear, a, s);
}

}  // namespace flbm
