// Access to the populations of two lattice sites per thread under the AA pattern, staged
// through shared memory, for the step kernels (step_kernels.cuh, batch.cu).
//
// Sites are taken in flat pair slots, so that every lane of every warp has work whatever the
// row length. From an even step count (PARITY 0) a site reads and writes its own slots only:
// slot k of the updated range is the sites first + 2k and first + 2k + 1, rows do not matter.
// From an odd count (PARITY 1) row r = y + ny z holds ceil(nx / 2) slots, numbered row-major.
//
// ALIGNED: pairs move as one word (8 bytes in FP32, 4 in the 16-bit types). PARITY 0 needs an
// even plane stride and range. PARITY 1 needs an even nx and pairs the sites x0 + 1 and x0 + 2
// (periodic; x0 even): an odd step reads slot opposite(i) of x - c_i and writes slot i of
// x + c_i, so with this pairing the populations with c_x = +-1 (18 of 27 on D3Q27) move as the
// aligned pairs at x0 or x0 + 2, and only those with c_x = 0 take two scalar accesses. Otherwise
// the pair is (x0, x0 + 1) with scalar accesses; the last slot of an odd row (or range) is one
// site, whose second lane repeats sites of the same row and is never stored.
//
// The reads go by cp.async (4 or 8 bytes) into a stage of the thread's own words
// (stage[word][thread]: no bank conflicts and no barrier), so that loads in flight hold no
// registers and on long launches the noise is formed while they travel. Without noise there is
// nothing to form meanwhile and the reads go to registers directly (STAGE false: 256^3 D3Q27 0.526 ms against 0.538
// staged), as do unaligned 16-bit elements (2 bytes, below cp.async's smallest size).
//
// ROWS (odd steps of aligned rows): the block's slots lie in one row, so that the row and plane
// offsets are the same for all of its threads.
//
// Offsets in a plane are bytes in O = uint32_t arithmetic modulo 2^32, for planes below 4 GB, or
// uint64_t. They are added up once per row (not per population) and kept from the compiler, which
// otherwise forms every address from its parts; the planes' bases are kernel arguments.
#pragma once

#include <cuda_runtime.h>

#include "cm.cuh"

namespace flbm {

__device__ __forceinline__ uint32_t shared_address(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch: lets the next kernel of the stream start its blocks as this
// one's drain, and waits for the kernels before this one (and their writes).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Quotient x / d by the multiply-shift constants of batch_magic (internal.h): exact for x < 2^31, or
// (ANY) for every x. ANY divides x / 2 and puts the last bit right, four more operations.
template <bool ANY>
__host__ __device__ __forceinline__ uint32_t udiv_magic(uint32_t x, uint32_t d, uint32_t m, int p) {
  if (!ANY) return (uint32_t)(((unsigned long long)x * m) >> p);
  const uint32_t q = 2u * (uint32_t)(((unsigned long long)(x >> 1) * m) >> p);
  return x - q * d >= d ? q + 1u : q;
}

// Row coordinates of pair slot `slot` (rows of hp = ceil(nx / 2) slots). ANY: the slots may number 2^31
// or more. That takes rows of odd length (nx = 1 has as many slots as sites, which are below 2^32) and
// a plane of 4 GB or more, so the step kernels, which send such planes to one site per thread, do without.
template <bool ANY>
__host__ __device__ __forceinline__ void slot_xyz(uint32_t slot, int nx, int ny, uint32_t m_hp, int p_hp, uint32_t m_ny,
                                                  int p_ny, int &x0, int &y, int &z) {
  const uint32_t hp = ((uint32_t)nx + 1u) >> 1;
  const uint32_t r = udiv_magic<ANY>(slot, hp, m_hp, p_hp);
  x0 = 2 * (int)(slot - r * hp);
  const uint32_t q = udiv_magic<ANY>(r, (uint32_t)ny, m_ny, p_ny);
  y = (int)(r - q * (uint32_t)ny);
  z = (int)q;
}

// First site of pair slot k of a row; false past the row's end. A row has up to 2^31 - 1 sites and a launch
// up to a block of slots more, whose sites are not ints any more.
__host__ __device__ __forceinline__ bool row_slot(uint32_t k, int nx, int &x0) {
  x0 = (int)(2u * k);
  return 2u * k < (uint32_t)nx;
}

template <int LAT>
__host__ __device__ constexpr bool has_velocity(int dx, int dy, int dz) {
  return LAT == 2 ? dz == 0 : LAT == 19 ? dx * dx + dy * dy + dz * dz < 3 : true;
}
template <int LAT>
struct ZRange {
  static constexpr int lo = Lat<LAT>::D == 3 ? -1 : 0, hi = Lat<LAT>::D == 3 ? 1 : 0;
};

// Words of one thread's stage: a pair per population; in the 16-bit types an aligned odd step
// also holds the second pair of each population with c_x = 0. None where the reads go to
// registers directly.
template <int LAT, typename S, int PARITY, bool ALIGNED, bool STAGE>
__host__ __device__ constexpr int stage_words() {
  if (!STAGE || (sizeof(S) == 2 && !ALIGNED)) return 0;
  return Lat<LAT>::Q + (sizeof(S) == 2 && PARITY == 1 ? (LAT == 2 ? 3 : 9) : 0);
}

// Address of byte `off` of population i's plane: from the planes' addresses in the kernel
// arguments (the constant bank), or from a lattice's array and the bytes of its plane. In the
// second form 32-bit offsets run over the whole array (below 4 GB), because i * plane in 64 bits
// costs an access as much of the FMA pipe as four packed operations (batch of 32 D3Q27 64^3:
// 0.307 ms a step with it, 0.281 with the 32-bit multiply-add, 0.313 with the planes' addresses
// in shared memory).
struct PlaneTable {
  char *const *p;
  template <typename O>
  __device__ __forceinline__ char *at(int i, O off) const { return p[i] + (size_t)off; }
};
struct PlaneStride {
  char *p;
  unsigned long long plane;
  __device__ __forceinline__ char *at(int i, uint32_t off) const {
    return p + (size_t)(off + (uint32_t)i * (uint32_t)plane);
  }
  __device__ __forceinline__ char *at(int i, uint64_t off) const { return p + i * plane + off; }
};

template <int LAT, typename S, int PARITY, bool ALIGNED, bool ROWS, typename O, bool STAGE, int THREADS,
          typename Base = PlaneTable>
struct PairAccess {
  static constexpr int E = (int)sizeof(S);
  static constexpr int WORDS = stage_words<LAT, S, PARITY, ALIGNED, STAGE>();
  static constexpr bool STAGED = WORDS > 0;
  using Word = typename std::conditional<E == 4, float2, uint32_t>::type;
  static_assert(!ROWS || (PARITY == 1 && ALIGNED), "rows of blocks are a form of the aligned odd step");

  Base base;
  // Byte offsets in a plane. PARITY 0: x[1], x[2] the two lanes' sites. PARITY 1 aligned: x[1]
  // the pair at x0, x[2] the pair at x0 + 2; else x[0 .. 3] the sites x0 - 1 .. x0 + 2.
  O x[4];
  O dy[3], dz[3];  // to the rows y -+ 1 and the planes z -+ 1 (periodic)
  bool two;                // the second lane is a site of its own
  uint32_t site0, dsite;   // local site index of lane x, and from it to lane y

  // PARITY 0: slot k of the range of n sites from `first`.
  __device__ __forceinline__ void init_flat(const Base &planes, uint32_t first, uint32_t n, uint32_t k) {
    base = planes;
    site0 = first + 2u * k;
    two = ALIGNED || 2u * k + 1u < n;
    dsite = two ? 1u : 0u;
    x[1] = (O)site0 * E;
    x[2] = x[1] + (two ? (O)E : (O)0);
  }
  // PARITY 1: the slot at (x0, y, z).
  __device__ __forceinline__ void init_row(const Base &planes, int x0, int y, int z, int nx, int ny, int nz) {
    base = planes;
    const uint32_t row = ((uint32_t)z * (uint32_t)ny + (uint32_t)y) * (uint32_t)nx;
    if (ALIGNED) {
      const uint32_t s0 = row + (uint32_t)x0, s2 = row + (x0 + 2 == nx ? 0u : (uint32_t)x0 + 2u);
      x[1] = (O)s0 * E;
      x[2] = (O)s2 * E;
      two = true;
      site0 = s0 + 1u;
      dsite = s2 - site0;
    } else {
      int x1 = x0 + 1;
      if (x1 >= nx) x1 -= nx;
      int x2 = x1 + 1;
      if (x2 >= nx) x2 -= nx;
      x[0] = (O)(row + (uint32_t)(x0 == 0 ? nx - 1 : x0 - 1)) * E;
      x[1] = (O)(row + (uint32_t)x0) * E;
      x[2] = (O)(row + (uint32_t)x1) * E;
      x[3] = (O)(row + (uint32_t)x2) * E;
      two = x0 + 1 < nx;
      site0 = row + (uint32_t)x0;
      dsite = (uint32_t)x1 - (uint32_t)x0;
    }
    const O rl = (O)nx * E, pl = rl * (O)ny;
    dy[0] = y == 0 ? rl * (O)(ny - 1) : (O)0 - rl;
    dy[1] = 0;
    dy[2] = y == ny - 1 ? (O)0 - rl * (O)(ny - 1) : rl;
    dz[0] = z == 0 ? pl * (O)(nz - 1) : (O)0 - pl;
    dz[1] = 0;
    dz[2] = z == nz - 1 ? (O)0 - pl * (O)(nz - 1) : pl;
  }

  // Hides where the offsets come from, so that the addresses of the stores are formed anew
  // instead of those of the reads staying in registers (two per population) across the collision.
  __device__ __forceinline__ void forget() {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (used(k)) hide(x[k]);
  }
  __device__ __forceinline__ static constexpr bool used(int k) {
    return k == 1 || (k == 2 && !(PARITY == 0 && ALIGNED)) || (PARITY == 1 && !ALIGNED);
  }
  __device__ __forceinline__ static void hide(O &v) {
    if constexpr (sizeof(O) == 4)
      asm volatile("" : "+r"(v));
    else
      asm volatile("" : "+l"(v));
  }

  // The thread's offsets in the row (y + ry, z + rz), opaque so that they are formed once per
  // row and joined to each population's uniform base by the access itself.
  struct Row {
    O x[4];
  };
  __device__ __forceinline__ Row row(int ry, int rz) const {
    Row r;
    const O d = PARITY == 0 ? (O)0 : dy[1 + ry] + dz[1 + rz];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!used(k)) continue;
      r.x[k] = x[k] + d;
      if (PARITY == 1 && (ry != 0 || rz != 0)) hide(r.x[k]);
    }
    return r;
  }
  __device__ __forceinline__ char *at(int i, const Row &r, int k) const { return base.at(i, r.x[k]); }

  // Starts the reads of the pair's arriving populations into the stage (at shared address
  // `st` of this thread's first word; words THREADS apart).
  __device__ __forceinline__ void fetch(uint32_t st) const {
    if constexpr (STAGED) {
      constexpr uint32_t W = THREADS * sizeof(Word);
#pragma unroll
      for (int dz_ = ZRange<LAT>::lo; dz_ <= ZRange<LAT>::hi; ++dz_)
#pragma unroll
        for (int dy_ = -1; dy_ <= 1; ++dy_) {
          const Row r = row(-dy_, -dz_);
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) {
            if (!has_velocity<LAT>(dx, dy_, dz_)) continue;
            const int i = Lat<LAT>::index(dx, dy_, dz_), o = opposite<LAT>(i);
            const uint32_t d = st + (uint32_t)i * W;
            if (PARITY == 0) {
              if (ALIGNED) {
                cp_async<2 * E>(d, at(i, r, 1));
              } else {
                cp_async<4>(d, at(i, r, 1));
                cp_async<4>(d + 4, at(i, r, 2));
              }
            } else if (!ALIGNED) {  // f_i(x) = A[opposite(i)][x - c_i]
              cp_async<4>(d, at(o, r, 1 - dx));
              cp_async<4>(d + 4, at(o, r, 2 - dx));
            } else if (dx != 0) {
              cp_async<2 * E>(d, at(o, r, dx == 1 ? 1 : 2));
            } else if (E == 4) {
              cp_async<4>(d, at(o, r, 1) + E);
              cp_async<4>(d + 4, at(o, r, 2));
            } else {  // the pairs that hold x0 + 1 and x0 + 2
              cp_async<4>(d, at(o, r, 1));
              cp_async<4>(st + (uint32_t)(Lat<LAT>::Q + extra(dy_, dz_)) * W, at(o, r, 2));
            }
          }
        }
    }
  }
  __device__ __forceinline__ static constexpr int extra(int dy_, int dz_) {
    return LAT == 2 ? dy_ + 1 : 3 * (dz_ + 1) + dy_ + 1;
  }

  // The pair's population of velocity (dx, dy_, dz_), once its read has arrived.
  __device__ __forceinline__ float2 get(const Word *stage, int dx, int dy_, int dz_) const {
    const int i = Lat<LAT>::index(dx, dy_, dz_);
    if constexpr (!STAGED) {
      const Row r = row(-dy_, -dz_);
      const int o = PARITY == 0 ? i : opposite<LAT>(i), a = PARITY == 0 ? 1 : 1 - dx;
      if (ALIGNED && (PARITY == 0 || dx != 0))
        return Storage2<S>::load(reinterpret_cast<const S *>(at(o, r, PARITY == 0 || dx == 1 ? 1 : 2)));
      if (ALIGNED)
        return make_float2(Storage<S>::load(reinterpret_cast<const S *>(at(o, r, 1) + E)),
                           Storage<S>::load(reinterpret_cast<const S *>(at(o, r, 2))));
      return make_float2(Storage<S>::load(reinterpret_cast<const S *>(at(o, r, a))),
                         Storage<S>::load(reinterpret_cast<const S *>(at(o, r, a + 1))));
    } else if constexpr (E == 4) {
      return stage[i * THREADS];
    } else {
      uint32_t w = stage[i * THREADS];
      if (PARITY == 1 && dx == 0)  // (high half, low half of the next pair)
        w = __funnelshift_r(w, stage[(Lat<LAT>::Q + extra(dy_, dz_)) * THREADS], 16);
      return Storage2<S>::load(reinterpret_cast<const S *>(&w));
    }
  }

  // Stores the pair's post-collision population of velocity (dx, dy_, dz_); r: row(dy_, dz_).
  __device__ __forceinline__ void put(const Row &r, int dx, int dy_, int dz_, float2 v) const {
    const int i = Lat<LAT>::index(dx, dy_, dz_), o = opposite<LAT>(i);
    if (PARITY == 0) {  // to the site's own slot opposite(i)
      if (ALIGNED)
        Storage2<S>::store(reinterpret_cast<S *>(at(o, r, 1)), v);
      else
        put_lanes(at(o, r, 1), at(o, r, 2), v);
    } else if (!ALIGNED) {  // to slot i of x + c_i
      put_lanes(at(i, r, 1 + dx), at(i, r, 2 + dx), v);
    } else if (dx != 0) {
      Storage2<S>::store(reinterpret_cast<S *>(at(i, r, dx == 1 ? 2 : 1)), v);
    } else {
      put_lanes(at(i, r, 1) + E, at(i, r, 2), v);
    }
  }
  __device__ __forceinline__ void put_lanes(char *p0, char *p1, float2 v) const {
    Storage<S>::store(reinterpret_cast<S *>(p0), v.x);
    if (two) Storage<S>::store(reinterpret_cast<S *>(p1), v.y);
  }

  __device__ __forceinline__ void load_tile(const Word *stage, float2 (&F)[3][3][3]) const {
#pragma unroll
    for (int dz_ = ZRange<LAT>::lo; dz_ <= ZRange<LAT>::hi; ++dz_)
#pragma unroll
      for (int dy_ = -1; dy_ <= 1; ++dy_)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) F[dz_ + 1][dy_ + 1][dx + 1] = get(stage, dx, dy_, dz_);
  }
  // Stores pop(dx, dy, dz) of every velocity.
  template <typename F>
  __device__ __forceinline__ void store_all(const F &pop) const {
#pragma unroll
    for (int dz_ = ZRange<LAT>::lo; dz_ <= ZRange<LAT>::hi; ++dz_)
#pragma unroll
      for (int dy_ = -1; dy_ <= 1; ++dy_) {
        const Row r = row(dy_, dz_);
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx)
          if (has_velocity<LAT>(dx, dy_, dz_)) put(r, dx, dy_, dz_, pop(dx, dy_, dz_));
      }
  }
  __device__ __forceinline__ void store_tile(const float2 (&F)[3][3][3]) const {
    store_all([&](int dx, int dy_, int dz_) { return F[dz_ + 1][dy_ + 1][dx + 1]; });
  }
  __device__ __forceinline__ void load_list(const Word *stage, float2 (&F)[19]) const {
#pragma unroll
    for (int i = 0; i < 19; ++i) F[i] = get(stage, Lat<19>::cx(i), Lat<19>::cy(i), Lat<19>::cz(i));
  }
  __device__ __forceinline__ void store_list(const float2 (&F)[19]) const {
    store_all([&](int dx, int dy_, int dz_) { return F[Lat<19>::index(dx, dy_, dz_)]; });
  }
};

}  // namespace flbm
