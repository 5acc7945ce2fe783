"""Slots of the pair kernels (csrc/pair.cuh): row coordinates by multiply-shift divisions, on the host.

A row of nx sites holds ceil(nx / 2) slots, so boxes of odd rows have up to as many slots as sites
(nx = 1), which may be anything below 2^32. The statistics, and the batches' forms with 64-bit offsets,
take all of them; a row or a plane that is not recognised as the last one would not wrap.
"""
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_16486_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "internal.h"
#include "pair.cuh"
// Reads lines "nx ny slot any" and prints "x0 y z"; any = 2: a slot of a row, "x0 in-the-row 0".
int main() {
  int nx, ny, any;
  unsigned slot;
  while (std::scanf("%d %d %u %d", &nx, &ny, &slot, &any) == 4) {
    uint32_t m_hp, m_ny;
    int p_hp, p_ny, x0, y, z;
    if (any == 2) {
      const bool in = flbm::row_slot(slot, nx, x0);
      std::printf("%d %d 0\n", in ? x0 : 0, int(in));
      continue;
    }
    flbm::batch_magic((uint32_t(nx) + 1) / 2, &m_hp, &p_hp);
    flbm::batch_magic(uint32_t(ny), &m_ny, &p_ny);
    if (any)
      flbm::slot_xyz<true>(slot, nx, ny, m_hp, p_hp, m_ny, p_ny, x0, y, z);
    else
      flbm::slot_xyz<false>(slot, nx, ny, m_hp, p_hp, m_ny, p_ny, x0, y, z);
    std::printf("%d %d %d\n", x0, y, z);
  }
  return 0;
}
"""


def _cases():
    rng = random.Random(3)
    boxes = [(1, 65534, 32773), (1, 65535, 65535), (1, 65533, 65535), (1, 40000, 65535), (3, 65535, 21845),
             (5, 60001, 14000), (4001, 1021, 1051), (2, 65535, 32767), (65535, 65535, 1), (7, 5, 3), (1, 1, 1),
             (2 ** 31 - 1, 1, 1), (2 ** 31 - 2, 2, 1)]
    for _ in range(60):
        nx, ny = 2 * rng.randrange(40) + 1, rng.randrange(1, 65536)
        boxes.append((nx, ny, max(1, min(65535, (2 ** 32 - 1) // (nx * ny)))))
    for nx, ny, nz in boxes:
        hp, slots = (nx + 1) // 2, (nx + 1) // 2 * ny * nz
        assert nx * ny * nz < 2 ** 32 and slots < 2 ** 32
        at = {0, slots - 1, slots // 2, min(slots - 1, 2 ** 31), min(slots - 1, 2147745781)}
        at |= {min(slots - 1, max(0, hp * ny * z + d)) for z in (1, nz // 2, nz - 1) for d in (-1, 0, 1, hp)}
        at |= {rng.randrange(slots) for _ in range(200)}
        for s in at:
            r = s // hp
            want = (2 * (s - r * hp), r % ny, r // ny)
            yield nx, ny, s, 1, want
            if s < 2 ** 31:
                yield nx, ny, s, 0, want
    # A launch over the rows covers their slots up to a whole block of 128.
    for nx in (2, 254, 256, 258, 2 ** 31 - 2, 2 ** 31 - 256, 2 ** 31 - 258):
        for k in [0, 1] + list(range(max(0, nx // 2 - 2), -(-nx // 2 // 128) * 128 + 128)):
            yield nx, 1, k, 2, (2 * k if k < nx // 2 else 0, int(k < nx // 2), 0)


def test_slots_of_every_box_the_library_accepts(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "slots.cu", tmp_path / "slots"
    src.write_text(DRIVER)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    cases = list(_cases())
    lines = "".join("%d %d %d %d\n" % c[:4] for c in cases)
    out = subprocess.run([str(exe)], input=lines, capture_output=True, text=True, check=True).stdout.split("\n")
    got = [tuple(int(v) for v in line.split()) for line in out if line]
    assert len(got) == len(cases)
    for c, g in zip(cases, got):
        assert g == c[4], c
