"""Host side of the staged step kernels (csrc/tiles.cpp), compiled on its own: no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_08515_gb300", "csrc")

# Lays out a ring lattice whose rows alternate between two patterns (stored places: the groups are no shifted copies)
# and, with patterns, one whose rows are all alike; the n-th allocation after the start fails, for every n.
PROBE = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include "kes_internal.h"
static std::atomic<long> left{-1};  // allocations until one fails; negative: none does
void* operator new(std::size_t n) {
  if (left >= 0 && left-- == 0) throw std::bad_alloc();
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
int main() {
  const int64_t slices = 256, rows = 32 * slices;
  for (int alike = 0; alike < 2; ++alike) {
    std::vector<int64_t> ptr(slices + 1);
    std::vector<int32_t> col(rows * 3), len(rows, 3);
    for (int64_t s = 0; s <= slices; ++s) ptr[s] = 96 * s;
    for (int64_t r = 0; r < rows; ++r) {
      const int64_t d = alike || r % 2 ? 1 : 2;
      const int64_t c[3] = {r < d ? 0 : r - d, r, r + d < rows ? r + d : rows - 1};
      int32_t* at = &col[ptr[r / 32] + r % 32];
      len[r] = 0;
      for (int k = 0; k < 3; ++k)
        if (len[r] == 0 || c[k] > at[32 * (len[r] - 1)]) at[32 * len[r]++] = static_cast<int32_t>(c[k]);
      for (int k = len[r]; k < 3; ++k) at[32 * k] = static_cast<int32_t>(r);
    }
    const int64_t row0 = 0;
    kes::TileInput in;
    in.n_slices = slices;
    in.slice_ptr = ptr.data();
    in.col = col.data();
    in.len = len.data();
    in.n_mesh = 1;
    in.mesh_row0 = &row0;
    in.mesh_rows = &rows;
    long failed = 0;
    for (long n = 0;; ++n) {
      bool done = false, ok = false;
      {
        kes::TileLayout lay;
        kes::TileHost h;
        left = n;
        try {
          ok = kes::build_tile_groups(in, lay) && kes::build_tiles(in, lay, 64, h);
          done = true;
        } catch (const std::bad_alloc&) {
          ++failed;
        }
        done = done && left >= 0;  // every allocation was within the budget
        left = -1;
      }
      if (done) {
        std::printf("%d %d %ld\n", alike, ok ? 1 : 0, failed);
        break;
      }
    }
  }
  return 0;
}
"""


def test_a_failed_allocation_is_an_exception_not_the_end_of_the_process(tmp_path):
    # kes_create turns std::bad_alloc into KES_ERR_OOM; one that leaves a thread of a parallel region would end the
    # caller's process instead
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fopenmp", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda,
                    str(src), os.path.join(CSRC, "tiles.cpp"), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, env=dict(os.environ, OMP_NUM_THREADS="4"))
    assert run.returncode == 0, run.stderr
    lines = [[int(v) for v in line.split()] for line in run.stdout.splitlines()]
    assert [(a, ok) for a, ok, _ in lines] == [(0, 1), (1, 1)]
    assert all(failed > 50 for _, _, failed in lines)
