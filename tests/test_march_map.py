"""Host check of the marching 3-D stage's shared-memory map (no GPU needed), for both shapes and every
ragged extent of a tile: within a level the owned cells and the x and y halo land on distinct
locations, each inside the level's own rows or the y halo (so the other four levels of the ring and
the right states parked in the oldest one are not touched), and every cell that an x or y window
reads was filled at the location it is read from."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <map>
#include <utility>
#include "paper_1901_02955_gb300/csrc/snap_march.cuh"
using namespace snap;

template <class T>
int check(int slot, int ex, int ey) {
  using M = MarchSmem<float, Lay<0, 0, true>, T>;
  const int cur = slot * M::NL;
  std::map<int, std::pair<int, int>> owner;
  std::map<std::pair<int, int>, int> place;
  int bad = 0;
  auto fill = [&](int x, int y) {
    const int i = M::at(cur, x, y);
    if (!(i >= cur && i < cur + M::NL) && !(i >= M::HY && i < M::NP)) ++bad;
    if (!owner.emplace(i, std::make_pair(x, y)).second) ++bad;
    place[{x, y}] = i;
  };
  auto read = [&](int x, int y) {
    const auto it = place.find({x, y});
    if (it == place.end() || it->second != M::at(cur, x, y)) ++bad;
  };
  for (int y = 0; y < ey; ++y)
    for (int x = 0; x < ex; ++x) {
      fill(x, y);
      // the thread's own column by the kernel's formula
      if (M::at(cur, x, y) != cur + y * M::BX + x + 3) ++bad;
    }
  for (int r = 0; r < 6; ++r) {
    for (int y = 0; y < ey; ++y) fill(r < 3 ? r - 3 : ex + r - 3, y);
    for (int x = 0; x < ex; ++x) fill(x, r < 3 ? r - 3 : ey + r - 3);
  }
  for (int k = -2; k <= 2; ++k) {
    for (int y = 0; y < ey; ++y)
      for (int x = -1; x <= ex; ++x) read(x + k, y);
    for (int y = -1; y <= ey; ++y)
      for (int x = 0; x < ex; ++x) read(x, y + k);
  }
  return bad;
}

template <class T>
int all_extents() {
  int bad = 0;
  for (int slot = 0; slot < 5; ++slot)
    for (int ey = 1; ey <= T::TY; ++ey)
      for (int ex = 1; ex <= T::TX; ++ex) bad += check<T>(slot, ex, ey);
  return bad;
}

int main() {
  const int bad = all_extents<MarchT<32, 8, 32, 3>>() + all_extents<MarchT<32, 16, 32, 1>>();
  printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_march_map_is_injective_and_covers_every_read(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "march_map.cu"
    src.write_text(DRIVER)
    exe = tmp_path / "march_map"
    subprocess.check_call([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                           "arch=compute_103a,code=sm_103a", "-I", ROOT, str(src), "-o", str(exe)],
                          cwd=ROOT)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.stdout.strip() == "bad 0" and out.returncode == 0, out.stdout + out.stderr
