"""Order of the additions of a warp's lanes into a tile's DoF buffer (csrc/turns.cuh).

The lanes of a warp are promised to be together only at __syncwarp; between two
of them one lane may run ahead of the others by any amount.  add_turns is
compiled for the host with every lane a thread, exactly one of them running at a
time, up to its next __syncwarp, in a chosen order of the lanes.  32 cells in a
row along x: node k of cell j and node 0 of cell j + 1 are one DoF, and in a
second case every pair of cells shares its interior nodes as siblings behind one
coarse face do.  The result must be the program's order of additions (slot by
slot, lanes by rank) bit for bit in whichever order the lanes run; the values
are large enough against each other that another order rounds differently.
"""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2203_12292_gb300" / "csrc"

SOURCE = r"""
#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
void __syncwarp();
#include "turns.cuh"

constexpr int W = 32, K = 4, N = K + 1;
std::mutex mu;
std::condition_variable cv;
int order_[W], at = 0;         // the lane of place `at` runs
thread_local int place;

void hand_on(std::unique_lock<std::mutex>& lk) {  // to the next place, wait for the next turn
  at = (at + 1) % W;
  cv.notify_all();
}
void my_turn(std::unique_lock<std::mutex>& lk) {
  cv.wait(lk, [] { return at == place; });
}
void __syncwarp() {  // all places pass once before this lane goes on
  std::unique_lock<std::mutex> lk(mu);
  hand_on(lk);
  my_turn(lk);
}

int main(int argc, char** argv) {
  const int mode = argv[1][0] - '0', siblings = argv[2][0] - '0';
  for (int i = 0; i < W; ++i) order_[i] = mode == 0 ? i : mode == 1 ? W - 1 - i : (i * 11) % W;
  // vertex j at x[j], j = 0 .. W; interior nodes of cell j after them
  std::vector<float> x(W + 1 + W * (K - 1), 0.f), ref(x);
  float v[W][N];
  for (int j = 0; j < W; ++j)
    for (int a = 0; a < N; ++a) v[j][a] = (1.f + 0.37f * a + 0.11f * j) * ((j + a) % 3 == 0 ? 3e7f : (j + a) % 3 == 1 ? 1.f : -3e7f);
  for (size_t i = 0; i < x.size(); ++i) x[i] = ref[i] = 0.1f * (i % 7);
  auto inner = [&](int j) { return W + 1 + (siblings ? j / 2 : j) * (K - 1); };
  const int turns = siblings ? 2 : 1;
  for (int line = 0; line < 2; ++line) {
    for (int j = 0; j < W; ++j) ref[j] += v[j][0];
    for (int q = 0; q < turns; ++q)
      for (int j = 0; j < W; ++j)
        if (!siblings || j % 2 == q)
          for (int a = 1; a < K; ++a) ref[inner(j) + a - 1] += v[j][a];
    for (int j = 0; j < W; ++j) ref[j + 1] += v[j][K];
  }
  std::vector<std::thread> t;
  for (int p = 0; p < W; ++p)
    t.emplace_back([&, p] {
      place = p;
      {
        std::unique_lock<std::mutex> lk(mu);
        my_turn(lk);
      }
      const int j = order_[p];
      for (int line = 0; line < 2; ++line) {
        gcmg::add_turns<1>(&x[j], v[j], 0, 1);
        gcmg::add_turns<K - 1>(&x[inner(j)], v[j] + 1, siblings ? j % 2 : 0, turns);
        gcmg::add_turns<1>(&x[j + 1], v[j] + K, 0, 1);
      }
      std::unique_lock<std::mutex> lk(mu);
      hand_on(lk);
    });
  for (auto& u : t) u.join();
  const bool same = std::memcmp(x.data(), ref.data(), x.size() * sizeof(float)) == 0;
  std::puts(same ? "same" : "different");
  return same ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("turns")
    (d / "turns.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-pthread", f"-I{CSRC}", "-o", str(d / "turns"),
                    str(d / "turns.cpp")], check=True)
    return str(d / "turns")


@pytest.mark.parametrize("siblings", [0, 1])
@pytest.mark.parametrize("order", [0, 1, 2])
def test_additions_keep_the_programs_order(program, order, siblings):
    r = subprocess.run([program, str(order), str(siblings)], timeout=60, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
