"""Plans are worked out once per size, whichever sizes a caller's layers have: razer_plan_cache.h compiled by itself."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_04052_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include "razer_plan_cache.h"
struct Plan { long long v; };
static long long made;
static long long plan(int N, int K, int M, int variant) {
  return razer::remembered<Plan>(N, K, M, variant, [&] { ++made; return Plan{((N * 40000LL + K) * 4000 + M) * 4 + variant}; }).v;
}
static int wrong;
static void use(int N, int K, int M, int variant) {
  wrong += plan(N, K, M, variant) != ((N * 40000LL + K) * 4000 + M) * 4 + variant;
}
static long long count() { long long n = made; made = 0; return n; }
int main() {
  const int shapes[][2] = {{4096, 4096}, {11008, 4096}, {4096, 11008}, {3584, 3584}, {18944, 3584}, {8192, 8192}, {28672, 8192}, {8192, 28672}};
  for (int M = 1; M <= 64; ++M) {                      // a loop over a model's layers: worked out in its first pass
    for (int pass = 0; pass < 3; ++pass) {
      for (auto& s : shapes) use(s[0], s[1], M, 0);
      printf("%lld ", count());
    }
  }
  for (int i = 0; i < 1000; ++i) use(256 + i, 256 + 16 * i, 1 + i % 64, i % 3);   // many sizes, each its own plan
  printf("\n%lld ", count());
  for (int i = 968; i < 1000; ++i) use(256 + i, 256 + 16 * i, 1 + i % 64, i % 3);  // the last 32 are still there
  printf("%lld ", count());
  use(1255, 256 + 16 * 999, 1 + 999 % 64, 1);           // a variant of one of them is not
  printf("%lld ", count());
  long long other = 0;
  std::thread([&] { use(4096, 4096, 1, 0); other = count(); }).join();   // another thread remembers for itself
  printf("%lld %d\n", other, wrong);
}
"""


def test_every_size_of_a_layer_loop_is_remembered(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")],
                   check=True, timeout=120)
    loop, rest = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=60).stdout.splitlines()
    assert [int(v) for v in loop.split()] == [8, 0, 0] * 64
    assert [int(v) for v in rest.split()] == [1000, 0, 1, 1, 0]
