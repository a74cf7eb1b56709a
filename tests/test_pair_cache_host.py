"""The kept answers about a kernel's resident CTA pairs (csrc/pair_cache.h) on the
host: one per device, kernel and shared-memory size - kernels of one signature are
told apart -, none for a failure, the right one also past the capacity and from many
threads."""
import os
import subprocess

HARNESS = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "pair_cache.h"
using jet::PairCache;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

template <int K> void kernel(int) {}

int main() {
  const void* a = reinterpret_cast<const void*>(&kernel<1>);
  const void* b = reinterpret_cast<const void*>(&kernel<2>);
  PairCache c;
  int asked = 0;
  auto ask = [&](int answer) { return [&asked, answer] { ++asked; return answer; }; };
  CHECK(c.get(0, a, 100, ask(76)) == 76 && asked == 1);
  CHECK(c.get(0, a, 100, ask(-5)) == 76 && asked == 1);    // kept
  CHECK(c.get(0, b, 100, ask(38)) == 38 && asked == 2);    // another kernel of its type
  CHECK(c.get(0, a, 200, ask(70)) == 70 && asked == 3);    // another size
  CHECK(c.get(1, a, 100, ask(74)) == 74 && asked == 4);    // another device
  CHECK(c.get(0, b, 300, ask(0)) == 0 && asked == 5);      // a failure is asked again
  CHECK(c.get(0, b, 300, ask(12)) == 12 && asked == 6);
  for (int i = 0; i < 3 * PairCache::kEntries; ++i)
    CHECK(c.get(2, a, size_t(i), ask(1000 + i)) == 1000 + i);
  CHECK(c.get(2, a, 3 * PairCache::kEntries - 1, ask(-1)) == 1000 + 3 * PairCache::kEntries - 1);
  CHECK(c.get(0, a, 100, ask(76)) == 76);
  PairCache t;
  std::vector<std::thread> threads;
  std::vector<int> wrong(8, 0);
  for (int w = 0; w < 8; ++w)
    threads.emplace_back([&, w] {
      for (int i = 0; i < 20000; ++i) {
        const size_t k = size_t(i * (w + 3)) % 97;
        if (t.get(int(k % 3), a, k, [k] { return int(k) + 1; }) != int(k) + 1) ++wrong[size_t(w)];
      }
    });
  for (auto& x : threads) x.join();
  for (int x : wrong) CHECK(x == 0);
  return 0;
}
"""


def test_answers_belong_to_their_kernel(tmp_path, repo_root):
    src, exe = tmp_path / "cache.cpp", tmp_path / "cache"
    src.write_text(HARNESS)
    inc = os.path.join(repo_root, "paper_2609_33874_gb300", "csrc")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread",
                    "-I", inc, str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
