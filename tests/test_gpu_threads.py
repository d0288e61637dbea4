"""Calls of several host threads at once, whose launches of one kernel need
different amounts of shared memory: each succeeds with the results it has
alone. Driven from C++ threads (Python's lock keeps calls too far apart)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <dlfcn.h>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>
#include "gramsci_gb300.h"

#define ENTRY(name) decltype(&::name) p_##name = (decltype(&::name))dlsym(lib, #name)

int main(int argc, char** argv) {
  void* lib = dlopen(argv[1], RTLD_NOW);
  if (!lib) { std::puts(dlerror()); return 2; }
  ENTRY(gs_build_graph);
  ENTRY(gs_disconnected_4pcf);
  ENTRY(gs_count_3pcf);
  ENTRY(gs_count_3pcf_equilateral);
  ENTRY(gs_count_3pcf_mu);
  ENTRY(gs_count_4pcf);
  const std::string query = argv[2];
  const int many = std::atoi(argv[3]), calls = std::atoi(argv[4]);
  const int n = 300, box = 40000;
  std::vector<int32_t> xyz(3 * n);
  std::vector<float> w(n);
  unsigned r = 1;
  for (auto& x : xyz) x = (int32_t)((r = r * 1664525u + 1013904223u) >> 8) % box;
  for (auto& x : w) x = 0.5f + (float)((r = r * 1664525u + 1013904223u) >> 8) / 16777216.0f;
  gs_graph* g[2];
  for (int k = 0; k < 2; ++k) {
    const int nb = k ? 3 : many;
    std::vector<int64_t> e(nb + 1);
    for (int b = 0; b <= nb; ++b) e[b] = 9000 * b / nb;
    if (p_gs_build_graph(xyz.data(), n, box, e.data(), nb, nullptr, &g[k])) return 3;
  }
  auto call = [&](int k, std::vector<uint64_t>& out) -> int {
    out.assign(1 << 16, 0);
    std::vector<double> sums(1 << 16);
    if (query == "pairs") return p_gs_disconnected_4pcf(g[k], w.data(), nullptr, out.data(), nullptr, nullptr, nullptr);
    if (query == "triangles") return p_gs_count_3pcf(g[k], w.data(), out.data(), sums.data(), nullptr);
    if (query == "equilateral") return p_gs_count_3pcf_equilateral(g[k], w.data(), out.data(), sums.data(), nullptr);
    if (query == "mu") return p_gs_count_3pcf_mu(g[k], nullptr, 4, out.data(), nullptr, nullptr);
    return p_gs_count_4pcf(g[k], nullptr, out.data(), nullptr, nullptr);
  };
  std::vector<uint64_t> ref[2];
  for (int k = 0; k < 2; ++k)
    if (call(k, ref[k])) return 4;
  std::atomic<int> failed{0}, wrong{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 6; ++t)
    threads.emplace_back([&, t] {
      std::vector<uint64_t> out;
      for (int c = 0; c < calls; ++c) {
        if (call(t % 2, out)) ++failed;
        else if (out != ref[t % 2]) ++wrong;
      }
    });
  for (auto& t : threads) t.join();
  std::printf("failed %d wrong %d\n", (int)failed, (int)wrong);
  return failed || wrong ? 1 : 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    import torch
    assert torch.cuda.is_available()
    d = tmp_path_factory.mktemp("threads")
    (d / "t.cpp").write_text("#include <string>\n" + PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), str(d / "t.cpp"),
                    "-o", str(d / "t"), "-ldl", "-lpthread"], check=True)
    return str(d / "t")


@pytest.mark.parametrize("query,bins", [("pairs", 254), ("triangles", 20), ("equilateral", 200),
                                        ("mu", 18), ("tetrahedra", 9)])
def test_threads_with_few_and_many_bins(program, query, bins):
    import paper_2607_06604_gb300 as gs
    r = subprocess.run([program, gs.lib_path, query, str(bins), "1500"], capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
