"""Host copies of a graph's row starts and lengths (csrc/gs_host_copy.h) with a
fetch that fails: the status reaches the caller, nothing of the failed fetch is
kept, and the next call fetches again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include "gs_host_copy.h"
#include <cstdio>
#include <cstdint>
int main() {
  std::mutex mu;
  std::vector<int32_t> kept;
  const int32_t* p = nullptr;
  int calls = 0;
  auto fails = [&](int32_t* d) { ++calls; d[0] = 7; return (int)GS_ECUDA; };
  auto works = [&](int32_t* d) { ++calls; for (int k = 0; k < 5; ++k) d[k] = 10 + k; return (int)GS_OK; };
  if (gs::host_copy(mu, kept, 5, fails, &p) != GS_ECUDA || p || !kept.empty()) return 1;
  if (gs::host_copy(mu, kept, 5, works, &p) != GS_OK || !p || p[0] != 10 || p[4] != 14) return 2;
  if (gs::host_copy(mu, kept, 5, fails, &p) != GS_OK || p[4] != 14 || calls != 2) return 3;
  std::vector<int64_t> huge;
  const int64_t* q = nullptr;
  auto unused = [&](int64_t*) { return (int)GS_OK; };
  if (gs::host_copy(mu, huge, (size_t)1 << 58, unused, &q) != GS_ENOMEM || q) return 4;
  std::vector<int64_t> none;
  if (gs::host_copy(mu, none, 0, unused, &q) != GS_OK) return 5;
  std::puts("ok");
  return 0;
}
'''


def test_failed_copy_is_not_kept(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2607_06604_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.returncode
