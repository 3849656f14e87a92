"""The record of raised shared-memory limits (csrc/smem_limit.h) against a fake runtime whose
limits, like CUDA's, belong to a kernel and a device."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <utility>
#include "smem_limit.h"

// the fake: 48 KB unasked, 227 KB at most, both with the kernel's static memory
static std::map<std::pair<int, const void*>, size_t> g_limit;
static std::map<const void*, size_t> g_static;
static int g_fail = 0, g_raised = 0;
static bool launch(int dev, const void* k, size_t bytes) {
  auto it = g_limit.find({dev, k});
  const size_t lim = it == g_limit.end() ? 48 * 1024 - g_static[k] : it->second;
  return bytes <= lim;
}
struct Handle {
  int dev;
  pinn::SmemLimits smem;
  int allow(const void* k, size_t bytes) {
    return smem.allow(k, bytes, 0, 9, [&](size_t* limit) {
      if (g_fail) { --g_fail; return 2; }
      ++g_raised;
      g_limit[{dev, k}] = *limit = 227 * 1024 - g_static[k];
      return 0;
    });
  }
  bool run(const void* k, size_t bytes) { return allow(k, bytes) == 0 && launch(dev, k, bytes); }
};
#define CHECK(x) do { if (!(x)) { printf("failed: %s\n", #x); return 1; } } while (0)

int main() {
  int kern[100];
  const void *a = &kern[0], *b = &kern[1];
  g_static[b] = 4656;
  Handle h0{0, {}}, h1{1, {}}, h0b{0, {}};
  CHECK(!launch(0, a, 65536));
  CHECK(h0.run(a, 65536));                      // raised on device 0 ...
  CHECK(h1.run(a, 65536));                      // ... and on its own account on device 1
  CHECK(g_raised == 2);
  for (int i = 0; i < 3; ++i) CHECK(h0.run(a, 65536) && h1.run(a, 150000));
  CHECK(g_raised == 2);                         // once per handle
  CHECK(h0.run(b, 150000) && h0b.run(b, 50000) && h0.run(b, 150000));   // a smaller need lowers nothing
  CHECK(h0b.run(b, 48 * 1024 - 100));           // below 48 KB only without the static memory
  CHECK(h0.allow(b, 227 * 1024) == 9);          // dynamic and static together are past the device
  CHECK(h0.allow(b, 227 * 1024 - 4656) == 0);
  Handle h2{2, {}};
  g_fail = 1;
  CHECK(h2.allow(a, 65536) == 2);               // an error is reported, and not kept
  CHECK(h2.run(a, 65536));
  for (int r = 0; r < 2; ++r)                   // more kernels than the record holds
    for (int i = 2; i < 100; ++i) CHECK(h2.run(&kern[i], 60000));
  printf("ok\n");
  return 0;
}
"""


def test_limits_are_kept_per_handle(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2604_15645_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_no_limit_is_kept_per_process():
    """Every raised limit goes through the handle's record."""
    csrc = os.path.join(ROOT, "paper_2604_15645_gb300", "csrc")
    found = {f: open(os.path.join(csrc, f)).read().count("cudaFuncSetAttribute(")
             for f in sorted(os.listdir(csrc)) if f.endswith((".cu", ".cuh", ".h"))}
    assert {f: n for f, n in found.items() if n} == {"api.cu": 1}


SHARED = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "smem_limit.h"
#define CHECK(x) do { if (!(x)) { printf("failed: %s\n", #x); return 1; } } while (0)

int main() {
  static pinn::ContextLimits contexts;
  static int kern[96];
  pinn::SmemLimits* a = contexts.of(7);
  CHECK(a && contexts.of(8) && contexts.of(8) != a && contexts.of(7) == a);   // one record per context
  std::atomic<int> raised{0}, wrong{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 8; ++t)
    threads.emplace_back([&] {
      pinn::SmemLimits* mine = contexts.of(7);
      for (int r = 0; r < 200; ++r)
        for (int i = 0; i < 96; ++i)
          wrong += mine->allow(&kern[i], (size_t)(1000 + i), 0, 9, [&](size_t* limit) {
            ++raised;
            *limit = (size_t)(1000 + i);
            return 0;
          }) != 0;
    });
  for (auto& t : threads) t.join();
  CHECK(wrong == 0 && raised >= 96 && raised <= 8 * 96);
  const int before = raised;
  for (int i = 0; i < 96; ++i)   // what one handle raised serves the context's next one
    CHECK(contexts.of(7)->allow(&kern[i], 1000, 0, 9, [&](size_t*) { ++raised; return 2; }) == 0);
  CHECK(raised == before);
  CHECK(contexts.of(8)->allow(&kern[0], 1000, 0, 9, [&](size_t*) { return 2; }) == 2);   // not another context's
  int more = 0;
  for (uint64_t c = 100; c < 200; ++c) more += contexts.of(c) != nullptr;
  CHECK(more == 30 && contexts.of(7) == a);   // bounded; the known ones stay
  printf("ok\n");
  return 0;
}
"""


def test_handles_of_a_context_share_its_record(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "shared.cpp", tmp_path / "shared"
    src.write_text(SHARED)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2604_15645_gb300", "csrc"), str(src), "-o", str(exe)], check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
