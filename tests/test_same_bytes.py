"""The threaded comparison of pointings (same_bytes.cuh), compiled by itself: what it finds, and that it
neither throws nor ends the process where a thread cannot be made (C callers cannot catch)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>
#include "same_bytes.cuh"

static int g_fail_at = -1, g_count = 0;      // the allocation that fails, from the mark on
void* operator new(std::size_t n) {
  if (g_fail_at >= 0 && g_count++ >= g_fail_at) throw std::bad_alloc();
  if (void* p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

int main() {
  for (std::size_t n : {std::size_t(0), std::size_t(1), std::size_t(1000), std::size_t(1) << 20,
                        (std::size_t(2) << 20) + 3, (std::size_t(5) << 20) + 7}) {
    std::vector<unsigned char> a(n + 1, 7), b(n + 1, 7);
    std::vector<std::size_t> at = {0, n / 4, n / 3, n / 2, 3 * n / 4, n ? n - 1 : 0};
    for (int fail : {-1, 0, 1, 2, 3}) {
      g_count = 0, g_fail_at = fail;
      bool ok = fftbf::same_bytes(a.data(), b.data(), n);
      for (std::size_t k : at) {
        if (k >= n) continue;
        b[k] ^= 1;
        g_count = 0;
        ok = ok && !fftbf::same_bytes(a.data(), b.data(), n);
        b[k] ^= 1;
      }
      g_fail_at = -1;
      if (!ok) { std::printf("wrong at %zu bytes, failing allocation %d\n", n, fail); return 1; }
    }
  }
  return 0;
}
"""


def test_same_bytes_without_threads_or_memory(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    inc = os.path.join(ROOT, "paper_1710_08591_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
