"""The gather of host requests (csrc/host_pack.h) on its own: ragged requests, several jobs on one packer, and processes that may
start only some threads, or none (pthread_create is replaced by one that fails from a given call on)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <dlfcn.h>
#include <pthread.h>
#include "host_pack.h"

static int allowed = 1 << 30;
extern "C" int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) noexcept {
  if (allowed-- <= 0) return EAGAIN;
  using Fn = int (*)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*);
  static const Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "pthread_create"));
  return real(t, a, f, x);
}

int main(int argc, char** argv) {
  allowed = atoi(argv[1]);
  phyai::HostPacker packer;
  const size_t rows[] = {64, 512, 6};
  for (size_t row : rows) {
    const uint32_t lens[] = {9, 0, 1, 100, 33};
    const int planes = 7, batch = 5;
    size_t total = 0;
    for (uint32_t n : lens) total += n;
    std::vector<std::vector<uint8_t>> src(batch);
    std::vector<const void*> ptr(batch);
    for (int b = 0; b < batch; ++b) {
      src[b].resize((size_t)planes * lens[b] * row);
      for (size_t i = 0; i < src[b].size(); ++i) src[b][i] = (uint8_t)(i * 31 + b * 7 + 1);
      ptr[b] = src[b].data();
    }
    std::vector<uint8_t> dst((size_t)planes * total * row + 64, 0xee);
    if (!packer.start(dst.data(), ptr.data(), lens, batch, planes, row)) return 2;
    for (int n : {1, 4, planes}) packer.wait(n);
    const uint8_t* d = dst.data();
    for (int p = 0; p < planes; ++p)
      for (int b = 0; b < batch; ++b)
        for (size_t i = 0; i < (size_t)lens[b] * row; ++i)
          if (*d++ != src[b][(size_t)p * lens[b] * row + i]) return 3;
    for (int i = 0; i < 64; ++i)
      if (*d++ != 0xee) return 4;
  }
  puts("ok");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_pack")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2608_03682_b200", "csrc"), str(src), "-o", str(exe),
                    "-pthread", "-ldl"], check=True)
    return str(exe)


@pytest.mark.parametrize("threads", [100, 3, 1, 0])
def test_gather_with_any_number_of_threads(program, threads):
    r = subprocess.run([program, str(threads)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stderr)
