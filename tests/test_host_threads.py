"""The host loops of the mesh builder where threads or memory run out: a process that cannot start
threads builds the mesh all the same (no abort at the C entry point), and an exception of any part of
a parallel loop reaches the caller after the other parts have ended. No GPU is
visible to it: the mesh ends with the status of the failed device allocation, after all host work."""
import os
import subprocess

import pytest

SRC = r"""
#include <pthread.h>
#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <new>
#include "hostutil.h"

// a process in which no thread can be started after the first `allowed` ones
static std::atomic<int> allowed(-1);
using Create = int (*)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*);
#include <dlfcn.h>
extern "C" int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) {
  static const Create real = (Create)dlsym(RTLD_NEXT, "pthread_create");
  if (allowed.load() >= 0 && allowed.fetch_sub(1) <= 0) {
    allowed.store(0);
    return EAGAIN;
  }
  return real(t, a, f, x);
}

int main(int argc, char** argv) {
  allowed.store(atoi(argv[2]));
  if (argv[1][0] == 'm') {  // uniform octree of level 6
    const int l = 6, n = 1 << (3 * l);
    std::vector<uint32_t> a((size_t)3 * n);
    std::vector<uint8_t> lev((size_t)n, (uint8_t)l);
    for (int i = 0; i < n; ++i)
      for (int d = 0; d < 3; ++d)
        a[3 * (size_t)i + d] = (uint32_t)(chns::host::compact3((uint64_t)i >> d) << (CHNS_MAXD - l));
    const double ext[3] = {1.0, 1.0, 1.0};
    chns_mesh* m = nullptr;
    const int st = chns_mesh_create(a.data(), lev.data(), n, ext, nullptr, &m);
    printf("status %d\n", st);
    if (m) chns_mesh_destroy(m);
    return 0;
  }
  const int bad = atoi(argv[3]);
  std::atomic<int> ended(0);
  try {
    chns::host::parallel_parts(1000, 8, [&](int t, int64_t b, int64_t e) {
      if (t == bad) throw std::bad_alloc();
      ended += (int)(e - b);
    });
  } catch (const std::bad_alloc&) {
    printf("caught after %d\n", ended.load());
    return 0;
  }
  printf("all %d\n", ended.load());
}
"""


@pytest.fixture(scope="module")
def exe(root, tmp_path_factory):
    from paper_2107_05123_gb300 import build as b
    lib = b.build()
    d = tmp_path_factory.mktemp("threads")
    src, out = d / "threads.cu", d / "threads"
    src.write_text(SRC)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-Xcompiler", "-rdynamic", "-I", b.CSRC, "-I",
                    os.path.join(root, "include"), "-o", str(out), str(src), lib, "-Xlinker",
                    "-rpath", "-Xlinker", os.path.dirname(lib), "-Xcompiler", "-pthread", "-ldl"],
                   check=True, capture_output=True)
    return str(out)


def _run(exe, *args):
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stderr
    return r.stdout.strip()


@pytest.mark.parametrize("allowed", [0, 2])
def test_mesh_without_threads(exe, allowed):
    assert _run(exe, "mesh", allowed) == _run(exe, "mesh", -1)


@pytest.mark.parametrize("bad", [0, 3, 7])
@pytest.mark.parametrize("allowed", [-1, 0])
def test_exception_of_a_part(exe, allowed, bad):
    assert _run(exe, "parts", allowed, bad) == "caught after 875"
    assert _run(exe, "parts", allowed, -1) == "all 1000"
