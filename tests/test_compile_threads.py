"""Compiling a mechanism's launch configurations where the process can start no further thread."""
import os
import subprocess

from tests import emulated
from tests.conftest import GOLDEN

MAIN = r"""
#include <pthread.h>
static bool none = false;
extern "C" int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) {
  static auto real = (int (*)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*))dlsym(RTLD_NEXT, "pthread_create");
  return none ? EAGAIN : real(t, a, f, x);
}
int main(int, char** v) {
  chem_mech m;
  if (read_spec(v[1], &m.data)) return 2;
  m.cache_dir = v[2];
  const std::vector<std::pair<int, int>> cfg = {{32, 32}, {16, 64}};
  auto a = build_cubins(&m, cfg, false);
  none = true;  // the second time from the cache
  auto b = build_cubins(&m, cfg, false);
  return a == b && !a[0].empty() && !a[1].empty() ? 0 : 3;
}
"""


def test_no_thread_to_be_had(tmp_path):
    exe = emulated.host_program(tmp_path, MAIN, flags=("-D_GNU_SOURCE",))
    r = subprocess.run([exe, os.path.join(GOLDEN, "tiny_hon7.mech"), str(tmp_path)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
