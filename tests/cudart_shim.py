"""A stand-in for single CUDA runtime calls, preloaded into a child process:
it makes the allocation of one size fail, and keeps a list of the kernel
attributes that were set."""
import os
import subprocess
import sys

SOURCE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
static void* real(const char* name) {
  void* lib = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  void* f = lib ? dlsym(lib, name) : NULL;
  if (!f) abort();
  return f;
}
int cudaMalloc(void** p, size_t n) {
  const char* e = getenv("SHIM_FAIL_BYTES");
  if (e && strtoull(e, NULL, 10) == n) n = (size_t)1 << 60; /* the runtime refuses it */
  return ((int (*)(void**, size_t))real("cudaMalloc"))(p, n);
}
int cudaFuncSetAttribute(const void* f, int attr, int value) {
  const char* e = getenv("SHIM_ATTR_LOG");
  FILE* log = e ? fopen(e, "a") : NULL;
  if (log) {
    fprintf(log, "%p %d %d\n", f, attr, value);
    fclose(log);
  }
  return ((int (*)(const void*, int, int))real("cudaFuncSetAttribute"))(f, attr, value);
}
"""


def run(tmp_path, code, **env):
    """Runs the Python source `code` in a child with the stand-in and `env`; its standard output."""
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=root, **env)
    r = subprocess.run([sys.executable, "-c", code], env=env, cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
