"""A host-side fake of the CUDA allocation calls for tests of what the library
does without memory: a preloaded shim that passes them on while the bytes held
through it stay within a budget, and otherwise returns
cudaErrorMemoryAllocation without calling CUDA.  run(script) runs Python code
in a child process with the shim loaded as `fake`:
fake_budget(bytes) sets the budget over what is held at that moment (< 0: none),
fake_largest(bytes, k) the largest single allocation from a memory pool (< 0:
any) after k more that are larger,
fake_peak(1) returns the most held since the last such call and starts anew,
fake_refused() the number of refusals; fake_free(bytes) what cudaMemGetInfo
reports as free (< 0: the truth)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <pthread.h>
#include <stdlib.h>

enum { SLOTS = 1 << 16, NOMEM = 2 };
static struct { void* p; size_t n; } slot[SLOTS];
static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static long long held, peak, budget = -1, largest = -1, over, refused;

static int room(size_t n, int pool) {
  int ok;
  pthread_mutex_lock(&mu);
  ok = budget < 0 || held + (long long)n <= budget;
  if (ok && pool && largest >= 0 && (long long)n > largest) ok = over-- > 0;
  if (!ok) ++refused;
  pthread_mutex_unlock(&mu);
  return ok;
}
static void add(void* p, size_t n) {
  size_t h = ((size_t)p >> 8) % SLOTS;
  pthread_mutex_lock(&mu);
  for (int i = 0; i < SLOTS; ++i, h = (h + 1) % SLOTS)
    if (!slot[h].p) { slot[h].p = p; slot[h].n = n; held += (long long)n; break; }
  if (held > peak) peak = held;
  pthread_mutex_unlock(&mu);
}
static void drop(void* p) {
  pthread_mutex_lock(&mu);
  for (int h = 0; p && h < SLOTS; ++h)
    if (slot[h].p == p) { slot[h].p = 0; held -= (long long)slot[h].n; break; }
  pthread_mutex_unlock(&mu);
}

int cudaMalloc(void** p, size_t n) {
  static int (*f)(void**, size_t);
  if (!f) f = dlsym(RTLD_NEXT, "cudaMalloc");
  if (!room(n, 0)) return NOMEM;
  int e = f(p, n);
  if (!e) add(*p, n);
  return e;
}
int cudaFree(void* p) {
  static int (*f)(void*);
  if (!f) f = dlsym(RTLD_NEXT, "cudaFree");
  drop(p);
  return f(p);
}
int cudaMallocFromPoolAsync(void** p, size_t n, void* pool, void* st) {
  static int (*f)(void**, size_t, void*, void*);
  if (!f) f = dlsym(RTLD_NEXT, "cudaMallocFromPoolAsync");
  if (!room(n, 1)) return NOMEM;
  int e = f(p, n, pool, st);
  if (!e) add(*p, n);
  return e;
}
int cudaFreeAsync(void* p, void* st) {
  static int (*f)(void*, void*);
  if (!f) f = dlsym(RTLD_NEXT, "cudaFreeAsync");
  drop(p);
  return f(p, st);
}

static long long free_bytes = -1;
int cudaMemGetInfo(size_t* fr, size_t* tot) {
  static int (*f)(size_t*, size_t*);
  if (!f) f = dlsym(RTLD_NEXT, "cudaMemGetInfo");
  int e = f(fr, tot);
  if (!e && free_bytes >= 0) *fr = (size_t)free_bytes;
  return e;
}

void fake_free(long long n) { free_bytes = n; }
void fake_budget(long long n) {
  pthread_mutex_lock(&mu);
  budget = n < 0 ? -1 : held + n;
  pthread_mutex_unlock(&mu);
}
void fake_largest(long long n, long long k) {
  largest = n;
  over = k;
}
long long fake_peak(int reset) {
  pthread_mutex_lock(&mu);
  long long r = peak;
  if (reset) peak = held;
  pthread_mutex_unlock(&mu);
  return r;
}
long long fake_held(void) { return held; }
long long fake_refused(void) { return refused; }
"""

HEAD = r"""
import ctypes, os, sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
fake = ctypes.CDLL({shim!r})
fake.fake_budget.argtypes = fake.fake_free.argtypes = [ctypes.c_longlong]
fake.fake_largest.argtypes = [ctypes.c_longlong] * 2
for f in ("fake_peak", "fake_held", "fake_refused"):
    getattr(fake, f).restype = ctypes.c_longlong
import numpy as np, torch
import gpu_util as gu, workloads as w
from paper_1810_04125_gb300 import build, hss
build.build()
"""


def run(script, tmp_path, timeout=600):
    src, shim = os.path.join(tmp_path, "fake.c"), os.path.join(tmp_path, "fake.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", shim, src, "-ldl", "-lpthread"], check=True)
    p = subprocess.run([sys.executable, "-c", HEAD.format(root=ROOT, shim=shim) + script], capture_output=True, text=True,
                       timeout=timeout, env=dict(os.environ, LD_PRELOAD=shim))
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout
