"""Idle workspaces of a server's size buckets go back in time: after a second of real time whether
or not the server is stepped again, and at once for an allocation that would fail without them."""
import os
import subprocess
import sys
import time

import pytest

from paper_2311_04435_gb300 import api

pytestmark = pytest.mark.gpu


def _serve_one(srv, now=0.0):
    p = api.Params(32, 16, U=4.0, T=0.3, delta=0.5, prec="bf16x3")
    rid = srv.submit(p, api.AdamConfig(lr=0.01, grad_tol=1e-9, max_steps=2, seed=1))
    while any(srv.step(now)):
        now += 0.01
    assert srv.poll(rid, p.N) is not None
    return now


def test_manual_server_frees_without_further_steps():
    torch = pytest.importorskip("torch")
    torch.cuda.init()
    with api.Server(hbm_budget_bytes=64 << 30, max_slots=2, manual=True) as srv:
        free0 = torch.cuda.mem_get_info()[0]
        _serve_one(srv)
        kept = free0 - torch.cuda.mem_get_info()[0]
        assert kept > 1 << 30  # the bucket of 256 slots waits for another request
        time.sleep(2.0)
        assert free0 - torch.cuda.mem_get_info()[0] < kept // 8
        _serve_one(srv, 1.0)  # and is made anew


# cudaMalloc calls of 64 MB and more fail from arm() on until a cudaFree of such a block
_SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int armed;
void shim_arm(void) { armed = 1; }
static void* real_fn(const char* name) {
  void* fn = dlsym(RTLD_NEXT, name);
  if (!fn) {
    void* h = dlopen("libcudart.so.13", RTLD_NOLOAD | RTLD_LAZY);
    if (h) fn = dlsym(h, name);
  }
  return fn;
}
static void* big[256];
int cudaMalloc(void** p, size_t n) {
  int (*fn)(void**, size_t) = (int (*)(void**, size_t))real_fn("cudaMalloc");
  if (armed && n >= (64u << 20)) return 2; /* cudaErrorMemoryAllocation */
  const int err = fn(p, n);
  if (!err && n >= (64u << 20))
    for (int k = 0; k < 256; ++k)
      if (!big[k]) { big[k] = *p; break; }
  return err;
}
int cudaFree(void* p) {
  for (int k = 0; k < 256; ++k)
    if (p && big[k] == p) { big[k] = 0; armed = 0; }
  return ((int (*)(void*))real_fn("cudaFree"))(p);
}
"""

_CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
from paper_2311_04435_gb300 import api, inputs
shim = ctypes.CDLL(sys.argv[2])
p = api.Params(32, 16, U=4.0, T=0.3, delta=0.5, prec="bf16x3")
with api.Server(hbm_budget_bytes=64 << 30, max_slots=2, manual=True) as srv:
    srv.submit(p, api.AdamConfig(lr=0.01, grad_tol=1e-9, max_steps=2, seed=1))
    now = 0.0
    while any(srv.step(now)):
        now += 0.01
    shim.shim_arm()  # no memory left but what the server keeps for later
    with api.Context(p) as c:
        om, g = c.grad(inputs.seed_phi(1, p.N))
print("reclaimed ok")
"""


def test_failed_allocation_takes_idle_workspaces(tmp_path):
    src, shim = tmp_path / "shim.c", tmp_path / "libshim.so"
    src.write_text(_SHIM)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(shim), str(src), "-ldl"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _CHILD, root, str(shim)], capture_output=True,
                       text=True, timeout=300, env=dict(os.environ, LD_PRELOAD=str(shim)))
    assert r.returncode == 0 and "reclaimed ok" in r.stdout, r.stdout + r.stderr
