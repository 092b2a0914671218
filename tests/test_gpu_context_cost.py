"""What creating a context costs: contexts that never take the nested elimination upload no tables
for it, and those whose densities of states do get them then; the memory that a context takes is
what sca_workspace_bytes says, which the server's admission goes by."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# counts the runtime's copies and stream creations made through the dynamic linker
_SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static long copies, streams;
static unsigned long long allocated;
unsigned long long shim_allocated(void) { return allocated; }
int cudaMalloc(void** p, size_t n);
long shim_copies(void) { return copies; }
long shim_streams(void) { return streams; }
static void* real_fn(const char* name) {
  void* fn = dlsym(RTLD_NEXT, name);
  if (!fn) {
    void* h = dlopen("libcudart.so.13", RTLD_NOLOAD | RTLD_LAZY);
    if (h) fn = dlsym(h, name);
  }
  return fn;
}
int cudaMalloc(void** p, size_t n) {
  const int err = ((int (*)(void**, size_t))real_fn("cudaMalloc"))(p, n);
  if (!err) allocated += n;
  return err;
}
int cudaMemcpy(void* d, const void* s, size_t n, int k) {
  ++copies;
  return ((int (*)(void*, const void*, size_t, int))real_fn("cudaMemcpy"))(d, s, n, k);
}
int cudaStreamCreateWithFlags(void** s, unsigned f) {
  ++streams;
  return ((int (*)(void**, unsigned))real_fn("cudaStreamCreateWithFlags"))(s, f);
}
int cudaStreamCreateWithPriority(void** s, unsigned f, int p) {
  ++streams;
  return ((int (*)(void**, unsigned, int))real_fn("cudaStreamCreateWithPriority"))(s, f, p);
}
"""

_CHILD = r"""
import ctypes, os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_2311_04435_gb300 import api, inputs
shim = ctypes.CDLL(sys.argv[2])
shim.shim_copies.restype = shim.shim_streams.restype = ctypes.c_long

def create(**kw):
    c0, s0 = shim.shim_copies(), shim.shim_streams()
    c = api.Context(api.Params(16, 100, U=4.0, delta=0.5, **kw))
    return c, shim.shim_copies() - c0, shim.shim_streams() - s0

phi, w = inputs.seed_phi(1, 256), np.linspace(-3, 3, 7)
c, copies, _ = create(T=0.2, prec="fp64")
rho = c.dos(phi, w, 0.1)
c.close()
assert copies == 1, copies  # the tables, in one piece
# 200 blocks: its own, the side stream and one for the second half (float64: no tensor-core path)
c, copies, streams = create(T=0.2, prec="fp64")
c.close()
assert streams == 3, streams
c, copies, streams = create(T=0.2, prec="bf16x3")
c.close()
assert (copies, streams) == (1, 3), (copies, streams)
# below the line: none, until a density of states above it
c, copies, _ = create(T=0.005, prec="fp64")
assert copies == 0, copies
c.blocks(phi)
assert np.array_equal(c.dos(phi, w, 0.1), rho)
c.close()
os.environ["SCA_REFINE_LOWER"] = "1"
c, copies, _ = create(T=0.2, prec="bf16x3")
assert copies == 0, copies
c.close()
print("context cost ok")
"""


_MEMORY_CHILD = r"""
import ctypes, os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_2311_04435_gb300 import api, inputs
shim = ctypes.CDLL(sys.argv[2])
shim.shim_allocated.restype = ctypes.c_ulonglong
api.Context(api.Params(4, 1, U=4.0, T=0.1)).close()
for resident in (None, "3"):
    if resident:
        os.environ["SCA_MAX_BLOCKS_RESIDENT"] = resident
    for L, nw, T, prec in ((4, 64, 0.1, "fp64"), (6, 40, 0.012, "fp64"), (8, 40, 0.05, "fp64"),
                           (8, 20, 0.02, "fp32"), (14, 20, 0.1, "fp32"), (16, 30, 0.005, "bf16x3"),
                           (20, 100, 0.1, "3xtf32"), (40, 8, 0.1, "bf16x3"), (64, 2, 0.1, "bf16x3")):
        p = api.Params(L, nw, U=4.0, T=T, delta=0.5, prec=prec)
        said, a0 = api.workspace_bytes(p), shim.shim_allocated()
        with api.Context(p) as c:
            c.set_site_energy(np.zeros(p.N))
            c.blocks(inputs.seed_phi(1, p.N))
            c.dos(inputs.seed_phi(1, p.N), np.array([0.1, 0.2]), 0.2)
        took = shim.shim_allocated() - a0
        assert 0 <= said - took <= 64, (L, nw, T, prec, resident, said, took)
print("context cost ok")
"""


@pytest.mark.parametrize("child", [_CHILD, _MEMORY_CHILD], ids=["tables", "memory"])
def test_cost_of_a_context(tmp_path, child):
    src, shim = tmp_path / "shim.c", tmp_path / "libshim.so"
    src.write_text(_SHIM)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(shim), str(src), "-ldl"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", child, root, str(shim)], capture_output=True,
                       text=True, timeout=300, env=dict(os.environ, LD_PRELOAD=str(shim)))
    assert r.returncode == 0 and "context cost ok" in r.stdout, r.stdout + r.stderr
