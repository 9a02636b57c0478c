"""A kernel's dynamic shared memory limit belongs to all threads that launch it: one call must not lower it
between another call's setting and its launch.  A small library, preloaded into a child process, stands
before cudaFuncSetAttribute and compares the limits that the library sets for each kernel over calls of
different sizes: they have to be the same."""

import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
#include <string.h>
typedef int (*set_fn)(const void*, int, int);
int shim_kernels = 0, shim_changed = 0;
static const void* seen[256];
static int limit[256];
int cudaFuncSetAttribute(const void* kernel, int attr, int value) {
  Dl_info caller = {0};
  dladdr(__builtin_return_address(0), &caller);
  if (attr == 8 && caller.dli_fname && strstr(caller.dli_fname, "libgs_sketch")) {
    int n = 0;  /* cudaFuncAttributeMaxDynamicSharedMemorySize */
    while (n < shim_kernels && seen[n] != kernel) ++n;
    if (n < shim_kernels && limit[n] != value) ++shim_changed;
    if (n == shim_kernels && n < 256) seen[shim_kernels++] = kernel;
    limit[n & 255] = value;
  }
  void* lib = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  set_fn f = lib ? (set_fn)dlsym(lib, "cudaFuncSetAttribute") : 0;
  if (!f) abort();
  return f(kernel, attr, value);
}
"""

CHILD = r"""
import ctypes, sys
import torch
sys.path.insert(0, sys.argv[2])
import paper_2108_06004_gb300 as gs
gs.load_library()
shim = ctypes.CDLL(sys.argv[1])
for d, r, c in ((1000, 5, 64), (100_003, 5, 4096), (3 << 19, 5, 1 << 14), ((1 << 22) + 1, 5, 1 << 14),
                ((1 << 22) + 1, 5, 1 << 16), ((1 << 22) + 1, 12, 1 << 12), ((1 << 22) + 1, 12, 1 << 14)):
    k = 100
    sk = gs.gs_sketch_create(r, c, d, 1)
    u, e, g = (torch.randn(d, device="cuda") for _ in range(3))
    if c <= 4096:
        gs.gs_accumulate_insert_staged(sk, 0, [u], [e], [g], d, 0.9)
    else:
        gs.gs_accumulate_insert(sk, 0, [u], [e], [g], d, 0.9)
    gs.gs_sketch_merge_tree(sk, 1)
    ws = torch.empty(gs.gs_query_heavymix_workspace_size(d, k), dtype=torch.uint8, device="cuda")
    idx = torch.empty(k, dtype=torch.int64, device="cuda")
    gs.gs_query_topk(sk, d, k, idx, None, ws)
    gs.gs_query_heavymix(sk, d, k, 7, idx, None, None, ws)
    torch.cuda.synchronize()
    gs.gs_sketch_destroy(sk)
kernels, changed = (ctypes.c_int.in_dll(shim, n).value for n in ("shim_kernels", "shim_changed"))
assert kernels >= 4, "the selection, the query and the staged insert set a limit"
assert changed == 0, "a limit followed one call's sizes"
print("checked")
"""


def test_shared_memory_limits(tmp_path):
    gcc = shutil.which("gcc")
    if gcc is None:
        pytest.skip("no host compiler")
    (tmp_path / "shim.c").write_text(SHIM)
    (tmp_path / "child.py").write_text(CHILD)
    shim = str(tmp_path / "shim.so")
    subprocess.run([gcc, "-O1", "-shared", "-fPIC", str(tmp_path / "shim.c"), "-o", shim, "-ldl"], check=True)
    res = subprocess.run([sys.executable, str(tmp_path / "child.py"), shim, ROOT], env=dict(os.environ, LD_PRELOAD=shim),
                         capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and "checked" in res.stdout, res.stderr[-3000:]
