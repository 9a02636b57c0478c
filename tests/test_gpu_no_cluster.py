"""Short selections where the device cannot hold the one-cluster selection.  A small library, preloaded
into a child process, stands before two calls of the CUDA runtime and refuses the cluster, as a partition
with too few SMs does: every call has to give the same selection by the kernels for long vectors."""

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
typedef int (*max_fn)(int*, const void*, const void*);
int shim_asked = 0;
static void* real(const char* name) {
  void* lib = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  void* f = lib ? dlsym(lib, name) : 0;
  if (!f) abort();
  return f;
}
static int refuse(const char* at) { return getenv("NO_CLUSTER") && !strcmp(getenv("NO_CLUSTER"), at); }
int cudaFuncSetAttribute(const void* kernel, int attr, int value) {
  if (attr == 14 && refuse("attribute")) {  /* cudaFuncAttributeNonPortableClusterSizeAllowed */
    ++shim_asked;
    return 801;                  /* cudaErrorNotSupported */
  }
  return ((set_fn)real("cudaFuncSetAttribute"))(kernel, attr, value);
}
int cudaOccupancyMaxActiveClusters(int* n, const void* kernel, const void* config) {
  if (refuse("occupancy")) {
    ++shim_asked;
    *n = 0;
    return 0;
  }
  return ((max_fn)real("cudaOccupancyMaxActiveClusters"))(n, kernel, config);
}
"""

CHILD = r"""
import ctypes, os, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[2])
import oracle
import paper_2108_06004_gb300 as gs
gs.load_library()
shim = ctypes.CDLL(sys.argv[1])

def check(d, k, r, c, kind):
    rng = np.random.default_rng(d + k)
    x = (np.zeros(d) if kind == "zero" else rng.standard_normal(d)).astype(np.float32)
    sk = gs.gs_sketch_create(r, c, d, 1)
    g = torch.from_numpy(x).cuda()
    gs.gs_sketch_insert(sk, 0, g, d)
    gs.gs_sketch_merge_tree(sk, 1)
    size = max(gs.gs_query_heavymix_workspace_size(d, k), gs.gs_step_workspace_size(d, k))
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    est = torch.empty(d, device="cuda")
    l2 = torch.empty(1, dtype=torch.float64, device="cuda")
    got = [torch.full((k,), -1, dtype=torch.int64, device="cuda") for _ in range(5)]
    gs.gs_query_topk(sk, d, k, got[0], est, ws)
    gs.gs_query_topk(sk, d, k, got[1], None, ws)
    gs.gs_query_topk_noalloc(sk, d, k, got[2], est)
    gs.gs_query_heavymix(sk, d, k, 77, got[3], est, l2, ws)
    key = est.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
    want = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
    for i in got[:3]:
        assert np.array_equal(i.cpu().numpy(), want), (d, k, kind)
    assert np.array_equal(got[3].cpu().numpy(), oracle.heavymix_select(est.cpu().numpy(), float(l2.item()), k, 77))
    # a captured step selects from the same sums
    u, e = torch.zeros(d, device="cuda"), torch.zeros(d, device="cuda")
    vals = torch.empty(k, device="cuda")
    plan = gs.gs_step_plan_create(sk, [u], [e], [g], d, 0.9, k, got[4], vals, est, None, 0.0, ws)
    gs.gs_plan_launch(plan)
    key = est.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
    want = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
    assert np.array_equal(got[4].cpu().numpy(), want)
    gs.gs_plan_destroy(plan)
    gs.gs_sketch_destroy(sk)

for case in ((1, 1, 5, 64, "normal"), (1000, 999, 3, 64, "normal"), (100_003, 100, 5, 4096, "normal"),
             (300_001, 777, 4, 3001, "normal"), (700_001, 9_999, 5, 4096, "zero"),
             (3 << 19, 1500, 5, 1 << 14, "normal")):
    check(*case)
torch.cuda.synchronize()
asked = ctypes.c_int.in_dll(shim, "shim_asked").value
assert (asked > 0) == ("NO_CLUSTER" in os.environ), "the refusal was not met"
print("checked")
"""


@pytest.mark.parametrize("refused_at", [None, "attribute", "occupancy"])
def test_short_selection(tmp_path, refused_at):
    gcc = shutil.which("gcc")
    if gcc is None:
        pytest.skip("no host compiler")
    (tmp_path / "shim.c").write_text(SHIM)
    (tmp_path / "child.py").write_text(CHILD)
    shim = str(tmp_path / "shim.so")
    subprocess.run([gcc, "-O1", "-shared", "-fPIC", str(tmp_path / "shim.c"), "-o", shim, "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=shim)
    env.pop("NO_CLUSTER", None)
    if refused_at:
        env["NO_CLUSTER"] = refused_at
    res = subprocess.run([sys.executable, str(tmp_path / "child.py"), shim, ROOT], env=env, capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0 and "checked" in res.stdout, res.stderr[-3000:]
