"""The query along a walk, at shapes where the walk is in fact taken: tables too large for the classified
query and two rows that share a walk (at most one new cell per coordinate for both, by choose_pair in
csrc/chain_plan.h, evaluated here on the sketch's own coefficients).  Every number of rows that it serves,
in the pruning form and, from 5 rows on, with every estimate returned, against the per-index query."""

import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06004_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "chain_plan.h"
using namespace gs;
int main(int, char** v) {
  std::vector<Convergent> l[2];
  const uint32_t c = (uint32_t)atoll(v[3]);
  const int64_t d = atoll(v[4]), steps = std::min<int64_t>(64, d / (atoll(v[5]) * 2048));
  for (int j = 0; j < 2; ++j) l[j] = slow_strides(rotation_convergents(strtoull(v[1 + j], nullptr, 10), c), 4096);
  double best = 2.0;
  for (int f = 0; f < 2; ++f) best = std::min(best, choose_pair(l[f], l[1 - f], d, 8, steps).changes);
  std::printf("%.6f\n", best);
}
"""


@pytest.fixture(scope="module")
def changes(tmp_path_factory):
    """Bucket changes per coordinate of the best walk that serves the first two rows of a sketch."""
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    path = tmp_path_factory.mktemp("walk")
    (path / "walk.cpp").write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(path / "walk.cpp"), "-o", str(path / "walk")], check=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def of(a, c, d):
        args = [str(int(x)) for x in (a[0], a[1], c, d, sms)]
        return float(subprocess.run([str(path / "walk"), *args], check=True, capture_output=True, text=True).stdout)
    return of


@pytest.mark.parametrize("r,c,seed", [(3, 1 << 19, 53), (4, 1 << 19, 54), (5, 1 << 19, 55), (5, 1 << 21, 72), (6, 1 << 18, 56),
                                      (7, 1 << 18, 57), (8, 1 << 18, 58), (9, 1 << 18, 59)])
def test_walk_taken(changes, r, c, seed):
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    d, k = 12_000_003, 9000
    assert (r // 2 + 1) * c // 4 > 192 << 10, "the classified query serves this table"
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r)
    x = torch.empty(d, device="cuda").normal_(0.0, 1e-3, generator=gen)
    x[torch.randint(0, d, (4 * k,), generator=gen, device="cuda")] *= 300
    sk = gs.gs_sketch_create(r, c, seed, 1)
    try:
        assert changes(gs.gs_sketch_coefficients(sk)[0], c, d) <= 1.0, "no walk serves these rows: choose another seed"
        gs.gs_sketch_insert(sk, 0, x, d)
        gs.gs_sketch_merge_tree(sk, 1)
        ws = torch.empty(gs.gs_query_topk_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        want = torch.empty(d, device="cuda")
        gs.gs_sketch_query_at(sk, torch.arange(d, device="cuda"), d, want)
        full = want.cpu().numpy().view(np.uint32)
        key = full & np.uint32(0x7FFFFFFF)
        top = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
        idx = torch.empty(k, dtype=torch.int64, device="cuda")
        gs.gs_query_topk(sk, d, k, idx, None, ws)
        assert np.array_equal(idx.cpu().numpy(), top)
        inner = ws[: 4 * d].view(torch.float32).cpu().numpy().view(np.uint32)
        marker = (inner > 0x80000000) & (inner < 0x80000400)
        assert marker.mean() > 0.5, "rows were not skipped"
        assert np.array_equal(inner[~marker], full[~marker])
        assert key[marker].max() < key[top].min()
        if r >= 5:
            est = torch.empty(d, device="cuda")
            idx.fill_(-1)
            gs.gs_query_topk(sk, d, k, idx, est, ws)
            assert torch.equal(est, want)
            assert np.array_equal(idx.cpu().numpy(), top)
    finally:
        gs.gs_sketch_destroy(sk)


@pytest.mark.parametrize("r,c", [(6, 1 << 18), (9, 1 << 19)])
def test_large_k(r, c):
    """A pruning query of a short vector on either side of the k from which it does not walk."""
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    d = 4_200_001
    gen = torch.Generator(device="cuda")
    gen.manual_seed(c + r)
    x = torch.empty(d, device="cuda").normal_(0.0, 1e-3, generator=gen)
    sk = gs.gs_sketch_create(r, c, 50 + r, 1)
    try:
        gs.gs_sketch_insert(sk, 0, x, d)
        gs.gs_sketch_merge_tree(sk, 1)
        want = torch.empty(d, device="cuda")
        gs.gs_sketch_query_at(sk, torch.arange(d, device="cuda"), d, want)
        key = want.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
        order = np.lexsort((np.arange(d), -key.astype(np.int64)))
        for k in (d // 200, d // 200 + 1, d // 3):
            ws = torch.empty(gs.gs_query_topk_workspace_size(d, k), dtype=torch.uint8, device="cuda")
            idx = torch.empty(k, dtype=torch.int64, device="cuda")
            gs.gs_query_topk(sk, d, k, idx, None, ws)
            assert np.array_equal(idx.cpu().numpy(), np.sort(order[:k]))
    finally:
        gs.gs_sketch_destroy(sk)
