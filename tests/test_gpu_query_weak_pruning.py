"""The classified query where few coordinates settle early: k a large part of d, many rows, few columns.
Every CTA then evaluates all rows of four coordinates per lane; the selection, the estimates kept in the
workspace and the markers are those of the per-index query and the settle rule.  HEAVYMIX with thresholds
from far above the cells' noise to within it, where the classified query leaves the work to k_query."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests import gpu_harness as H  # noqa: E402

pytestmark = pytest.mark.gpu


def _sketch(gs, r, c, d, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.empty(d, device="cuda").normal_(0.0, 1e-3, generator=gen)
    sk = gs.gs_sketch_create(r, c, seed, 1)
    gs.gs_sketch_insert(sk, 0, x, d)
    gs.gs_sketch_merge_tree(sk, 1)
    return sk


@pytest.mark.parametrize("r,c", [(3, 64), (3, 1 << 18), (4, 1 << 16), (5, 1 << 14), (8, 1 << 12), (10, 1 << 10), (13, 1 << 14),
                                 (16, 1 << 14), (16, 128)])
@pytest.mark.parametrize("frac", [3, 40])
def test_topk(r, c, frac):
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    d = (1 << 22) + 4 * r + 3
    k = d // frac
    sk = _sketch(gs, r, c, d, 7 * r + frac)
    try:
        ws = torch.empty(gs.gs_query_topk_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        idx = torch.empty(k, dtype=torch.int64, device="cuda")
        want = torch.empty(d, device="cuda")
        gs.gs_query_topk(sk, d, k, idx, None, ws)
        gs.gs_sketch_query_at(sk, torch.arange(d, device="cuda"), d, want)
        full = want.cpu().numpy().view(np.uint32)
        key = full & np.uint32(0x7FFFFFFF)
        top = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
        assert np.array_equal(idx.cpu().numpy(), top)
        inner = ws[: 4 * d].view(torch.float32).cpu().numpy()
        marker, _ = H.pruned_rows(inner, r)
        assert np.array_equal(inner.view(np.uint32)[~marker], full[~marker])
        assert not marker.any() or key[marker].max() < key[top].min()
    finally:
        gs.gs_sketch_destroy(sk)


@pytest.mark.parametrize("r,c", [(3, 64), (4, 1 << 14), (5, 1 << 12), (9, 1 << 14), (13, 1 << 12), (16, 1 << 12)])
def test_heavymix(r, c):
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    d = (1 << 22) + 9
    sk = _sketch(gs, r, c, d, r)
    try:
        for k in (1, c // 8 + 1, c // 2, c, 4 * c, 64 * c):
            ws = torch.empty(gs.gs_query_heavymix_workspace_size(d, k), dtype=torch.uint8, device="cuda")
            full, inner = (torch.empty(k, dtype=torch.int64, device="cuda") for _ in range(2))
            est = torch.empty(d, device="cuda")
            gs.gs_query_heavymix(sk, d, k, 2**50 + 1, full, est, None, ws)
            gs.gs_query_heavymix(sk, d, k, 2**50 + 1, inner, None, None, ws)
            assert torch.equal(full, inner)
    finally:
        gs.gs_sketch_destroy(sk)
