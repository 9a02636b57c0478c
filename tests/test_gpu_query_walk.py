"""The query along a walk that serves two rows, against the per-index query (gs_sketch_query_at), which
shares none of its path: every estimate bit-equal, for each number of rows the walk serves (3 and 4 only
where it prunes), ragged d, the smallest and a large number of columns; the pruning form (its estimate
internal) selects the same coordinates, with every unpruned estimate equal and every marker below the
k-th largest."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,c,d", [(3, 1 << 20, 4_194_304), (4, 1 << 19, 4_194_307), (5, 1 << 16, 4_200_001),
                                   (5, 1 << 21, 6_000_003), (6, 1 << 18, 4_200_002), (7, 1 << 18, 4_194_304),
                                   (8, 1 << 17, 4_300_001), (9, 1 << 18, 5_000_007)])
def test_query_walk(r, c, d):
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    k = 3000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r + d)
    x = torch.empty(d, device="cuda").normal_(0.0, 1e-3, generator=gen)
    x[torch.randint(0, d, (4 * k,), generator=gen, device="cuda")] *= 300
    sk = gs.gs_sketch_create(r, c, d % 1000 + r, 1)
    try:
        gs.gs_sketch_insert(sk, 0, x, d)
        gs.gs_sketch_merge_tree(sk, 1)
        ws = torch.empty(gs.gs_query_topk_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        idx = torch.empty(k, dtype=torch.int64, device="cuda")
        est = torch.empty(d, device="cuda")
        gs.gs_query_topk(sk, d, k, idx, est, ws)
        want = torch.empty(d, device="cuda")
        gs.gs_sketch_query_at(sk, torch.arange(d, device="cuda"), d, want)
        assert torch.equal(est, want)
        key = want.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
        top = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
        assert np.array_equal(idx.cpu().numpy(), top)
        idx2 = torch.empty_like(idx)
        gs.gs_query_topk(sk, d, k, idx2, None, ws)
        assert torch.equal(idx, idx2)
        inner = ws[: 4 * d].view(torch.float32).cpu().numpy().view(np.uint32)
        marker = (inner > 0x80000000) & (inner < 0x80000400)
        full = want.cpu().numpy().view(np.uint32)
        assert np.array_equal(inner[~marker], full[~marker])
        assert not marker.any() or key[marker].max() < key[top].min()
    finally:
        gs.gs_sketch_destroy(sk)
