"""The one-cluster selection (d up to 1.5 * 2^20) against the exact top-k of the returned estimate:
lengths around a bitmap word, a CTA's share and the path's limit, more candidates than a CTA's list
holds, and a plateau of equal keys; with a workspace and without."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LIMIT = 3 << 19


@pytest.fixture(scope="module")
def gs():
    import paper_2108_06004_gb300 as lib
    lib.load_library()
    torch.cuda.set_device(0)
    return lib


@pytest.mark.parametrize("d,k,c,kind", [(1, 1, 64, "normal"), (31, 31, 64, "normal"), (33, 5, 64, "normal"),
                                        (511, 17, 64, "normal"), (513, 400, 64, "normal"), (65_537, 1, 4096, "normal"),
                                        (1_000_003, 300_000, 1 << 20, "flat"), (700_001, 12_345, 4096, "zero"),
                                        (LIMIT, 1500, 1 << 14, "normal"), (LIMIT + 1, 1500, 1 << 14, "normal")])
def test_small_selection(gs, d, k, c, kind):
    rng = np.random.default_rng(d + k)
    # "flat": magnitudes within a factor of 1.2, so that one level-1 bin holds nearly all of them
    x = {"normal": lambda: rng.standard_normal(d), "flat": lambda: rng.uniform(1.0, 1.2, d) * rng.choice([-1, 1], d),
         "zero": lambda: np.zeros(d)}[kind]().astype(np.float32)
    r = 1 if kind == "flat" else 5
    sk = gs.gs_sketch_create(r, c, d, 1)
    try:
        gs.gs_sketch_insert(sk, 0, torch.from_numpy(x).cuda(), d)
        gs.gs_sketch_merge_tree(sk, 1)
        ws = torch.empty(gs.gs_query_topk_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        est = torch.empty(d, device="cuda")
        for noalloc in (False, True):
            idx = torch.full((k,), -1, dtype=torch.int64, device="cuda")
            if noalloc:
                gs.gs_query_topk_noalloc(sk, d, k, idx, est)
            else:
                gs.gs_query_topk(sk, d, k, idx, est, ws)
            key = est.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
            want = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
            assert np.array_equal(idx.cpu().numpy(), want)
    finally:
        gs.gs_sketch_destroy(sk)
