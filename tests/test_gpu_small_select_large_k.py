"""Selections on either side of the line between the one-cluster selection and the kernels for long vectors
when k is large, against the exact top-k of the returned estimate; with a workspace and without, and
HEAVYMIX against its rule on the same estimate."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

ANY_K, LIMIT = 25 << 15, 3 << 19


@pytest.mark.parametrize("d,k", [(ANY_K, ANY_K // 2), (ANY_K, ANY_K), (ANY_K + 1, ANY_K // 100), (ANY_K + 1, ANY_K // 100 + 1),
                                 (ANY_K + 1, ANY_K + 1), (1 << 20, 10_485), (1 << 20, 10_486), (LIMIT, 15_728),
                                 (LIMIT, 15_729), (LIMIT, LIMIT)])
@pytest.mark.parametrize("kind", ["normal", "flat", "zero"])
def test_large_k(d, k, kind):
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    rng = np.random.default_rng(d + k)
    # "flat": magnitudes within a factor of 1.2, so that one level-1 bin holds nearly all of them
    x = {"normal": lambda: rng.standard_normal(d), "flat": lambda: rng.uniform(1.0, 1.2, d) * rng.choice([-1, 1], d),
         "zero": lambda: np.zeros(d)}[kind]().astype(np.float32)
    sk = gs.gs_sketch_create(*((1, 1 << 20) if kind == "flat" else (5, 1 << 14)), d, 1)
    try:
        gs.gs_sketch_insert(sk, 0, torch.from_numpy(x).cuda(), d)
        gs.gs_sketch_merge_tree(sk, 1)
        size = max(gs.gs_query_topk_workspace_size(d, k), gs.gs_query_heavymix_workspace_size(d, k))
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        est = torch.empty(d, device="cuda")
        l2 = torch.empty(1, dtype=torch.float64, device="cuda")
        got = [torch.full((k,), -1, dtype=torch.int64, device="cuda") for _ in range(3)]
        gs.gs_query_topk(sk, d, k, got[0], est, ws)
        gs.gs_query_topk_noalloc(sk, d, k, got[1], est)
        gs.gs_query_heavymix(sk, d, k, 99, got[2], est, l2, ws)
        key = est.cpu().numpy().view(np.uint32) & np.uint32(0x7FFFFFFF)
        want = np.sort(np.lexsort((np.arange(d), -key.astype(np.int64)))[:k])
        assert np.array_equal(got[0].cpu().numpy(), want)
        assert np.array_equal(got[1].cpu().numpy(), want)
        assert np.array_equal(got[2].cpu().numpy(), oracle.heavymix_select(est.cpu().numpy(), float(l2.item()), k, 99))
    finally:
        gs.gs_sketch_destroy(sk)
