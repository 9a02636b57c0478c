"""HEAVYMIX on estimates that share their bits with the pruning markers: small negative subnormals.
Cell additions in global memory flush subnormals, the merge does not, so two workers whose values
nearly cancel leave one.  With the threshold at that scale the coordinate belongs to H, whether the
estimate is returned or stays in the workspace."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -149  # the smallest positive fp32


@pytest.mark.parametrize("r,c", [(3, 1 << 16), (4, 1 << 16), (5, 1 << 16), (5, 1 << 19), (7, 1 << 16)])
@pytest.mark.parametrize("units,k", [((5,), 1), ((-5,), 1), ((1, 1023, -7), 3), ((1024, 133), 2)])
def test_heavymix_subnormal_estimates(r, c, units, k):
    """units: the merged values at a few coordinates, in multiples of -2^-149."""
    import paper_2108_06004_gb300 as gs
    gs.load_library()
    d, seed, fill_seed = (1 << 22) + 5, 31 + r, 2**40 + 9
    at = np.array([123_457, 2_000_003, d - 1])[:len(units)]
    x = [torch.zeros(d, device="cuda") for _ in range(2)]
    for i, n in zip(at, units):
        big = 2.0 ** -126 + abs(n) * TINY
        x[0][i], x[1][i] = (2.0 ** -126, -big) if n > 0 else (big, -(2.0 ** -126))
    sk = gs.gs_sketch_create(r, c, seed, 2)
    try:
        for p in range(2):
            gs.gs_sketch_insert(sk, p, x[p], d)
        gs.gs_sketch_merge_tree(sk, 2)
        ws = torch.empty(gs.gs_query_heavymix_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        l2 = torch.empty(1, dtype=torch.float64, device="cuda")
        est = torch.empty(d, device="cuda")
        full, inner = (torch.empty(k, dtype=torch.int64, device="cuda") for _ in range(2))
        gs.gs_query_heavymix(sk, d, k, fill_seed, full, est, l2, ws)
        gs.gs_query_heavymix(sk, d, k, fill_seed, inner, None, l2, ws)
        e = est.cpu().numpy()
        assert np.array_equal(e[at], np.array(units) * np.float64(-TINY)), "the estimates are those planted"
        want = oracle.heavymix_select(e, float(l2.item()), k, fill_seed)
        assert np.array_equal(full.cpu().numpy(), want)
        assert np.array_equal(inner.cpu().numpy(), want)
    finally:
        gs.gs_sketch_destroy(sk)
