"""The chained insert (c a power of two) against the CPU oracle where its walk has edges: lengths
around a CTA, around the shortest stride and with several segments, one column, every cell width."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

REL = 1e-5  # of a cell's sum of |contributions|, the bar of every sketch cell


@pytest.fixture(scope="module")
def gs():
    import paper_2108_06004_gb300 as lib
    lib.load_library()
    torch.cuda.set_device(0)
    return lib


def _table(gs, sk, worker, r, c):
    buf = np.empty(r * c, dtype=np.float32)
    gs.gs_sketch_copy_to_host(sk, worker, buf)
    return buf.reshape(r, c).astype(np.float64)


@pytest.mark.parametrize("P,W,r,c", [(1, 1, 5, 4096), (2, 2, 3, 1), (3, 4, 1, 1 << 16), (7, 8, 4, 2), (16, 16, 2, 256)])
@pytest.mark.parametrize("d", [1, 3, 255, 256, 257, 4095, 4096, 4097, 300_001])
def test_chained_insert_edges(gs, P, W, r, c, d):
    seed = d + 31 * W
    rng = np.random.default_rng(seed)
    coeffs = oracle.derive_coefficients(r, seed)
    xs = [(rng.standard_normal(d) * 10.0 ** rng.integers(-6, 1, d)).astype(np.float32) for _ in range(P)]
    want = [oracle.sketch(x, coeffs, c) for x in xs]
    dev = [torch.from_numpy(x).cuda() for x in xs]
    zero = [torch.zeros(d, device="cuda") for _ in range(2 * P)]
    sk = gs.gs_sketch_create(r, c, seed, P, W)
    try:
        # one vector at a time, then the group at once (momentum and error zero: e becomes x)
        for p in range(P):
            gs.gs_sketch_insert(sk, p, dev[p], d)
        single = [_table(gs, sk, p, r, c) for p in range(P)]
        gs.gs_sketch_zero(sk)
        gs.gs_accumulate_insert(sk, 0, zero[:P], zero[P:], dev, d, 0.9)
        group = [_table(gs, sk, p, r, c) for p in range(P)]
        for p, (T, A) in enumerate(want):
            assert np.all(np.abs(single[p] - T) <= REL * A), f"worker {p}, inserted alone"
            assert np.all(np.abs(group[p] - T) <= REL * A), f"worker {p}, inserted with its group"
            assert np.array_equal(zero[P + p].cpu().numpy(), xs[p])
    finally:
        gs.gs_sketch_destroy(sk)
