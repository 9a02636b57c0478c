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


@pytest.mark.parametrize("P,W,r,c,offset", [(1, 1, 3, 1 << 15, 0), (2, 2, 4, 1 << 15, 0), (3, 4, 3, 1 << 14, 1),
                                            (7, 8, 6, 1 << 15, 0), (8, 8, 2, 1 << 21, 0), (11, 16, 3, 64, 0)])
def test_accumulate_walking_chains(gs, P, W, r, c, offset):
    """The accumulate pass that walks chains (from d = 2^22 on), with ragged d, lanes without a worker,
    vectors off the 16-byte boundary, and rows beyond L2: momentum and error bit-exact, every cell
    within 1e-5 of its magnitude.  The vectors are zero but for 200,000 coordinates, the last among
    them, so that the oracle's sketch is quick."""
    d, rho, seed = (1 << 22) + 3, 0.9, 7 * W + r
    rng = np.random.default_rng(seed)
    coeffs = oracle.derive_coefficients(r, seed)
    at = np.unique(np.concatenate([rng.integers(0, d, 200_000), [0, d - 4, d - 3, d - 1]]))
    mk = lambda: (rng.standard_normal(at.size) * 1e-2).astype(np.float32)  # noqa: E731
    bufs = [[torch.zeros(d + 4, device="cuda") for _ in range(3)] for _ in range(P)]
    views = [[b[offset:offset + d] for b in trio] for trio in bufs]
    vals = [[mk() for _ in range(3)] for _ in range(P)]
    dev_at = torch.from_numpy(at).cuda()
    for v, x in zip(views, vals):
        for a, b in zip(v, x):
            a[dev_at] = torch.from_numpy(b).cuda()
    sk = gs.gs_sketch_create(r, c, seed, P, W)
    try:
        gs.gs_accumulate_insert(sk, 0, [v[0] for v in views], [v[1] for v in views], [v[2] for v in views], d, rho)
        for p in range(P):
            u, e = oracle.accumulate(*vals[p], rho)
            assert np.array_equal(views[p][0][dev_at].cpu().numpy().view(np.uint32), u.view(np.uint32))
            assert np.array_equal(views[p][1][dev_at].cpu().numpy().view(np.uint32), e.view(np.uint32))
            assert int(torch.count_nonzero(bufs[p][0])) == np.count_nonzero(u)
            assert int(torch.count_nonzero(bufs[p][1])) == np.count_nonzero(e)
            T, A = oracle.sketch(e, coeffs, c, idx=at)
            assert np.all(np.abs(_table(gs, sk, p, r, c) - T) <= REL * A), f"worker {p}"
    finally:
        gs.gs_sketch_destroy(sk)
