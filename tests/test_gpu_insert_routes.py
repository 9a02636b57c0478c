"""Inserts of vectors of middling length (c a power of two), where the expected savings of a row's chains
decide whether it goes along them or by one reduction per coordinate: shapes on either side of each line
(number of rows, columns, workers per cell, length), tables beyond one pass, groups with a lane missing
and vectors off the 16-byte boundary, against the CPU oracle.  The vectors are zero but for a few
thousand coordinates, so that the oracle's sketch is quick."""

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


def _sparse(rng, d, n, count):
    at = np.unique(np.concatenate([rng.integers(0, d, n), [0, d - 1, d // 2, min(65_535, d - 1)]]))
    return at, [(rng.standard_normal(at.size) * 1e-2).astype(np.float32) for _ in range(count)]


def _check(gs, sk, worker, r, c, coeffs, at, x, what):
    buf = np.empty(r * c, dtype=np.float32)
    gs.gs_sketch_copy_to_host(sk, worker, buf)
    T, A = oracle.sketch(x, coeffs, c, idx=at)
    assert np.all(np.abs(buf.reshape(r, c).astype(np.float64) - T) <= REL * A), what


@pytest.mark.parametrize("d", [33_001, 65_535, 65_536, 100_003, 230_001, 420_001, 1_400_001])
@pytest.mark.parametrize("W,r,c", [(1, 1, 256), (1, 1, 1 << 19), (2, 5, 1 << 14), (4, 3, 1 << 21), (16, 9, 1)])
def test_single_inserts(gs, W, r, c, d):
    rng = np.random.default_rng(d + r)
    coeffs = oracle.derive_coefficients(r, d + W)
    at, (x,) = _sparse(rng, d, 20_000, 1)
    full = torch.zeros(d + 1, device="cuda")
    v = full[1:]  # 4 bytes off a 16-byte boundary
    v[torch.from_numpy(at).cuda()] = torch.from_numpy(x).cuda()
    sk = gs.gs_sketch_create(r, c, d + W, W, W)
    try:
        gs.gs_sketch_insert(sk, W // 2, v, d)
        _check(gs, sk, W // 2, r, c, coeffs, at, x, "inserted alone")
    finally:
        gs.gs_sketch_destroy(sk)


@pytest.mark.parametrize("P,W,r,c", [(1, 1, 9, 1 << 17), (1, 1, 1, 1 << 21), (2, 2, 5, 1 << 17), (3, 4, 9, 1 << 17),
                                     (4, 4, 2, 1 << 21), (8, 8, 2, 1 << 14), (7, 8, 9, 1 << 18), (8, 8, 1, 1 << 16),
                                     (15, 16, 5, 1 << 18), (16, 16, 16, 1 << 16)])
@pytest.mark.parametrize("d,offset", [(70_001, 0), (130_003, 0), (130_003, 1), (600_001, 0), (1_500_003, 0)])
def test_group_inserts(gs, P, W, r, c, d, offset):
    """The accumulate pass with its rows, and the sketched state's insert of already accumulated vectors."""
    rho, seed, k = 0.9, d + 7 * W + r, 20
    rng = np.random.default_rng(seed)
    coeffs = oracle.derive_coefficients(r, seed)
    at, vals = _sparse(rng, d, 3000, 3 * P)
    dev_at = torch.from_numpy(at).cuda()
    bufs = [torch.zeros(d + 4, device="cuda") for _ in range(3 * P)]
    views = [b[offset:offset + d] for b in bufs]
    for v, x in zip(views, vals):
        v[dev_at] = torch.from_numpy(x).cuda()
    sketches = [gs.gs_sketch_create(r, c, seed, n, w) for n, w in ((P, W), (1, 0), (1, 0))]
    try:
        gs.gs_accumulate_insert(sketches[0], 0, views[:P], views[P:2 * P], views[2 * P:], d, rho)
        for p in range(P):
            u, e = oracle.accumulate(vals[p], vals[P + p], vals[2 * P + p], rho)
            assert np.array_equal(views[p][dev_at].cpu().numpy().view(np.uint32), u.view(np.uint32))
            assert np.array_equal(views[P + p][dev_at].cpu().numpy().view(np.uint32), e.view(np.uint32))
            assert int(torch.count_nonzero(bufs[P + p])) == np.count_nonzero(e)
            _check(gs, sketches[0], p, r, c, coeffs, at, e, f"worker {p}, accumulated")
        ws = torch.empty(gs.gs_step_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        idx, out = torch.empty(k, dtype=torch.int64, device="cuda"), torch.empty(k, device="cuda")
        gs.gs_sketched_state_step(*sketches, views[2 * P:], d, rho, k, idx, out, None, 0.0, ws)
        for p in range(P):
            _check(gs, sketches[0], p, r, c, coeffs, at, vals[2 * P + p], f"worker {p}, inserted as it is")
    finally:
        for sk in sketches:
            gs.gs_sketch_destroy(sk)
