"""Inserts whose rows do not all go the same way, against the CPU oracle: c not a power of two with a table
beyond one pass (later passes re-read the error vectors), the same for the insert of already accumulated
vectors, and gradients in host memory with a table beyond one pass (some rows directly, the others along
chains)."""

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


def _vectors(rng, P, d):
    return [(rng.standard_normal(d) * 1e-3).astype(np.float32) for _ in range(P)]


def _check_tables(gs, sk, es, r, c, seed):
    coeffs = oracle.derive_coefficients(r, seed)
    buf = np.empty(r * c, dtype=np.float32)
    for p, e in enumerate(es):
        gs.gs_sketch_copy_to_host(sk, p, buf)
        T, A = oracle.sketch(e, coeffs, c)
        assert np.all(np.abs(buf.reshape(r, c).astype(np.float64) - T) <= REL * A), f"worker {p}"


SHAPES = [(8, 8, 7, 299_993, 2), (2, 2, 5, 1_600_001, 2), (3, 4, 3, 1_999_999, 3), (1, 1, 3, 7_000_001, 3),
          (11, 16, 4, 250_007, 2)]


@pytest.mark.parametrize("P,W,r,c,passes", SHAPES)
def test_accumulate_insert_in_passes(gs, P, W, r, c, passes):
    d, rho, seed = 200_003, 0.9, c % 1000 + P
    rng = np.random.default_rng(seed)
    us, es, grads = (_vectors(rng, P, d) for _ in range(3))
    dev = [[torch.from_numpy(x).cuda() for x in xs] for xs in (us, es, grads)]
    sk = gs.gs_sketch_create(r, c, seed, P, W)
    try:
        assert -(-r // gs.gs_sketch_info(sk)["rows_per_pass"]) == passes
        gs.gs_accumulate_insert(sk, 0, dev[0], dev[1], dev[2], d, rho)
        want = [oracle.accumulate(u, e, g, rho) for u, e, g in zip(us, es, grads)]
        for p, (u, e) in enumerate(want):
            assert np.array_equal(dev[0][p].cpu().numpy().view(np.uint32), u.view(np.uint32))
            assert np.array_equal(dev[1][p].cpu().numpy().view(np.uint32), e.view(np.uint32))
        _check_tables(gs, sk, [e for _, e in want], r, c, seed)
    finally:
        gs.gs_sketch_destroy(sk)


@pytest.mark.parametrize("P,W,r,c,passes", SHAPES)
def test_insert_all_in_passes(gs, P, W, r, c, passes):
    """The sketched-state step's insert of every worker's gradient."""
    d, k, seed = 150_001, 50, c % 1000 + P
    rng = np.random.default_rng(seed)
    grads = _vectors(rng, P, d)
    sketches = [gs.gs_sketch_create(r, c, seed, n, w) for n, w in ((P, W), (1, 0), (1, 0))]
    try:
        assert -(-r // gs.gs_sketch_info(sketches[0])["rows_per_pass"]) == passes
        ws = torch.empty(gs.gs_step_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        idx = torch.empty(k, dtype=torch.int64, device="cuda")
        vals = torch.empty(k, device="cuda")
        gs.gs_sketched_state_step(*sketches, [torch.from_numpy(g).cuda() for g in grads], d, 0.9, k, idx, vals, None, 0.0, ws)
        _check_tables(gs, sketches[0], grads, r, c, seed)
    finally:
        for sk in sketches:
            gs.gs_sketch_destroy(sk)


@pytest.mark.parametrize("P,W,r,c", [(8, 8, 5, 1 << 19), (2, 2, 7, 1 << 21), (4, 4, 3, 1 << 21), (1, 1, 5, 1 << 22)])
def test_host_gradients_with_rows_beyond_one_pass(gs, P, W, r, c):
    d, k, rho, seed = 400_001, 300, 0.9, 3 * W + r
    rng = np.random.default_rng(seed)
    us, es, grads = (_vectors(rng, P, d) for _ in range(3))
    u_dev, e_dev = ([torch.from_numpy(x).cuda() for x in xs] for xs in (us, es))
    pinned = [torch.from_numpy(g).pin_memory() for g in grads]
    buf = [torch.empty(d, device="cuda") for _ in range(P)]
    sk = gs.gs_sketch_create(r, c, seed, P, W)
    try:
        assert gs.gs_sketch_info(sk)["rows_per_pass"] < r and d * r > 1 << 20
        ws = torch.empty(gs.gs_step_workspace_size(d, k), dtype=torch.uint8, device="cuda")
        idx = torch.empty(k, dtype=torch.int64).pin_memory()
        vals = torch.empty(k).pin_memory()
        gs.gs_step_host(sk, u_dev, e_dev, pinned, buf, d, rho, k, idx, vals, ws)
        want = [oracle.accumulate(u, e, g, rho) for u, e, g in zip(us, es, grads)]
        _check_tables(gs, sk, [e for _, e in want], r, c, seed)
        keep = np.ones(d, dtype=bool)
        keep[idx.numpy()] = False
        for p, (u, e) in enumerate(want):
            assert np.array_equal(u_dev[p].cpu().numpy()[keep].view(np.uint32), u[keep].view(np.uint32))
            assert np.array_equal(e_dev[p].cpu().numpy()[keep].view(np.uint32), e[keep].view(np.uint32))
    finally:
        gs.gs_sketch_destroy(sk)
