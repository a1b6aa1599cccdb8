"""Batches of very many tiny instances: more than the 65,535 that fit the second
dimension of a grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_more_instances_than_a_grid_has_rows():
    """70,000 instances of 2 x 2 cells in one call give what two halves give, bit for
    bit: predictions, prolonged fields, and gradients (whose sums differ in order)."""
    from paper_2103_02119_gb300 import lbm as L
    n, half = 70000, 35000
    rng = np.random.default_rng(1)
    x = rng.standard_normal((n, 2, 2, 4)).astype(np.float32)
    x[..., 0] = rng.random((n, 2, 2)) < 0.2
    t = rng.standard_normal((n, 2, 2, 3)).astype(np.float32)
    fluid = (x[..., 0] < 0.5).astype(np.uint8)
    fine = (rng.random((n, 4, 4)) < 0.8).astype(np.uint8)
    nn = L.lbm_nn_create([8], n, 2, 2, seed=2)
    y = L.lbm_nn_forward(nn, x)
    z = L.lbm_nn_prolong(nn, y, 2, fine)
    loss, g = L.lbm_nn_gradients(nn, x, t, fluid)
    losses, grads, cells = [], [], []
    for s in (slice(0, half), slice(half, n)):
        assert np.array_equal(y[s], L.lbm_nn_forward(nn, x[s]))
        assert np.array_equal(z[s], L.lbm_nn_prolong(nn, y[s], 2, fine[s]))
        part = L.lbm_nn_gradients(nn, x[s], t[s], fluid[s])
        losses.append(part[0])
        grads.append(part[1])
        cells.append(float(fluid[s].sum()))
    w = np.array(cells) / sum(cells)
    assert abs(loss - w @ np.array(losses)) <= 1e-5 * loss
    # the output gradients are scaled by 1 / (3 cells) and rounded to bfloat16 in the
    # halves (2^-8 of each term)
    want = np.tensordot(w, np.array(grads, np.float64), 1)
    scale = np.abs(np.array(grads)).max()
    assert np.abs(g - want).max() <= 2.0 ** -7 * scale
    L.lbm_nn_destroy(nn)


def test_many_instances_cost_what_their_cells_cost():
    """The output stage of 60,000 instances of 2 x 2 cells takes at most twice as long
    as of 60 instances with as many cells in all (the same transfers): no blocks for
    parts that an instance does not have."""
    import time

    from paper_2103_02119_gb300 import lbm as L
    times = []
    for n, h, w in ((60000, 2, 2), (60, 40, 100)):
        y = np.zeros((n, h, w, 3), np.float32)
        fluid = np.ones((n, h, w), np.uint8)
        nn = L.lbm_nn_create([8], n, h, w, seed=2)
        best = 1e9
        for _ in range(12):
            t0 = time.perf_counter()
            L.lbm_nn_prolong(nn, y, 1, fluid)
            best = min(best, time.perf_counter() - t0)
        times.append(best)
        L.lbm_nn_destroy(nn)
    assert times[0] <= 2.0 * times[1], times
