"""Convolutions over tiles of pixels, at the edges of the tile: images of fewer
positions than a tile and rows as long as one, tiles that end in a padding column
or row, 48 channels (three steps of 16) and 24 (none: the GEMM form), output
columns that fill no tile, and channels whose tile does not fit shared memory
(the GEMM form again).

A few weights of +-1 per output channel and inputs of small integers make every
sum exact, so the reference rounds the same values to bfloat16 and no decision
falls the other way: the outputs agree to the FP32 output stage (a 3 x 3 average
and a projection, about 20 roundings of 2^-24), and the gradients to the bound of
the surrogate's other tests (their sums start from the output stage's rounded
values)."""
import numpy as np
import pytest

from test_gpu_nn import S, allowed, outliers

pytestmark = pytest.mark.gpu

EDGES = [([16], 1, (2, 3)), ([16], 3, (5, 127)), ([16], 2, (3, 128)), ([32], 1, (1, 300)), ([16], 2, (63, 7)),
         ([48, 32], 3, (24, 18)), ([24, 16], 2, (10, 14)), ([16, 160], 2, (16, 16)), ([16, 272], 1, (16, 16))]


@pytest.mark.parametrize("channels,n,hw", EDGES)
def test_convolution_tiles_match_reference(channels, n, hw):
    from paper_2103_02119_gb300 import lbm as L
    rng = np.random.default_rng(4)
    params = []
    for w, b in S.init_params(channels, seed=4):
        w, b = np.zeros_like(w), np.zeros_like(b)
        for co in range(w.shape[3]):
            for _ in range(4):
                w[rng.integers(3), rng.integers(3), rng.integers(w.shape[2]), co] = rng.choice([-1.0, 1.0, 1.0])
            b[co] = rng.integers(0, 3)
        params.append((w, b))
    x = rng.integers(-4, 5, (n, *hw, 4)).astype(np.float64)
    x[..., 0] = rng.random((n, *hw)) > 0.85
    t = rng.standard_normal((n, *hw, 3))
    fluid = x[..., 0] < 0.5
    nn = L.lbm_nn_create(channels, n, *hw, seed=0)
    L.lbm_nn_set_params(nn, L.params_to_vec(params).astype(np.float32))
    ref = S.WarmNet(channels, params, bf16_storage=True)
    y = L.lbm_nn_forward(nn, x)
    yr, tape = ref.forward(x)
    assert np.abs(y - yr).max() <= 20 * 2.0 ** -24 * 9 * max(1.0, np.abs(yr).max())
    loss, g = L.lbm_nn_gradients(nn, x, t, fluid)
    lr, gy = ref.loss(yr, t, fluid)
    gr = ref.backward(tape, gy)
    assert abs(loss - lr) <= 1e-5 * lr
    got = L.params_to_list(g, S.layer_shapes(channels))
    for k, (a, b) in enumerate(zip(got, gr)):
        for j in (0, 1):
            assert outliers(a[j], b[j]) <= allowed(b[j].size), (k, j)
    L.lbm_nn_destroy(nn)
