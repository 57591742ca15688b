"""Gradient of the learned law's training step over one tile of 128 points,
several, a count beside the batches of sixteen that the update sums, and more
tiles than the GPU runs at once, against FP64 backpropagation with the same
bf16 rounding points.  Tolerance: that of the two-tile gradient (2e-3 of a
block's norm: FP32 sums, and single bf16 flips where an FP32 sum lands on a
rounding boundary); the loss is a mean of FP32 partials (1e-5)."""
import numpy as np
import pytest

import mlp_reference as R
import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [1, 3, 16, 17, 160])
def test_gradient_over_tiles(tiles):
    import paper_2301_05552_gb300 as pkg
    s = pkg.pdn_sur_create(pi.material_im7_like_config(t_ply=0.275, spread=0.0), 0.552, seed=7)
    p = pkg.pdn_sur_get_params(s)[0].astype(np.float64)
    rng = np.random.default_rng(tiles)
    n = 128 * tiles
    xn = rng.normal(size=(n, 10)).astype(np.float32)
    tn = rng.normal(size=(n, 10)).astype(np.float32)
    g, loss = pkg.pdn_sur_gradient(s, xn, tn)
    lb, gb = R.loss_and_grad(p, xn.astype(np.float64), tn.astype(np.float64), bf=True)
    assert abs(loss - lb) <= 1e-5 * lb
    o = 0
    for shape in R.SHAPES:
        k = int(np.prod(shape))
        a, b = g[o:o + k].astype(np.float64), gb[o:o + k]
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b) + 1e-12
        o += k
    s.close()
