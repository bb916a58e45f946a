"""TV prox around the edges of its tiles and of the iterations one launch takes
(needs a GB300): sides below, at and above the tile of 16 or 32, five
iterations per launch and remainders.  Bound: 1e-5 relative, the FP32 operator
bound (each iteration is a projection, its errors do not grow)."""
import numpy as np
import pytest

from oracle import tv as otv
from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,iters,weighted", [(8, 1, False), (12, 4, True), (16, 5, False), (24, 6, True),
                                              (48, 11, False), (96, 10, True), (384, 7, False), (512, 9, True),
                                              (768, 5, True), (16, 0, False)])
def test_prox_tv_tiles(n, iters, weighted):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(n + iters)
    ctx = binding.Context(n, inputs.uniform_uv(8, rng).astype(np.float32), J=4, levels=2)
    x = inputs.random_image(n, rng)
    w = rng.uniform(0.2, 1.5, (n, n)).astype(np.float32) if weighted else None
    lam = np.float32(0.37)
    got = host(ctx.prox_tv(dev(x, torch), dev(w, torch) if weighted else None, float(lam), iters))
    want = otv.prox_tv(x, float(lam), None if w is None else w.astype(np.float64), iters)
    assert rel_err(got, want) <= 1e-5
    # a zero weight of the prior is the identity
    assert np.array_equal(host(ctx.prox_tv(dev(x, torch), None, 0.0, iters)), x)
