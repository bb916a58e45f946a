"""CG steps on both sides of the Gram pass's dense-tile rule (needs a GB300).

G^T G of a tile is a stored half stencil or a gather, chosen by its entries,
the kernel support and what fits L2; small grids with J <= 4 use stencils only.
Whatever the choice the steps must be those of the oracle's CG (1e-5 relative,
the bound of the FP32 operators).
"""
import numpy as np
import pytest

from oracle import cg as ocg, measurement as me
from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,J,kind", [(64, 1, 4, "uniform"), (64, 700, 2, "uniform"), (64, 9000, 4, "gauss"),
                                        (96, 3000, 4, "gauss"), (256, 20000, 4, "gauss"), (256, 20000, 6, "gauss"),
                                        (256, 3001, 8, "uniform"), (192, 60000, 4, "gauss")])
def test_cg_steps(n, M, J, kind):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(n + M)
    uv = inputs.uniform_uv(M, rng) if kind == "uniform" else \
        inputs.uv_variable_density(M, n, rng).astype(np.float32).astype(np.float64)
    ctx = binding.Context(n, uv.astype(np.float32), J=J)
    b, x0 = inputs.random_image(n, rng), inputs.random_image(n, rng)
    x, _ = ctx.cg_solve(dev(b, torch), dev(x0, torch), 4)
    want, _ = ocg.cg(lambda v: me.phi_adj(me.phi(v, uv, J), uv, n, J) + 2.0 * v, b, x0, 4)
    assert rel_err(host(x), want) <= 1e-5
