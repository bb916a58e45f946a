"""The largest 3 2^a side (needs a GB300): n = 1536, rows and columns of 3072
points in the compile-time FFT engine (column CTAs of 1024 threads, one row per
CTA, step sizes by the one-block kernel), with ragged visibilities, against the
FP64 oracle at the bound of the FP32 operators.
"""
import numpy as np

import pytest

from oracle import cg as ocg, measurement as me
from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, rel_err, require_gpu

pytestmark = pytest.mark.gpu


def test_1536():
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    n, M, J = 1536, 5003, 6
    rng = np.random.default_rng(1536)
    uv = inputs.uniform_uv(M, rng).astype(np.float32).astype(np.float64)
    ctx = binding.Context(n, uv.astype(np.float32), J=J)
    x, v = inputs.random_image(n, rng), inputs.random_vis(M, rng)
    assert rel_err(host(ctx.phi(dev(x, torch))), me.phi(x, uv, J)) <= 1e-5
    assert rel_err(host(ctx.phi_adj(dev(v, torch))), me.phi_adj(v, uv, n, J)) <= 1e-5
    x0 = inputs.random_image(n, rng)
    got, _ = ctx.cg_solve(dev(x, torch), dev(x0, torch), 3)
    want, _ = ocg.cg(lambda u: me.phi_adj(me.phi(u, uv, J), uv, n, J) + 2.0 * u, x, x0, 3)
    assert rel_err(host(got).reshape(n, n), want) <= 1e-5
