"""Contexts whose grid tile is the whole grid (needs a GB300): the footprints
that wrap at the grid's edges have all their parts in one tile's list.  Phi,
Phi^H, CG steps (the Gram pass as a gather and from stored stencils) and SDMM
iterations against the FP64 oracle (1e-5 relative for the FP32 operators, 1e-4
for the iterations, the bounds of the other tests).
"""
import numpy as np
import pytest

from oracle import cg as ocg, measurement as me, sdmm as osdmm, simulate
from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,M", [(8, 2, 300), (8, 8, 12), (8, 8, 2000), (16, 6, 40), (16, 4, 900), (32, 6, 200),
                                   (32, 6, 9000), (32, 8, 1)])
def test_operators_and_cg(n, J, M):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(n + M)
    uv = inputs.uniform_uv(M, rng).astype(np.float32).astype(np.float64)
    ctx = binding.Context(n, uv.astype(np.float32), J=J, levels=3, tile=2 * n)
    x, v = inputs.random_image(n, rng), inputs.random_vis(M, rng)
    out = torch.full((M,), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.phi(dev(x, torch), out=out)
    assert rel_err(host(out), me.phi(x, uv, J)) <= 1e-5
    assert rel_err(host(ctx.phi_adj(dev(v, torch))), me.phi_adj(v, uv, n, J)) <= 1e-5
    b, x0 = inputs.random_image(n, rng), inputs.random_image(n, rng)
    got, _ = ctx.cg_solve(dev(b, torch), dev(x0, torch), 4)
    want, _ = ocg.cg(lambda u: me.phi_adj(me.phi(u, uv, J), uv, n, J) + 2.0 * u, b, x0, 4)
    assert rel_err(host(got).reshape(n, n), want) <= 1e-5


def test_sdmm_iterations():
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    w = inputs.Workload("one tile", n=32, M=1024, J=4, n_src=8, diffuse=False, seed=2024)
    p = inputs.make_problem(w)
    y, eps = simulate.visibilities(p.x_true, p.uv, w.J, p.noise_unit, w.isnr_db)
    y = y.astype(np.complex64).astype(np.complex128)
    ref = osdmm.solve(simulate.operators(p.uv, w.n, w.J), y, eps, (w.n, w.n), (9, w.n, w.n), iters=5, cg_iters=10)
    ctx = binding.Context(w.n, p.uv.astype(np.float32), J=w.J, tile=64)
    x, _ = ctx.sdmm_solve(dev(y, torch), eps, max_iters=5, cg_iters=10)
    assert rel_err(host(x), ref.x_hat) <= 1e-4
