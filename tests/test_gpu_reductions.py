"""Device reductions at the sizes where their trees change shape (needs a GB300).

The norms sum FP32-exact terms (float pairs within a warp, FP64 beyond), so
they must match FP64 sums of the same float32 values to FP64 rounding; values
whose sum of squares leaves FP32's range take the FP64 tree of the warp.
"""
import numpy as np
import pytest

from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 3e18])
@pytest.mark.parametrize("count", [1, 31, 33, 255, 257, 70001])
def test_norm_against_fp64(count, scale):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(count)
    ctx = binding.Context(16, inputs.uniform_uv(8, rng).astype(np.float32), J=4)
    # moduli within [0.6, 1.4]: with scale 3e18 every square fits FP32 and the sum over a warp does not
    a = (rng.uniform(0.4, 1.0, count) + 1j * rng.uniform(0.4, 1.0, count)) * scale
    a = a.astype(np.complex64)
    nrm = torch.zeros(1, dtype=torch.float64, device="cuda")
    ctx.proj_l2ball(dev(a, torch), dev(np.zeros(count, np.complex64), torch), 1.0, norm_out=nrm)
    want = np.sqrt(np.sum(a.real.astype(np.float64) ** 2 + a.imag.astype(np.float64) ** 2))
    # exact products; at most 2^-47 per warp sum and a few FP64 roundings
    assert float(nrm.item()) == pytest.approx(want, rel=1e-13)


@pytest.mark.parametrize("R", [1, 7, 64, 65, 300])
def test_block_norms(R):
    """nu and nu_min of the distributed form around the switch of its last summation (64 blocks)."""
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(R)
    n, M = 16, 90001 if R == 7 else 3001  # seven blocks: more chunks per block than lanes of a few warps
    ctx = binding.Context(n, inputs.uniform_uv(M, rng).astype(np.float32), J=4, levels=2)
    y = dev(inputs.random_vis(M, rng), torch)
    off = np.concatenate([[0], np.sort(rng.choice(np.arange(1, M), R - 1, replace=False)), [M]])
    eps = rng.uniform(0.5, 1.5, R)
    st = ctx.sdmm_state()
    st.set_blocks(off, eps)
    st.init(y, 1.0)
    st.step()
    st.step()
    rep = st.report()
    d = host(y) - host(ctx.phi(st.get_image()))
    nu = np.array([np.linalg.norm(d[off[b]:off[b + 1]]) / eps[b] for b in range(R)])
    # the residual is rounded to FP32 here (2^-24 of each term), exact in the library
    assert rep["nu"] == pytest.approx(nu.max(), rel=1e-6)
    assert rep["nu_min"] == pytest.approx(nu.min(), rel=1e-6)
