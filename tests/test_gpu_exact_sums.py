"""Reductions whose exact value an FP64 sum holds (needs a GB300).

The terms are integers (or multiples of 2^-25) that need more than the 48 bits
of a float pair but fit FP64's 53, so the library's sums, FP64 once they leave
a thread's few terms, must be exact: no tolerance.
"""
import math

import numpy as np
import pytest

from paper_1307_4370_gb300 import inputs

from gpu_util import dev, require_gpu

pytestmark = pytest.mark.gpu

BIG, SMALL = 2.0 ** 25, 2.0 ** 13 + 1.0  # squares 2^50 and 2^26 + 2^14 + 1


@pytest.mark.parametrize("count,at", [(32, 5), (33, 32), (4096, 1234), (70001, 40000)])
def test_norm(count, at):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    ctx = binding.Context(16, inputs.uniform_uv(8, np.random.default_rng(0)).astype(np.float32), J=4)
    a = np.full(count, SMALL, np.complex64)
    a[at] = BIG
    nrm = torch.zeros(1, dtype=torch.float64, device="cuda")
    ctx.proj_l2ball(dev(a, torch), dev(np.zeros(count, np.complex64), torch), 1.0, norm_out=nrm)
    assert float(nrm.item()) == math.sqrt(int(BIG) ** 2 + (count - 1) * int(SMALL) ** 2)


@pytest.mark.parametrize("n,M,at", [(64, 3000, 11), (768, 60000, 7), (768, 60000, 30000), (768, 60000, 59999)])
def test_sdmm_norms(n, M, at):
    """nu of an iteration at x_hat = 0 (no CG step): ||y|| alone, over one and over several units per CTA."""
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    ctx = binding.Context(n, inputs.uniform_uv(M, np.random.default_rng(n)).astype(np.float32), J=4)
    y = np.full(M, SMALL, np.complex64)
    y[at] = BIG
    st = ctx.sdmm_state()
    st.init(dev(y, torch), 1.0, cg_iters=0)
    st.step()
    assert st.report()["nu"] == math.sqrt(int(BIG) ** 2 + (M - 1) * int(SMALL) ** 2)


def test_sdmm_norms_beyond_float():
    """Terms whose sum over a warp leaves FP32's range (the warp's FP64 tree)."""
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    M = 3000
    ctx = binding.Context(64, inputs.uniform_uv(M, np.random.default_rng(1)).astype(np.float32), J=4)
    st = ctx.sdmm_state()
    st.init(dev(np.full(M, 2.0 ** 62, np.complex64), torch), 1.0, cg_iters=0)
    st.step()
    assert st.report()["nu"] == math.sqrt(M * 2.0 ** 124)


HEADER = 48  # bytes before x_hat in an exported state


@pytest.mark.parametrize("n,levels", [(64, 4), (32, 3)])
def test_f1(n, levels):
    """f1 = sum w |Psi^H x_hat| with the weights of the Dirac plane alone, moduli 1 and 2^-25 mixed."""
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(n)
    M, N = 40, n * n
    ctx = binding.Context(n, inputs.uniform_uv(M, rng).astype(np.float32), J=4, levels=levels, bases_mask=0xF)
    st = ctx.sdmm_state()
    st.init(dev(inputs.random_vis(M, rng), torch), 1.0, cg_iters=0)
    one = rng.integers(0, 2, N).astype(bool)
    blob = bytearray(st.export())
    blob[HEADER:HEADER + 8 * N] = np.where(one, 2.0, 2.0 ** -24).astype(np.complex64).tobytes()  # x / sqrt(4 planes)
    st.import_(bytes(blob))
    w = np.zeros((4, N), np.float32)
    w[0] = 1.0
    st.set_weights(dev(w, torch))
    st.step()
    assert st.report()["f1"] == float(one.sum()) + float((~one).sum()) * 2.0 ** -25


def test_cg_direction_update_is_the_fp64_quotient():
    """beta of the last CG step of an iteration, against the two <r, r> it is the quotient of."""
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(3)
    n, M = 32, 500
    ctx = binding.Context(n, inputs.uniform_uv(M, rng).astype(np.float32), J=4, levels=3)
    st = ctx.sdmm_state()
    st.init(dev(inputs.random_vis(M, rng), torch), 1.0, cg_iters=3)
    N, D = n * n, 9 * n * n
    st.step()  # (starts from a zero residual)
    for _ in range(24):
        st.step()
        # the scalars end the exported state: beta is the third, the last steps' <r, r> the 19th (even steps) and 20th
        sc = np.frombuffer(st.export()[HEADER + 8 * (5 * N + D + 2 * M) + 4 * D:], np.float64, 22)
        assert sc[2] == sc[18] / sc[19]
