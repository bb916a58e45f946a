"""SARA levels whose tiles take the blocked and the plain filter loops (needs a GB300).

The analysis filters four outputs per thread on tiles of a multiple of four
and the synthesis on even tiles; sides 2^a and 3 2^a with up to six levels
reach tiles of 16, 12, 8, 6, 4, 3, 2 and 1.  Bound: FP32 filter arithmetic,
1e-5 relative as for the other operators; the synthesis is the exact
transpose, so Psi Psi^H x = x to the same bound.
"""
import numpy as np
import pytest

from oracle import sara as osara
from paper_1307_4370_gb300 import inputs

from gpu_util import dev, host, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels,mask", [(64, 6, 0x1FF), (128, 6, 0x1FF), (192, 6, 0x1FF), (48, 4, 0x1FF),
                                           (24, 3, 0x1FE), (96, 5, 0x181), (12, 2, 0x1FF), (8, 1, 0x010),
                                           (768, 4, 0x003), (256, 1, 0x100)])
def test_sara_levels(n, levels, mask):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    rng = np.random.default_rng(n + 31 * levels)
    bases = tuple(b for b in range(9) if mask >> b & 1)
    ctx = binding.Context(n, inputs.uniform_uv(16, rng).astype(np.float32), J=4, levels=levels, bases_mask=mask)
    x = inputs.random_image(n, rng)
    al = host(ctx.sara_analysis(dev(x, torch)))
    assert rel_err(al, osara.sara_analysis(x, levels, bases)) <= 1e-5
    a = rng.standard_normal((len(bases), n, n)) + 1j * rng.standard_normal((len(bases), n, n))
    a = a.astype(np.complex64).astype(np.complex128)
    assert rel_err(host(ctx.sara_synthesis(dev(a, torch))), osara.sara_synthesis(a, levels, bases)) <= 1e-5
    assert rel_err(host(ctx.sara_synthesis(ctx.sara_analysis(dev(x, torch)))), x) <= 1e-5
