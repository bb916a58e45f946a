"""Contexts of different sizes used from several host threads at once (needs a
GB300).  A kernel's shared-memory limit belongs to the kernel, not to a context
or a thread, so a launch must not depend on the size another thread asked for
last.  Each thread has its own context and stream; results equal the ones of
the same calls made alone, bit for bit (the kernels are deterministic).
"""
import threading

import numpy as np
import pytest

from paper_1307_4370_gb300 import inputs

from gpu_util import dev, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["sara", "phi_adj"])
def test_sizes_in_threads(call):
    torch = require_gpu()
    from paper_1307_4370_gb300 import binding

    jobs = []
    for n, J, tile in ((64, 4, 16), (96, 8, 64)):  # SARA tails of 64 and 48; gridding tiles of 16 and 64
        rng = np.random.default_rng(n)
        ctx = binding.Context(n, inputs.uniform_uv(3000, rng).astype(np.float32), J=J, tile=tile)
        x, v = dev(inputs.random_image(n, rng), torch), dev(inputs.random_vis(3000, rng), torch)
        jobs.append((lambda s, ctx=ctx, x=x: ctx.sara_analysis(x, stream=s)) if call == "sara" else
                    (lambda s, ctx=ctx, v=v: ctx.phi_adj(v, stream=s)))
    want = [j(None).clone() for j in jobs]
    torch.cuda.synchronize()
    errors, got = [], [None, None]

    def work(k):
        s = torch.cuda.Stream()
        try:
            with torch.cuda.stream(s):
                for _ in range(3000):
                    out = jobs[k](s)
                got[k] = out
            s.synchronize()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, w in zip(got, want):
        assert torch.equal(torch.view_as_real(g), torch.view_as_real(w))
