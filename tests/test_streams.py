"""Handles on CUDA streams of their own."""
import time

import numpy as np
import pytest

from paper_0912_3824_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def md():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0912_3824_gb300 import build
    build.build()
    from paper_0912_3824_gb300 import md as m
    return m


@pytest.mark.parametrize("n", [864, 2000, 4000])
def test_small_systems_on_streams_of_their_own_overlap(md, n):
    """Four handles stepped together: the states of handles stepped alone, bit for
    bit, in clearly less than four times one handle's time (0.28 to 0.56 of it
    measured; 1 if the launches exclude one another)."""
    import torch
    s = synth.ka_mixture(n=n, temperature=0.8, seed=3)
    sims = [md.System(md.make_params(s.params, 0.002), [n], [s.box], s.species, s.pos, (k + 1) * 0.25 * s.vel,
                      stream=torch.cuda.Stream()) for k in range(4)]
    alone, together = [], []
    for rep in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for x in sims:
            x.step(300)
            torch.cuda.synchronize()
        t1 = time.perf_counter()
        for x in sims:
            x.step(300)
        torch.cuda.synchronize()
        alone.append(t1 - t0)
        together.append(time.perf_counter() - t1)
    got = [x.get_state() for x in sims]
    assert all(x.sync() == md.MD_OK for x in sims)
    for x in sims:
        x.close()
    assert min(together) < 0.8 * min(alone)
    for k in (0, 3):
        ref = md.System(md.make_params(s.params, 0.002), [n], [s.box], s.species, s.pos, (k + 1) * 0.25 * s.vel)
        for _ in range(12):
            ref.step(300)
        for a, b in zip(got[k], ref.get_state()):
            assert np.array_equal(a, b)
        ref.close()
