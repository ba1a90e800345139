"""Handles on CUDA streams of their own."""
import ctypes as C
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


def _green_stream(cu, min_sms):
    """A stream of a green context of at least min_sms SMs: (stream, context, SMs), or None
    where the driver offers no such context."""
    dev, res, part, rest = C.c_int(), (C.c_uint8 * 512)(), (C.c_uint8 * 512)(), (C.c_uint8 * 512)()
    groups, desc, ctx, stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    if (cu.cuDeviceGet(C.byref(dev), 0) or cu.cuDeviceGetDevResource(dev, res, 1) or
            cu.cuDevSmResourceSplitByCount(part, C.byref(groups), res, rest, 0, min_sms) or
            cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1) or cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1) or
            cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0)):      # (1: non-blocking)
        return None
    return stream, ctx, C.cast(C.addressof(part) + 96, C.POINTER(C.c_uint))[0]    # CUdevResource.sm.smCount


@pytest.mark.parametrize("n", [864, 4000, 40000])
def test_a_stream_with_part_of_the_sms(md, n):
    """A handle on a stream that has 64 of the GPU's SMs: one block on each of these,
    and the states of a handle with all of them, bit for bit."""
    import torch
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    got = _green_stream(cu, 64)
    if got is None:
        pytest.skip("no green contexts")
    stream, ctx, sms = got
    assert 64 <= sms < torch.cuda.get_device_properties(0).multi_processor_count
    s = synth.ka_mixture(n=n, temperature=0.8, seed=3)
    runs = []
    for st in (torch.cuda.ExternalStream(stream.value), None):
        sim = md.System(md.make_params(s.params, 0.002, threads_per_particle=2), [n], [s.box], s.species, s.pos, s.vel,
                        stream=st)
        sim.step(200)
        assert sim.sync() == md.MD_OK
        runs.append(sim.get_state())
        sim.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)
