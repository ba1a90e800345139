"""What a handle does after a failure has been reported: its lists belong to its
state again, and a state that was lost is asked for."""
import numpy as np
import pytest

import oracle
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


def _sim(md, s, **kw):
    kw.setdefault("sample_interval", 10)
    return md.System(md.make_params(s.params, 0.002, **kw), [s.n], [s.box], s.species, s.pos, s.vel)


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_calls_made_while_a_failure_is_pending_change_nothing(md, prec, use_graph):
    """md_step stops at its step budget; a force call and a further md_step before
    the report do nothing but (the force call) report it; the run then goes on
    bit for bit as in a handle that was only asked for its status."""
    s = synth.perturb(synth.ka_mixture(n=2000, temperature=1.5, seed=3), 0.05, 103)
    got = []
    for call in (False, True):
        sim = _sim(md, s, precision=md.PRECISIONS[prec], step_budget=37, use_graph=use_graph)
        sim.step(100)
        if call:
            sim.step(20)
            with pytest.raises(md.MDError) as ei:
                sim.forces()
            assert ei.value.code == md.MD_E_TIMEOUT
        else:
            assert sim.sync() == md.MD_E_TIMEOUT
        assert sim.sync() == md.MD_OK
        sim.step(30)
        assert sim.sync() == md.MD_OK
        got.append(sim.get_state() + (sim.info()["step"], sim.info()["rebuilds"]))
        sim.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-5), ("fp64", 1e-12)])
def test_state_set_while_a_failure_is_pending(md, prec, tol):
    """md_set_state before the report: the new state is there after it, and the
    lists and the forces that open the next md_step are the new state's."""
    s = synth.perturb(synth.ka_mixture(n=2000, temperature=1.0, seed=3), 0.05, 103)
    t = synth.perturb(synth.ka_mixture(n=2000, temperature=1.0, seed=3), 0.05, 104)
    sim = _sim(md, s, precision=md.PRECISIONS[prec], step_budget=37)
    sim.step(100)
    sim.set_state(t.pos, t.vel)
    assert sim.sync() == md.MD_E_TIMEOUT
    counts, lists = sim.neighbours()
    inner, inner_l = oracle.neighbours_brute(s.params, s.box, s.species, t.pos, 0.3 - 1e-4, kmax=512)
    for i in range(s.n):
        assert set(inner_l[i, :inner[i]].tolist()) <= set(lists[i, :counts[i]].tolist())
    sim.step(30)
    assert sim.sync() == md.MD_OK
    a = sim.get_state()
    sim.close()
    ref = _sim(md, s, precision=md.PRECISIONS[prec])
    ref.set_state(t.pos, t.vel)
    ref.step(30)
    b = ref.get_state()
    ref.close()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_a_list_past_the_cap_fails_again_until_the_state_changes(md):
    """A state whose lists exceed the cap: the build fails, and so does going on (the
    lists written then are not those of the state's order).  After a state whose
    lists fit, forces and steps are right."""
    s = synth.perturb(synth.ka_mixture(n=2000, temperature=0.7, seed=3), 0.02, 103)
    probe = _sim(md, s)
    cap = (probe.info()["max_neighbours"] + 7) // 8 * 8
    probe.close()
    sim = _sim(md, s, neigh_capacity=cap, neigh_capacity_max=cap)
    sim.set_state(0.9 * s.pos, s.vel)
    assert sim.sync() == md.MD_E_CAPACITY
    for _ in range(2):
        sim.step(1)
        assert sim.sync() == md.MD_E_CAPACITY and sim.info()["step"] == 0
    p, _, _ = sim.get_state()
    assert np.abs(p - 0.9 * s.pos).max() < 1e-9
    sim.set_state(s.pos, s.vel)
    f, _, _ = sim.forces()
    fr, _, _ = oracle.forces_cells(s.params, s.box, s.species, s.pos)
    assert np.abs(f - fr).max() <= 1e-5 * np.sqrt((fr ** 2).sum(axis=1).mean())
    sim.step(20)
    assert sim.sync() == md.MD_OK and sim.info()["step"] == 20
    sim.close()


@pytest.mark.parametrize("prec", ["mixed", "fp64", "fp32"])
@pytest.mark.parametrize("where", ["step", "rebuild"])
def test_a_wait_that_ran_out_is_reported_and_a_new_state_mends_it(md, prec, where):
    """The barriers' limit set to one poll: a launch ends with MD_E_TIMEOUT inside a
    step or inside a rebuild (after its binning has counted the particles).  The
    handle then refuses what needs the state it lost, and goes on bit for bit like
    a fresh one once a state has been loaded."""
    s = synth.perturb(synth.ka_mixture(n=2000, temperature=1.0, seed=3), 0.05, 103)
    sim = _sim(md, s, precision=md.PRECISIONS[prec])
    sim.step(20)
    assert sim.sync() == md.MD_OK
    for reported in (True, False):
        md.md_set_wait_limit(sim.h, 1)
        if where == "step":
            sim.step(20)
            sim.step(20)
        else:
            sim.set_state(s.pos, s.vel)
        md.md_set_wait_limit(sim.h, 0)
        if reported:
            assert sim.sync() == md.MD_E_TIMEOUT
            assert sim.sync() == md.MD_OK
            for call in (lambda: sim.step(1), sim.get_state, sim.forces, sim.neighbours, lambda: sim.rescale(1.0),
                         lambda: sim.andersen(1.0, 1, 0)):
                with pytest.raises(md.MDError) as ei:
                    call()
                assert ei.value.code == md.MD_E_TIMEOUT and "md_set_state" in str(ei.value)
        else:
            with pytest.raises(md.MDError) as ei:            # (the read-back reports it)
                sim.get_state()
            assert ei.value.code == md.MD_E_TIMEOUT
        sim.set_state(s.pos, s.vel)
        f, _, _ = sim.forces()
        ref = _sim(md, s, precision=md.PRECISIONS[prec])
        fr, _, _ = ref.forces()
        assert np.array_equal(f, fr)
        sim.step(40)
        ref.step(40)
        assert sim.sync() == md.MD_OK and ref.sync() == md.MD_OK
        for x, y in zip(sim.get_state(), ref.get_state()):
            assert np.array_equal(x, y)
        ref.close()
    sim.close()
