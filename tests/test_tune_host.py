"""The autotuner's choice of candidates, with the GPU trials replaced by a table of
times (host logic only)."""
import pytest

from paper_0912_3824_gb300 import md, synth, tune


def _tuned(monkeypatch, n, precision, times, auto, **kw):
    """autotune over fake handles: `times` by lanes, `auto` lanes by default."""
    class Fake:
        def __init__(self, p, *a, **k):
            self.lanes = p.threads_per_particle or auto

        def step(self, n):
            pass

        def sync(self):
            return md.MD_OK

        def info(self):
            return {"max_neighbours": 100, "neigh_capacity": 160, "threads_per_particle": self.lanes}

        def close(self):
            pass

    monkeypatch.setattr(md, "System", Fake)
    monkeypatch.setattr(tune, "_time", lambda torch, sim, steps, repeats: times[sim.lanes])
    s = synth.ka_mixture(n=n, temperature=0.7, seed=1)
    base = md.make_params(s.params, 0.001, precision=precision)
    return tune.autotune(base, [s.n], [s.box], s.species, s.pos, s.vel, **kw)


@pytest.mark.parametrize("precision,auto,times", [
    # us per MD step of the Kob-Andersen mixture at 1000 particles
    (md.MD_PREC_MIXED, 16, {1: 11.0, 2: 9.57, 4: 8.60, 8: 7.30, 16: 7.28}),
    (md.MD_PREC_FP64, 16, {2: 68.8, 4: 36.5, 8: 23.5, 16: 18.5})])
def test_tuned_is_never_slower_than_the_default(monkeypatch, precision, auto, times):
    p, trials = _tuned(monkeypatch, 1000, precision, times, auto, skins=(0.2, 0.3))
    assert p.threads_per_particle == auto
    seen = [(t["skin"], t["threads_per_particle"]) for t in trials]
    assert len(seen) == len(set(seen)) == 8                  # auto and the list, none twice


def test_the_automatic_lanes_are_not_timed_twice(monkeypatch):
    p, trials = _tuned(monkeypatch, 1000, md.MD_PREC_MIXED, {1: 3.0, 2: 2.0, 4: 2.5}, 2, skins=(0.3,))
    assert p.threads_per_particle == 2 and [t["threads_per_particle"] for t in trials] == [2, 1, 4]


def test_lanes_given_by_the_caller_are_the_only_ones(monkeypatch):
    p, trials = _tuned(monkeypatch, 1000, md.MD_PREC_MIXED, {1: 3.0, 2: 2.0, 16: 1.0}, 16, lanes=(1, 2), skins=(0.3,))
    assert [t["threads_per_particle"] for t in trials] == [1, 2] and p.threads_per_particle == 2
