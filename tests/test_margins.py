"""Margins of the single-precision tests that precede exact work: the FP64 pair
loop's cutoff test and the list distances, in boxes and with cutoffs large
enough for their rounding to count.  Lengths are in whatever unit the caller
takes: argon in picometres has sigma = 340 and r_c = 850."""
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


def _params(sigma, h=0.0):
    p = synth.lj_params()
    for k in ("sigma", "rcut"):
        p[k] = [[sigma * v for v in row] for row in p[k]]
    if h:
        p["smooth"] = h
    return p


def _pairs(L, m, sep, offset, rng):
    """m^3 pairs, first particles on a grid of spacing L / m shifted by `offset`,
    second particles at the distances sep() in random directions."""
    g = np.arange(m) * (L / m)
    c = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + offset
    u = rng.standard_normal((len(c), 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    pos = np.empty((2 * len(c), 3))
    pos[0::2] = c
    pos[1::2] = c + u * sep(len(c))[:, None]
    return np.mod(pos, L)


@pytest.mark.parametrize("tpp,h", [(0, 0.0), (4, 0.0), (1, 0.0), (4, 0.005)])
@pytest.mark.parametrize("sigma,L", [(1.0, 24.0), (3.4, 100.0), (34.0, 850.0), (340.0, 8500.0)])
def test_fp64_finds_pairs_just_inside_a_large_cutoff(md, sigma, L, tpp, h):
    """Pairs 1e-10 to 1e-7 of r_c inside the cutoff, a quarter of them near the
    upper box faces, where a coordinate cut to 24 bits is off by most.  Without
    smoothing a pair that the first test drops misses the force at the cutoff.
    Bound on the rest: separations are off by 2 ulp of L (L <= 30 sigma), 5e-15 of
    r_c, forces by seven times that, and the sums have a few terms: 1e-13, taken as
    1e-12 of the largest force; energies by the force times 1.4e-14 sigma."""
    rc = 2.5 * sigma
    fcut = 24.0 / rc * 0.4 ** 6
    p = _params(sigma, h)
    for seed in range(4):
        rng = np.random.default_rng(seed)
        pos = _pairs(L, 4, lambda k: rc * (1.0 - 10.0 ** rng.uniform(-10, -7, k)), rng.uniform(-0.4 * rc, 0.4 * rc, 3), rng)
        n = len(pos)
        sp = np.zeros(n, dtype=np.int32)
        fr, er, _ = oracle.forces_brute(p, L, sp, pos)
        tol = 1e-12 * max(np.abs(fr).max(), fcut)
        assert fcut > 1e3 * tol
        q = md.make_params(p, 0.001, precision=md.MD_PREC_FP64, threads_per_particle=tpp)
        sim = md.System(q, [n], [L], sp, pos, np.zeros((n, 3)))
        f, e, _ = sim.forces()
        sim.close()
        assert np.abs(f - fr).max() <= tol
        assert np.abs(e - er).max() <= 1e-13 * max(np.abs(er).max(), 1.0)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("form", [1, 2])
def test_lists_hold_every_pair_within_the_list_radius_of_a_large_box(md, prec, form):
    """r_c 50, skin 0.3, L 1500, where a single-precision coordinate is good to
    6e-5: isolated pairs up to 2e-5 inside the list radius, at and away from the
    box faces, are all listed (the margin of 1e-4 is there for the rounding of
    the distances alone), and pairs 1e-3 outside it are not."""
    sigma, L, rl = 20.0, 1500.0, 50.3
    p = _params(sigma)
    for seed in range(3):
        rng = np.random.default_rng(seed)
        sep = lambda k: np.where(np.arange(k) % 8 == 7, rl + 1e-3, rl - rng.uniform(1e-8, 2e-5, k))
        pos = _pairs(L, 8, sep, rng.uniform(-40.0, 40.0, 3), rng)
        n = len(pos)
        q = md.make_params(p, 0.001, precision=md.PRECISIONS[prec], build_form=form)
        sim = md.System(q, [n], [L], np.zeros(n, dtype=np.int32), pos, np.zeros((n, 3)))
        held, _, _ = sim.get_state()
        counts, lists = sim.neighbours()
        sim.close()
        d = held[0::2] - held[1::2]
        d -= L * np.round(d / L)
        r = np.repeat(np.sqrt((d ** 2).sum(1)), 2)           # distances of the positions held
        listed = np.array([counts[i] == 1 and lists[i, 0] == (i ^ 1) for i in range(n)])
        assert listed[r < rl].all()
        assert not listed[r > rl + 4e-4].any()
