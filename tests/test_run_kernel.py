"""The run kernel's phases and the kernels beside it at the sizes where they can
go wrong: cells beyond the direct scan, rows shorter than the lanes, boxes of
fewer than three cells, samples at every interval, more replicas than groups of
threads, coordinates on the box faces and far outside the box, copies shared
out over threads."""
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


def _ferr(f, ref):
    return np.abs(f - ref).max() / np.sqrt((ref ** 2).sum(axis=1).mean())


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_cells_beyond_the_direct_scan(md, prec, tol):
    """A droplet in a box of 21^3 = 9261 cells, most of them empty: forces equal
    the oracle's, and 80 steps with rebuilds agree bit for bit between one launch
    and a launch per phase."""
    s = synth.perturb(synth.lj_fluid(n=864, temperature=0.722, seed=4), 0.05, 104)
    box = 60.0
    runs = []
    for use_graph in (True, False):
        # (the droplet's lists are a liquid's, up to ~110 entries; the automatic capacity goes by
        # the mean density of the box)
        p = md.make_params(s.params, 0.005, precision=md.PRECISIONS[prec], use_graph=use_graph, neigh_capacity=160)
        sim = md.System(p, [s.n], [box], s.species, s.pos + 24.0, s.vel)
        assert sim.info()["cells_per_edge"] == 21
        f, _, _ = sim.forces()
        fr, _, _ = oracle.forces_cells(s.params, box, s.species, s.pos + 24.0)
        assert _ferr(f, fr) <= tol
        sim.step(80)
        assert sim.sync() == md.MD_OK and sim.info()["rebuilds"] >= 4
        runs.append(sim.get_state())
        sim.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("tpp", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("kind,n,density", [("ka", 700, 1.2), ("lj", 333, 0.05), ("ka", 1500, 1.2)])
def test_fp64_pair_queue(md, tpp, kind, n, density):
    """FP64 forces at every number of lanes: rows of ~100 entries in several
    rounds, rows shorter than the lanes, particles exactly on the box faces."""
    params = synth.ka_params() if kind == "ka" else synth.lj_params()
    s = synth.perturb(synth.make_system(n, density, 0.7, 6, params), 0.08, 106)
    s.pos[0, 0] = 0.0
    s.pos[1, 1] = 0.0
    s.pos[2, 2] = np.nextafter(s.box, 0.0)
    p = md.make_params(s.params, 0.001, precision=md.MD_PREC_FP64, threads_per_particle=tpp)
    sim = md.System(p, [s.n], [s.box], s.species, s.pos, s.vel)
    f, e, tot = sim.forces()
    sim.close()
    fr, er, w7 = oracle.forces_brute(s.params, s.box, s.species, s.pos)
    # FP64 sums of ~60 pairs of up to |F| ~ 1e3: 60 eps against an rms force of order 10
    assert _ferr(f, fr) <= 1e-12 * max(1.0, np.abs(fr).max() / np.sqrt((fr ** 2).sum(axis=1).mean()))
    assert abs(tot["e_pot"][0] - er.sum()) <= 1e-12 * np.abs(er).sum()


@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("n,density", [(200, 0.8442), (150, 0.5), (2, 0.01)])
def test_build_forms_in_boxes_of_fewer_than_three_cells(md, prec, n, density):
    """One cell that is its own stencil: nearest images are taken pair by pair.
    Both build forms give the same lists, and those of the definition."""
    s = synth.perturb(synth.make_system(n, density, 0.7, 8, synth.lj_params()), 0.1 if n > 2 else 0.0, 108)
    box = max(s.box, 5.8)
    lists = []
    for form in (1, 2):
        p = md.make_params(s.params, 0.001, precision=md.PRECISIONS[prec], build_form=form)
        sim = md.System(p, [n], [box], s.species, s.pos, s.vel)
        lists.append(sim.neighbours())
        sim.close()
    assert np.array_equal(lists[0][0], lists[1][0]) and np.array_equal(lists[0][1], lists[1][1])
    inner, _ = oracle.neighbours_brute(s.params, box, s.species, s.pos, 0.3 - 1e-4, kmax=512)
    outer, _ = oracle.neighbours_brute(s.params, box, s.species, s.pos, 0.3 + 1e-3, kmax=512)
    assert (lists[0][0] >= inner).all() and (lists[0][0] <= outer).all()


@pytest.mark.parametrize("interval", [1, 2, 3, 7])
def test_samples_and_energies_at_short_intervals(md, interval):
    """Consecutive samples (every step, so that one step's sums are added up while
    the next is sampled), md_step calls of 1 to 20 steps: the records of one launch
    and of a launch per phase are equal, and a sample's energy is the series'."""
    s = synth.perturb(synth.ka_mixture(n=1500, temperature=0.9, seed=9), 0.05, 109)
    got = []
    for use_graph in (True, False):
        p = md.make_params(s.params, 0.002, sample_interval=interval, use_graph=use_graph)
        sim = md.System(p, [s.n], [s.box], s.species, s.pos, s.vel)
        for k in (1, 2, 20, 5, 1):
            sim.step(k)
        assert sim.sync() == md.MD_OK
        obs = sim.observables()
        st, e = sim.epot_series()
        sim.close()
        assert np.array_equal(st, np.arange(30))
        assert np.array_equal(obs["step"][:, 0], np.arange(0, 30, interval))
        assert np.array_equal(e[obs["step"][:, 0], 0], obs["e_pot"][:, 0])
        assert (obs["max_disp"] >= 0).all() and (obs["max_disp"] > 0).any()   # (0 right after a rebuild)
        got.append((obs, e))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


def test_more_replicas_than_groups(md):
    """1100 copies of one small system (more than the 1064 groups of a GB300):
    every copy has the same energies."""
    s = synth.perturb(synth.ka_mixture(n=160, temperature=0.7, seed=3), 0.05, 103)
    box, r = max(s.box, 5.7), 1100
    p = md.make_params(s.params, 0.001, sample_interval=10)
    sim = md.System(p, [s.n] * r, [box] * r, np.tile(s.species, r), np.tile(s.pos, (r, 1)), np.tile(s.vel, (r, 1)))
    sim.step(30)
    assert sim.sync() == md.MD_OK
    obs = sim.observables()
    st, e = sim.epot_series()
    sim.close()
    assert obs.shape == (4, r) and e.shape == (31, r)
    assert (e == e[:, :1]).all()
    for k in ("e_pot", "e_kin", "virial"):
        assert (obs[k] == obs[k][:, :1]).all()


@pytest.mark.parametrize("prec,tpp", [("mixed", 1), ("mixed", 8), ("fp64", 4), ("fp32", 2)])
def test_chunks_shared_out_over_one_and_over_many_sweeps(md, prec, tpp):
    """One system alone (a chunk per group at most, sums per group) and as one of
    enough copies that every group sweeps several chunks (sums per chunk): equal
    states of every copy after 60 steps with rebuilds, bit for bit, and the same
    energies up to the order of their sums."""
    n, steps = 2000, 60
    s = synth.perturb(synth.ka_mixture(n=n, temperature=1.5, seed=5), 0.05, 105)
    r = 3 * 1064 * 128 // tpp // n + 1                         # > 3 chunks per group of a GB300
    # (the maxima behind the rebuild decision are those of all replicas, here the same)
    p = md.make_params(s.params, 0.002, precision=md.PRECISIONS[prec], threads_per_particle=tpp, check_interval=4,
                       sample_interval=20, obs_capacity=128)
    one = md.System(p, [n], [s.box], s.species, s.pos, s.vel)
    all_ = md.System(p, [n] * r, [s.box] * r, np.tile(s.species, r), np.tile(s.pos, (r, 1)), np.tile(s.vel, (r, 1)))
    for sim in (one, all_):
        sim.step(steps)
        assert sim.sync() == md.MD_OK and sim.info()["rebuilds"] >= 3
    for a, b in zip(one.get_state(), all_.get_state()):
        assert np.array_equal(np.tile(a, (r, 1)), b)
    o1, o2 = one.observables(), all_.observables()
    e1, e2 = one.epot_series()[1], all_.epot_series()[1]
    one.close()
    all_.close()
    assert np.array_equal(o1["step"], o2["step"][:, :1])
    # sums of 2000 terms in double, or energies in double-single (2^-44 a sum)
    for k in ("e_pot", "e_kin", "virial"):
        assert np.abs(o2[k] / o1[k] - 1.0).max() <= 1e-10
    assert np.abs(e2 / e1 - 1.0).max() <= 1e-10


@pytest.mark.parametrize("n", [2, 31, 33, 513, 1030])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("far", [0.0, 2.0e3, 1.0e6])
def test_noalloc_sizes_and_far_coordinates(md, n, prec, far):
    """Edges of the tiles and warps, and coordinates up to `far` boxes away (beyond
    2^18 boxes every pair goes through the exact evaluation)."""
    import torch
    s = synth.perturb(synth.make_system(n, min(1.2, n / 6.0 ** 3), 0.7, 12, synth.ka_params()), 0.05, 112)
    shift = np.round(np.random.RandomState(1).uniform(-far, far, (n, 3)))
    pos = s.pos + s.box * shift
    d = {k: torch.from_numpy(v).cuda() for k, v in (("species", s.species), ("pos", pos))}
    f = torch.empty(n, 3, dtype=torch.float64, device="cuda")
    e = torch.empty(n, dtype=torch.float64, device="cuda")
    t = torch.empty(8, dtype=torch.float64, device="cuda")
    p = md.make_params(s.params, 0.001, precision=md.PRECISIONS[prec])
    md.md_forces_noalloc(p, n, s.box, d["species"].data_ptr(), d["pos"].data_ptr(), f.data_ptr(), e.data_ptr(),
                         t.data_ptr(), torch.cuda.current_stream().cuda_stream)
    fr, er, w7 = oracle.forces_brute(s.params, s.box, s.species, np.mod(pos, s.box))
    # separations are off by a few ulp of the coordinates; the force changes by at most ~|F| 40 / r per
    # length (r >= 0.7)
    ulp = np.abs(pos).max() * 2.0 ** -51
    scale = max(np.abs(fr).max(), 1e-3)
    tol = (1e-12 if prec == "fp64" else 5e-6) * scale + 100.0 * scale * ulp
    assert np.abs(f.cpu().numpy() - fr).max() <= tol
    assert abs(t[0].item() - er.sum()) <= (1e-12 if prec == "fp64" else 5e-6) * np.abs(er).sum() + 50 * n * scale * ulp + 1e-12


@pytest.mark.parametrize("n", [30000, 150001])
def test_state_copies_shared_over_threads(md, n):
    """Arrays large enough for several copying threads, sizes that they do not
    divide: what goes in comes out."""
    s = synth.make_system(n, 0.8442, 1.0, 2, synth.lj_params())
    img = np.random.RandomState(3).randint(-5, 6, (n, 3)).astype(np.int32)
    p = md.make_params(s.params, 0.001, precision=md.MD_PREC_FP64)
    sim = md.System(p, [n], [s.box], s.species, s.pos, s.vel, img)
    pos, vel, im = sim.get_state()
    assert np.array_equal(pos, s.pos) and np.array_equal(vel, s.vel) and np.array_equal(im, img)
    sim.set_state(pos[::-1], vel[::-1], im[::-1])
    pos, vel, im = sim.get_state()
    sim.close()
    assert np.array_equal(pos, s.pos[::-1]) and np.array_equal(vel, s.vel[::-1]) and np.array_equal(im, img[::-1])
