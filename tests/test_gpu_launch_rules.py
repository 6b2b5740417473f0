"""Launch shapes the library chooses by itself (GPU): the +-1 cubic and chain
sweeps and the Gaussian cubic sweep with one and with two replicas per thread
against the oracle."""
import time

import numpy as np
import pytest

from oracle import oracle as o
from paper_1006_0252_gb300 import inputs, pa

pytestmark = pytest.mark.gpu


# (L, R0, threads per replica): the largest odd populations that take one
# replica a thread (R0 P <= 900 x 152) and the smallest that take two, whose
# last columns hold one replica; L = 12 also past 50000, where it splits less.
@pytest.mark.parametrize("L,R0,split", [(2, 4001, 1), (4, 34199, 4), (4, 34201, 4), (6, 45601, 3), (8, 17099, 8),
                                        (8, 17101, 8), (10, 27361, 5), (12, 11401, 12), (12, 50001, 6),
                                        (14, 19543, 7), (16, 17101, 8)])
def test_chosen_shape_bit_exact(L, R0, split):
    """One sweep each where every compare runs, where the thr(8) and thr(12)
    compares are mostly skipped, and where the minimum skips all of them."""
    J = inputs.couplings_3d(L, 2, 9)
    cap = R0 + 4000
    g = pa.Run(J, L, 3, R0, 23, R_cap=cap)
    assert pa.pa_sweep_shape(g._h)[1] == split
    c = o.Run(J, 3, L, L, L, 7, R0=R0, R_cap=cap, seed=23)
    for beta, sweeps in ((0.1, 1), (0.5, 0), (0.9, 0), (1.2, 0), (1.5, 1), (1.9, 0), (2.6, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
    go, co = g.observables(), c.state()
    assert go["R"] == co.R and go["sumE"] == co.sumE and go["sumE2"] == co.sumE2
    assert np.array_equal(g.energies(), c.energies())
    assert np.array_equal(g.spins(), c.spins())
    assert abs(go["minus_beta_F"] - co.minus_beta_F) <= 1e-12 * abs(co.minus_beta_F)


# (N, open, R0): chains of 3, 5, 8, 32 and 128 words, short last words, odd
# length, one and two replicas a thread.
@pytest.mark.parametrize("N,is_open,R0", [(70, False, 40001), (130, True, 34201), (256, False, 17099),
                                          (256, False, 17101), (1001, True, 17101), (1000, False, 17101),
                                          (4096, True, 17101), (4094, False, 17103)])
def test_chosen_chain_shape_bit_exact(N, is_open, R0):
    J = inputs.couplings_chain(N, 2, 9, open_chain=is_open)
    J[N // 3] = 0  # a diluted chain: two sites inside have one bond
    cap = R0 + 4000
    g = pa.Run(J, N, 1, R0, 29, R_cap=cap)
    c = o.Run(J, 1, N, R0=R0, R_cap=cap, seed=29)
    for beta, sweeps in ((0.1, 1), (0.5, 0), (1.0, 1), (1.5, 0), (2.0, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
    go, co = g.observables(), c.state()
    assert go["R"] == co.R and go["sumE"] == co.sumE and go["sumE2"] == co.sumE2
    assert np.array_equal(g.energies(), c.energies())
    assert np.array_equal(g.spins(), c.spins())


# (L, R0): Gaussian couplings; the largest odd populations that take one replica
# a thread and the smallest that take two (600 threads an SM; 400 at L = 6, 10).
# The betas give thresholds of 2^24 to rises (1e-6), ordinary ones, and 0 (60).
@pytest.mark.parametrize("L,R0,split", [(4, 22799, 4), (4, 22801, 4), (6, 20265, 3), (6, 20267, 3), (8, 301, 8),
                                        (8, 11399, 8), (8, 11401, 8), (10, 12159, 5), (10, 12161, 5)])
def test_chosen_gauss_shape_bit_exact(L, R0, split):
    J = inputs.gaussian_couplings_3d(L, 4, 1)
    cap = R0 + 4000
    g = pa.Run(J, L, 3, R0, 31, R_cap=cap, gaussian=True)
    assert pa.pa_sweep_shape(g._h) == (1024, split)
    c = o.GaussRun(J, 3, L, L, L, 7, R0=R0, R_cap=cap, seed=31)
    for beta, sweeps in ((1e-6, 1), (0.4, 1), (0.9, 0), (1.5, 1), (3.0, 0), (8.0, 0), (20.0, 0), (60.0, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
        assert g.observables()["R"] == c.state().R, beta
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.energies(), c.energies())
    assert np.array_equal(g.spins(), c.spins())


# (N, open, R0, threads per replica): Gaussian chains of 1, 2, 4, 8, 32 and 128
# words, short last words, odd length, one and two replicas a thread.
@pytest.mark.parametrize("N,is_open,R0,split", [(30, False, 501, 1), (64, False, 501, 2), (34, False, 68401, 2),
                                                (103, True, 34201, 4), (256, False, 17099, 8), (258, False, 17101, 8),
                                                (1001, True, 17101, 8), (4096, False, 301, 8)])
def test_chosen_gauss_chain_shape_bit_exact(N, is_open, R0, split):
    J = inputs.gaussian_couplings_chain(N, 2, 9, open_chain=is_open)
    J[N // 3] = 0  # both neighbours' alignments give the same energy change
    cap = R0 + 4000
    g = pa.Run(J, N, 1, R0, 37, R_cap=cap, gaussian=True)
    assert pa.pa_sweep_shape(g._h)[1] == split
    c = o.GaussRun(J, 1, N, R0=R0, R_cap=cap, seed=37)
    for beta, sweeps in ((1e-6, 1), (0.5, 1), (1.0, 0), (2.0, 1), (5.0, 0), (12.0, 0), (30.0, 0), (80.0, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
        assert g.observables()["R"] == c.state().R, beta
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.energies(), c.energies())
    assert np.array_equal(g.spins(), c.spins())


# (Lx, Ly, Lz, periodic mask, R0): general boxes whose words hold 4, 6, 8, 9, 12,
# 15 and 16 sites of a colour (uniforms that start a call again after 1, 2 and 4
# words), with 1, 2 and 4 replicas a thread.
@pytest.mark.parametrize("gaussian", [False, True])
@pytest.mark.parametrize("Lx,Ly,Lz,mask,R0", [(8, 6, 5, 3, 20001), (8, 6, 5, 3, 1999), (4, 4, 3, 3, 30001),
                                              (4, 8, 8, 3, 5003), (6, 4, 3, 3, 20003), (8, 4, 3, 3, 9001),
                                              (6, 8, 5, 3, 8009), (8, 8, 8, 3, 7001), (2, 3, 2, 0, 40001),
                                              (32, 2, 3, 1, 2503)])
def test_chosen_box_shape_bit_exact(Lx, Ly, Lz, mask, R0, gaussian):
    J = inputs.gaussian_couplings_lattice(Lx, Ly, Lz, 6) if gaussian else inputs.couplings_lattice(Lx, Ly, Lz, 6, 3)
    cap = R0 + 4000
    g = pa.Run(J, Lx, 3, R0, 41, R_cap=cap, gaussian=gaussian, Ls=(Lx, Ly, Lz), periodic_mask=mask)
    assert pa.pa_sweep_shape(g._h)[0] == 1024
    c = (o.GaussRun if gaussian else o.Run)(J, 3, Lx, Ly, Lz, mask, R0=R0, R_cap=cap, seed=41)
    for beta, sweeps in ((1e-6, 1), (0.4, 1), (0.9, 0), (1.5, 1), (2.5, 0), (5.0, 0), (12.0, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
        assert g.observables()["R"] == c.state().R, beta
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.energies().astype(np.int64), c.energies().astype(np.int64))
    assert np.array_equal(g.spins(), c.spins())


# Populations resampled by one block (capacity up to 2048: passes of 1024
# replicas) and by one block per 256 replicas; heavy replicas, a step that
# changes nothing, and the state after a step that outgrows the capacity.
@pytest.mark.parametrize("R0,cap", [(40, 400), (1024, 1500), (1025, 2048), (1600, 2048), (1600, 2049), (5121, 8000)])
def test_resampling_paths_bit_exact(R0, cap):
    J = inputs.couplings_3d(4, 3, 9)
    g = pa.Run(J, 4, 3, R0, 43, R_cap=cap)
    c = o.Run(J, 3, 4, 4, 4, 7, R0=R0, R_cap=cap, seed=43)
    for beta in (0.2, 0.2, 1.6, 5.0):
        Rprev = c.state().R
        g.step(beta, 1)
        c.step(beta, 1, R0)
        assert np.array_equal(g.copies(Rprev), c.copies(Rprev)), beta
        assert g.observables()["R"] == c.state().R, beta
        assert np.array_equal(g.energies(), c.energies()), beta
    assert np.array_equal(g.spins(), c.spins())
    E = g.energies()
    with pytest.raises(pa.PAError) as e:
        g.step(5.1, 1, R_target=40 * cap)
        g.sync()
    assert e.value.code == pa.PA_ERR_CAPACITY
    assert np.array_equal(pa.pa_copy_energies(g._h, cap), E)


# A schedule of small runs commits a step at the start of the next: the same states as steps
# committed one by one, with and without a graph.
@pytest.mark.parametrize("gaussian,R0", [(False, 900), (False, 5000), (True, 900)])
@pytest.mark.parametrize("use_graph", [False, True])
def test_schedule_commits_every_step(gaussian, R0, use_graph):
    J = inputs.gaussian_couplings_3d(4, 3, 9) if gaussian else inputs.couplings_3d(4, 3, 9)
    betas = np.array([0.1, 0.3, 0.3, 0.7])
    a, b = (pa.Run(J, 4, 3, R0, 47, gaussian=gaussian) for _ in range(2))
    a.run_schedule(betas, np.full(4, 2), use_graph=use_graph)
    a.sync()
    for beta in betas:
        b.step(float(beta), 2)
    assert a.observables() == b.observables()
    ta, tb = a.trajectory(), b.trajectory()
    assert all(np.array_equal(ta[k], tb[k]) for k in tb)
    assert np.array_equal(a.spins(), b.spins())


# Bootstrap with tabulated weights: one run, a lane's worth and more of them,
# population factors and the observable given or not, and weights so far apart
# that most resamples miss the runs that carry them (1e-200 of the largest).
@pytest.mark.parametrize("M,B", [(1, 2), (2, 33), (33, 129), (200, 64)])
@pytest.mark.parametrize("spread", [0.9, 3000.0])
def test_bootstrap_weights(M, B, spread):
    rng = np.random.default_rng(M)
    x, A = rng.normal(2500.0, spread, M), rng.normal(-600.0, 4.0, M)
    R = rng.integers(20000, 80000, M).astype(np.float64)
    for args in ((x, A, R), (x, A, None), (x, None, R), (x, None, None)):
        g, want = pa.pa_bootstrap(*args, B=B, seed=9), o.bootstrap(*args, B=B, seed=9)
        # values of ~3e3 agree to a few units of 2^-53 a draw; their spread may
        # cancel to zero where every resample is the same
        for a, b in zip(g, want):
            assert abs(a - b) <= 1e-9 * abs(b) + 1e-10, (M, B, spread, a, b)


# Weighted averages by a warp (up to 32 runs) and by a block of 256 threads.
@pytest.mark.parametrize("M", [32, 33, 256, 257, 1000])
def test_weighted_average_sizes(M):
    rng = np.random.default_rng(M)
    x, x2, A = rng.normal(2500.0, 0.9, M), rng.normal(2500.0, 0.9, M), rng.normal(-600.0, 4.0, M)
    R = rng.integers(20000, 80000, M).astype(np.float64)
    for Rw in (R, None):
        # sums of M terms in FP64, relative to their own size: 1e-12
        for got, want in ((pa.pa_weighted_average(x, A, Rw), o.weighted_average(x, A, Rw)),
                          (pa.pa_weighted_average_pairs(x, x2, A, Rw, Rw),
                           o.weighted_average(x + x2, A, None if Rw is None else Rw * Rw))):
            assert all(abs(a - b) <= 1e-12 * abs(b) for a, b in zip(got, want)), (M, got, want)


# Classes swept side by side, in a graph and (from 2^20 spins outside the
# largest class) launch by launch: every run ends as it does alone.
@pytest.mark.parametrize("use_graph", [False, True])
def test_classes_side_by_side(use_graph):
    betas = np.array([0.2, 0.5, 0.9])
    sizes = [(8, 3001), (6, 6001), (8, 2999), (4, 3000)]
    specs = [inputs.RunSpec(3, L, 0, 50 + i, R0, betas, 2) for i, (L, R0) in enumerate(sizes)]
    b = pa.Batch(specs)
    b.run(betas, thetas=2, use_graph=use_graph)
    assert not b.sync().any()
    res = b.results()
    for r, (L, R0) in enumerate(sizes):
        g = pa.Run(specs[r].couplings(), L, 3, R0, 50 + r)
        g.run_schedule(betas, np.full(3, 2))
        ob = g.observables()
        assert res["R"][r] == ob["R"] and res["sumE"][r] == ob["sumE"] and res["sumE2"][r] == ob["sumE2"], r
        assert np.array_equal(b.spins(r, ob["R"]), g.spins()), r


# Uniforms of exactly 0 (found by search: seed, slot, sweep, colour, call) at
# thresholds of 0: such a site must stay, where any other threshold lets it go.
@pytest.mark.parametrize("seed,slot,T,c,q", [(699, 356, 1, 0, 5), (3247, 1167, 3, 0, 8), (3332, 1187, 1, 1, 19),
                                             (3760, 1084, 0, 0, 22), (3878, 231, 3, 0, 2), (3932, 1324, 4, 1, 3)])
def test_uniform_zero_against_threshold_zero(seed, slot, T, c, q):
    R0, beta = 1600, 200.0  # e^{-beta dE} is below 2^-32 for every rise of +-1 and almost every Gaussian one
    made = []
    for g in (False, True):
        J = inputs.gaussian_couplings_lattice(8, 6, 5, 3) if g else inputs.couplings_lattice(8, 6, 5, 3, 1)
        made.append((J, g, (8, 6, 5), 3))
    made += [(inputs.gaussian_couplings_3d(L, 3, 1), True, (L, L, L), 7) for L in (6, 8, 10)]
    made += [(inputs.couplings_3d(8, 3, 1), False, (8, 8, 8), 7)]
    for J, g, (Lx, Ly, Lz), mask in made:
        a = pa.Run(J, Lx, 3, R0, seed, R_cap=3000, gaussian=g, Ls=(Lx, Ly, Lz), periodic_mask=mask)
        b = (o.GaussRun if g else o.Run)(J, 3, Lx, Ly, Lz, mask, R0=R0, R_cap=3000, seed=seed)
        a.step(beta, 6)
        b.step(beta, 6, R0)
        assert a.observables()["R"] > slot
        assert np.array_equal(a.spins(), b.spins()), (Lx, Ly, Lz, g)
    J = inputs.gaussian_couplings_chain(256, 3, 1, open_chain=False)
    a, b = pa.Run(J, 256, 1, R0, seed, R_cap=3000, gaussian=True), o.GaussRun(J, 1, 256, R0=R0, R_cap=3000, seed=seed)
    a.step(beta, 6)
    b.step(beta, 6, R0)
    assert np.array_equal(a.spins(), b.spins())


# Gaussian cubic lattices with every number of threads per replica that their
# rows split into, in every block size: what the threshold tables have no shape
# for (L = 10 with one thread a replica) runs in a smaller block.
@pytest.mark.parametrize("L,split", [(4, 1), (4, 2), (4, 4), (6, 1), (8, 1), (8, 2), (8, 4), (10, 1), (12, 1), (12, 2)])
@pytest.mark.parametrize("tpb", [0, 128, 512, 1024])
def test_gauss_cubic_asked_shape_bit_exact(L, split, tpb):
    J = inputs.gaussian_couplings_3d(L, 4, 1)
    g = pa.Run(J, L, 3, 301, 53, gaussian=True, threads_per_block=tpb, threads_per_replica=split)
    assert pa.pa_sweep_shape(g._h)[1] == split
    c = o.GaussRun(J, 3, L, L, L, 7, R0=301, seed=53)
    for beta in (0.4, 1.5):
        g.step(beta, 1)
        c.step(beta, 1, 301)
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.spins(), c.spins())


# More runs than SMs: blocks of 256 threads, here with up to six passes over a population and
# runs of a few replicas among them.
def test_many_small_runs_bit_exact():
    betas = np.array([0.2, 0.7, 2.5])
    specs = [inputs.RunSpec(3, 4, r % 5, 100 + r, (40, 255, 256, 700, 1400)[r % 5], betas, 1) for r in range(160)]
    b = pa.Batch(specs)
    b.run(betas, thetas=1)
    assert not b.sync().any()
    res = b.results()
    for r in (0, 1, 2, 3, 4, 77, 158, 159):
        R0 = specs[r].R0
        c = o.Run(specs[r].couplings(), 3, 4, 4, 4, 7, R0=R0, seed=100 + r)
        for beta in betas:
            c.step(float(beta), 1, R0)
        assert res["R"][r] == c.state().R and res["sumE"][r] == c.state().sumE, r
        assert np.array_equal(b.spins(r, c.state().R), c.spins()), r


# ... and they take no longer than with the launches apart (capacities above
# 2048), where blocks of 1024 threads took 1.15 times as long.
def test_many_small_runs_take_no_longer():
    betas = np.linspace(0.05, 4.0, 40)

    def seconds(cap):
        b = pa.Batch([inputs.RunSpec(3, 4, 0, 50 + r, 100, betas, 10, R_cap=cap) for r in range(3000)], max_steps=64)
        times = []
        for _ in range(5):
            b.reset()
            b.sync()
            t = time.perf_counter()
            b.run(betas, thetas=10)
            b.sync()
            times.append(time.perf_counter() - t)
        return min(times)

    assert seconds(2048) <= 1.05 * seconds(2049)


# Boxes of up to four sites: site at a time in small populations.
@pytest.mark.parametrize("Lx,Ly,Lz,R0,tpb", [(2, 1, 1, 5000, 64), (2, 2, 1, 19999, 64), (2, 2, 1, 20000, 1024),
                                             (4, 2, 1, 5000, 1024)])
@pytest.mark.parametrize("gaussian", [False, True])
def test_tiny_box_shape_bit_exact(Lx, Ly, Lz, R0, tpb, gaussian):
    J = inputs.gaussian_couplings_lattice(Lx, Ly, Lz, 6) if gaussian else inputs.couplings_lattice(Lx, Ly, Lz, 6, 3)
    g = pa.Run(J, Lx, 3, R0, 41, R_cap=R0 + 4000, gaussian=gaussian, Ls=(Lx, Ly, Lz), periodic_mask=0)
    assert pa.pa_sweep_shape(g._h)[0] == tpb
    c = (o.GaussRun if gaussian else o.Run)(J, 3, Lx, Ly, Lz, 0, R0=R0, R_cap=R0 + 4000, seed=41)
    for beta, sweeps in ((0.4, 1), (1.5, 2)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.spins(), c.spins())


# Chains whose words the finest split leaves places idle for: coarser splits in large
# populations (the last range short, one and two replicas a thread).
@pytest.mark.parametrize("N,R0,split", [(130, 20000, 4), (130, 80001, 1), (190, 70001, 2), (260, 17400, 8),
                                        (260, 17501, 4), (260, 70001, 1), (340, 36001, 4)])
def test_coarser_chain_split_bit_exact(N, R0, split):
    J = inputs.couplings_chain(N, 2, 9, open_chain=True)
    J[N // 3] = 0
    g, c = pa.Run(J, N, 1, R0, 59), o.Run(J, 1, N, R0=R0, seed=59)
    assert pa.pa_sweep_shape(g._h)[1] == split
    for beta, sweeps in ((0.1, 1), (1.5, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.spins(), c.spins())


@pytest.mark.parametrize("N,R0,split", [(96, 18001, 2), (96, 70001, 1), (130, 40001, 2), (260, 18001, 4),
                                        (260, 40001, 2), (1100, 17501, 8), (1100, 76001, 4)])
def test_coarser_gauss_chain_split_bit_exact(N, R0, split):
    J = inputs.gaussian_couplings_chain(N, 2, 9, open_chain=False)
    g, c = pa.Run(J, N, 1, R0, 59, gaussian=True), o.GaussRun(J, 1, N, R0=R0, seed=59)
    assert pa.pa_sweep_shape(g._h)[1] == split
    for beta, sweeps in ((0.1, 1), (1.5, 1)):
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.spins(), c.spins())
