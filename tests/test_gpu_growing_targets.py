"""Population targets far above R0 (GPU): the launch shapes follow them.  The
runs agree with the oracle before, at and after the change, and take the time
of a run that was made for the larger population."""
import numpy as np
import pytest

from oracle import oracle as o
from paper_1006_0252_gb300 import inputs, pa

pytestmark = pytest.mark.gpu


def _lattice(kind, L):
    """(couplings, dim, Ls, periodic mask, gaussian)."""
    gaussian = kind.startswith("gauss")
    if kind.endswith("cubic"):
        return (inputs.gaussian_couplings_3d if gaussian else inputs.couplings_3d)(L, 2, 9), 3, (L, L, L), 7, gaussian
    if kind.endswith("chain"):
        J = (inputs.gaussian_couplings_chain if gaussian else inputs.couplings_chain)(L, 2, 9, open_chain=not gaussian)
        return J, 1, (L, 1, 1), 7, gaussian
    return (inputs.gaussian_couplings_lattice if gaussian else inputs.couplings_lattice)(*L, 6), 3, L, 3, gaussian


def _run(kind, L, R0, seed, cap):
    J, dim, Ls, mask, gaussian = _lattice(kind, L)
    if kind.endswith("box"):
        return pa.Run(J, Ls[0], 3, R0, seed, R_cap=cap, gaussian=gaussian, Ls=Ls, periodic_mask=mask)
    return pa.Run(J, L, dim, R0, seed, R_cap=cap, gaussian=gaussian)


def _oracle(kind, L, R0, seed, cap):
    J, dim, Ls, mask, gaussian = _lattice(kind, L)
    return (o.GaussRun if gaussian else o.Run)(J, dim, *Ls, mask, R0=R0, R_cap=cap, seed=seed)


def _same(g, c):
    assert g.observables()["R"] == c.state().R
    assert np.array_equal(g.energies().astype(np.int64), c.energies().astype(np.int64))
    assert np.array_equal(g.spins(), c.spins())


# (lattice, R0, target): from one replica a thread to two, from small to large
# blocks and work items, with table entries to spare and without.
GROWN = [("cubic", 4, 300, 36000), ("cubic", 6, 300, 16000), ("cubic", 8, 300, 18000), ("cubic", 10, 300, 9000),
         ("cubic", 12, 200, 5000), ("gauss cubic", 4, 300, 24000), ("gauss cubic", 6, 300, 21000),
         ("gauss cubic", 8, 300, 12000), ("gauss cubic", 10, 100, 5000), ("gauss cubic", 12, 100, 1500),
         ("chain", 256, 300, 18000), ("gauss chain", 256, 300, 18000), ("box", (8, 6, 5), 300, 12000),
         ("gauss box", (6, 4, 3), 300, 12000)]


@pytest.mark.parametrize("kind,L,R0,target", GROWN)
def test_growing_targets_bit_exact(kind, L, R0, target):
    cap = target + 6000
    g, c = _run(kind, L, R0, 71, cap), _oracle(kind, L, R0, 71, cap)
    for beta, Rt in ((0.1, R0), (0.2, target // 3), (0.3, target), (0.4, R0)):
        g.step(beta, 1, R_target=Rt)
        c.step(beta, 1, Rt)
    _same(g, c)
    # the schedule's graph, captured before the change and after it; the reset
    # initialises the population with the larger work items
    betas, low, high = np.array([0.1, 0.2]), np.array([R0, R0]), np.array([R0, target])
    g = _run(kind, L, R0, 72, cap)
    for targets, seed in ((low, 72), (high, 73), (low, 74)):
        g.reset(seed)
        g.run_schedule(betas, np.full(2, 1), targets)
        c = _oracle(kind, L, R0, seed, cap)
        for beta, Rt in zip(betas, targets):
            c.step(float(beta), 1, int(Rt))
        _same(g, c)


@pytest.mark.parametrize("tune", [False, True])
def test_growing_batch_bit_exact(tune):
    sizes = [(8, 300, 9000), (10, 200, 4000), (8, 400, 400)]
    betas = np.array([0.1, 0.2, 0.3])
    specs = [inputs.RunSpec(3, L, 0, 80 + i, R0, betas, 1, R_cap=Rt + 6000) for i, (L, R0, Rt) in enumerate(sizes)]
    b = pa.Batch(specs)
    if tune:
        b.autotune(1)
    targets = np.array([[R0, Rt, Rt] for _, R0, Rt in sizes])
    b.run(np.broadcast_to(betas, (3, 3)).copy(), thetas=1, R_targets=targets)
    assert not b.sync().any()
    res = b.results()
    for r, (L, R0, Rt) in enumerate(sizes):
        c = o.Run(specs[r].couplings(), 3, L, L, L, 7, R0=R0, R_cap=Rt + 6000, seed=80 + r)
        for beta, t in zip(betas, targets[r]):
            c.step(float(beta), 1, int(t))
        assert res["R"][r] == c.state().R and res["sumE"][r] == c.state().sumE, r
        assert np.array_equal(b.spins(r, c.state().R), c.spins()), r


# Sweep time at a target 20 to 100 times R0 against a run made for it: at most
# half as much again (in the first shape it took 2 to 10 times as much).
@pytest.mark.parametrize("kind,L,R0,target", [("gauss cubic", 6, 1000, 50000), ("gauss cubic", 8, 1000, 100000),
                                              ("cubic", 8, 1000, 100000), ("chain", 256, 1000, 100000),
                                              ("gauss chain", 256, 1000, 100000), ("box", (8, 6, 5), 1000, 20000)])
def test_grown_run_takes_the_time_of_a_large_one(kind, L, R0, target):
    cap = target + 6000

    def sweep_ms(first):
        g = _run(kind, L, first, 75, cap)
        g.step(0.05, 1, R_target=target)
        best = float("inf")
        for k in range(4):
            g.sync()
            pa.pa_kernel_time(g._h, True)
            for i in range(3):
                g.step(0.05 + 0.01 * (3 * k + i + 1), 10, R_target=target)
            g.sync()
            best = min(best, pa.pa_kernel_time(g._h, False)[0])
        return best

    large, grown = sweep_ms(target), sweep_ms(R0)
    assert grown <= 1.5 * large, (grown, large)
