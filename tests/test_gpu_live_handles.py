"""Several live handles (GPU): what one holds of the process -- the
shared-memory limits of the kernels above all -- must not depend on what was
made after it.  Every run is compared with the oracle."""
import numpy as np
import pytest

from oracle import oracle as o
from paper_1006_0252_gb300 import inputs, pa

pytestmark = pytest.mark.gpu

SCHEDULE = ((0.3, 1), (0.9, 1))


def _run(kind, L, R0, seed):
    """A run and its oracle."""
    if kind == "cubic":
        J = inputs.couplings_3d(L, 2, 9)
        return pa.Run(J, L, 3, R0, seed), o.Run(J, 3, L, L, L, 7, R0=R0, seed=seed)
    if kind == "gauss cubic":
        J = inputs.gaussian_couplings_3d(L, 2, 9)
        return pa.Run(J, L, 3, R0, seed, gaussian=True), o.GaussRun(J, 3, L, L, L, 7, R0=R0, seed=seed)
    if kind == "chain":
        J = inputs.couplings_chain(L, 2, 9, open_chain=True)
        return pa.Run(J, L, 1, R0, seed), o.Run(J, 1, L, R0=R0, seed=seed)
    if kind == "gauss chain":
        J = inputs.gaussian_couplings_chain(L, 2, 9, open_chain=False)
        return pa.Run(J, L, 1, R0, seed, gaussian=True), o.GaussRun(J, 1, L, R0=R0, seed=seed)
    Lx, Ly, Lz = L
    gaussian = kind == "gauss box"
    J = inputs.gaussian_couplings_lattice(*L, 6) if gaussian else inputs.couplings_lattice(*L, 6, 3)
    return (pa.Run(J, Lx, 3, R0, seed, gaussian=gaussian, Ls=L, periodic_mask=3),
            (o.GaussRun if gaussian else o.Run)(J, 3, Lx, Ly, Lz, 3, R0=R0, seed=seed))


def _step_and_compare(g, c, R0, schedule=SCHEDULE):
    for beta, sweeps in schedule:
        g.step(beta, sweeps)
        c.step(beta, sweeps, R0)
        assert g.observables()["R"] == c.state().R, beta
    assert g.observables()["sumE"] == c.state().sumE
    assert np.array_equal(g.energies().astype(np.int64), c.energies().astype(np.int64))
    assert np.array_equal(g.spins(), c.spins())


# Pairs that share a kernel but not its shared memory: the first is stepped
# after the second was made, then reset (its initial-state kernel) and stepped
# again.  The boxes have equal words (4 and 16 sites of a colour) in lattices of
# different size.
@pytest.mark.parametrize("kind,first,second", [
    ("cubic", (8, 1000), (8, 3000)),
    ("cubic", (6, 2000), (6, 9000)),
    ("gauss cubic", (8, 300), (8, 2000)),
    ("chain", (4096, 300), (3500, 300)),
    ("chain", (256, 1000), (512, 3000)),
    ("gauss chain", (4096, 300), (3500, 300)),
    ("gauss chain", (256, 1000), (256, 9000)),
    ("box", ((8, 8, 7), 1000), ((8, 6, 5), 1000)),
    ("gauss box", ((8, 8, 8), 1000), ((4, 8, 8), 1000)),
])
def test_second_handle_leaves_the_first_alone(kind, first, second):
    g, c = _run(kind, *first, 61)
    g2, c2 = _run(kind, *second, 62)
    _step_and_compare(g, c, first[1])
    _step_and_compare(g2, c2, second[1])
    g.reset(63)
    _step_and_compare(g, _run(kind, *first, 63)[1], first[1])


# The same for a batch that was tuned (every shape of its classes tried) beside
# a live run, and for the batch itself beside a run made after it.
@pytest.mark.parametrize("kind", ["cubic", "chain"])
def test_autotuned_batch_beside_a_run(kind):
    betas = np.array([0.3, 0.9])
    L, dim = (8, 3) if kind == "cubic" else (256, 1)
    g, c = _run(kind, L, 1000, 64)
    specs = [inputs.RunSpec(dim, L, 0, 70 + i, 3000, betas, 1) for i in range(2)]
    b = pa.Batch(specs)
    b.autotune(1)
    _step_and_compare(g, c, 1000)
    late = _run(kind, L, 9000, 65)
    b.run(betas, thetas=1, use_graph=False)
    assert not b.sync().any()
    _step_and_compare(*late, 9000)
    res = b.results()
    for r, spec in enumerate(specs):
        alone = (o.Run(spec.couplings(), 3, L, L, L, 7, R0=3000, seed=70 + r) if dim == 3
                 else o.Run(spec.couplings(), 1, L, R0=3000, seed=70 + r))
        for beta in betas:
            alone.step(float(beta), 1, 3000)
        assert res["R"][r] == alone.state().R and res["sumE"][r] == alone.state().sumE, r


# Chains of different length share their kernel within one batch or server.
CHAINS = ((256, 1000), (512, 3000), (4096, 200), (3500, 200))


@pytest.mark.parametrize("gaussian", [False, True])
@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_of_chains_of_several_lengths(gaussian, use_graph):
    betas = np.array([0.3, 0.9])
    specs = [inputs.RunSpec(1, N, 0, 80 + i, R0, betas, 1, gaussian=gaussian, open_chain=not gaussian)
             for i, (N, R0) in enumerate(CHAINS)]
    b = pa.Batch(specs)
    b.run(betas, thetas=1, use_graph=use_graph)
    assert not b.sync().any()
    res = b.results()
    for r, (N, R0) in enumerate(CHAINS):
        c = (o.GaussRun if gaussian else o.Run)(specs[r].couplings(), 1, N, R0=R0, seed=80 + r)
        for beta in betas:
            c.step(float(beta), 1, R0)
        assert res["R"][r] == c.state().R and res["sumE"][r] == c.state().sumE, r


def test_server_of_chains_of_several_lengths():
    betas = np.array([0.3, 0.9])
    srv = pa.Server(max_runs=4)
    J = [inputs.couplings_chain(N, i, 1) for i, (N, _) in enumerate(CHAINS)]
    ids = [srv.submit(1, N, J[i], R0, 90 + i, betas, 1) for i, (N, R0) in enumerate(CHAINS)]
    for _ in range(4):
        srv.tick(1)
    for i, (N, R0) in enumerate(CHAINS):
        res = srv.result(ids[i])
        c = o.Run(J[i], 1, N, R0=R0, seed=90 + i)
        for beta in betas:
            c.step(float(beta), 1, R0)
        assert res["status"] == 2 and res["R"] == c.state().R and res["sumE"] == c.state().sumE, i
