"""Pair search with a cell's atoms dealt to several warps (grids of few cells) and the two-edges-at-a-
time reverse search: the pair set equals the oracle's bit for bit for one crowded cell, cells of more
than 32 and more than 64 atoms, and grids on both sides of every number of warps per cell; energies
and forces, which use the reverse edges, are those of the oracle."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import compare, engine, model

pytestmark = pytest.mark.gpu


def _pairs(sy_x, cell, cutoff, skin):
    eng = engine()
    with eng.Potential(64, T=1, n_species=1) as pot:
        n = pot.build_neighbors(sy_x, cell, cutoff=cutoff, skin=skin)
        return pot.get_pairs(n)


@pytest.mark.parametrize("n,box", [(1, 9.0), (2, 9.0), (33, 11.0), (200, 11.0), (200, 17.0), (1500, 29.0), (900, 48.0),
                                   (3000, 66.0), (4000, 84.0)])
def test_pairs_exact(orc, n, box):
    """Uniform gas: 1 to 14^3 cells of the search grid (R = 6 A), 1 to 32 warps per cell."""
    rng = np.random.default_rng(n)
    x = rng.uniform(0.0, box, size=(n, 3))
    cell = np.diag([box] * 3)
    got = _pairs(x, cell, 5.0, 1.0)
    xw, _ = orc.wrap(x, cell)
    for a, b in zip(got, orc.pairs_cells(xw, cell, 6.0)):
        np.testing.assert_array_equal(a, b)


def test_rows_longer_than_one_reverse_scan(orc):
    """A dense blob: rows of more than 96 Verlet edges, of even and odd length."""
    rng = np.random.default_rng(2)
    x = np.concatenate([20.0 + rng.uniform(-3.6, 3.6, size=(131, 3)), rng.uniform(0.0, 40.0, size=(30, 3))])
    cell, species = np.diag([40.0] * 3), rng.integers(0, 2, 161).astype(np.int32)
    vals, blob = model(64, 2, 2, seed=3, bias=0.2)
    with engine().Potential(64, T=2, n_species=2, params=blob) as pot:
        out = pot.compute(species, x, cell, energies=True)
    compare(out, orc.painn(vals, 64, 20, 2, 2, species, x, cell))


def test_replica_sums_at_slice_edges():
    """Served replicas of 4 to 192 atoms (slices of 64) against the single-system loop."""
    eng = engine()
    F, T, S, steps, dt = 64, 2, 2, 3, 0.5
    _, blob = model(F, T, S, seed=7, bias=0.1)
    systems = [syn.fcc(1, 1, 1, jitter=0.05, seed=1), syn.fcc(4, 2, 2, jitter=0.05, seed=2)]
    systems += [syn.water_box(k, seed=k) for k in (21, 22, 43, 64)]
    srv = eng.Server(F, blob, T=T, n_species=S, max_replicas=len(systems), dt=dt)
    vel = [syn.maxwell_boltzmann(sy.masses, 300.0, seed=k) for k, sy in enumerate(systems)]
    ids = [srv.submit(sy.species, sy.masses, sy.positions, v, sy.cell, nsteps=steps) for sy, v in zip(systems, vel)]
    left = len(ids)
    while left:
        left -= srv.step()[2]
    for r, sy, v in zip(ids, systems, vel):
        got = srv.poll(r)
        with eng.Potential(F, T=T, n_species=S, params=blob) as pot:
            pot.md_set_state(sy.species, sy.masses, sy.positions, v, sy.cell, skin=1.0)
            ep, ek, _ = pot.md_run(steps, dt)
            x, _ = pot.md_get_state()
            w = pot.compute(sy.species, x, sy.cell, rebuild=True)["virial"]
        # the same FP32 per-atom terms summed in FP64 in another order, over trajectories that agree
        # to FP64 rounding
        scale = np.abs(got["epot"]).max() + 1e-3 * sy.n
        np.testing.assert_allclose(got["epot"], ep, rtol=0, atol=1e-9 * scale)
        np.testing.assert_allclose(got["ekin"], ek, rtol=1e-9)
        assert np.linalg.norm(got["virial"] - w) <= 1e-5 * np.linalg.norm(w)
