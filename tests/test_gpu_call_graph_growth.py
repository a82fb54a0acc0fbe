"""The recorded forces step when the list grows under it: an earlier build that no step followed has made
the list's own buffers large, so a denser system with the same atom count allocates nothing while its
list is built, and the buffers that the step itself writes must still grow.  Results equal a fresh
context's bit for bit; under a budget a call that does not fit says so."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, model

pytestmark = pytest.mark.gpu

N = 1000


def _gas():
    """1,000 atoms 5.5 A apart: six list entries each, few of them within the cutoff."""
    rng = np.random.default_rng(1)
    k = np.stack(np.meshgrid(*[np.arange(10)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    return 5.5 * k + rng.uniform(-0.4, 0.4, size=(N, 3)), np.diag([55.0] * 3)


def _same(a, b):
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(np.asarray(a[k]), np.asarray(b[k]), err_msg=k)


def _eager(eng, F, prec, blob, z, x, cell):
    with eng.Potential(F, T=2, n_species=1, precision=prec, params=blob) as pot:
        pot.profile(True)
        return pot.compute(z, x, cell, energies=True)


def _build_large(pot, how):
    large = syn.fcc(8, 8, 8, jitter=0.05, seed=2)
    if how == "build":
        pot.build_neighbors(large.positions, large.cell)
    else:
        pot.md_set_state(large.species, large.masses, large.positions, 0.0 * large.positions, large.cell)


@pytest.mark.parametrize("how", ["build", "md_state"])
@pytest.mark.parametrize("F,prec", [(64, "fp32"), (128, "bf16")])
def test_denser_system_under_a_recorded_step(F, prec, how):
    eng = engine()
    dense = syn.fcc(5, 5, 10, jitter=0.05, seed=3)
    assert dense.n == N
    x, cell = _gas()
    _, blob = model(F, 2, 1, seed=3, bias=0.1)
    thin = _eager(eng, F, prec, blob, dense.species, x, cell)
    want = _eager(eng, F, prec, blob, dense.species, dense.positions, dense.cell)
    with eng.Potential(F, T=2, n_species=1, precision=prec, params=blob) as pot:
        _build_large(pot, how)
        for _ in range(5):
            _same(pot.compute(dense.species, x, cell, energies=True), thin)
        for _ in range(5):
            _same(pot.compute(dense.species, dense.positions, dense.cell, energies=True), want)
        _same(pot.compute(dense.species, x, cell, energies=True), thin)


def test_growth_under_a_budget():
    """Budgets from too small to ample: every call gives the eager result or reports the budget, and a context
    whose steps are recorded takes exactly the budgets that an eager one takes."""
    eng = engine()
    from paper_2506_04055_gb300 import _lib
    dense = syn.fcc(5, 5, 10, jitter=0.05, seed=3)
    x, cell = _gas()
    _, blob = model(64, 2, 1, seed=3, bias=0.1)
    thin = _eager(eng, 64, "fp32", blob, dense.species, x, cell)
    want = _eager(eng, 64, "fp32", blob, dense.species, dense.positions, dense.cell)
    with eng.Potential(64, T=2, n_species=1, params=blob) as pot:
        _build_large(pot, "build")
        held = [pot.compute(dense.species, p, c, stats=True)["stats"]["bytes_allocated"]
                for p, c in ((x, cell), (dense.positions, dense.cell))]

    def calls_done(budget, eager):
        done = 0
        with eng.Potential(64, T=2, n_species=1, params=blob, hbm_budget_bytes=int(budget)) as pot:
            pot.profile(eager)
            try:
                _build_large(pot, "build")
                for _ in range(5):
                    _same(pot.compute(dense.species, x, cell, energies=True), thin)
                    done += 1
                for _ in range(3):
                    _same(pot.compute(dense.species, dense.positions, dense.cell, energies=True), want)
                    done += 1
            except _lib.CtdError as e:
                assert e.code == _lib.CTD_ERR_OUT_OF_BUDGET
        return done

    counts = []
    for budget in np.linspace(0.5 * held[0], 1.03 * held[1], 60).astype(int):
        counts.append(calls_done(budget, False))
        assert counts[-1] == calls_done(budget, True), budget
    assert counts[0] == 0 and counts[-1] == 8
