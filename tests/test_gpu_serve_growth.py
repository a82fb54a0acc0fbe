"""Served steps recorded and replayed while a replica's list grows from a few pairs per atom to hundreds
(a lattice of heavy atoms that moves towards its centre): the trajectory equals the eager one bit for
bit, and under a budget it either does so too or the step reports the budget."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, model

pytestmark = pytest.mark.gpu

NSTEPS = 40


def _system():
    rng = np.random.default_rng(2)
    k = np.stack(np.meshgrid(np.arange(7), np.arange(7), np.arange(6), indexing="ij"), axis=-1).reshape(-1, 3)
    x = 10.0 + 5.5 * k + rng.uniform(-0.2, 0.2, size=k.shape)
    z = rng.integers(0, 2, len(x)).astype(np.int32)
    return z, np.full(len(x), 1e6), x, -0.02 * (x - x.mean(0)), np.diag([60.0] * 3)


def _run(eng, blob, graph, budget=0):
    z, m, x, v, cell = _system()
    srv = eng.Server(32, blob, T=2, n_species=2, dt=1.0, hbm_budget_bytes=budget)
    try:
        srv.use_graph(graph)
        rid = srv.submit(z, m, x, v, cell, NSTEPS, skin=1.0)
        for _ in range(NSTEPS + 3):
            srv.step()
        return srv.poll(rid), srv.graph_stats()
    finally:
        srv.close()


def test_growing_lists_under_a_recorded_step():
    eng = engine()
    from paper_2506_04055_gb300 import _lib
    _, blob = model(32, 2, 2, seed=5, bias=0.1)
    want, gs = _run(eng, blob, False)
    assert want["state"] == 2 and gs["graph_steps"] == 0

    def check(got):
        assert got["state"] == 2
        for k in ("epot", "ekin", "positions", "velocities"):
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)

    got, gs = _run(eng, blob, True)
    check(got)
    assert gs["graph_steps"] > 0
    for mb in range(8, 49, 4):
        try:
            got, _ = _run(eng, blob, True, budget=mb << 20)
        except _lib.CtdError as e:
            assert e.code == _lib.CTD_ERR_OUT_OF_BUDGET
            continue
        check(got)
