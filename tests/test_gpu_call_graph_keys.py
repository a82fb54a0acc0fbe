"""Recorded forces steps of several keys side by side in one context: systems of different sizes and
different outputs in turn, more of them than are kept, equal eager calls bit for bit."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, model

pytestmark = pytest.mark.gpu


def _same(a, b):
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(np.asarray(a[k]), np.asarray(b[k]), err_msg=k)


@pytest.mark.parametrize("F,prec", [(64, "fp32"), (128, "bf16")])
@pytest.mark.parametrize("count", [2, 6])
def test_systems_and_outputs_in_turn(F, prec, count):
    eng = engine()
    _, blob = model(F, 2, 2, seed=3, bias=0.1)
    jobs = []
    for k in range(count):
        sy = syn.water_box(50 + 10 * (k // 2), seed=k // 2)
        jobs.append((sy, dict(forces=k % 2 == 0, virial=k % 2 == 0)))
    want = []
    for sy, kw in jobs:
        with eng.Potential(F, T=2, n_species=2, precision=prec, params=blob) as pot:
            pot.profile(True)
            want.append(pot.compute(sy.species, sy.positions, sy.cell, energies=True, **kw))
    with eng.Potential(F, T=2, n_species=2, precision=prec, params=blob) as pot:
        for turn in range(5):
            for (sy, kw), ref in zip(jobs, want):
                for _ in range(1 + turn % 2):
                    _same(pot.compute(sy.species, sy.positions, sy.cell, energies=True, **kw), ref)
