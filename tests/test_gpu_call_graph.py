"""The recorded forces step of calls and MD steps: replays equal eager calls bit for bit, and follow
every change of positions, list, size, outputs asked for, options and parameters (an eager call is
one with launch profiling on)."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, model

pytestmark = pytest.mark.gpu

CASES = {"fp32": (64, "fp32"), "bf16_F64": (64, "bf16"), "bf16_F128": (128, "bf16")}


def _eager(eng, F, prec, blob, sy, x, **kw):
    with eng.Potential(F, T=2, n_species=2, precision=prec, params=blob) as pot:
        pot.profile(True)
        return pot.compute(sy.species, x, sy.cell, energies=True, **kw)


def _same(a, b):
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(np.asarray(a[k]), np.asarray(b[k]), err_msg=k)


@pytest.mark.parametrize("case", sorted(CASES))
def test_replays_follow_their_inputs(case):
    F, prec = CASES[case]
    eng = engine()
    sy, big = syn.water_box(60, seed=1), syn.water_box(90, seed=2)
    _, blob = model(F, 2, 2, seed=3, bias=0.1)
    _, other = model(F, 2, 2, seed=4, bias=0.2, e_scale=0.5)
    rng = np.random.default_rng(0)
    moved = [sy.positions + rng.uniform(-0.6, 0.6, size=sy.positions.shape) for _ in range(3)]
    with eng.Potential(F, T=2, n_species=2, precision=prec, params=blob) as pot:
        ref = _eager(eng, F, prec, blob, sy, sy.positions)
        for _ in range(4):   # eager, recorded, replayed
            _same(pot.compute(sy.species, sy.positions, sy.cell, energies=True), ref)
        for x in moved:      # past skin / 2: new lists under the recorded step
            _same(pot.compute(sy.species, x, sy.cell, energies=True, rebuild=True), _eager(eng, F, prec, blob, sy, x))
        quiet = _eager(eng, F, prec, blob, sy, moved[0], forces=False, virial=False)
        for _ in range(3):
            _same(pot.compute(sy.species, moved[0], sy.cell, energies=True, forces=False, virial=False, rebuild=True), quiet)
        ref = _eager(eng, F, prec, blob, big, big.positions)
        for _ in range(3):   # another size, larger buffers
            _same(pot.compute(big.species, big.positions, big.cell, energies=True), ref)
        pot.load_params(other)
        ref = _eager(eng, F, prec, other, big, big.positions)
        for _ in range(3):
            _same(pot.compute(big.species, big.positions, big.cell, energies=True), ref)
        ref = _eager(eng, F, prec, other, sy, moved[1])
        for _ in range(3):   # back to the smaller size
            _same(pot.compute(sy.species, moved[1], sy.cell, energies=True, rebuild=True), ref)


def test_option_changes_leave_the_recorded_step():
    from paper_2506_04055_gb300 import _lib
    eng = engine()
    sy = syn.fcc(4, 4, 4, jitter=0.05, seed=1)
    _, blob = model(128, 2, 1, seed=3, bias=0.1)
    with eng.Potential(128, T=2, n_species=1, precision="bf16", params=blob) as pot:
        for opt in (_lib.CTD_OPT_TC_ADJOINT, _lib.CTD_OPT_TC_MESSAGE):
            for value in (1, 0):
                pot.set_option(opt, value)
                got = [pot.compute(sy.species, sy.positions, sy.cell, energies=True) for _ in range(3)]
                with eng.Potential(128, T=2, n_species=1, precision="bf16", params=blob) as ref:
                    ref.set_option(opt, value)
                    ref.profile(True)
                    want = ref.compute(sy.species, sy.positions, sy.cell, energies=True)
                for g in got:
                    _same(g, want)
            pot.set_option(opt, 1)


def test_md_and_launch_counts():
    """An MD run with recorded steps (rebuilds among them) equals an eager one, launches included."""
    eng = engine()
    sy = syn.water_box(64, seed=5)
    _, blob = model(64, 2, 2, seed=6, bias=0.1)
    v = syn.maxwell_boltzmann(sy.masses, 2000.0, seed=1)
    out = []
    for eager in (True, False):
        with eng.Potential(64, T=2, n_species=2, params=blob) as pot:
            pot.md_set_state(sy.species, sy.masses, sy.positions, v, sy.cell, skin=0.1)
            pot.profile(eager)
            pot.profile_read(reset=True)
            ep, ek, nreb = pot.md_run(30, 0.5)
            counts = {k: c for k, (_, c) in pot.profile_read().items()}
            out.append((ep, ek, *pot.md_get_state(), nreb, counts))
    assert out[0][4] > 0 and out[0][4:] == out[1][4:]
    for a, b in zip(out[0][:4], out[1][:4]):
        np.testing.assert_array_equal(a, b)
