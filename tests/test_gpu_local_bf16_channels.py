"""Strictly local model on the BF16 path at the channel counts whose tensor products run in separate passes
(48, 64; 16 beside them), against the oracle.  Tolerance: about 4 L + 4 products on BF16 operands forward and as many in
the adjoint, each rounding two operands to 2^-9: sqrt(4 (4 L + 4)) 2^-9, doubled for what the layers amplify."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, rel_force_rmse

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::UserWarning")]


@pytest.mark.parametrize("F,C,L", [(64, 16, 2), (64, 48, 1), (64, 48, 2), (64, 64, 3), (128, 48, 2), (128, 64, 2)])
def test_matches_oracle(F, C, L):
    import oracle.local as ol
    sy = syn.water_box(64, seed=2)
    vals = syn.local_xavier_params(F, 20, L, 2, C, seed=F + C + L, bias_scale=0.1)
    blob = syn.local_params_blob(F, 20, L, 2, C, values=vals)
    ref = ol.local_model(vals, F, 20, L, 2, C, sy.species, sy.positions, sy.cell)
    with engine().Potential(F, K=20, T=L, n_species=2, precision="bf16", params=blob, family="local", channels=C) as pot:
        out = pot.compute(sy.species, sy.positions, sy.cell, energies=True)
        again = pot.compute(sy.species, sy.positions, sy.cell, energies=True)
    tol = 2.0 * np.sqrt(4.0 * (4 * L + 4)) * 2.0 ** -9
    assert rel_force_rmse(out["forces"], ref["forces"]) <= tol
    scale = np.sqrt(np.mean(ref["energies"] ** 2))
    assert np.sqrt(np.mean((out["energies"] - ref["energies"]) ** 2)) <= tol * scale
    np.testing.assert_array_equal(out["forces"], again["forces"])
