"""The one-pass tensor-product, channel-mixing and readout kernels of the strictly local model against
its oracle: the channel counts they are built for (16, 32) and one they are not (12), one to
three layers, rows of no, one, an odd and a large number of edges, FP32."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import compare, engine

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::UserWarning")]


def _uneven():
    """A dense blob in a sparse gas: rows of 0 to over 60 edges."""
    rng = np.random.default_rng(9)
    x = np.concatenate([22.0 + rng.uniform(-3.5, 3.5, size=(61, 3)), rng.uniform(0.0, 44.0, size=(60, 3))])
    return rng.integers(0, 2, 121).astype(np.int32), x[rng.permutation(121)], np.diag([44.0] * 3)


@pytest.mark.parametrize("F,C,L", [(64, 16, 1), (64, 16, 3), (64, 32, 2), (64, 12, 2), (40, 32, 3), (256, 16, 2)])
@pytest.mark.parametrize("system", ["water", "uneven"])
def test_matches_oracle(F, C, L, system):
    import oracle.local as ol
    sy = syn.water_box(64, seed=2)
    species, x, cell = (sy.species, sy.positions, sy.cell) if system == "water" else _uneven()
    vals = syn.local_xavier_params(F, 20, L, 2, C, seed=F + C + L, bias_scale=0.1)
    blob = syn.local_params_blob(F, 20, L, 2, C, values=vals)
    ref = ol.local_model(vals, F, 20, L, 2, C, species, x, cell)
    with engine().Potential(F, K=20, T=L, n_species=2, params=blob, family="local", channels=C) as pot:
        out = pot.compute(species, x, cell, energies=True)
        again = pot.compute(species, x, cell, energies=True)
    compare(out, ref)
    np.testing.assert_array_equal(out["forces"], again["forces"])
