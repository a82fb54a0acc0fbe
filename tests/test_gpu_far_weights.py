"""FP32 message step and adjoint with filter weights that are a million times larger at centres far below every
distance of the system than near them: what such a Gaussian adds beyond six widths counts, and the FP32 path's bars
for forces and virial hold.  (The bar for the energy is for weights of one scale: with all Gaussians visited it is
missed here, 1.04e-6 at F = 32, K = 32.)"""
import math

import numpy as np
import pytest

import synthetic as syn
from gpu_common import FP32_FORCE_RMSE, FP32_VIRIAL_REL, engine, rel_force_rmse, virial_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,far", [(16, 4), (20, 8), (32, 12)])
@pytest.mark.parametrize("F", [32, 64, 128])
def test_far_weights(orc, F, K, far):
    T = 2
    d = (far - 1 + 6.33) * 5.0 / (K - 1)   # the last far centre is 6.33 widths below the nearest neighbours
    sy = syn.fcc(4, 4, 4, a=d * math.sqrt(2.0), jitter=0.05, seed=1)
    vals = syn.xavier_params(F, K, T, 1, seed=F + K, bias_scale=0.1)
    off = 0
    for name, shape in syn.param_shapes(F, K, T, 1):
        n = int(np.prod(shape))
        if name.startswith("Wf"):
            vals[off:off + n].reshape(shape)[:, :far] *= 1e6
        off += n
    ref = orc.painn(vals, F, K, T, 1, sy.species, sy.positions, sy.cell)
    with engine().Potential(F, K=K, T=T, n_species=1, params=syn.params_blob(F, K, T, 1, values=vals)) as pot:
        out = pot.compute(sy.species, sy.positions, sy.cell)
    assert rel_force_rmse(out["forces"], ref["forces"]) <= FP32_FORCE_RMSE
    assert virial_rel(out["virial"], ref["virial"]) <= FP32_VIRIAL_REL
