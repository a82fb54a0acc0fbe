"""FP32 message step and adjoint with a basis of a few Gaussians (all of their weights in registers), against the
FP64 oracle at the FP32 path's tolerances: dimers at every distance and a water box, both sides of the line to the
larger basis, filters recomputed and stored."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import compare, engine, model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [32, 64, 128, 256])
@pytest.mark.parametrize("K", [2, 4, 5, 8, 9])
def test_small_basis(orc, F, K):
    eng = engine()
    from paper_2506_04055_gb300 import _lib
    d = np.linspace(0.3, 4.95, 60)
    rng = np.random.default_rng(F + K)
    u = rng.normal(size=(60, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    k = np.arange(60)
    base = 20.0 * np.stack([k % 4, (k // 4) % 4, k // 16], axis=1) + 10.0
    dimers = np.concatenate([base, base + u * d[:, None]]), np.repeat(np.array([0, 1], np.int32), 60), np.diag([80.0] * 3)
    sy = syn.water_box(60, seed=K)
    vals, blob = model(F, 2, 2, seed=F + K, bias=0.2, K=K)
    for x, z, cell in (dimers, (sy.positions, sy.species, sy.cell)):
        ref = orc.painn(vals, F, K, 2, 2, z, x, cell)
        for store in (0, 1):
            with eng.Potential(F, K=K, T=2, n_species=2, params=blob) as pot:
                pot.set_option(_lib.CTD_OPT_EDGE_STORE, store)
                compare(pot.compute(z, x, cell, energies=True), ref)
