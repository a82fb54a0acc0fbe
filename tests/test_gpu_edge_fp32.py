"""FP32 message step and adjoint (edge_fp32.cu) where their tiling can go wrong, against the FP64
oracle at the FP32 path's tolerances: every width and basis-size class, pairs at every distance
(which groups of centres are visited), rows of no, one and several stages of edges, and more rows
than one chunk per warp."""
import numpy as np
import pytest

import synthetic as syn
from gpu_common import compare, engine, model

pytestmark = pytest.mark.gpu


def _both(orc, F, K, T, species, x, cell, seed):
    vals, blob = model(F, T, 2, seed=seed, bias=0.2, K=K)
    ref = orc.painn(vals, F, K, T, 2, species, x, cell)
    with engine().Potential(F, K=K, T=T, n_species=2, params=blob) as pot:
        out = pot.compute(species, x, cell, energies=True)
    compare(out, ref)


@pytest.mark.parametrize("F,K", [(32, 20), (64, 2), (64, 16), (64, 17), (64, 20), (64, 21), (64, 32), (128, 20),
                                 (128, 32), (256, 16), (256, 20), (256, 32)])
def test_dimers_at_every_distance(orc, F, K):
    """60 dimers 20 A apart, 0.3 to 4.95 A long: rows of one edge, every first group of centres."""
    d = np.linspace(0.3, 4.95, 60)
    rng = np.random.default_rng(F + K)
    u = rng.normal(size=(60, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    k = np.arange(60)
    base = 20.0 * np.stack([k % 4, (k // 4) % 4, k // 16], axis=1) + 10.0
    x = np.concatenate([base, base + u * d[:, None]])
    species = np.concatenate([np.zeros(60, np.int32), np.ones(60, np.int32)])
    _both(orc, F, K, 2, species, x, np.diag([80.0, 80.0, 80.0]), seed=F + K)


@pytest.mark.parametrize("F", [32, 64, 128, 256])
def test_uneven_rows(orc, F):
    """A dense blob in a sparse gas: rows of 0 to over 100 edges, chunks that mix them."""
    rng = np.random.default_rng(5)
    blob_x = 24.0 + rng.uniform(-4.0, 4.0, size=(90, 3))
    gas = rng.uniform(0.0, 48.0, size=(70, 3))
    x = np.concatenate([blob_x, gas])[rng.permutation(160)]
    _both(orc, F, 20, 3, rng.integers(0, 2, 160).astype(np.int32), x, np.diag([48.0] * 3), seed=F)


def test_several_rows_per_chunk(orc):
    """5,000 atoms, F = 64: more rows than one per warp of the grid."""
    sy = syn.water_box(1667, seed=4)
    _both(orc, 64, 20, 2, sy.species, sy.positions, sy.cell, seed=1)
