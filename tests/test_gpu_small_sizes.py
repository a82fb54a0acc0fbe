"""FP32 path at the sizes where its tile rules change (16 x 32 GEMM tiles, 24 to 48 rows by 64, the
readout's 32-atom tiles and their remainders, blocks of the partial sums), against the FP64 oracle at
the FP32 tolerances."""
import pytest

import synthetic as syn
from gpu_common import compare, engine, model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [64, 128])
@pytest.mark.parametrize("molecules", [3, 11, 43, 300, 820])
def test_water(orc, F, molecules):
    sy = syn.water_box(molecules, seed=molecules)
    vals, blob = model(F, 2, 2, seed=F, bias=0.2)
    ref = orc.painn(vals, F, 20, 2, 2, sy.species, sy.positions, sy.cell)
    with engine().Potential(F, T=2, n_species=2, params=blob) as pot:
        out = pot.compute(sy.species, sy.positions, sy.cell, energies=True)
    compare(out, ref)
