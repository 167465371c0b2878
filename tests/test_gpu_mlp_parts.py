"""FP32 networks whose tiles are split over 4, 2 or 1 blocks: remainders of every kind.

Element counts just below, at and above 16, 32 and 64 rows (with 4 blocks per tile), and
systems on either side of the tile counts where the split changes, against the oracle.
"""

from __future__ import annotations

import pytest

import oracle
from gpu_helpers import assert_parity, gpu_eval
from synth import make_model, water_box

pytestmark = pytest.mark.gpu


# 2 n H and n O atoms; 38 / 39 and 76 / 77 tiles of 64 rows for the last four
@pytest.mark.parametrize("n", [5, 8, 16, 17, 32, 33, 65, 800, 833, 1600, 1633])
def test_remainders(n):
    spec = make_model(T=2)
    s = water_box(n, seed=n)
    assert_parity(gpu_eval(spec, s), oracle.energy_forces(spec, s.pos, s.species, s.cell), s.n_atoms)


@pytest.mark.parametrize("n", [8, 33, 833])
def test_remainders_pairs_and_one_layer(n):
    s = water_box(n, seed=n)
    for spec in (make_model(T=2, pairs=True), make_model(T=1)):
        assert_parity(gpu_eval(spec, s), oracle.energy_forces(spec, s.pos, s.species, s.cell), s.n_atoms)
