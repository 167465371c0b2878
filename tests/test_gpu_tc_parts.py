"""Tensor-core backward networks whose tiles are split over clusters of 4 or 2 blocks:
remainders of the row quarters and the tile counts where the split changes, against the
oracle.  A row that lands in the wrong block is off by its whole force; split BF16 keeps 16
significant bits per operand, so the relative error stays below a few times 2^-17 per
product (measured 9e-6 on the force vector; 5e-5 allowed); BF16 measured 6e-3 and FP8 3e-2
(2e-2 and 1e-1 allowed).
"""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import make_model, water_box

pytestmark = pytest.mark.gpu

TOL = {1: 2e-2, 2: 5e-5, 3: 1e-1}  # BF16, split BF16, FP8


# 2 n H and n O atoms; 32 / 33 and 76 / 77 tiles of 128 rows for the last four
@pytest.mark.parametrize("precision", [1, 2, 3])
@pytest.mark.parametrize("n", [8, 16, 17, 33, 48, 65, 1365, 1366, 3200, 3300])
def test_remainders(n, precision):
    import torch

    from paper_2505_06711_gb300 import Potential, binding

    assert (binding.REANN_MLP_BF16, binding.REANN_MLP_BF16X3, binding.REANN_MLP_FP8) == (1, 2, 3)
    spec, s = make_model(T=2), water_box(n, seed=n)
    pot = Potential(spec, precision=precision)
    sy = pot.system(s.pos, s.species, s.cell)
    sy.evaluate()
    sy.check()
    torch.cuda.synchronize()
    got = sy.forces.double().cpu().numpy()
    sy.close()
    pot.close()
    want = oracle.energy_forces(spec, s.pos, s.species, s.cell)["forces"]
    assert np.linalg.norm(got - want) <= TOL[precision] * np.linalg.norm(want)
