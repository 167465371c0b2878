"""Virial W = -dE/d(strain) from the reverse edge pass, against the FP64 oracle
(whose virial is pinned by central differences under strain).

Each directed edge of each layer contributes -(dE/dr_e) r_e^T once, from the
pass over its centre atom's list.  Tolerance: the FP32 energy bar (1e-6 eV
per atom) scaled by the ratio of the per-atom virial to the per-atom energy,
at most 20 on these boxes, gives 2e-5 eV per atom on every component
(measured on GB300: <= 2.2e-6 at T = 3, 6.3e-6 on the Cu crystal at T = 5).
"""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import fcc_box, hea_box, make_model, water_box

pytestmark = pytest.mark.gpu

W_TOL_PER_ATOM = 2e-5  # eV

CASES = {
    "water192-T3": (lambda: water_box(64, seed=0), 3, 3),
    "water24576-T3": (lambda: water_box(8192, seed=0), 3, 3),
    "cu4000-T3": (lambda: fcc_box(10, seed=0), 3, 3),
    "cu4000-T5": (lambda: fcc_box(10, seed=0), 5, 3),
    "hea4000-T3": (lambda: hea_box(10, seed=0), 3, 8),
    "cu32000-T2": (lambda: fcc_box(20, seed=0), 2, 3),  # beyond 28,672 atoms the reverse pass has 8 lanes per atom
}


def _virial(spec, s, ranks=None, precision=0):
    import torch

    from paper_2505_06711_gb300 import Potential

    pot = Potential(spec, precision=precision)
    try:
        sy = pot.system(s.pos, s.species, s.cell, ranks=ranks)
        sy.evaluate(virial=True, atom_virial=True)
        sy.check()
        torch.cuda.synchronize()
        out = (sy.virial.cpu().numpy(), sy.atom_virial.double().cpu().numpy(), sy.forces.cpu().numpy())
        sy.close()
        return out
    finally:
        pot.close()


@pytest.mark.parametrize("case", list(CASES))
def test_virial_matches_oracle(case):
    make, T, ne = CASES[case]
    s = make()
    spec = make_model(T=T, n_elem=ne)
    W, Wa, _ = _virial(spec, s)
    ref = oracle.energy_forces(spec, s.pos, s.species, s.cell)["virial"]
    dw = float(np.abs(W - ref).max()) / s.n_atoms
    print(f"[virial] {case} max|dW|/N={dw:.3e} eV  max|W|/N={np.abs(ref).max() / s.n_atoms:.3e} eV  "
          f"asym={np.abs(W - W.T).max() / s.n_atoms:.2e}")
    assert np.abs(ref).max() / s.n_atoms > 1e-4  # not vacuous
    assert dw <= W_TOL_PER_ATOM
    # the per-atom shares sum to the total (FP64 sums of the same FP32 values)
    np.testing.assert_allclose(Wa.sum(0).reshape(3, 3), W, rtol=1e-9, atol=1e-9 * s.n_atoms)


def test_virial_decomposed_and_forces_unchanged():
    import torch

    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=3)
    s = water_box(8192, seed=1)
    W1, Wa1, F1 = _virial(spec, s)
    W2, Wa2, F2 = _virial(spec, s, ranks=(2, 2, 2))
    assert np.array_equal(Wa1, Wa2) and np.array_equal(F1, F2)
    np.testing.assert_allclose(W1, W2, rtol=1e-12, atol=1e-12 * s.n_atoms)
    # the virial request leaves the forces of the plain entry point unchanged
    pot = Potential(spec)
    try:
        sy = pot.system(s.pos, s.species, s.cell)
        sy.evaluate()
        torch.cuda.synchronize()
        assert np.array_equal(sy.forces.cpu().numpy(), F1)
        sy.close()
    finally:
        pot.close()


def test_virial_bf16x3_within_bound():
    spec = make_model(T=3)
    s = water_box(64, seed=0)
    W, _, _ = _virial(spec, s, precision=2)
    ref = oracle.energy_forces(spec, s.pos, s.species, s.cell)["virial"]
    assert float(np.abs(W - ref).max()) / s.n_atoms <= W_TOL_PER_ATOM


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 545])
def test_virial_sums_over_rows(n):
    # block and warp edges of the sums: the total is the FP64 sum of the rows, and the rows come in caller order
    from synth import Structure

    spec = make_model(T=1)
    full = water_box(200, seed=3)
    s = Structure(full.pos[:n], full.species[:n], full.cell)
    W, Wa, _ = _virial(spec, s)
    np.testing.assert_allclose(W, Wa.sum(0).reshape(3, 3), rtol=1e-12, atol=1e-12 * n)
    p = np.random.default_rng(n).permutation(n)
    _, Wp, _ = _virial(spec, Structure(s.pos[p], s.species[p], s.cell))
    # another order of the atoms changes the order of each row's sums only: FP32 roundings of ~200 terms
    np.testing.assert_allclose(Wp, Wa[p], rtol=0, atol=2e-5 * max(1e-3, np.abs(Wa).max()))
