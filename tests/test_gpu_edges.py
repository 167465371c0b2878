"""Edge passes at the sizes where their dispatch and their batches can go wrong.

* one system per lane layout (forward 16, 8, 4 lanes per atom; reverse 32, 16, 8), with
  row lengths that are no multiple of a batch, against the oracle;
* isolated atoms, a dimer near the cutoff and a lone pair (rows of 0 and 1 live edges);
* records kept for a part of the rows only, recomputed per run of rows in every pass:
  bitwise the same results as with all of them kept.
"""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_helpers import assert_parity, gpu_eval
from synth import Structure, fcc_box, make_model, water_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize(
    "make",
    [lambda: water_box(67, seed=1), lambda: water_box(1366, seed=2), lambda: fcc_box(12, seed=3),
     lambda: fcc_box(16, seed=4), lambda: water_box(5462, seed=5), lambda: fcc_box(20, seed=6)],
    ids=["201", "4098", "6912", "16384", "16386", "32000"],
)
def test_lane_layouts(make):
    spec = make_model(T=2)
    s = make()
    assert_parity(gpu_eval(spec, s), oracle.energy_forces(spec, s.pos, s.species, s.cell), s.n_atoms)


def test_short_rows():
    pos = np.array([[1.0, 1.0, 1.0], [1.0, 1.0, 5.9], [20.0, 20.0, 20.0], [30.0, 30.0, 30.0], [31.1, 30.2, 30.3],
                    [39.9, 10.0, 10.0], [0.4, 10.0, 10.0]])
    s = Structure(pos, np.array([0, 1, 2, 1, 0, 2, 2], dtype=np.int32), np.eye(3) * 40.0)
    for pairs in (False, True):
        spec = make_model(T=3, pairs=pairs)
        assert_parity(gpu_eval(spec, s), oracle.energy_forces(spec, s.pos, s.species, s.cell), s.n_atoms)


def test_narrow_gaussians_keep_their_range():
    # alpha r_c^2 = 80, the largest accepted: exp(-80) times a small cutoff stays a normal float
    import torch

    from paper_2505_06711_gb300 import Potential

    s = water_box(32, seed=7)
    spec = make_model(T=2, alpha=3.2)
    pot = Potential(spec)  # not gpu_eval's, whose potentials are kept by T and parameters
    sy = pot.system(s.pos, s.species, s.cell)
    sy.evaluate()
    sy.check()
    torch.cuda.synchronize()
    gpu = {"energy": float(sy.energy), "forces": sy.forces.double().cpu().numpy(),
           "atom_energy": sy.atom_energy.double().cpu().numpy()}
    assert_parity(gpu, oracle.energy_forces(spec, s.pos, s.species, s.cell), s.n_atoms)
    sy.close()
    pot.close()


@pytest.mark.parametrize("virial", [False, True])
def test_records_of_a_part_of_the_rows(virial):
    import torch

    from paper_2505_06711_gb300 import Potential, binding

    s = water_box(400, seed=8)
    pot = Potential(make_model(T=3))
    got = []
    for rows in (1 << 40, 1199, 512, 7):
        sy = pot.system(s.pos, s.species, s.cell)
        assert binding.lib().reann_test_limit_edge_rows(sy.nl, binding._i64(rows)) == 0
        for _ in range(3):  # direct, captured, replayed
            sy.evaluate(virial=virial)
        sy.check()
        torch.cuda.synchronize()
        got.append((float(sy.energy), sy.forces.cpu().numpy().copy(), sy.info()[3]))
        sy.close()
    pot.close()
    for e, f, live in got[1:]:
        assert e == got[0][0] and np.array_equal(f, got[0][1]) and live == got[0][2]
