"""Edge passes at the sizes where their dispatch and their batches can go wrong.

* one system per lane layout (forward 16, 8, 4 lanes per atom; reverse 32, 16, 8), with
  row lengths that are no multiple of a batch, against the oracle;
* isolated atoms, a dimer near the cutoff and a lone pair (rows of 0 and 1 live edges);
* records kept for a part of the rows only, recomputed per run of rows in every pass:
  bitwise the same results as with all of them kept.
"""

from __future__ import annotations

import dataclasses

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


def test_many_rows():
    # beyond 65,536 rows the forward pass prefetches its records; a supercell repeats its cell's forces
    spec = make_model(T=2)
    one = fcc_box(13, seed=7)
    shift = np.stack(np.meshgrid(*[np.arange(2)] * 3, indexing="ij"), -1).reshape(-1, 1, 3) @ one.cell
    s = Structure((one.pos + shift).reshape(-1, 3), np.tile(one.species, 8), 2 * one.cell)
    assert s.n_atoms > 1 << 16
    ref = gpu_eval(spec, one)
    assert_parity(gpu_eval(spec, s), {"energy": 8 * ref["energy"], "forces": np.tile(ref["forces"], (8, 1)),
                                      "atom_energy": np.tile(ref["atom_energy"], 8)}, s.n_atoms)


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


def _evaluated(s, T, rows, virial, precision=0):
    import torch

    from paper_2505_06711_gb300 import Potential, binding

    pot = Potential(make_model(T=T), precision=precision)
    sy = pot.system(s.pos, s.species, s.cell)
    assert binding.lib().reann_test_limit_edge_rows(sy.nl, binding._i64(rows)) == 0
    for _ in range(3):  # direct, captured, replayed
        sy.evaluate(virial=virial, atom_virial=virial)
    sy.check()
    torch.cuda.synchronize()
    out = [np.array(sy.info()[3])] + [x.cpu().numpy().copy() for x in (sy.energy, sy.forces, sy.atom_energy)]
    if virial:
        out += [sy.virial.cpu().numpy().copy(), sy.atom_virial.cpu().numpy().copy()]
    sy.close()
    pot.close()
    return out


def _assert_same(a, b):
    assert len(a) == len(b)
    for k, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x, y), k


@pytest.mark.parametrize("virial", [False, True])
def test_records_of_a_part_of_the_rows(virial):
    s = water_box(400, seed=8)
    whole = _evaluated(s, 3, 1 << 40, virial)
    for rows in (1199, 512, 7):
        _assert_same(_evaluated(s, 3, rows, virial), whole)


@pytest.mark.parametrize("virial,precision", [(False, 0), (True, 0), (False, 3)])
@pytest.mark.parametrize("molecules,rows", [(1400, 3000), (2800, 4096), (5600, 9000), (9600, 20000), (9600, 700)])
def test_sums_do_not_depend_on_the_run(molecules, rows, virial, precision):
    # the order of a row's sums follows the list's atoms (forward 16, 8, 4 lanes up to 4,096, 8,192, beyond;
    # reverse 32, 16, 8 up to 16,384, 28,672, beyond), not the run's rows, which here lie across a line
    s = water_box(molecules, seed=9)
    _assert_same(_evaluated(s, 2, rows, virial, precision), _evaluated(s, 2, 1 << 40, virial, precision))


@pytest.mark.parametrize("m,alpha", [(3, 1.3), (6, 1.3), (2, 3.2), (4, 3.2), (5, 3.2), (6, 3.2)])
def test_radial_derivative_near_a_gaussian_centre(m, alpha):
    # lone pairs on an axis, at distances that FP32 holds, which see one radial channel of l = 0 only: |F| is
    # |phi_m'| times a smooth factor.  phi_m' is a difference that is small where phi_m is largest; its rms error,
    # relative to its rms, is up to 1.1e-7 in FP32 with d - mu_m taken first, and 1.3e-7 to 5.3e-7 with
    # 2 alpha mu_m / d - 2 alpha rounded term by term (both from an FP32 emulation).  phi_m enters the force twice
    # and the recurrence's factor phi_m m times: with that factor within an ulp, 6e-8, 1.2e-7 m at most.
    import torch

    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=1, n_elem=1, alpha=alpha)
    p = np.array(spec.params)
    p[:8] = 0.0
    p[m] = 1.0
    W = p[8 : 8 + 3 * 8 * 16].reshape(3, 8, 16)
    W[1:] = 0.0
    p[8 + W.size :] = np.abs(p[8 + W.size :])  # networks without cancellation
    spec = dataclasses.replace(spec, params=p)
    rng = np.random.default_rng(m)
    at = 13.0 * np.stack(np.meshgrid(*[np.arange(10)] * 3, indexing="ij"), -1).reshape(-1, 3) + 4.0
    mu = m * 5.0 / 7.0
    w = 2.0 / np.sqrt(2.0 * alpha)
    d = np.round(rng.uniform(max(0.7, mu - w), min(4.9, mu + w), len(at)) * 2**20) / 2**20
    s = Structure(np.concatenate([at, at + d[:, None] * [1.0, 0.0, 0.0]]), np.zeros(2 * len(at), np.int32), np.eye(3) * 130.0)
    pot = Potential(spec)
    sy = pot.system(s.pos, s.species, s.cell)
    sy.evaluate()
    sy.check()
    torch.cuda.synchronize()
    f = sy.forces.double().cpu().numpy()
    sy.close()
    pot.close()
    ref = oracle.energy_forces(spec, s.pos, s.species, s.cell)["forces"]
    err = np.sqrt(((f - ref) ** 2).mean()) / np.sqrt((ref**2).mean())
    print(f"[radial] m={m} alpha={alpha} rms error {err:.2e}")
    assert err <= 1.1e-7 + 1.2e-7 * m
