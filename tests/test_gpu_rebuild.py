"""Neighbour sets bit-exact against the oracle's brute force where the rebuild's kernels
can go wrong, at the build and after device rebuilds at displaced positions:

* cells so small that an atom has hundreds of images, more than a warp's 32 at a time,
  with atoms of differing numbers of images in one warp; rectangular and triclinic cells,
  positions on faces and many cells away;
* atom counts around the scan's 4,096-entry tile, the 2,048 atoms that one block sorts, a
  warp's 32 atoms and its last lane;
* few atoms in a cell of more than 65,536 bins (the scan with look-back) and in a long
  thin one (columns of very different bin counts per axis).
"""

from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_helpers import potential
from synth import Structure, make_model

pytestmark = pytest.mark.gpu

SKEW = np.array([[1.0, 0.0, 0.0], [0.3, 0.9, 0.0], [-0.2, 0.25, 1.1]])
TURNED = np.array([[0.1, 0.9, 0.2], [-0.8, 0.2, 0.3], [0.2, -0.1, 1.0]])


def _grid(n, cell, seed):
    """n atoms on a jittered grid over the cell, some of them exactly on faces and some
    many cells away."""
    rng = np.random.default_rng(seed)
    k = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    frac = (g[rng.permutation(len(g))[:n]] + 0.5 * (rng.random((n, 3)) < 0.7)) / k
    frac = frac + (rng.random((n, 1)) < 0.5) * rng.integers(-3, 4, (n, 3))
    pos = frac @ cell + (rng.random((n, 1)) < 0.8) * rng.normal(0, 0.05, (n, 3))
    return Structure(pos, rng.integers(0, 3, n).astype(np.int32), cell)


CASES = {
    "1_tiny": (1, np.eye(3) * 3.0),
    "2_tiny_skew": (2, SKEW * 3.6),
    "5_flat": (5, np.diag([3.0, 5.5, 21.0])),
    "31_turned": (31, TURNED * 10.0),
    "33": (33, np.diag([9.0, 10.0, 12.0])),
    "64_skew": (64, SKEW * 13.0),
    "2048": (2048, np.diag([29.0, 29.0, 31.0])),
    "2049_skew": (2049, SKEW * 29.0),
    "4095": (4095, np.diag([39.0, 36.0, 33.0])),
    "4096_skew": (4096, SKEW * 37.0),
    "4097": (4097, np.diag([36.0, 36.0, 37.0])),
    "8000_many_bins": (8000, np.eye(3) * 160.0),
    "300_long": (300, np.diag([9.0, 11.0, 4000.0])),
}


def _rows(i, j, s):
    a = np.concatenate([i[:, None], j[:, None], s], axis=1).astype(np.int64)
    return a[np.lexsort(a.T)]


@pytest.mark.parametrize("name", list(CASES))
def test_neighbor_sets(name):
    import torch

    n, cell = CASES[name]
    s = _grid(n, cell, seed=n)
    spec = make_model(T=1)
    sy = potential(spec).system(s.pos, s.species, s.cell, skin=1.0)
    for step in range(10):  # the eighth rebuild sorts the atoms again
        pos = s.pos + (0 if step == 0 else np.random.default_rng(step).normal(0, 0.1, s.pos.shape))
        if step:
            sy.rebuild(torch.as_tensor(pos, device="cuda").contiguous())
            sy.check()
        if step not in (0, 1, 8, 9):
            continue
        got, want = _rows(*sy.neighbors()), _rows(*oracle.neighbors(pos, s.cell, spec.r_c + 1.0))
        assert len(want) > 0 and np.array_equal(got, want)
    sy.close()
