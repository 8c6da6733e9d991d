"""Tables that a sector Hamiltonian builds on the host: the segment kernel's rank
tables and the bond-major kernel's lists, through products of every basis vector
of small sectors (a wrong rank shows as a wrong column), against the oracle's
dense matrix.  Exact: one nonzero term per entry."""
import itertools
import random

import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import pair
from paper_2307_13222_gb300 import hphi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nup", [(2, 1), (3, 1), (7, 3), (9, 2), (11, 9), (21, 2)])
@pytest.mark.parametrize("variant", [-1, 3])
def test_every_column(N, nup, variant):
    rng = random.Random(N)
    pairs = list(itertools.combinations(range(N), 2))
    pairs = rng.sample(pairs, min(len(pairs), 3 * N))
    m, b, h = pair("SPIN_HALF", N, nup, 0, [("XXZ", i, j, 0, rng.choice([-2.0, 1.0, 4.0]), rng.choice([0.0, 2.0, -1.0]))
                                            for i, j in pairs])
    h.set_tuning(variant=variant)
    want = O.dense_matrix(m)
    eye = torch.eye(m.dim, dtype=torch.float64, device="cuda")
    y = torch.empty(m.dim, dtype=torch.float64, device="cuda")
    for c in range(m.dim):
        hphi.hphi_apply_H(h, eye[c], y)
        assert np.array_equal(y.cpu().numpy(), want[:, c]), c
