"""Tiled block kernel by items of rows (full space, 32 real columns): the
smallest space, one tile, a tile set one site short of the space (two
separated single sites), several tiles, bonds with none, one and both sites in
an item, and the cTPQ and real-time forms.  FP64 1e-13, FP32 2e-6 of max|y|."""
import itertools
import random

import numpy as np
import pytest
import torch

from gpu_util import pair, rel_err
from paper_2307_13222_gb300 import hphi
from workloads import chain, random_vectors

pytestmark = pytest.mark.gpu


def _terms(N, seed, bonds):
    rng = random.Random(seed)
    return [("XXZ", i, j, 0, rng.uniform(-1, 2), rng.uniform(-1, 2) if k % 5 else 0.0)
            for k, (i, j) in enumerate(bonds)]


@pytest.mark.parametrize("N,dense", [(5, True), (6, True), (11, True), (18, False), (19, False), (20, False)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_items(N, dense, dtype):
    bonds = list(itertools.combinations(range(N), 2)) if dense else chain(N)
    m, b, h = pair("SPIN_HALF_GC", N, 0, 0, _terms(N, 3 * N, bonds))
    X = torch.from_numpy(random_vectors(m.dim, 32, N, normalize=False)).to(dtype)
    Y = torch.from_numpy(random_vectors(m.dim, 32, N + 1, normalize=False)).to(dtype)
    for alpha, beta in ((0.7, 0.0), (-1.2, 0.4)):
        y = Y.cuda()
        hphi.hphi_apply_H(h, X.cuda(), y, alpha, beta)
        assert h.ctx.last_kernel().startswith("k_tile<")
        cols = [0, 1, 13, 31]  # every lane layout's first, middle and last columns
        want = np.stack([m.apply(np.ascontiguousarray(X[:, c].double().numpy()), alpha, beta,
                                 np.ascontiguousarray(Y[:, c].double().numpy())) for c in cols], axis=1)
        assert rel_err(y[:, cols].cpu().double().numpy(), want) < (1e-13 if dtype == torch.float64 else 2e-6)


@pytest.mark.parametrize("N", [8, 18])
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_steps(N, dtype):
    """Pair swap and fused reductions of 16 complex columns."""
    m, b, h = pair("SPIN_HALF_GC", N, 0, 0, _terms(N, N, chain(N)))
    tol = 1e-11 if dtype == torch.complex128 else 2e-5
    V0 = random_vectors(m.dim, 16, 7, complex_=True)
    Vg, Vo = torch.from_numpy(V0).to(dtype).cuda().contiguous(), V0[:, :2].copy()
    for _ in range(2):
        n2, e, h2, n2n = hphi.hphi_time_step(h, Vg, 0.02, 4)
        no, eo, noo = m.time_step(Vo, 0.02, 4)
        assert np.allclose(n2[:2], no, rtol=tol) and np.allclose(e[:2], eo, rtol=tol, atol=tol)
    assert rel_err(Vg[:, :2].cpu().numpy(), Vo) < tol
    norm2 = np.zeros(16)
    Vg, Vo = torch.from_numpy(V0).to(dtype).cuda().contiguous(), V0[:, :2].copy()
    for _ in range(2):
        e, h2, logd = hphi.hphi_tpq_step(h, Vg, 0.05, 3, norm2)
        eo, h2o, do = m.tpq_step(Vo, 0.05, 3)
        assert np.allclose(e[:2], eo, rtol=tol, atol=tol) and np.allclose(h2[:2], h2o, rtol=tol)
        assert np.allclose(logd[:2], np.log(do), atol=tol)
    assert rel_err(Vg[:, :2].cpu().numpy(), Vo / np.linalg.norm(Vo, axis=0) * np.sqrt(norm2[:2])) < tol


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_steps_over_many_tiles_repeat_bitwise(dtype):
    """Several tiles per pass: tickets in the first pass, paced thread blocks in the second
    (its sums in a fixed order), so a repeated step gives the same bits."""
    N = 20
    m, b, h = pair("SPIN_HALF_GC", N, 0, 0, _terms(N, N, chain(N)))
    tol = 1e-11 if dtype == torch.complex128 else 2e-5
    V0 = random_vectors(m.dim, 16, 7, complex_=True)
    runs = []
    for _ in range(2):
        V = torch.from_numpy(V0).to(dtype).cuda().contiguous()
        ev = hphi.hphi_time_step(h, V, 0.02, 3)
        norm2 = np.zeros(16)
        tp = hphi.hphi_tpq_step(h, V, 0.05, 2, norm2)
        assert h.ctx.last_kernel().startswith("k_tile<")
        runs.append((V, [np.asarray(a) for a in (*ev, *tp, norm2)]))
    assert torch.equal(torch.view_as_real(runs[0][0]), torch.view_as_real(runs[1][0]))
    assert all(np.array_equal(a, c) for a, c in zip(runs[0][1], runs[1][1]))
    Vo = V0[:, :1].copy()
    no, eo, noo = m.time_step(Vo, 0.02, 3)
    n2, e = runs[0][1][:2]
    assert np.allclose(n2[:1], no, rtol=tol) and np.allclose(e[:1], eo, rtol=tol, atol=tol)
    eo, h2o, do = m.tpq_step(Vo, 0.05, 2)
    e, h2, logd, norm2 = runs[0][1][4:]
    assert np.allclose(e[:1], eo, rtol=tol, atol=tol) and np.allclose(h2[:1], h2o, rtol=tol)
    assert rel_err(runs[0][0][:, :1].cpu().numpy(), Vo / np.linalg.norm(Vo, axis=0) * np.sqrt(norm2[:1])) < tol
