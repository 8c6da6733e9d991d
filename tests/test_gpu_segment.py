"""Segment H*x kernel (S^z sector, one column; the automatic choice there)
against the oracle and the bond-major kernel.  Tolerances as the other H*x
kernels: the same terms per row in another order (FP64 1e-13, FP32 2e-6 of
max|y|)."""
import itertools
import random

import numpy as np
import pytest
import torch

from gpu_util import pair, rel_err
from paper_2307_13222_gb300 import hphi
from workloads import chain, heisenberg_terms, random_vectors, square

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-13, torch.float32: 2e-6}


def _terms(N, seed):
    rng = random.Random(seed)
    pairs = list(itertools.combinations(range(N), 2))
    pairs = rng.sample(pairs, min(len(pairs), 3 * N))
    return [("XXZ", i, j, 0, rng.uniform(-1, 2), rng.uniform(-1, 2) if k % 7 else 0.0)
            for k, (i, j) in enumerate(pairs)]


# two sites to segments of 10 bits with and without further low bits, popcounts at
# both ends of the sector, a last row block shorter than a warp, one state
@pytest.mark.parametrize("N,nup", [(2, 0), (2, 1), (3, 3), (9, 4), (12, 6), (13, 1), (16, 8), (17, 8), (19, 3),
                                   (20, 10), (21, 20), (22, 11), (23, 9), (25, 5)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_segment_kernel(N, nup, dtype):
    m, b, h = pair("SPIN_HALF", N, nup, 0, _terms(N, N * 41 + nup))
    x = torch.from_numpy(random_vectors(m.dim, 1, N, normalize=False)[:, 0]).to(dtype)
    y = torch.from_numpy(random_vectors(m.dim, 1, N + 1, normalize=False)[:, 0]).to(dtype)
    for alpha, beta in ((0.8, 0.0), (-1.1, 0.35)):
        # x and y between guard values, at addresses that are no multiple of 16 bytes
        pad = torch.full((m.dim + 130,), float("nan"), dtype=dtype, device="cuda")
        xd = pad.clone()[65:65 + m.dim].copy_(x)
        yd = pad[65:65 + m.dim].copy_(y)
        hphi.hphi_apply_H(h, xd, yd, alpha, beta)
        want = m.apply(x.double().numpy(), alpha, beta, y.double().numpy().copy())
        assert rel_err(yd.cpu().double().numpy(), want) < TOL[dtype]
        assert pad[:65].isnan().all() and pad[65 + m.dim:].isnan().all()
        if dtype == torch.float64 or m.dim >= 16384:
            assert h.ctx.last_kernel().startswith("k_hvw<")
        h.set_tuning(variant=3)
        y3 = y.cuda()
        hphi.hphi_apply_H(h, xd, y3, alpha, beta)
        assert rel_err(yd.cpu().double().numpy(), y3.cpu().double().numpy()) < TOL[dtype]
        h.set_tuning(variant=-1)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_segment_kernel_reductions(dtype):
    """The fused reductions of every launch form: Lanczos steps (<x, y>) and
    one-column cTPQ steps (<x, Hx>, |Hx|^2, |x|^2; |y|^2)."""
    m, b, h = pair("SPIN_HALF", 18, 9, 0, heisenberg_terms(square(6, 3), 1.0))
    v0 = random_vectors(m.dim, 1, 8)[:, 0]
    r = hphi.hphi_lanczos(h, torch.from_numpy(v0).to(dtype).cuda(), 12, 0.0, 12)
    ro = m.lanczos(v0, 12, 0.0)
    tol = 1e-11 if dtype == torch.float64 else 2e-6
    assert np.allclose(r["alpha"], ro["alpha"], rtol=tol, atol=tol)
    assert np.allclose(r["beta"], ro["beta"][1:], rtol=tol, atol=tol)
    Vg = torch.from_numpy(v0[:, None].copy()).to(dtype).cuda().contiguous()
    Vo = v0[:, None].copy()
    norm2 = np.zeros(1)
    for _ in range(3):
        e, h2, logd = hphi.hphi_tpq_step(h, Vg, 0.05, 6, norm2)
        eo, h2o, do = m.tpq_step(Vo, 0.05, 6)
        assert np.allclose(e, eo, rtol=tol, atol=tol) and np.allclose(h2, h2o, rtol=tol)
        assert np.allclose(logd, np.log(do), rtol=10 * tol, atol=tol)


def test_segment_kernel_repeats_bitwise():
    m, b, h = pair("SPIN_HALF", 20, 10, 0, heisenberg_terms(chain(20), 1.0))
    x = torch.from_numpy(random_vectors(m.dim, 1, 3)[:, 0]).cuda()
    a = hphi.hphi_lanczos(h, x, 30, 0.0, 30)
    c = hphi.hphi_lanczos(h, x, 30, 0.0, 30)
    assert (a["alpha"] == c["alpha"]).all() and (a["beta"] == c["beta"]).all()


# Two strong Ising bonds that cancel on the rows where x lives, next to weak couplings: the
# grid of the fixed-point diagonal follows the strong ones.  FP64: S first in the site order
# and -S next, so that a sum over the bonds holds no trace of them.
@pytest.mark.parametrize("S", [1.0, 1e4, 1e8])
@pytest.mark.parametrize("dtype,pairs,sign,rows", [(torch.float32, ((0, 2), (4, 6)), -1, (0, 0)),
                                                   (torch.float32, ((0, 2), (4, 6)), 1, (0, 1)),
                                                   (torch.float64, ((0, 2), (0, 3)), -1, (0, 0))])
def test_weak_couplings_next_to_cancelling_strong_ones(S, dtype, pairs, sign, rows):
    N = 18
    terms = [("XXZ", *pairs[0], 0, S, 0.0), ("XXZ", *pairs[1], 0, sign * S, 0.0)] + heisenberg_terms(chain(N)[1:], 0.7)
    m, b, h = pair("SPIN_HALF", N, 9, 0, terms)
    s = b.states(0, b.dim)[0].cpu().numpy()
    anti = [((s >> i) ^ (s >> j)) & 1 for i, j in pairs]
    x = random_vectors(m.dim, 1, 5, normalize=False)[:, 0] * ((anti[0] == rows[0]) & (anti[1] == rows[1]))
    xt = torch.from_numpy(x).to(dtype)
    y = torch.empty(m.dim, dtype=dtype, device="cuda")
    hphi.hphi_apply_H(h, xt.cuda(), y)
    assert rel_err(y.cpu().double().numpy(), m.apply(xt.double().numpy())) < TOL[dtype]
    if dtype == torch.float32:
        assert h.ctx.last_kernel().startswith("k_hvw<f32")


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("model,ncol", [("SPIN_HALF", 1), ("SPIN_HALF_GC", 32)])
def test_coupling_that_is_not_finite_stays_on_its_rows(model, ncol, dtype):
    """An infinite exchange coupling marks the rows of its bond and no others (segment and
    tiled kernels)."""
    N = 18 if ncol == 1 else 9
    m, b, h = pair(model, N, N // 2, 0, heisenberg_terms(chain(N), 0.7)[1:] + [("XXZ", 0, 1, 0, 0.7, float("inf"))])
    s = b.states(0, b.dim)[0].cpu().numpy()
    x = torch.ones((m.dim, ncol), dtype=dtype, device="cuda")
    y = torch.empty_like(x)
    hphi.hphi_apply_H(h, x, y)
    assert (np.isfinite(y.cpu().numpy()) == (((s ^ (s >> 1)) & 1) == 0)[:, None]).all()


# FP32 (above 2^14 rows, below which the bond-major kernel takes the call) at both ends of the
# popcounts: segments of 0 to 4 and of 6 to 10 up spins, of one row to 210, most of them short.
@pytest.mark.parametrize("N,nup", [(27, 4), (27, 23), (31, 4), (20, 7)])
def test_segment_kernel_f32_sparse_sectors(N, nup):
    m, b, h = pair("SPIN_HALF", N, nup, 0, _terms(N, N * 41 + nup)[:64])
    x = torch.from_numpy(random_vectors(m.dim, 1, N, normalize=False)[:, 0]).float()
    y = torch.from_numpy(random_vectors(m.dim, 1, N + 1, normalize=False)[:, 0]).float()
    for alpha, beta in ((0.8, 0.0), (-1.1, 0.35)):
        pad = torch.full((m.dim + 130,), float("nan"), device="cuda")
        xd = pad.clone()[65:65 + m.dim].copy_(x)
        yd = pad[65:65 + m.dim].copy_(y)
        hphi.hphi_apply_H(h, xd, yd, alpha, beta)
        assert h.ctx.last_kernel().startswith("k_hvw<f32")
        want = m.apply(x.double().numpy(), alpha, beta, y.double().numpy().copy())
        assert rel_err(yd.cpu().double().numpy(), want) < TOL[torch.float32]
        assert pad[:65].isnan().all() and pad[65 + m.dim:].isnan().all()
