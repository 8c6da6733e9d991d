"""Hubbard H*x kernel (one column, or one pair of columns; the automatic choice
there) against the oracle and the generic kernel: numbers of up strings that
are no multiple of the strings per thread block, one down string, thread-block
sizes on both sides of their limits, V terms, hops of one species, the pair
swap and the reductions.  FP64 1e-13, FP32 2e-6 of max|y|, as the other kernels."""
import random

import numpy as np
import pytest
import torch

from gpu_util import pair, rel_err
from paper_2307_13222_gb300 import hphi
from workloads import chain, hubbard_terms, random_vectors, square

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-13, torch.float32: 2e-6, torch.complex128: 1e-13, torch.complex64: 2e-6}


def _terms(N, bonds, seed):
    rng = random.Random(seed)
    t = [("HOP", i, j, rng.choice([-1, -1, 0, 1]), rng.uniform(0.5, 1.5), 0.0) for i, j in bonds]
    t += [("HUBBARD_U", i, i, 0, rng.uniform(-2, 8), 0.0) for i in range(N)]
    return t + [("DENS_DENS", i, j, 0, rng.uniform(-1, 1), 0.0) for i, j in bonds[::2]]


# (sites, up, down): 1 up or down string; 5, 6, 9 up strings; D_dn = 495 .. 792 (64 and 256
# threads), 6435 (1024)
@pytest.mark.parametrize("lx,ly,nu,nd", [(5, 1, 1, 0), (5, 1, 0, 2), (4, 1, 2, 2), (9, 1, 8, 4), (6, 2, 1, 4),
                                         (6, 2, 11, 5), (5, 3, 1, 7), (7, 1, 3, 4)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
def test_hubbard_kernel(lx, ly, nu, nd, dtype):
    N = lx * ly
    m, b, h = pair("HUBBARD", N, nu, nd, _terms(N, square(lx, ly) if ly > 1 else chain(lx), N * 7 + nu))
    cplx = dtype.is_complex
    x = torch.from_numpy(random_vectors(m.dim, 1, N, complex_=cplx, normalize=False)[:, 0].copy()).to(dtype)
    y = torch.from_numpy(random_vectors(m.dim, 1, N + 1, complex_=cplx, normalize=False)[:, 0].copy()).to(dtype)
    for alpha, beta in ((0.8, 0.0), (-1.1, 0.35)):
        pad = torch.full((m.dim + 2,), float("nan"), dtype=dtype, device="cuda")
        xd = pad.clone()[1:1 + m.dim].copy_(x)
        yd = pad[1:1 + m.dim].copy_(y)
        hphi.hphi_apply_H(h, xd, yd, alpha, beta)
        assert h.ctx.last_kernel().startswith("k_hub<")
        f = torch.float64
        if cplx:
            xr, yr = torch.view_as_real(x).to(f).numpy(), torch.view_as_real(y).to(f).numpy()
            want = sum(u * m.apply(np.ascontiguousarray(xr[:, k]), alpha, beta, np.ascontiguousarray(yr[:, k]))
                       for k, u in ((0, 1.0), (1, 1j)))
        else:
            want = m.apply(x.to(f).numpy(), alpha, beta, y.to(f).numpy().copy())
        assert rel_err(yd.cpu().numpy(), want) < TOL[dtype]
        assert pad[:1].isnan().all() and pad[1 + m.dim:].isnan().all()
        h.set_tuning(variant=0)
        y0 = y.cuda()
        hphi.hphi_apply_H(h, xd, y0, alpha, beta)
        assert rel_err(yd.cpu().numpy(), y0.cpu().numpy()) < TOL[dtype]
        h.set_tuning(variant=-1)


def _h(m, x):
    return m.apply(np.ascontiguousarray(x.real)) + 1j * m.apply(np.ascontiguousarray(x.imag))


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_hubbard_kernel_pair_swap_and_reductions(dtype):
    """Real-time and cTPQ steps of one complex column (pair swap, fused
    reductions), and Lanczos scalars of one real column."""
    m, b, h = pair("HUBBARD", 8, 4, 3, hubbard_terms(8, chain(8), t=1.0, U=4.0, V=0.3))
    tol = 1e-12 if dtype == torch.complex128 else 2e-5
    V0 = random_vectors(m.dim, 1, 5, complex_=True)
    Vg = torch.from_numpy(V0[:, 0].copy()).to(dtype).cuda()
    Vo = V0.copy()
    for _ in range(4):
        n2, e, h2, n2n = hphi.hphi_time_step(h, Vg, 0.02, 6)
        no, eo, noo = m.time_step(Vo, 0.02, 6)
    assert h.ctx.last_kernel().startswith("k_hub<")
    assert rel_err(Vg.cpu().numpy(), Vo[:, 0]) < tol
    assert np.allclose(n2, no, rtol=tol) and np.allclose(e, eo, rtol=10 * tol) and np.allclose(n2n, noo, rtol=tol)
    assert abs(h2[0] - np.linalg.norm(_h(m, Vo[:, 0])) ** 2) < 1e-3 * h2[0]  # conserved to the step's order
    norm2 = np.zeros(1)
    Wg = torch.from_numpy(V0[:, 0].copy()).to(dtype).cuda()
    Wo = V0.copy()
    for _ in range(3):
        e, h2, logd = hphi.hphi_tpq_step(h, Wg, 0.05, 4, norm2)
        eo, h2o, do = m.tpq_step(Wo, 0.05, 4)
        assert np.allclose(e, eo, rtol=10 * tol) and np.allclose(h2, h2o, rtol=10 * tol)
        assert np.allclose(logd, np.log(do), atol=10 * tol)
    rd = torch.float64 if dtype == torch.complex128 else torch.float32
    v0 = np.ascontiguousarray(V0[:, 0].real)
    got = hphi.hphi_lanczos(h, torch.from_numpy(v0).to(rd).cuda(), 10, 0.0, 10)
    want = m.lanczos(v0, 10, 0.0)
    assert np.allclose(got["alpha"], want["alpha"], atol=10 * tol) and np.allclose(got["beta"], want["beta"][1:],
                                                                                   atol=10 * tol)


# One large coupling next to small ones: a row without a doubly occupied site (or without the
# large U's) has only small terms in its diagonal, and x lives on such rows.
@pytest.mark.parametrize("U", [1.0, 1e2, 1e4, 1e6, 1e8])
@pytest.mark.parametrize("one_site", [False, True])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
def test_small_couplings_next_to_a_large_one(U, one_site, dtype):
    N = 8
    terms = hubbard_terms(N, chain(N), t=1.0, U=0.3 if one_site else U, V=0.3)
    if one_site:
        terms.append(("HUBBARD_U", 2, 2, 0, U, 0.0))
    m, b, h = pair("HUBBARD", N, 4, 3, terms)
    up, dn = (s.cpu().numpy() for s in b.states(0, b.dim))
    keep = ((up & dn) & ((1 << 2) if one_site else (1 << N) - 1)) == 0
    cplx = dtype.is_complex
    x = random_vectors(m.dim, 1, 11, complex_=cplx, normalize=False)[:, 0] * keep
    xt = torch.from_numpy(x.copy()).to(dtype)
    f = xt.to(torch.complex128 if cplx else torch.float64).numpy()
    want = _h(m, f) if cplx else m.apply(f)
    yd = torch.empty(m.dim, dtype=dtype, device="cuda")
    hphi.hphi_apply_H(h, xt.cuda(), yd)
    assert rel_err(yd.cpu().numpy(), want) < TOL[dtype]
    if not cplx and dtype == torch.float32:
        assert h.ctx.last_kernel().startswith("k_hub<f32,C1,64,I")


# Few up strings: wider thread blocks, several of which share a group of up strings (1 to 6 here,
# more of them than up strings), the last with an incomplete round; the partial sums of all.
@pytest.mark.parametrize("N,nu,nd,threads", [(14, 0, 7, 1024), (14, 1, 7, 1024), (13, 1, 6, 1024), (16, 1, 7, 1024),
                                             (10, 2, 5, 256), (9, 8, 4, 256)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
def test_few_up_strings(N, nu, nd, threads, dtype):
    m, b, h = pair("HUBBARD", N, nu, nd, hubbard_terms(N, chain(N), t=1.0, U=4.0, V=0.5))
    cplx = dtype.is_complex
    tol = TOL[dtype]
    v0 = random_vectors(m.dim, 1, N + nd, complex_=cplx)
    Vg = torch.from_numpy(v0[:, 0].copy()).to(dtype).cuda()
    if cplx:
        Vo = Vg.cpu().to(torch.complex128).numpy()[:, None].copy()
        n2, e, h2, n2n = hphi.hphi_time_step(h, Vg, 0.02, 3)
        no, eo, noo = m.time_step(Vo, 0.02, 3)
        assert rel_err(Vg.cpu().numpy(), Vo[:, 0]) < 4 * tol
        assert np.allclose(n2, no, rtol=4 * tol) and np.allclose(n2n, noo, rtol=4 * tol)
        assert np.allclose(e, eo, rtol=4 * tol, atol=40 * tol)
    else:
        x = Vg.double().cpu().numpy()
        got, want = hphi.hphi_lanczos(h, Vg, 3, 0.0, 3), m.lanczos(x, 3, 0.0)
        assert np.allclose(got["alpha"], want["alpha"], atol=40 * tol)
        assert np.allclose(got["beta"], want["beta"][1:], atol=40 * tol)
        y = torch.empty_like(Vg)
        hphi.hphi_apply_H(h, Vg, y)
        assert rel_err(y.double().cpu().numpy(), m.apply(x)) < tol
    assert f",{threads},I" in h.ctx.last_kernel() and h.ctx.last_kernel().startswith("k_hub<")


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
def test_alpha_is_applied_once(dtype):
    """y = alpha (H x) rounds H x by alpha once: bit for bit alpha times the product with
    alpha = 1 (couplings that carry alpha would be rounded once more each).  Segment kernel
    in FP64 too."""
    hams = [pair("HUBBARD", 8, 4, 3, hubbard_terms(8, chain(8), t=0.7, U=3.3, V=0.3))]
    if dtype == torch.float64:
        hams.append(pair("SPIN_HALF", 14, 7, 0, [("XXZ", i, j, 0, 0.7, 1.1) for i, j in square(7, 2)]))
    for m, b, h in hams:
        x = torch.from_numpy(random_vectors(m.dim, 1, 9, complex_=dtype.is_complex, normalize=False)[:, 0].copy())
        xd = x.to(dtype).cuda()
        y1, ya = torch.empty_like(xd), torch.empty_like(xd)
        hphi.hphi_apply_H(h, xd, y1)
        for alpha in (0.8, -1.1, 0.123456789):
            hphi.hphi_apply_H(h, xd, ya, alpha)
            r = (lambda t: torch.view_as_real(t)) if dtype.is_complex else (lambda t: t)
            al = torch.tensor(alpha, dtype=r(y1).dtype, device="cuda")
            assert torch.equal(r(ya), al * r(y1)), (h.ctx.last_kernel(), alpha)


def test_autotune_tries_every_kernel_once():
    """One Hubbard column: the automatic kernel in its one form, the row kernel in 6 (split x
    hints), the bond-major kernel in 2 (hints)."""
    m, b, h = pair("HUBBARD", 8, 4, 3, hubbard_terms(8, chain(8), t=1.0, U=4.0))
    assert h.autotune(torch.float32, 1, reps=1)[1] == 9
    assert h.autotune(torch.complex64, 1, reps=1)[1] == 7  # (the bond-major kernel takes one column)


# What the automatic choice is around the limits of shared memory: 12,870 down strings of 16 bytes
# fit (k_hub), 19,448 do not, 24,310 of the FP32 bond-major kernel's 8 bytes do, 43,758 do not.
@pytest.mark.parametrize("N,nd,f32,f64", [(16, 8, "k_hub<", "k_hub<"), (17, 7, "k_hvp<", "k_hv<"),
                                          (17, 8, "k_hvp<", "k_hv<"), (18, 8, "k_hv<", "k_hv<")])
def test_automatic_kernel_by_down_strings(N, nd, f32, f64):
    m, b, h = pair("HUBBARD", N, 1, nd, hubbard_terms(N, chain(N), t=1.0, U=4.0))
    x = random_vectors(m.dim, 1, 3, normalize=False)[:, 0]
    for dtype, name in ((torch.float32, f32), (torch.float64, f64)):
        xt = torch.from_numpy(x).to(dtype)
        y = torch.empty(m.dim, dtype=dtype, device="cuda")
        hphi.hphi_apply_H(h, xt.cuda(), y, 0.9)
        assert h.ctx.last_kernel().startswith(name)
        assert rel_err(y.cpu().double().numpy(), m.apply(xt.double().numpy(), 0.9)) < TOL[dtype]


def test_bond_major_kernel_4x4_sampled():
    """165,636,900 rows through the bond-major kernel (on request there), FP32."""
    from test_gpu_hv import _sampled_rows
    m, b, h = pair("HUBBARD", 16, 8, 8, hubbard_terms(16, square(4, 4), t=1.0, U=8.0))
    h.set_tuning(variant=3)
    rows = np.concatenate([[0, m.dim - 1], np.random.default_rng(9).integers(0, m.dim, 300)])
    assert _sampled_rows(m, h, torch.float32, 1, rows, 44) < 1e-6
    assert h.ctx.last_kernel().startswith("k_hvp<f32")


@pytest.mark.parametrize("dtype", [torch.float64, torch.complex128])
def test_huge_hop_stays_finite(dtype):
    """Hops near the end of FP64's range (the kernel scales its couplings: not taken there)."""
    m, b, h = pair("HUBBARD", 6, 3, 2, hubbard_terms(6, chain(6), t=1e295, U=4.0))
    x = torch.from_numpy(random_vectors(m.dim, 1, 4, complex_=dtype.is_complex)[:, 0].copy())
    y = torch.empty(m.dim, dtype=dtype, device="cuda")
    hphi.hphi_apply_H(h, x.to(dtype).cuda(), y)
    want = _h(m, x.numpy()) if dtype.is_complex else m.apply(x.numpy())
    assert rel_err(y.cpu().numpy() / 1e295, want / 1e295) < TOL[dtype]
