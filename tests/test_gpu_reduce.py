"""Partial sums, the one-column dot and the multi-vector kernels at their
edges: lengths around a vector load, a tile and a grid, unaligned operands, and
stored-vector counts around the groups of 8 and 16.  FP64 sums agree with
numpy's to 1e-13 of the sum of magnitudes (another order of the same terms);
FP32 data to 1e-6 of it."""
import numpy as np
import pytest
import torch

from gpu_util import ctx, pair
from paper_2307_13222_gb300 import hphi
from workloads import chain, hubbard_terms, random_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 7, 1023, 1024 * 256 + 1, 3_000_001])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("shift", [0, 1])
def test_one_column_dot(n, dtype, shift):
    g = torch.Generator().manual_seed(n)
    a = torch.randn(n + 1, dtype=dtype, generator=g).cuda()[shift:shift + n]
    b = torch.randn(n + 1, dtype=dtype, generator=g).cuda()[shift:shift + n]
    got = hphi.hphi_dot(ctx(), a, b)[0]
    terms = a.cpu().double().numpy() * b.cpu().double().numpy()
    assert abs(got - terms.sum()) <= (1e-13 if dtype == torch.float64 else 1e-6) * np.abs(terms).sum()
    assert hphi.hphi_dot_static(0, a, b)[0] == got
    assert hphi.hphi_dot(ctx(), a, b)[0] == got


# rows: below one 16-byte load, not a multiple of it, more than one tile
@pytest.mark.parametrize("L,nu,nd,steps", [(3, 1, 1, 5), (5, 2, 1, 17), (7, 3, 3, 33), (9, 4, 4, 18)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_reorthogonalised_basis(L, nu, nd, steps, dtype):
    """alpha, beta of the reorthogonalised run are those of the oracle's projected
    matrix: T = V^T H V from a dense Krylov basis in FP64 (1e-10; FP32 storage
    1e-4, its rounding carried through the steps)."""
    m, b, h = pair("HUBBARD", L, nu, nd, hubbard_terms(L, chain(L), t=1.0, U=3.0, V=0.4))
    v0 = random_vectors(m.dim, 1, 4)[:, 0]
    gs = torch.empty(m.dim + 1, dtype=dtype, device="cuda")[1:]  # not on a 16-byte boundary
    r = hphi.hphi_lanczos(h, torch.from_numpy(v0).to(dtype).cuda(), steps, 0.0, steps, gs, True)
    V = [v0 / np.linalg.norm(v0)]
    al, be = [], []
    for _ in range(r["steps"]):
        u = m.apply(V[-1])
        al.append(V[-1] @ u)
        for _ in range(2):
            for w in V:
                u = u - (w @ u) * w
        be.append(np.linalg.norm(u))
        V.append(u / be[-1])
    tol = 1e-10 if dtype == torch.float64 else 1e-4
    assert np.allclose(r["alpha"], al, rtol=0, atol=tol) and np.allclose(r["beta"][:-1], be[:-1], rtol=0, atol=tol)
    assert abs(float(torch.linalg.vector_norm(gs.double())) - 1.0) < (1e-12 if dtype == torch.float64 else 1e-6)
