"""Gram-Schmidt passes at the sizes where a split of rows or columns can go
wrong, against the oracle's CGS2: one cluster (up to 2,048 unknowns), clusters
with partial sums (below 16,384), column-split passes, and one row per thread
(from 152 * 384 unknowns up); column counts at the edges of the warps' shares
and one past the last register pass.

Tolerance: operands are split to 2^-49, products and sums are pairs of about
2^-46 relative error, and at most 2^17 terms of size ||v|| ||w|| / n add up to
a coefficient: 1e-12 ||w|| leaves a factor of ten."""
import numpy as np
import pytest

import stab_inputs as si

pytestmark = pytest.mark.gpu
SIZES = [(8, 8), (16, 32), (9, 57), (32, 64), (63, 65), (64, 64), (37, 111), (121, 121)]
KS = (1, 4, 5, 16, 17, 33, 64, 65)


def _stab(nx, ny, **opts):
    from paper_1502_03701_gb300 import Stab
    g = si.Grid(2, nx, ny, 1, si.LX_04, -15, 15)
    f = si.Flow(0.3, 1000.0)
    return Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, **opts), g


@pytest.mark.parametrize("nx,ny", SIZES, ids=[f"{4 * a * b}" for a, b in SIZES])
def test_cgs2_at_edge_sizes(orc, nx, ny):
    import torch
    S, g = _stab(nx, ny)
    rng = np.random.default_rng(nx)
    Q = np.linalg.qr(rng.standard_normal((g.n, max(KS))) + 1j * rng.standard_normal((g.n, max(KS))))[0]
    for k in KS:
        V = torch.from_numpy(np.ascontiguousarray(Q[:, :k].T)).cuda()
        w = si.random_complex(40 + k, g.n)
        wn = np.linalg.norm(w)
        for scale in (1.0, 0.0):  # a generic vector, and one in the span up to 1e-6
            x = scale * w + (1.0 - scale) * (Q[:, :k] @ si.random_complex(k, k) + 1e-6 * w)
            wd = torch.from_numpy(x.copy()).cuda()
            h, nrm = S.orthogonalize(V, k, wd)
            href, wref = orc.krylov.cgs2(Q[:, :k], x)
            got = wd.cpu().numpy()
            assert np.abs(h - href).max() < 1e-12 * wn, k
            assert np.linalg.norm(got - wref) < 1e-12 * wn, k
            assert abs(nrm - np.linalg.norm(got)) < 1e-12 * wn, k
    S.close()


def test_batched_cgs2_equals_single_bit_for_bit():
    """The same bodies in one launch over all row splits."""
    import torch
    from paper_1502_03701_gb300 import JvBatch
    hs, Vs, ws, ks = [], [], [], [29, 3, 17, 64, 40, 33]
    for (nx, ny), k in zip([(16, 32), (8, 8), (9, 57), (63, 65), (37, 111), (121, 121)], ks):
        S, g = _stab(nx, ny)
        rng = np.random.default_rng(k)
        V = np.linalg.qr(rng.standard_normal((g.n, k)) + 1j * rng.standard_normal((g.n, k)))[0]
        hs.append(S)
        Vs.append(torch.from_numpy(np.ascontiguousarray(V.T)).cuda())
        ws.append(torch.from_numpy(si.random_complex(k, g.n)).cuda())
    single = []
    for S, V, k, w in zip(hs, Vs, ks, ws):
        w1 = w.clone()
        single.append((w1,) + tuple(S.orthogonalize(V, k, w1)))
    B = JvBatch(hs)
    w2 = [w.clone() for w in ws]
    hb, nb = B.orthogonalize(Vs, ks, w2)
    for (w1, h1, n1), wb, h, n in zip(single, w2, hb, nb):
        assert torch.equal(w1, wb) and np.array_equal(h1, h) and n1 == n
    B.close()
    for S in hs:
        S.close()


@pytest.mark.parametrize("nx,ny", [(65, 66), (121, 122)])
def test_gmres_reorthogonalises(nx, ny):
    """With a shift far above the spectrum of J every new Krylov vector lies
    almost in the span of the earlier ones, so the second pass of the selective
    reorthogonalisation runs at each step; the solution has the residual that
    GMRES reports."""
    import torch
    S, g = _stab(nx, ny, eps_mode=2, gmres_m=30, gmres_tol=1e-10)
    sigma = 2.0e4
    b = torch.from_numpy(si.random_complex(3, g.n)).cuda()
    x = torch.zeros_like(b)
    st, iters = S.solve(sigma, b, x)
    assert st == 0 and iters > 1
    r = torch.empty_like(b)
    S.apply_J(x, r, sigma)
    assert float(torch.linalg.vector_norm(r - b)) < 2e-10 * float(torch.linalg.vector_norm(b))
    S.close()
