"""Applies of the preconditioners at the sizes where a split can go wrong:
levels of the reduced operator from one row's threads to 256 unknowns (register
pieces, shared ring, unstaged), one level and level counts around the depth of
the prefetch; block-Jacobi blocks from four rows up in BF16, FP32 and FP64.

Tolerances are those of the storage: FP64 factors to rounding (1e-9), FP32 and
BF16 to their unit roundoff times the blocks' conditioning (1e-3, 3e-2)."""
import numpy as np
import pytest

import stab_inputs as si
from gpu_util import rel_err

pytestmark = pytest.mark.gpu
TOL = {64: 1e-9, 32: 1e-3, 16: 3e-2}


def _make(g, f, **opts):
    from paper_1502_03701_gb300 import Stab
    return Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, **opts)


def _apply(S, q):
    import torch
    z = torch.empty(q.size, dtype=torch.complex128, device="cuda")
    S.precond_apply(torch.from_numpy(q).cuda(), z)
    return z.cpu().numpy()


# (nx, ny, nz), tile: 8 tx unknowns per level in 2-D (10 tx tz in 3-D), ty / 2 levels
LEVELS = [
    ((8, 12, 1), (1, 12)), ((8, 14, 1), (2, 14)), ((6, 8, 1), (3, 2)), ((8, 10, 1), (4, 10)), ((10, 12, 1), (5, 6)),
    ((16, 10, 1), (8, 10)), ((16, 8, 1), (8, 4)), ((9, 8, 1), (9, 8)), ((16, 12, 1), (16, 12)), ((32, 8, 1), (32, 8)),
    ((6, 8, 6), (1, 8, 1)), ((6, 6, 6), (3, 6, 2)), ((8, 8, 6), (4, 8, 2)),
]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n,tile", LEVELS, ids=["x".join(map(str, n + t)) for n, t in LEVELS])
def test_reduced_apply_at_edge_levels(orc, n, tile, prec):
    dim = 3 if n[2] > 1 else 2
    g = si.Grid(dim, *n, si.LX_04, -15, 15, *((si.LX_04,) if dim == 3 else ()))
    f = si.Flow(0.4, 700.0)
    S = _make(g, f, precond=2, tile=tile, precond_prec=prec)
    sigma = 0.25 + 0.05j
    S.precond_build(sigma)
    P = orc.Problem.from_inputs(g, f, low_order=1)
    J = orc.core.dense_jacobian(P, si.tanh_base_flow(g, f))
    M = orc.stability.BlockJacobi(P, tile, orc.stability.blocks_from_dense(J, P, tile, sigma))
    q = si.random_complex(12, g.n)
    assert rel_err(_apply(S, q), M(q)) < TOL[prec]
    # a non-finite entry stays non-finite (results are converted without the conversion instruction)
    q[0] = float("nan")
    assert not np.isfinite(_apply(S, q)).all()
    S.close()


BLOCKS = [((6, 7), (1, 1)), ((6, 8), (2, 1)), ((9, 10), (3, 5)), ((16, 16), (8, 16)), ((32, 16), (16, 16))]


@pytest.mark.parametrize("n,tile", BLOCKS, ids=["x".join(map(str, n + t)) for n, t in BLOCKS])
def test_block_apply_at_edge_blocks(orc, n, tile):
    g = si.Grid(2, *n, 1, si.LX_04, -15, 15)
    f = si.Flow(0.3, 1000.0)
    P = orc.Problem.from_inputs(g, f)
    J = orc.core.dense_jacobian(P, si.tanh_base_flow(g, f))
    M = orc.stability.BlockJacobi(P, tile, orc.stability.blocks_from_dense(J, P, tile, 0.25))
    q = si.random_complex(7, g.n)
    ref = M(q)
    for prec, tol in TOL.items():
        S = _make(g, f, tile=tile, precond_prec=prec)
        S.precond_build(0.25)
        assert rel_err(_apply(S, q), ref) < tol, prec
        S.close()
