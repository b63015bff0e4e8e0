"""FP64 applies of the reduced-operator preconditioner with more tiles than SMs
(half the threads per tile): M z = q tile by tile, with the tiles' own blocks.

Tolerance: FP64 factors to rounding, as for the other level sizes (1e-9)."""
import numpy as np
import pytest

import stab_inputs as si

pytestmark = pytest.mark.gpu
# (nx, ny, nz), tile: 8 tx unknowns per level in 2-D (10 tx tz in 3-D), ty / 2 levels; 160 tiles and more
CASES = [((20, 40, 1), (1, 4)), ((48, 40, 1), (3, 4)), ((128, 96, 1), (8, 6)), ((160, 64, 1), (16, 4)),
         ((320, 64, 1), (32, 4)), ((32, 32, 16), (2, 8, 2)), ((160, 6, 6), (1, 6, 6))]


@pytest.mark.parametrize("n,tile", CASES, ids=["x".join(map(str, n + t)) for n, t in CASES])
def test_many_tiles(n, tile):
    import torch
    from paper_1502_03701_gb300 import Stab
    dim = 3 if n[2] > 1 else 2
    g = si.Grid(dim, *n, si.LX_04, -15, 15, *((si.LX_04,) if dim == 3 else ()))
    f = si.Flow(0.4, 700.0)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, precond=2, tile=tile, precond_prec=64)
    sigma = 0.25 + 0.05j
    S.precond_build(sigma)
    q = si.random_complex(5, g.n)
    z = torch.empty(g.n, dtype=torch.complex128, device="cuda")
    S.precond_apply(torch.from_numpy(q).cuda(), z)
    tx, ty, tz = tile + (1,) * (3 - len(tile))
    shape = (g.nvars, g.nz // tz, tz, g.ny // ty, ty, g.nx // tx, tx)
    q, z = q.reshape(shape), z.cpu().numpy().reshape(shape)
    count = shape[1] * shape[3] * shape[5]
    assert count > 152
    for t in (0, 1, 151, 152, count - 1):
        X, Y, Z = t % shape[5], t // shape[5] % shape[3], t // (shape[5] * shape[3])
        M = S.precond_block(sigma, t)
        r = M @ z[:, Z, :, Y, :, X].reshape(-1) - q[:, Z, :, Y, :, X].reshape(-1)
        size = np.linalg.norm(M, 2) * np.linalg.norm(z[:, Z, :, Y, :, X]) + np.linalg.norm(q[:, Z, :, Y, :, X])
        assert np.linalg.norm(r) < 1e-9 * size, t
    S.close()
