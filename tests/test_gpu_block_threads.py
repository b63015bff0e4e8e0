"""BF16 block applies whose thread count follows the block size: every class of
block rows (32 to 256 threads, one row per thread for sizes that are no multiple
of four), each against the FP64 inverses of the same blocks, and all of them in
one batch, bit for bit.

Tolerance: BF16 storage, as for the other applies (3e-2)."""
import pytest

import stab_inputs as si
from gpu_util import rel_err

pytestmark = pytest.mark.gpu
# (nx, ny, nz), tile: 4 (3-D: 5) unknowns per point
CASES = [((20, 18, 1), (1, 1)), ((20, 18, 1), (2, 1)), ((64, 60, 1), (2, 2)), ((20, 24, 1), (5, 1)), ((16, 18, 1), (4, 2)),
         ((20, 18, 1), (4, 3)), ((32, 24, 1), (4, 4)), ((10, 9, 1), (5, 3)), ((24, 24, 1), (8, 6)), ((48, 32, 1), (16, 16)),
         ((8, 9, 6), (1, 1, 1)), ((6, 9, 6), (3, 1, 1)), ((12, 9, 6), (3, 3, 1)), ((10, 10, 6), (5, 5, 3)),
         ((8, 8, 6), (2, 2, 1)), ((6, 6, 6), (3, 3, 3))]


def test_bf16_blocks_of_every_thread_count():
    import torch
    from paper_1502_03701_gb300 import JvBatch, Stab
    hs, qs, zs = [], [], []
    for n, tile in CASES:
        dim = 3 if n[2] > 1 else 2
        g = si.Grid(dim, *n, si.LX_04, -15, 15, *((si.LX_04,) if dim == 3 else ()))
        f = si.Flow(0.4, 700.0)
        q = torch.from_numpy(si.random_complex(len(hs), g.n)).cuda()
        z = {}
        for prec in (64, 16):
            S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, tile=tile, precond_prec=prec)
            S.precond_build(0.25)
            z[prec] = torch.empty_like(q)
            S.precond_apply(q, z[prec])
            if prec == 64:
                S.close()
        assert rel_err(z[16].cpu().numpy(), z[64].cpu().numpy()) < 3e-2, (n, tile)
        hs.append(S)
        qs.append(q)
        zs.append(z[16])
    B = JvBatch(hs)
    out = [torch.empty_like(q) for q in qs]
    B.precond_apply(qs, out)
    for o, z, c in zip(out, zs, CASES):
        assert torch.equal(o, z), c
    B.close()
    for S in hs:
        S.close()
