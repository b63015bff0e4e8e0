"""J v - shift v where the shift's term is far larger than J v (base flows that
depend on y only): that term is rounded to FP64, not to a pair's 48 bits.

Tolerance, relative to |shift| ||v||: two roundings of each component here, three
in the reference's complex product and one in its difference, 6 sqrt(2) 2^-53 =
9.4e-16; J v's own error, at most 1e-10 of its entries, with shifts so large that
||J v|| / ||shift v|| < 1e-6: below 1e-16 of the rest."""
import pytest

import stab_inputs as si
from gpu_util import rel_err

pytestmark = pytest.mark.gpu
# one output row per thread, all rows per thread; 2-D and 3-D
GRIDS = [si.Grid(2, 17, 33, 1, si.LX_04, -15, 15), si.Grid(2, 131, 190, 1, si.LX_04, -15, 15),
         si.Grid(3, 12, 18, 10, si.LX_04, -15, 15, si.LX_04), si.Grid(3, 40, 33, 20, si.LX_04, -15, 15, si.LX_04)]


@pytest.mark.parametrize("shift", [3.0e9, 2.0e9 - 1.0e9j, 5.0e9j], ids=["real", "complex", "imag"])
@pytest.mark.parametrize("g", GRIDS, ids=[f"{g.nx}x{g.ny}x{g.nz}" for g in GRIDS])
def test_large_shift_keeps_fp64(orc, g, shift):
    import torch
    from paper_1502_03701_gb300 import JvBatch, Stab
    f = si.Flow(0.5, 600.0)
    q0 = si.tanh_base_flow(g, f)
    v = si.random_complex(71, g.n)
    dv = torch.from_numpy(v).cuda()
    for mode in (2, 0):
        S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=mode)
        out = torch.empty_like(dv)
        S.apply_J(dv, out, shift)
        ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent" if mode == 2 else "quad",
                          None if mode == 2 else S.last_eps())
        assert rel_err(out.cpu().numpy(), ref - shift * v) < 9.5e-16
        B = JvBatch([S])
        one = torch.empty_like(dv)
        B.apply([dv], [one], [shift])
        assert torch.equal(one, out)
        B.close()
        S.close()
