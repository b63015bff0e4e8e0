"""J(s v) = s J(v) over the documented range of v, for base flows that depend on
y only: entries and derivative fields between 2^-74 and 2^100 keep full accuracy,
smaller ones FP32 accuracy of their own.

s is a power of two, so where nothing leaves that range the bits agree.  Below,
an entry of a field under 2^-74 is off by at most 2^-98, and J v weighs the fields
by coefficients: the largest are the heat conduction's, mu cp / Pr = 3,914 per
direction at Ma 0.3 and Re 0.01, all others add up to less than 1,500.  10^4 times
2^-98, over the largest entry of J v, bounds the error; where s is large, 1e-12.
The lines are long: differences of neighbours are 2^-11 of the derivatives, second
differences 2^-21."""
import numpy as np
import pytest

import stab_inputs as si
from gpu_util import max_rel_err

pytestmark = pytest.mark.gpu
GRIDS = [si.Grid(2, 16, 1500, 1, si.LX_04, -15, 15), si.Grid(2, 1500, 16, 1, si.LX_04, -15, 15),
         si.Grid(3, 8, 12, 1200, si.LX_04, -15, 15, si.LX_04), si.Grid(2, 300, 700, 1, si.LX_04, -15, 15)]


def _waves(g):
    """Smooth fields bounded away from zero, a few waves along every axis."""
    z, y, x = np.meshgrid(np.arange(g.nz) / g.nz, np.arange(g.ny) / g.ny, np.arange(g.nx) / g.nx, indexing="ij")
    out = []
    for a in range(g.nvars):
        w = np.cos(2 * np.pi * x + a) * np.cos(5 * y + a) * np.cos(2 * np.pi * z + 2 * a)
        out.append(1.5 + 0.4 * w + 1j * (1.4 - 0.3 * w ** 2))
    return np.stack(out).reshape(-1)


@pytest.mark.parametrize("mode", [2, 0], ids=["tangent", "quotient"])
@pytest.mark.parametrize("g", GRIDS, ids=[f"{g.nx}x{g.ny}x{g.nz}" for g in GRIDS])
def test_scaled_input_gives_scaled_output(g, mode):
    import torch
    from paper_1502_03701_gb300 import Stab
    f = si.Flow(0.3, 0.01)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, eps_mode=mode)
    v = torch.from_numpy(_waves(g)).cuda()
    one, out = torch.empty_like(v), torch.empty_like(v)
    S.apply_J(v, one)
    assert torch.isfinite(torch.view_as_real(one)).all()
    largest = float(one.abs().max())
    for p in (-60, -56, -30, 30, 60, 90):
        S.apply_J(v * 2.0 ** p, out)
        got = out * 2.0 ** -p
        if abs(p) == 30 and mode == 2:
            assert torch.equal(got, one), p
        assert max_rel_err(got.cpu().numpy(), one.cpu().numpy()) < 1e-12 + 1e4 * 2.0 ** (-98 - p) / largest, p
    S.close()
