"""Pair-arithmetic line passes and the sparse pointwise map of J v (base flows
that depend on y only) against the oracle, at the sizes where a chunk
partition can go wrong: the shortest lines, one point past a chunk, chunks of
uneven length, lines shorter than the reach of the sweeps, and every line
shape.  The base flow has all of its fields varying in y, so every coefficient
that the map keeps can differ from zero.

Tolerance: a value passes at most about 30 pair operations of 2^-47 relative
error, and the closure rows of a bounded line amplify by at most 13:
30 * 13 * 2^-47 = 2.8e-12 of the largest entry."""
import numpy as np
import pytest

import stab_inputs as si
from gpu_util import max_rel_err

pytestmark = pytest.mark.gpu
TOL = 2.8e-12


def _profile(g, f):
    q = si.tanh_base_flow(g, f)
    y = g.y()[None, :, None]
    q[0] *= 1.0 + 0.05 * np.tanh(y / 3.0)
    q[2] += 0.03 * np.exp(-y ** 2 / 9.0) - 0.01
    if g.dim == 3:
        q[3] += 0.2 * np.sin(0.4 * y)
    q[-1] += 0.02 * np.tanh(y / 2.0 + 0.3)
    return q


GRIDS = [
    (si.Grid(2, 6, 6, 1, si.LX_04, -15, 15), si.Flow(0.5, 300.0)),
    (si.Grid(2, 9, 7, 1, si.LX_04, -15, 15, 1.0, 1.2), si.Flow(0.5, 300.0)),
    (si.Grid(2, 17, 33, 1, si.LX_04, -15, 15), si.Flow(0.3, 800.0)),
    (si.Grid(2, 24, 41, 1, si.LX_04, -15, 15), si.Flow(0.7, 0.0)),
    (si.Grid(2, 131, 197, 1, si.LX_04, -15, 15, 1.0, 1.7), si.Flow(0.6, 500.0)),
    (si.Grid(3, 6, 9, 7, si.LX_04, -15, 15, si.LX_04), si.Flow(0.4, 500.0)),
    (si.Grid(3, 33, 20, 6, si.LX_04, -15, 15, 5.0, 0.9), si.Flow(0.6, 900.0)),
    (si.Grid(3, 12, 18, 34, si.LX_04, -15, 15, si.LX_04), si.Flow(0.5, 0.0)),
]


@pytest.mark.parametrize("tangent", [True, False])
@pytest.mark.parametrize("g,f", GRIDS, ids=[f"{g.nx}x{g.ny}x{g.nz}" for g, _ in GRIDS])
def test_profile_base_flow_matches_oracle(orc, g, f, tangent):
    import torch
    from paper_1502_03701_gb300 import Stab
    q0 = _profile(g, f)
    v = si.random_complex(900, g.n)
    S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2 if tangent else 0)
    dv = torch.from_numpy(v).cuda()
    out = torch.empty_like(dv)
    S.apply_J(dv, out)
    got, eps = out.cpu().numpy(), S.last_eps()
    ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent" if tangent else "quad", None if tangent else eps)
    assert max_rel_err(got, ref) < TOL
    # every chunk length; lines per CTA change nothing, bit for bit
    for C in (16, 32, 64):
        outs = []
        for L in (1, 3, 16):
            for ax in range(g.dim):
                S.set_line_config(ax, C, L, 3)
            o = torch.empty_like(dv)
            S.apply_J(dv, o)
            outs.append(o)
        assert max_rel_err(outs[0].cpu().numpy(), ref) < TOL, C
        assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2]), C
    S.close()


def test_non_finite_input_stays_non_finite():
    """A NaN or an Inf in v reaches J v (the solvers detect it there)."""
    import torch
    from paper_1502_03701_gb300 import Stab
    g, f = si.mixing_layer_2d(32, 48)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, eps_mode=2)
    for bad in (float("nan"), float("inf")):
        v = torch.from_numpy(si.random_complex(5, g.n)).cuda()
        v[777] = complex(bad, 0.0)
        out = torch.empty_like(v)
        S.apply_J(v, out)
        assert not bool(torch.isfinite(torch.view_as_real(out)).all())
    S.close()
