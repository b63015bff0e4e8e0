"""The FP64 line passes (general base flows) at every admissible launch shape, with
FP64 and pair right-hand sides, against the oracle, and the tuner on them.  Base
flows that depend on y only take the pair passes, which ignore ``kinds``.

Tolerance: 1e-10 of the largest entry, as for every other J v of these passes."""
import pytest

import stab_inputs as si
from gpu_util import max_rel_err, rel_err

pytestmark = pytest.mark.gpu
TOL = 1e-10

CASES = [
    ("ragged2d_stretched", si.Grid(2, 70, 67, 1, si.LX_04, -15, 15, 1.0, 1.7), si.Flow(0.6, 500.0)),
    ("small3d", si.Grid(3, 12, 16, 8, si.LX_04, -15, 15, si.LX_04), si.Flow(0.5, 800.0)),
    ("ragged_y33", si.Grid(2, 20, 33, 1, si.LX_04, -15, 15), si.Flow(0.4, 700.0)),
    ("inviscid", si.Grid(2, 130, 49, 1, si.LX_04, -15, 15), si.Flow(0.5, 0.0)),
]


@pytest.mark.parametrize("stencil_prec", [64, 48])
@pytest.mark.parametrize("name,g,f", CASES, ids=[c[0] for c in CASES])
def test_every_line_shape_of_a_general_flow(orc, name, g, f, stencil_prec):
    import torch
    from paper_1502_03701_gb300 import Stab, StabError
    q0 = si.perturbed_base_flow(g, f, seed=17)
    v = si.random_complex(311, g.n)
    ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent")
    S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2, stencil_prec=stencil_prec)
    dv = torch.from_numpy(v).cuda()
    out = torch.empty_like(dv)
    tried = set()
    for kinds in (1, 2, 3):
        for C in (16, 32, 64):
            for L in (1, 3, 8, 32):
                try:
                    for ax in range(g.dim):
                        S.set_line_config(ax, C, L, kinds)
                except StabError:
                    continue
                S.apply_J(dv, out)
                got = out.cpu().numpy()
                assert max_rel_err(got, ref) < TOL, (C, L, kinds)
                assert rel_err(got, ref) < TOL, (C, L, kinds)
                tried.add((kinds, C))
    assert len(tried) == 9
    S.close()


def test_tuner_on_a_general_flow(orc):
    import torch
    from paper_1502_03701_gb300 import Stab
    g, f = CASES[0][1], CASES[0][2]
    q0 = si.perturbed_base_flow(g, f, seed=18)
    v = si.random_complex(312, g.n)
    dv = torch.from_numpy(v).cuda()
    S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    res = S.autotune(force=True)
    for C, L, kinds, ms in res.values():
        assert C in (16, 32, 64) and 1 <= L <= 32 and kinds in (1, 2, 3) and ms > 0
    out, again = torch.empty_like(dv), torch.empty_like(dv)
    S.apply_J(dv, out)
    ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent")
    assert max_rel_err(out.cpu().numpy(), ref) < TOL
    T = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2)  # takes the cached shape at creation
    T.apply_J(dv, again)
    assert torch.equal(out, again)
    S.close()
    T.close()
