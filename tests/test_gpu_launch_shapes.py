"""J v at the sizes where the default launch shapes change, against the oracle:
both components of a pair per thread (large grids, base flows that depend on y
only), and the three ranges of the FP64 passes of general base flows.

Tolerances: pair arithmetic as derived for the pair passes (30 operations of
2^-47, closure rows amplify by 13: 2.8e-12 of the largest entry); FP64 passes
1e-10 element by element, scaled by the largest entry, as for every other J v."""
import pytest

import stab_inputs as si
from gpu_util import max_rel_err

pytestmark = pytest.mark.gpu
CASES = [
    ("packed", si.Grid(3, 64, 72, 48, si.LX_04, -15, 15, si.LX_04), False, 2.8e-12),
    ("fp64_middle", si.Grid(2, 130, 250, 1, si.LX_04, -15, 15), True, 1e-10),
    ("fp64_large", si.Grid(2, 250, 510, 1, si.LX_04, -15, 15), True, 1e-10),
    ("fp64_short_lines", si.Grid(3, 60, 45, 28, si.LX_04, -15, 15, si.LX_04), True, 1e-10),
]


@pytest.mark.parametrize("name,g,general,tol", CASES, ids=[c[0] for c in CASES])
def test_default_shapes_match_oracle(orc, name, g, general, tol):
    import torch
    from paper_1502_03701_gb300 import Stab
    f = si.Flow(0.5, 600.0)
    q0 = si.perturbed_base_flow(g, f, seed=31) if general else si.tanh_base_flow(g, f)
    v = si.random_complex(11, g.n)
    S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    dv = torch.from_numpy(v).cuda()
    out = torch.empty_like(dv)
    S.apply_J(dv, out)
    ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent", None)
    assert max_rel_err(out.cpu().numpy(), ref) < tol
    S.close()


def test_chained_launches_keep_stream_order():
    """J v reads a vector written just before on the same stream, by another
    library's kernel and by the call's own last kernel, and the next writer of
    that vector comes after it: 50 applications in a row equal 50 with a
    synchronisation after each, bit for bit."""
    import torch
    from paper_1502_03701_gb300 import Stab
    g, f = si.mixing_layer_2d(32, 64)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr)
    results = []
    for sync in (False, True):
        v = torch.from_numpy(si.random_complex(2, g.n)).cuda()
        out = torch.empty_like(v)
        for _ in range(50):
            S.apply_J(v, out)
            if sync:
                torch.cuda.synchronize()
            torch.div(out, 100.0, out=v)
            if sync:
                torch.cuda.synchronize()
        results.append(v.clone())
    assert torch.equal(results[0], results[1])
    assert torch.isfinite(torch.view_as_real(results[0])).all()
    S.close()
