"""GMRES cycles that end inside the cycle, at sizes whose Givens step and scaling
share a launch of two to many blocks (k_gm_step_scale): the cycle's last basis
vector is not read again, so the same solve gives the same bits every time, and
the solution has the residual that GMRES reports.  Also the cycle that ends at
its first step (b an eigenvector up to rounding: a shift far above the spectrum)
and solves of one column each.

Tolerance: GMRES stops at a relative residual of 1e-10 by its own estimate; the
true residual adds rounding of J x, below 1e-11 of ||b|| here: 2e-10."""
import pytest

import stab_inputs as si

pytestmark = pytest.mark.gpu
# unknowns: one more than a cluster takes (2,048), clusters, column-split passes, and row passes
SIZES = [(16, 33), (40, 50), (64, 64), (66, 65), (128, 130)]


@pytest.mark.parametrize("m", [1, 40])
@pytest.mark.parametrize("nx,ny", SIZES, ids=[f"{4 * a * b}" for a, b in SIZES])
def test_cycle_that_ends_early_is_repeatable(nx, ny, m):
    import torch
    from paper_1502_03701_gb300 import Stab
    g, f = si.mixing_layer_2d(nx, ny)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr, eps_mode=2, gmres_m=m, gmres_tol=1e-10)
    b = torch.from_numpy(si.random_complex(nx, g.n)).cuda()
    for sigma in (2.0e4, 3.0e13):  # several steps; one step
        first, its = None, None
        for _ in range(10):
            x = torch.full_like(b, float("nan"))
            st, iters = S.solve(sigma, b, x)
            assert st == 0
            if first is None:
                first, its = x.clone(), iters
            assert torch.equal(x, first) and iters == its
        r = torch.empty_like(b)
        S.apply_J(first, r, sigma)
        assert float(torch.linalg.vector_norm(r - b)) < 2e-10 * float(torch.linalg.vector_norm(b))
        assert its == 1 if sigma > 1e12 else its > 1
    S.close()
