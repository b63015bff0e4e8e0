"""The tuner's cache keeps the shapes of the pair passes (base flows that depend
on y only) and of the FP64 passes (general ones) apart, on the same grid, in the
process and in its file; a line written before the kinds were told apart is an
entry of the FP64 passes.  Both kinds' J v stay within the oracle's bounds of the
other tests (2.8e-12 and 1e-10 of the largest entry) with any loaded shape."""
import pytest

import stab_inputs as si
from gpu_util import max_rel_err

pytestmark = pytest.mark.gpu


def _pair(g, f):
    return si.tanh_base_flow(g, f), si.perturbed_base_flow(g, f, seed=5)


def _lines(path, n, nlines):
    rows = [[int(x) for x in r.split()] for r in open(path).read().splitlines()]
    return [r for r in rows if r[0] == n and r[1] == nlines]


@pytest.mark.parametrize("first", ["layer", "general"])
def test_one_kind_does_not_take_the_other_kinds_shape(first, tmp_path):
    from paper_1502_03701_gb300 import Stab, binding
    g, f = (si.Grid(2, 36, 51, 1, si.LX_04, -15, 15), si.Flow(0.4, 600.0)) if first == "layer" else \
        (si.Grid(2, 38, 53, 1, si.LX_04, -15, 15), si.Flow(0.4, 600.0))
    layer, general = _pair(g, f)
    a, b = (layer, general) if first == "layer" else (general, layer)
    A = Stab(a, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    A.autotune(force=True)
    B = Stab(b, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    again = B.autotune(force=False)
    assert all(ms > 0 for _, _, _, ms in again.values())  # timed, not taken from the other kind's entry
    C = Stab(a, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    assert all(r[3] == -1.0 for r in C.autotune(force=False).values())
    path = str(tmp_path / "cache")
    binding.autotune_save(path)
    assert sorted(r[8:] for r in _lines(path, g.ny, g.nx)) == [[], [1]]
    for s in (A, B, C):
        s.close()


def test_file_of_the_older_format(orc, tmp_path):
    import torch
    from paper_1502_03701_gb300 import Stab, binding
    g, f = si.Grid(2, 34, 57, 1, si.LX_04, -15, 15), si.Flow(0.4, 600.0)
    path = str(tmp_path / "old")
    open(path, "w").write("57 34 5 0 64 2 1\n34 57 7 1 32 3 2 0\n")
    assert binding.autotune_load(path) == 2
    P = orc.Problem.from_inputs(g, f)
    v = si.random_complex(8, g.n)
    for q0, tol, taken in zip(_pair(g, f), (2.8e-12, 1e-10), (False, True)):
        S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2)
        out = torch.empty(g.n, dtype=torch.complex128, device="cuda")
        S.apply_J(torch.from_numpy(v).cuda(), out)
        assert max_rel_err(out.cpu().numpy(), orc.core.jv(P, q0, v, "tangent")) < tol
        got = S.autotune(force=False)
        assert (got["y"] == (64, 2, 1, -1.0)) == taken and (got["x"] == (32, 3, 2, -1.0)) == taken
        S.close()


@pytest.mark.parametrize("C,L", [(1, 1), (2, 7), (3, 100000), (7, 3), (1000, 2000000000)])
def test_loaded_shapes_outside_the_tuned_ones(orc, C, L, tmp_path):
    """Any positive C and L in the file: the pair passes keep chunks of four points or more."""
    import torch
    from paper_1502_03701_gb300 import Stab, binding
    g, f = si.Grid(2, 9 + C % 5, 22 + 2 * (C % 7), 1, si.LX_04, -15, 15), si.Flow(0.4, 600.0)
    path = str(tmp_path / "odd")
    open(path, "w").write(f"{g.ny} {g.nx} 5 0 {C} {L} 3 0 1\n{g.nx} {g.ny} 7 1 {C} {L} 3 0 1\n")
    assert binding.autotune_load(path) == 2
    q0 = si.tanh_base_flow(g, f)
    S = Stab(q0, g, f.Ma, f.Re, f.Pr, eps_mode=2)
    v = si.random_complex(9, g.n)
    out = torch.empty(g.n, dtype=torch.complex128, device="cuda")
    S.apply_J(torch.from_numpy(v).cuda(), out)
    ref = orc.core.jv(orc.Problem.from_inputs(g, f), q0, v, "tangent")
    assert max_rel_err(out.cpu().numpy(), ref) < 2.8e-12
    S.close()
