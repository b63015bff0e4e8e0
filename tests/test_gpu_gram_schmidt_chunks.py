"""CGS2 with one row per thread where a block takes several chunks of 512 rows
(above 152 * 512 = 77,824 unknowns), a ragged last chunk, and the column counts at
which the warps' shares of a chunk change, against FP64 sums.

Tolerance: operands are split to 2^-49 and products and sums are pairs of about
2^-46 relative error.  The first pass's coefficients are corrected by the second,
so the vector and the coefficients are off by the update's rounding, at most k
terms of ||w|| |V_ij| <= ||w|| per row in the Euclidean norm: k 2^-46 < 2.5e-13
||w|| for k <= 17, and 1e-12 for the column sums, as in the smaller sizes."""
import numpy as np
import pytest

import stab_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(140, 139), (256, 256), (211, 331), (512, 512)],
                         ids=["one_chunk_and_a_bit", "262144", "279364", "1048576"])
def test_several_chunks_per_block(nx, ny):
    import torch
    from paper_1502_03701_gb300 import Stab
    g, f = si.mixing_layer_2d(nx, ny)
    S = Stab(si.tanh_base_flow(g, f), g, f.Ma, f.Re, f.Pr)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(nx)
    kmax = 17
    a = torch.view_as_complex(torch.randn(g.n, kmax, 2, dtype=torch.float64, device="cuda", generator=gen))
    for _ in range(2):  # Cholesky QR twice: orthonormal to working precision
        low = torch.linalg.cholesky(a.mH @ a)
        a = torch.linalg.solve_triangular(low.mH, a, upper=True, left=False)
    Q = a.T.contiguous()
    w = torch.from_numpy(si.random_complex(ny, g.n)).cuda()
    wn = float(torch.linalg.vector_norm(w))
    for k in (1, 4, 5, 8, 9, 16, 17):
        V = Q[:k]
        span = V.T @ torch.from_numpy(si.random_complex(k, k)).cuda() * wn + 1e-6 * w
        for x in (w, span):
            href, wref = torch.zeros(k, dtype=torch.complex128, device="cuda"), x.clone()
            for _ in range(2):
                t = V.conj() @ wref
                wref = wref - V.T @ t
                href = href + t
            got = x.clone()
            h, nrm = S.orthogonalize(V, k, got)
            size = float(torch.linalg.vector_norm(x))
            assert np.abs(h - href.cpu().numpy()).max() < 1e-12 * size, k
            assert float(torch.linalg.vector_norm(got - wref)) < 1e-12 * size, k
            assert abs(nrm - float(torch.linalg.vector_norm(got))) < 1e-12 * size, k
            assert float((V.conj() @ got).abs().max()) < 1e-12 * size, k
    S.close()
