"""FGMRES passes: the operator's short form between the absorbing layers, and the second projection."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fdfd_oracle as O

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


@pytest.mark.parametrize("nx,ny,npml", [(40, 33, (7, 5)), (40, 33, (0, 6)), (33, 40, (8, 0)), (12, 12, (6, 6)),
                                        (3, 40, (0, 0)), (1, 9, (0, 3)), (30, 21, (1, 10))])
@pytest.mark.parametrize("transpose", [False, True])
def test_apply_matches_the_assembled_operator(nx, ny, npml, transpose):
    """Every row against the oracle's matrix: 2^-52 times a few operations per entry."""
    rng = np.random.default_rng(nx)
    eps = rng.uniform(1.0, 12.0, nx * ny)
    k0dx = np.array([0.16, 0.21])
    s = FD.Solver(nx, ny, 0.05, k0dx / 0.05, npml)
    s.factor(torch.from_numpy(eps).cuda())
    x = W.random_complex((2, 2, nx * ny), 3)
    y = s.apply(torch.from_numpy(x).cuda(), transpose=transpose).cpu().numpy()
    for w in range(2):
        A = O.assemble(nx, ny, eps.reshape(nx, ny), s.k0[w] * 0.05, npml)
        A = A.T if transpose else A
        scale = abs(A) @ np.ones(nx * ny)
        for r in range(2):
            assert np.max(np.abs(y[w, r] - A @ x[w, r]) / scale) <= 2e-15 * np.max(np.abs(x))
    s.close()


@pytest.mark.parametrize("transpose", [False, True])
def test_repeated_solves_on_a_weak_preconditioner(transpose):
    """C2 with TF32 update matrices in every front takes cycles of nine or more Krylov vectors: the
    orthogonality watch and, in the solves after the first, the second projection must leave the
    FP64 residual at the tolerance and need no complex128 factors."""
    wl = W.make("c2")
    s = FD.Solver(wl.nx, wl.ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                  options=FD.default_options(tensor_form=1, tensor_min_m=1, tensor_min_tiles=1, gmres_restart=16,
                                             ir_tol=1e-13))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    b = torch.from_numpy(W.random_complex((1, 3, wl.n), 8)).cuda()
    for _ in range(3):
        x = s.solve(b, transpose=transpose)
        r = b - s.apply(x, transpose=transpose)
        rel = torch.linalg.vector_norm(r, dim=2) / torch.linalg.vector_norm(b, dim=2)
        assert rel.max().item() <= 2e-13
        assert s.stats()["ir_iters"] <= 24
    assert s.stats()["fallbacks"] == 0
    s.close()
