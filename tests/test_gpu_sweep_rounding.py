"""Rounding of the sweeps where factors have grown: the symmetric form takes no pivots, and on these grids its
multipliers reach 2e4 and 1.2e5.  What the L^T sweep rounds in a front with a small pivot is the noise that
FGMRES has to remove: with neighbouring rows one after the other in a sum a solve needs 9 vectors, with the rows
dealt out in turn it needed 12 to 14.  The bound is one more than the 9."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


@pytest.mark.parametrize("n_omega", [1, 4])
@pytest.mark.parametrize("restart", [8, 16])
@pytest.mark.parametrize("transpose", [False, True])
def test_krylov_vectors_on_grown_symmetric_factors(n_omega, restart, transpose):
    wl = W.make_small(540, 540, 8, (135, 135, 180, 180), n_omega=n_omega, seed=540)
    s = FD.Solver(540, 540, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                  options=FD.default_options(factor_form=FD.FORM_SYMMETRIC, gmres_restart=restart))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    b = torch.from_numpy(W.random_complex((n_omega, 1, wl.n), 540)).cuda()
    for _ in range(3):
        x = s.solve(b, transpose=transpose)
        st = s.stats()
        assert st["factor_form"] == FD.FORM_SYMMETRIC and st["growth"] > 1e4 and st["fallbacks"] == 0
        assert st["ir_iters"] <= 10
        r = b - s.apply(x, transpose=transpose)
        assert (torch.linalg.vector_norm(r, dim=2) / torch.linalg.vector_norm(b, dim=2)).max().item() <= 2e-9
    s.close()
