"""Panel steps of the large fronts (32 pivots each) at the edges of their tiles: pivot blocks one below,
at and one above multiples of 32, last panels of one column, fronts with little or nothing below the
pivots, levels that take one launch a step and levels of several waves.

A solve on complex128 factors must reach the oracle to 1e-10; a refined solve on complex64 factors must
leave an FP64 residual below its tolerance of 1e-10, checked through fdfd_apply."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fdfd_oracle as O

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


def _solver(wl, mode, **kw):
    s = FD.Solver(wl.nx, wl.ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                  options=FD.default_options(mode=mode, **kw))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    return s


def _workload(nx, ny, n_omega):
    npml = min(8, nx // 4, ny // 4)
    return W.make_small(nx, ny, npml, (nx // 4, ny // 4, max(1, nx // 3), max(1, ny // 3)), n_omega=n_omega, seed=nx)


@pytest.mark.parametrize("nx,ny,n_omega", [(63, 70, 1), (64, 64, 1), (65, 66, 2), (97, 98, 1), (128, 40, 1), (33, 120, 3)])
def test_f64_factors_reach_the_oracle(nx, ny, n_omega):
    wl = _workload(nx, ny, n_omega)
    s = _solver(wl, FD.MODE_F64)
    b = W.random_complex((n_omega, 1, wl.n), ny)
    x = s.solve(torch.from_numpy(b).cuda()).cpu().numpy()
    for w, k0dx in enumerate(wl.k0dx()):
        fac = O.Factor(O.assemble(nx, ny, wl.eps_full(), k0dx, wl.npml), (nx, ny))
        assert O.rel_err(x[w, 0], fac.solve(b[w, 0])) <= 1e-10
    s.close()


@pytest.mark.parametrize("nx,ny,n_omega", [
    (97, 98, 1), (128, 129, 1), (160, 161, 2), (225, 226, 1),   # one launch a step on most levels
    (129, 130, 24), (192, 190, 12),                             # several waves on most levels
])
@pytest.mark.parametrize("transpose", [False, True])
def test_refined_residual(nx, ny, n_omega, transpose):
    wl = _workload(nx, ny, n_omega)
    s = _solver(wl, FD.MODE_MIXED, ir_tol=1e-10)
    b = torch.from_numpy(W.random_complex((n_omega, 1, wl.n), ny)).cuda()
    x = s.solve(b, transpose=transpose)
    r = b - s.apply(x, transpose=transpose)
    rel = torch.linalg.vector_norm(r, dim=2) / torch.linalg.vector_norm(b, dim=2)
    assert rel.max().item() <= 2e-10
    assert s.stats()["fallbacks"] == 0
    s.close()
