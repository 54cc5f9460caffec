"""Dataflow sweeps at the edges of their units: fronts of every class (a warp's, a CTA's, cut into rows
or columns with one or several parts), odd sizes, right-hand sides in pairs, odd counts and more than one
launch takes, both CTA shapes.

A solve on complex128 factors is one sweep pair, so it must reach the oracle to 1e-10; a refined solve
on complex64 factors must leave an FP64 residual below its tolerance of 1e-10, checked through
fdfd_apply (whose stencil the parity tests pin)."""
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


@pytest.mark.parametrize("nx,ny,n_omega,nrhs,leaf", [
    (53, 47, 2, 1, 96),      # packed leaves of up to 96 unknowns
    (53, 47, 1, 9, 32),      # more right-hand sides than one launch takes, an odd one in each chunk
    (97, 131, 2, 3, 5),      # tiny leaves, an odd count
    (31, 400, 1, 2, 64),     # a long grid
    (3, 5, 1, 2, 32),        # one front
    (200, 200, 8, 1, 32),    # the shape of large problems (320 thousand unknowns), single right-hand sides
    (331, 251, 4, 3, 64),    # ... pairs, large fronts in several parts
    (380, 360, 1, 2, 32),    # the shape of small problems, fronts above 700 unknowns
])
@pytest.mark.parametrize("form", [FD.FORM_LU, FD.FORM_SYMMETRIC])
@pytest.mark.parametrize("transpose", [False, True])
def test_refined_residual(nx, ny, n_omega, nrhs, leaf, form, transpose):
    npml = min(8, nx // 4, ny // 4)
    wl = W.make_small(nx, ny, npml, (nx // 4, ny // 4, max(1, nx // 3), max(1, ny // 3)), n_omega=n_omega, seed=nx)
    s = _solver(wl, FD.MODE_MIXED, leaf_area=leaf, factor_form=form, ir_tol=1e-10)
    b = torch.from_numpy(W.random_complex((n_omega, nrhs, wl.n), ny)).cuda()
    x = s.solve(b, transpose=transpose)
    r = b - s.apply(x, transpose=transpose)
    rel = torch.linalg.vector_norm(r, dim=2) / torch.linalg.vector_norm(b, dim=2)
    assert rel.max().item() <= 2e-10
    s.close()


@pytest.mark.parametrize("nx,ny,n_omega,nrhs,leaf", [(53, 47, 2, 9, 96), (97, 131, 1, 3, 5), (3, 5, 1, 2, 32)])
@pytest.mark.parametrize("transpose", [False, True])
def test_f64_factors_reach_the_oracle(nx, ny, n_omega, nrhs, leaf, transpose):
    npml = min(8, nx // 4, ny // 4)
    wl = W.make_small(nx, ny, npml, (nx // 4, ny // 4, max(1, nx // 3), max(1, ny // 3)), n_omega=n_omega, seed=nx)
    s = _solver(wl, FD.MODE_F64, leaf_area=leaf)
    b = W.random_complex((n_omega, nrhs, wl.n), ny)
    x = s.solve(torch.from_numpy(b).cuda(), transpose=transpose).cpu().numpy()
    for w, k0dx in enumerate(wl.k0dx()):
        fac = O.Factor(O.assemble(nx, ny, wl.eps_full(), k0dx, npml), (nx, ny))
        for r in range(nrhs):
            ref = (fac.solve_T if transpose else fac.solve)(b[w, r])
            assert O.rel_err(x[w, r], ref) <= 1e-10
    s.close()
