"""A sweep whose dependency never completes must end by itself: its CTAs decide together (a producer warp as
a whole, the working warps of a CTA as a whole), so that no warp is left at a barrier, the launch returns with the
error status and the next solve on the same context is right.

Fronts of every class are held back in turn: a warp's, a CTA's and large ones (whose second phase waits for
the front itself), near the leaves, in the middle and next to the root."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fdfd_oracle as O

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


@pytest.mark.parametrize("nx,ny,n_omega,mode,form", [
    (150, 170, 1, FD.MODE_MIXED, FD.FORM_LU),            # every front whole: the warps' and the CTAs' units
    (200, 200, 8, FD.MODE_MIXED, FD.FORM_LU),            # large fronts, two CTAs per SM
    (200, 200, 8, FD.MODE_MIXED, FD.FORM_SYMMETRIC),
    (150, 170, 1, FD.MODE_F64, FD.FORM_LU),              # large fronts of several units
])
def test_a_front_that_never_completes(nx, ny, n_omega, mode, form):
    wl = W.make_small(nx, ny, 8, (nx // 4, ny // 4, nx // 3, ny // 3), n_omega=n_omega, seed=nx)
    s = FD.Solver(nx, ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                  options=FD.default_options(mode=mode, factor_form=form))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    b = W.random_complex((n_omega, 1, wl.n), ny)
    bt = torch.from_numpy(b).cuda()
    s.solve(bt)
    k, m, parent, level, _, _ = s.plan_fronts()
    n = k + m
    root = int(np.argmax(level))
    pick = [int(np.argmin(n)), int(np.flatnonzero((parent == root) & (n > 96))[-1])]
    for lo, hi in [(33, 64), (65, 96), (97, 1 << 20)]:      # the packed classes and the others
        pick.append(int(np.flatnonzero((n >= lo) & (n <= hi) & (parent >= 0))[0]))
    has_child = np.isin(np.arange(len(k)), parent)
    sweeps = (0, 3) if form == FD.FORM_SYMMETRIC else (0, 1, 2, 3)
    for i, f in enumerate(pick):
        for sweep in sweeps[i % 2::2]:
            st = s.selftest_sweep(sweep, f)
            # bottom-up a front's parent waits for it, top-down its children do (a leaf has none)
            assert st == 7 or (st == 0 and sweep in (1, 3) and not has_child[f]), (sweep, f, st)
    assert s.selftest_sweep(4, 0) == 1 and s.selftest_sweep(0, len(k)) == 1
    x = s.solve(bt).cpu().numpy()
    fac = O.Factor(O.assemble(nx, ny, wl.eps_full(), wl.k0dx()[0], wl.npml), (nx, ny))
    assert O.rel_err(x[0, 0], fac.solve(b[0, 0])) <= 1e-7
    s.close()
