"""Figures that the library reports about itself, against counts made from the plan."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


def _solver(n_omega=2, **kw):
    wl = W.make_small(120, 110, 8, (30, 28, 40, 36), n_omega=n_omega, seed=3)
    s = FD.Solver(wl.nx, wl.ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                  options=FD.default_options(**kw))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    return wl, s


@pytest.mark.parametrize("mode,es", [(FD.MODE_MIXED, 8), (FD.MODE_F64, 16)])
@pytest.mark.parametrize("nrhs", [1, 2, 5, 11])
@pytest.mark.parametrize("transpose", [False, True])
def test_sweep_bytes_count_a_factor_entry_once_a_launch(mode, es, nrhs, transpose):
    """Eight right-hand sides at most share a launch's staged factors, so the factor's part of the bytes grows
    with the launches and the vectors' part with the right-hand sides; flops grow with the right-hand sides."""
    wl, s = _solver(mode=mode, ir_max_iter=0)
    k, m, *_ = (v.astype(float) for v in s.plan_fronts())
    low, up, rect = (k * (k - 1) / 2).sum(), (k * (k + 1) / 2).sum(), (k * m).sum()
    vec = (np.ceil((k + m) / 4) * 4).sum()
    b = torch.from_numpy(W.random_complex((2, nrhs, wl.n), 4)).cuda()
    s.solve(b, transpose=transpose)
    s.profile(True)
    s.solve(b, transpose=transpose)
    p = s.profile_get()
    s.close()
    groups = -(-nrhs // 8)
    for name, ent in (("sweep_Ut", up), ("sweep_Lt", low)) if transpose else (("sweep_L", low), ("sweep_U", up)):
        assert p[name]["launches"] == groups
        assert p[name]["bytes"] == es * 2 * ((ent + rect) * groups + vec * nrhs)
        assert p[name]["flops"] == 8 * 2 * (ent + rect) * nrhs


@pytest.mark.parametrize("mode,es", [(FD.MODE_MIXED, 8), (FD.MODE_F64, 16)])
def test_store_bytes_cover_the_factors(mode, es):
    """At least L21, U12 and the update matrix of every front, wherever they are kept."""
    _, s = _solver(n_omega=3, mode=mode)
    k, m, *_ = (v.astype(float) for v in s.plan_fronts())
    assert s.stats()["store_bytes"] >= es * 3 * (2 * k * m + m * m).sum()
    s.close()


@pytest.mark.parametrize("nrhs", [1, 3])
def test_fgmres_flops_count_what_a_cell_takes(nrhs):
    """Per cell: the operator between the absorbing layers, the difference and the norm 18, each projection or
    update 8 a vector, the norm after it 4."""
    wl, s = _solver()
    b = torch.from_numpy(W.random_complex((2, nrhs, wl.n), 4)).cuda()
    s.solve(b)
    s.profile(True)
    s.solve(b)
    p, its = s.profile_get(), s.stats()["ir_iters"]
    s.close()
    assert p["stencil_f64"]["launches"] == 1 and p["gmres_arnoldi"]["launches"] == 2 * its      # one cycle
    cells = 2 * nrhs * wl.n
    assert p["stencil_f64"]["flops"] == 18 * cells
    assert p["gmres_arnoldi"]["flops"] == sum(18 + 8 * j + 8 * j + 4 for j in range(1, its + 1)) * cells
