"""The sweeps themselves, not what refinement makes of them.

Raw solves (no refinement) against a refined one whose FP64 residual is checked through fdfd_apply: at these
sizes complex64 factors give 1e-5 to 1e-3 (the bound is 5e-3), complex128 factors 1e-13 (1e-10), and a
unit, a part or a source left out gives an error of order one.  The unit counts are asserted, so that the sizes go on
covering what they are listed for."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


def _solver(nx, ny, n_omega, **kw):
    npml = min(8, nx // 4, ny // 4)
    wl = W.make_small(nx, ny, npml, (nx // 4, ny // 4, max(1, nx // 3), max(1, ny // 3)), n_omega=n_omega, seed=nx)
    s = FD.Solver(nx, ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box, options=FD.default_options(**kw))
    s.factor(torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda())
    return wl, s


def _rel(x, ref):
    return (torch.linalg.vector_norm(x - ref, dim=2) / torch.linalg.vector_norm(ref, dim=2)).max().item()


def _reference(s, b, transpose):
    """A refined solve on the same factors, to a residual of 1e-12."""
    s.set_options(ir_tol=1e-12, ir_max_iter=40)
    x = s.solve(b, transpose=transpose)
    assert _rel(s.apply(x, transpose=transpose), b) <= 2e-12 and s.stats()["fallbacks"] == 0
    s.set_options(ir_max_iter=0)
    return x


@pytest.mark.parametrize("nx,ny,n_omega,nrhs,tri,rect", [
    (700, 701, 1, 2, {0, 1, 2, 3}, {0, 1, 2, 3}),     # two CTAs per SM, both kinds of units in parts in every sweep
    (540, 540, 8, 1, {0, 2, 3}, {0, 1, 2, 3}),
    (380, 360, 1, 3, set(), {3}),                      # one CTA per SM
    (97, 131, 2, 5, set(), set()),                     # the root one whole front without boundary rows
])
@pytest.mark.parametrize("transpose", [False, True])
def test_raw_complex64_solves(nx, ny, n_omega, nrhs, tri, rect, transpose):
    wl, s = _solver(nx, ny, n_omega)
    units = [s.sweep_units(q) for q in range(4)]
    assert {q for q in range(4) if units[q]["tri_parts"]} >= tri
    assert {q for q in range(4) if units[q]["rect_parts"]} >= rect
    b = torch.from_numpy(W.random_complex((n_omega, nrhs, wl.n), ny)).cuda()
    ref = _reference(s, b, transpose)
    assert _rel(s.solve(b, transpose=transpose), ref) <= 5e-3
    s.close()


@pytest.mark.parametrize("nx,ny,n_omega,nrhs,tri,rect", [
    (540, 540, 1, 1, {0, 2, 3}, {0, 1, 2, 3}),
    (200, 200, 1, 3, set(), {3}),
])
@pytest.mark.parametrize("transpose", [False, True])
def test_complex128_solves(nx, ny, n_omega, nrhs, tri, rect, transpose):
    wl, s = _solver(nx, ny, n_omega, mode=FD.MODE_F64)
    units = [s.sweep_units(q, f64=True) for q in range(4)]
    assert {q for q in range(4) if units[q]["tri_parts"]} >= tri
    assert {q for q in range(4) if units[q]["rect_parts"]} >= rect
    b = torch.from_numpy(W.random_complex((n_omega, nrhs, wl.n), ny)).cuda()
    x = s.solve(b, transpose=transpose)
    assert _rel(s.apply(x, transpose=transpose), b) <= 1e-10
    s.close()


@pytest.mark.parametrize("nx,ny,n_omega", [(97, 131, 2), (331, 251, 1), (331, 251, 4)])
@pytest.mark.parametrize("transpose", [False, True])
def test_a_source_does_not_depend_on_its_neighbours(nx, ny, n_omega, transpose):
    """The first sources of 11 (two launches: four pairs, one pair and a single) in calls of one, two, three and eight."""
    wl, s = _solver(nx, ny, n_omega, ir_max_iter=0)
    b = torch.from_numpy(W.random_complex((n_omega, 11, wl.n), ny)).cuda()
    full = s.solve(b, transpose=transpose)
    for n in (1, 2, 3, 8):
        x = s.solve(b[:, 11 - n:].contiguous(), transpose=transpose)
        assert _rel(x, full[:, 11 - n:]) <= 1e-3
    s.close()


@pytest.mark.parametrize("nx,ny,n_omega,nrhs,leaf", [
    (53, 47, 2, 1, 96), (53, 47, 1, 9, 32), (97, 131, 2, 3, 5), (31, 400, 1, 2, 64), (3, 5, 1, 2, 32),
    (200, 200, 8, 1, 32), (331, 251, 4, 3, 64), (380, 360, 1, 2, 32)])
@pytest.mark.parametrize("form,most", [(FD.FORM_LU, 5), (FD.FORM_SYMMETRIC, 9)])
@pytest.mark.parametrize("transpose", [False, True])
def test_refinement_stays_short(nx, ny, n_omega, nrhs, leaf, form, most, transpose):
    """Every class of front at the edges of its units: a damaged sweep would still converge on FP64 factors, or in
    many more vectors (sound ones take 2 to 4 in the LU form, some more where the symmetric form's factors grow)."""
    wl, s = _solver(nx, ny, n_omega, leaf_area=leaf, factor_form=form, ir_tol=1e-10)
    b = torch.from_numpy(W.random_complex((n_omega, nrhs, wl.n), ny)).cuda()
    for scale in (1.0, 1e-3):            # other sources on the same context, then the first again
        x = s.solve(scale * b.flip(1), transpose=transpose)
        x = s.solve(b, transpose=transpose)
        assert _rel(s.apply(x, transpose=transpose), b) <= 2e-10
        st = s.stats()
        assert st["fallbacks"] == 0 and st["repivots"] == 0 and st["ir_iters"] <= most
    s.close()
