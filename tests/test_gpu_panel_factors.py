"""The complex64 panel steps' factors themselves, front by front: the complex128 factorisation of the same problem
pivots in another order, so what is compared is free of the order of the pivots.  With P F11 = L11 U11 and the
stored X_L = L11^-1, X_U = U11^-1:
  S = F22 - F21 F11^-1 F12;  X_U U12 = F11^-1 F12;  G G^H with G = L21 X_L (F21 F11^-1 up to the order of its
  columns);  H H^H with H = X_U X_L (F11^-1 likewise).
complex64 rounding through the levels below gives 1e-6 to 1e-4 while a front's pivot block is well conditioned (in
FP64: singular values of F11^-1 within 1e4; the others, two of all fronts here, are left out: what is compared moves
by the condition number times the rounding, whatever the kernels do); a panel, a tile or an
update left out gives an error of order one.  The bound is 5e-3."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402


def _pieces(s, f, w, k, m, f64):
    F, X = s.front_data(f, w, f64=f64)
    X = X[:, :k].astype(np.complex128)
    XL, XU = np.tril(X, -1) + np.eye(k), np.triu(X)
    H = XU @ XL
    out = {"H": H @ H.conj().T}
    if m:
        F = F.astype(np.complex128)
        G = F[k:k + m, :k] @ XL
        out.update(S=F[k:k + m, k:k + m], W=XU @ F[:k, k:k + m], G=G @ G.conj().T)
    return out


@pytest.mark.parametrize("nx,ny,n_omega", [
    (97, 98, 1), (128, 129, 1), (160, 161, 2), (225, 226, 1),   # one launch a step on most levels
    (129, 130, 24), (192, 190, 12),                             # several waves on most levels
])
def test_factors_of_the_large_fronts(nx, ny, n_omega):
    wl = W.make_small(nx, ny, 8, (nx // 4, ny // 4, nx // 3, ny // 3), n_omega=n_omega, seed=nx)
    eps = torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda()
    s = {}
    for mode in (FD.MODE_MIXED, FD.MODE_F64):
        s[mode] = FD.Solver(nx, ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                            options=FD.default_options(mode=mode))
        s[mode].factor(eps)
    k, m, *_ = s[FD.MODE_MIXED].plan_fronts()
    n = k + m
    fronts = set(np.argsort(n)[-8:].tolist())
    fronts |= set(np.flatnonzero(n > 96)[:4].tolist())           # the smallest of the panel steps' fronts ...
    fronts |= set(np.flatnonzero((n > 96) & (k % 32 == 1))[:2].tolist())   # ... and last panels of one column
    checked = 0
    for f in sorted(fronts):
        for w in {0, n_omega - 1}:
            b = _pieces(s[FD.MODE_F64], f, w, k[f], m[f], True)
            ev = np.linalg.eigvalsh(b["H"])
            if ev[0] <= 1e-8 * ev[-1]:
                continue
            checked += 1
            a = _pieces(s[FD.MODE_MIXED], f, w, k[f], m[f], False)
            for key in b:
                err = np.linalg.norm(a[key] - b[key]) / np.linalg.norm(b[key])
                assert err <= 5e-3, (f, w, key, k[f], m[f], err)
    assert checked >= 10
    for v in s.values():
        v.close()
