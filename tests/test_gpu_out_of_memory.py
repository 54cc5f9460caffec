"""Device memory that runs out inside fdfd_factor: the call reports it, a solve on the context is refused (there
is no factorisation to sweep), and once there is memory again the next fdfd_factor allocates what the failed one
left out.  The rest of the memory is taken by one buffer that nothing touches; what is left is swept over the
context's needs, so that the failure falls on the plan, the factors, the inverses and the packed store in turn."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2307_05388_gb300 import fdfd as FD  # noqa: E402

OOM, STATE = 3, 2


def _solver(wl, mode):
    return FD.Solver(wl.nx, wl.ny, wl.dx, 2 * np.pi / wl.wavelengths, wl.npml, box=wl.box,
                     options=FD.default_options(mode=mode))


@pytest.mark.parametrize("mode", [FD.MODE_MIXED, FD.MODE_F64])
def test_factor_after_running_out_of_memory(mode):
    wl = W.make_small(340, 330, 8, (85, 82, 113, 110), n_omega=3, seed=1)
    eps = torch.from_numpy(wl.eps_full().reshape(-1).copy()).cuda()
    b = torch.from_numpy(W.random_complex((3, 1, wl.n), 2)).cuda()
    # kernels loaded, and what a context takes
    s = _solver(wl, mode)
    s.factor(eps)
    s.solve(b)
    s.apply(b)
    s.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    s = _solver(wl, mode)
    s.factor(eps)
    torch.cuda.synchronize()
    need = before - torch.cuda.mem_get_info()[0]
    s.close()
    failed = 0
    for share in (0.02, 0.1, 0.3, 0.5, 0.6, 0.7, 0.8, 0.9, 0.97):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        spare = torch.cuda.mem_get_info()[0] - int(share * need)
        rest = torch.empty(spare, dtype=torch.uint8, device="cuda")
        s = _solver(wl, mode)
        out = torch.empty_like(b)
        try:
            s.factor(eps)
        except FD.FdfdError as e:
            assert e.status == OOM, e
            failed += 1
            with pytest.raises(FD.FdfdError) as err:
                s.solve(b, out=out)
            assert err.value.status == STATE
        del rest
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        s.factor(eps)
        x = s.solve(b, out=out)
        r = b - s.apply(x)
        assert (torch.linalg.vector_norm(r, dim=2) / torch.linalg.vector_norm(b, dim=2)).max().item() <= 2e-9
        assert s.stats()["fallbacks"] == 0
        s.close()
    assert failed >= 6
