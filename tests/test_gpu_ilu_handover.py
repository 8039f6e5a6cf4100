"""The ILU(0) strips' hand-over when it fails: a strip that hands nothing over makes the (shortened) wait
for it run out.  The step then ends with a status that the host reads, and the device stays usable."""
import ctypes as C

import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu


def _context(shape, mg, galerkin, wait=-1, mute=-1):
    from paper_0912_0180_gb300 import _lib as L
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, (shape[0] + 2, shape[1] + 2), 0, extent=((shape[0] + 1) / 32, (shape[1] + 1) / 32), k0=6.0,
                        phi_kind="bump", rhs="zero", bump_centre=(0.4, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.4, smoother=hi.SM_ILU, galerkin=galerkin, nu1=0, nu2=1, coarse_max=2)
    lim = L.load().helm_test_limits
    lim.argtypes, lim.restype = [C.c_longlong, C.c_int], None
    lim(wait, mute)
    try:
        return Helm(p, pc, mg_dtype=mg), Oracle(p, pc)
    finally:
        lim(-1, -1)


# three strips in three blocks; 19 strips, two warps a block; more strips than a cluster holds
@pytest.mark.parametrize("shape,mute,mg,galerkin", [((70, 80), 1, "c64", False), ((40, 600), 7, "c128", False),
                                                    ((40, 600), 8, "c64", True), ((20, 4200), 40, "c64", False)])
def test_missing_handover_ends_with_a_status(shape, mute, mg, galerkin):
    import paper_0912_0180_gb300._lib as L
    from paper_0912_0180_gb300.helm import HelmError
    h, o = _context(shape, mg, galerkin, wait=1 << 20, mute=mute)
    lvl = 1 if galerkin else 0
    dt = torch.complex64 if mg == "c64" else torch.complex128
    f = hi.random_vector(o.level_size(1, lvl), 6).astype(np.complex64)
    b = torch.from_numpy(f).cuda().to(dt)
    u = torch.zeros_like(b)
    h.level_op(L.HELM_OP_SMOOTH0, lvl, u, b, None, count=1)
    torch.cuda.synchronize()
    assert not torch.isfinite(torch.view_as_real(u)).all()
    r = torch.from_numpy(hi.random_vector(h.n, 7)).cuda()
    with pytest.raises(HelmError) as e:  # the earlier call's, reported once
        h.vcycle(r)
    assert e.value.status == L.HELM_ERR_TIMEOUT
    h.vcycle(r)
    torch.cuda.synchronize()
    with pytest.raises(HelmError) as e:
        h.level_op(L.HELM_OP_SMOOTH0, lvl, u, b, None, count=1)
    assert e.value.status == L.HELM_ERR_TIMEOUT
    with pytest.raises(HelmError) as e:
        h.solve(r, maxmv=20)
    assert e.value.status == L.HELM_ERR_TIMEOUT
    if mg == "c128":
        with pytest.raises(HelmError) as e:
            h.mg_iterate(r, 2)
        assert e.value.status == L.HELM_ERR_TIMEOUT
    h.close()
    # the device is usable: the same step on a context without the limits
    h, o = _context(shape, mg, galerkin)
    u = torch.zeros_like(b)
    h.level_op(L.HELM_OP_SMOOTH0, lvl, u, b, None, count=1)
    ref = o.smooth(lvl, np.zeros(len(f), complex), f.astype(complex), 1)
    assert np.linalg.norm(u.cpu().numpy() - ref) <= (1e-10 if mg == "c128" else 5e-5) * np.linalg.norm(ref)
    h.vcycle(r)
    h.close()
