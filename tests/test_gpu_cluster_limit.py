"""Devices that grant smaller thread-block clusters: a test limit stands in for them."""
import ctypes as C

import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu


def _limited(blocks, *args, **kw):
    from paper_0912_0180_gb300 import _lib as L
    from paper_0912_0180_gb300.helm import Helm
    lim = L.load().helm_test_cluster
    lim.argtypes, lim.restype = [C.c_int], None
    lim(blocks)
    try:
        return Helm(*args, **kw)
    finally:
        lim(0)


@pytest.mark.parametrize("blocks", [8, 3, 1])
@pytest.mark.parametrize("shape,mg", [((40, 290), "c64"), ((33, 600), "c128"), ((20, 4200), "c64")])
@pytest.mark.parametrize("galerkin", [False, True])
def test_ilu_strips_in_smaller_clusters(shape, mg, galerkin, blocks):
    """The ILU(0) strips where fewer than 16 blocks a cluster are granted: more warps a block, then several launches."""
    import paper_0912_0180_gb300._lib as L
    p = hi.make_problem(2, (shape[0] + 2, shape[1] + 2), 0, extent=((shape[0] + 1) / 32, (shape[1] + 1) / 32), k0=6.0,
                        phi_kind="bump", rhs="zero", bump_centre=(0.4, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.4, smoother=hi.SM_ILU, galerkin=galerkin, nu1=0, nu2=1, coarse_max=2)
    o = Oracle(p, pc)
    h = _limited(blocks, p, pc, mg_dtype=mg)
    dt = torch.complex128 if mg == "c128" else torch.complex64
    tol = 1e-10 if mg == "c128" else 5e-5
    lvl = 1 if galerkin else 0
    f = hi.random_vector(o.level_size(1, lvl), 6).astype(np.complex64)
    u = torch.zeros(len(f), dtype=dt, device="cuda")
    h.level_op(L.HELM_OP_SMOOTH0, lvl, u, torch.from_numpy(f).cuda().to(dt), None, count=1)
    ref = o.smooth(lvl, np.zeros(len(f), complex), f.astype(complex), 1)
    d = u.cpu().numpy() - ref
    h.close()
    assert np.linalg.norm(d) <= tol * np.linalg.norm(ref) and np.max(np.abs(d)) <= tol * np.max(np.abs(ref))
