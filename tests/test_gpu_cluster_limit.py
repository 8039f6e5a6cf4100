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


@pytest.mark.parametrize("blocks", [8, 4])
@pytest.mark.parametrize("mg", ["c128", "c64"])
@pytest.mark.parametrize("sm,galerkin", [(hi.SM_JACOBI, False), (hi.SM_RBGS, False), (hi.SM_JACOBI, True)])
@pytest.mark.parametrize("shape", [(10, 10), (26, 26), (5, 202), (66, 39), (98, 98), (163, 250)])
def test_tail_in_a_smaller_cluster(shape, sm, galerkin, mg, blocks):
    """2D V(1,1) cycles with the tail in 8 blocks (an operator level whose rows fit them) and without a cluster."""
    p = hi.make_problem(2, shape, ((0, 0), (0, 0)), k0=0.3 * (max(shape) - 1), phi_kind="bump", rhs="zero",
                        bump_centre=(0.3, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=sm, galerkin=galerkin)
    r = hi.random_vector(p.n, 31)
    ref = Oracle(p, pc).vcycle(r)
    tol = 1e-10 if mg == "c128" else 5e-5
    for autotune in (True, False):
        h = _limited(blocks, p, pc, mg_dtype=mg, autotune=autotune)
        z = h.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        h.close()
        assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref) and np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("mg", ["c128", "c64"])
def test_group_without_a_cluster_is_refused(mg):
    """Hierarchies whose tail is not the one-cluster one run alone but not as a group; in 8 blocks they do, bitwise."""
    from paper_0912_0180_gb300 import _lib as L
    from paper_0912_0180_gb300.helm import HelmError, solve_group
    p = hi.make_problem(2, 40, 6, k0=12.0, rhs="gauss")
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=hi.SM_RBGS)
    b = torch.from_numpy(p.b).cuda()
    for blocks, others in ((4, 4), (8, 16), (8, 8)):
        hs = [_limited(n, p, pc, mg_dtype=mg, autotune=False) for n in (blocks, others)]
        lone = [h.solve(b, tol=1e-6)[0] for h in hs]
        if (blocks, others) == (8, 8):
            xs, _ = solve_group(hs, [b, b], tol=1e-6)
            assert torch.equal(xs[0], lone[0]) and torch.equal(xs[1], lone[1])
        else:
            with pytest.raises(HelmError) as e:
                solve_group(hs, [b, b], tol=1e-6)
            assert e.value.status == L.HELM_ERR_ARG and "cluster" in str(e.value)
        for h in hs:
            h.close()
