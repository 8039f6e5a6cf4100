"""Coarsest levels between the operator limit of the one-cluster tail and the largest one that a tail ends in."""
import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu


def _instance(shape, mg, sm, **kw):
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, [n + 2 for n in shape], 0, k0=0.3 * (max(shape) + 1), phi_kind="bump", rhs="gauss",
                        bump_centre=(0.4, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.4, smoother=sm, **kw)
    return p, pc, Helm(p, pc, mg_dtype=mg)


@pytest.mark.parametrize("sm", [hi.SM_JACOBI, hi.SM_RBGS])
@pytest.mark.parametrize("mg", ["c128", "c64"])
def test_group_takes_single_levels(mg, sm):
    """A hierarchy of one level, solved directly, joins a group up to 256 unknowns (FP64): the whole cycle is the tail;
    bitwise the lone solve's iterates (which a direct solve of M need not bring to the tolerance in 50 matvecs)."""
    from paper_0912_0180_gb300.helm import solve_group
    inst = [_instance(s, mg, sm, max_levels=1) for s in ((13, 12), (16, 16), (7, 9), (51, 5))]
    hs = [h for _, _, h in inst]
    bs = [torch.from_numpy(p.b).cuda() for p, _, _ in inst]
    lone = [h.solve(b, tol=1e-8, maxmv=50) for h, b in zip(hs, bs)]
    xs, infos = solve_group(hs, bs, tol=1e-8, maxmv=50)
    for (x, i), xg, ig in zip(lone, xs, infos):
        assert (i.status, i.matvecs) == (ig.status, ig.matvecs) and torch.equal(x, xg)
    for h in hs:
        h.close()


@pytest.mark.parametrize("sm", [hi.SM_JACOBI, hi.SM_RBGS])
@pytest.mark.parametrize("mg", ["c128", "c64"])
@pytest.mark.parametrize("shape,coarse", [((31, 31), 15), ((33, 32), 16), ((30, 27), 15), ((62, 65), 16), ((85, 7), 128),
                                          ((86, 3), 128), ((20, 13), 20)])
def test_cycle_ends_in_a_large_coarsest_level(shape, coarse, mg, sm):
    """Coarsest levels of 151 to 256 unknowns and just beyond (260), alone or below other levels."""
    p, pc, h = _instance(shape, mg, sm, coarse_max=coarse)
    r = hi.random_vector(p.n, 12)
    ref = Oracle(p, pc).vcycle(r)
    z = h.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    h.close()
    tol = 1e-10 if mg == "c128" else 5e-5
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref) and np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))
