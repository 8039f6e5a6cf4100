"""ILU(0) levels of few rows: one strip that stores only the rows it has (a 1D level has one)."""
import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

PC = dict(kind=hi.PC_CSG_UNIFORM, theta_beta=0.4, smoother=hi.SM_ILU, nu1=0, nu2=1, coarse_max=2)


@pytest.mark.parametrize("mg,esz", [("c64", 8), ("c128", 16)])
def test_estimate_of_a_1d_level(mg, esz):
    """Per unknown of a level 9 FP64 entries while the factors are made and at most 10 values in the cycle's precision;
    the levels' unknowns add up to twice the finest's (and 128 bytes a level of skew and chunk ends)."""
    from paper_0912_0180_gb300.helm import estimate_bytes
    p = hi.make_problem(1, 60000, 0, k0=10.0, rhs="zero")
    more = estimate_bytes(p, hi.Precond(**PC), mg) - estimate_bytes(p, hi.Precond(**{**PC, "smoother": hi.SM_JACOBI}), mg)
    assert 0 < more <= 2 * p.n * (9 * 16 + 10 * esz) + 16 * 10 * 8 * esz


@pytest.mark.gpu
@pytest.mark.parametrize("mg,esz", [("c64", 8), ("c128", 16)])
def test_memory_of_a_1d_hierarchy(mg, esz):
    """A context holds 6 values an unknown for ILU(0) on 5-point (1D: 3-point) levels."""
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(1, 30000, 0, k0=10.0, rhs="zero")
    size = {}
    for sm in (hi.SM_ILU, hi.SM_JACOBI):
        h = Helm(p, hi.Precond(**{**PC, "smoother": sm}), mg_dtype=mg, autotune=False)
        size[sm] = h.workspace_bytes
        h.close()
    assert size[hi.SM_ILU] - size[hi.SM_JACOBI] <= 2 * p.n * 6 * esz + 16 * 6 * 8 * esz


@pytest.mark.gpu
@pytest.mark.parametrize("mg", ["c64", "c128"])
@pytest.mark.parametrize("galerkin", [False, True])
@pytest.mark.parametrize("shape", [(100,), (1,), (6, 1), (1, 6), (41, 2), (200, 5), (9, 31), (70, 31), (70, 32), (70, 33), (64, 63)])
def test_few_rows(shape, galerkin, mg):
    """One smoothing step from a guess and from zero on every level above the coarsest, against the oracle's."""
    import paper_0912_0180_gb300._lib as L
    from paper_0912_0180_gb300.helm import Helm
    if galerkin and len(shape) == 1:
        pytest.skip("Galerkin coarse operators need 2D")
    p = hi.make_problem(len(shape), tuple(n + 2 for n in shape), 0, extent=tuple((n + 1) / 32 for n in shape), k0=6.0,
                        phi_kind="bump", rhs="zero", bump_centre=(0.4, 0.6))
    pc = hi.Precond(**PC, galerkin=galerkin)
    o = Oracle(p, pc)
    h = Helm(p, pc, mg_dtype=mg)
    dt = torch.complex128 if mg == "c128" else torch.complex64
    tol = 1e-10 if mg == "c128" else 5e-5
    for lvl in range(o.nlev - 1):
        n = o.level_size(1, lvl)
        a, b = hi.random_vector(n, 5).astype(np.complex64), hi.random_vector(n, 6).astype(np.complex64)
        for op, start in ((L.HELM_OP_SMOOTH, a), (L.HELM_OP_SMOOTH0, 0 * a)):
            u = torch.from_numpy(start).cuda().to(dt)
            h.level_op(op, lvl, u, torch.from_numpy(b).cuda().to(dt), None, count=1)
            ref = o.smooth(lvl, start.astype(complex), b.astype(complex), 1)
            d = u.cpu().numpy() - ref
            if len(shape) == 1:  # ILU(0) is the LU of a tridiagonal M: the error carries its condition (4e3 at 100
                d = o.apply(d, 1, lvl)  # unknowns), the residual does not
                ref = np.max(np.abs(o.dense(1, lvl))) * ref
            assert np.linalg.norm(d) <= tol * np.linalg.norm(ref) and np.max(np.abs(d)) <= tol * np.max(np.abs(ref))
    h.close()
