"""The one-cluster tail of 2D V(1,1) cycles (levels split over the blocks of one cluster, the rest of
the cycle as a dense operator) against the oracle's V-cycle, where its split can go wrong: the whole
cycle as the operator, fewer rows than blocks, one row a block, thin grids, odd sizes, the largest
level that fits, with and without a launch level above it."""
import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu

# unknowns per axis are n_int - 2 without layers
SHAPES = [(10, 10), (26, 26), (27, 26), (5, 202), (202, 5), (39, 66), (66, 39), (98, 35), (35, 98), (131, 129), (163, 250),
          (322, 162)]


@pytest.mark.parametrize("mg", ["c128", "c64"])
@pytest.mark.parametrize("sm,galerkin", [(hi.SM_JACOBI, False), (hi.SM_RBGS, False), (hi.SM_JACOBI, True)])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_tail_vcycle(shape, sm, galerkin, mg):
    """FP64 to 1e-10, FP32 to 5e-5 relative (rounding 2^-24 an operation through a few dozen chained
    ones), as for the other V-cycle kernels; and the same result whichever level the tail begins at
    (the tuner's choice or the rule's): FP32 bit for bit, FP64 to a few units of its rounding (whether
    f - a s is one fused operation is the compiler's choice in each kernel)."""
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, shape, ((0, 0), (0, 0)), k0=0.3 * (max(shape) - 1), phi_kind="bump", rhs="zero",
                        bump_centre=(0.3, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=sm, galerkin=galerkin)
    r = hi.random_vector(p.n, 31)
    ref = Oracle(p, pc).vcycle(r)
    tol = 1e-10 if mg == "c128" else 5e-5
    zs = []
    for autotune in (True, False):
        h = Helm(p, pc, mg_dtype=mg, autotune=autotune)
        zs.append(h.vcycle(torch.from_numpy(r).cuda()))
        h.close()
    if mg == "c64":
        assert torch.equal(zs[0], zs[1])
    else:
        assert torch.linalg.norm(zs[0] - zs[1]) <= 1e-13 * torch.linalg.norm(zs[1])
    z = zs[0].cpu().numpy()
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref)
    assert np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))
