"""HELM_PF_UNFUSED on 3D FP32 red-black levels: every component in a launch of its own."""
import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,levels,kind", [((35, 20, 23), 2, "const"), ((66, 33, 31), 32, "bump"), ((30, 32, 34), 32, "const")])
def test_unfused_components_have_their_own_launches(shape, levels, kind):
    """The oracle's V-cycle in either output type (5e-5, as every FP32 V-cycle), and more launches a solve than the
    default: the residual and its weighting are two kernels instead of one on each x-split level."""
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(3, shape, 0, k0=6.0, phi_kind=kind, rhs="gauss", bump_centre=(0.3, 0.6, 0.4))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=hi.SM_RBGS, max_levels=levels)
    r = torch.from_numpy(hi.random_vector(p.n, 51)).cuda()
    ref = Oracle(p, pc).vcycle(hi.random_vector(p.n, 51))
    info = {}
    for fused in (True, False):
        h = Helm(p, pc, mg_dtype="c64", fused=fused, autotune=False)
        for dt in (torch.complex64, torch.complex128):
            z = h.vcycle(r, dtype=dt).cpu().numpy()
            assert np.linalg.norm(z - ref) <= 5e-5 * np.linalg.norm(ref) and np.max(np.abs(z - ref)) <= 5e-5 * np.max(np.abs(ref))
        _, info[fused] = h.solve(torch.from_numpy(p.b).cuda(), tol=1e-6, maxmv=200)
        h.close()
    assert info[False].kernels / info[False].matvecs >= info[True].kernels / info[True].matvecs + 1
