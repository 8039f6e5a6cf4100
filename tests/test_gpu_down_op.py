"""HELM_OP_DOWN: the first half of a level, with its iterate, in one launch."""
import ctypes

import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu


def _launches(fn):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    n = ctypes.c_size_t()
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("mg", ["c64", "c128"])
@pytest.mark.parametrize("sm", [hi.SM_JACOBI, hi.SM_RBGS])
@pytest.mark.parametrize("shape", [(24, 19), (122, 33), (300, 131), (700, 620)])
def test_down_is_one_launch(shape, sm, mg):
    import paper_0912_0180_gb300._lib as L
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, shape, 0, k0=10.0, phi_kind="bump", rhs="zero", bump_centre=(0.3, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=sm, omega=0.5)
    h, o = Helm(p, pc, mg_dtype=mg, autotune=False), Oracle(p, pc)
    dt, tol = (torch.complex64, 5e-5) if mg == "c64" else (torch.complex128, 1e-10)
    f = hi.random_vector(p.n, 42).astype(np.complex64)
    F = torch.from_numpy(f).cuda().to(dt)
    u = torch.zeros(p.n, dtype=dt, device="cuda")
    fc = torch.zeros(o.level_size(1, 1), dtype=dt, device="cuda")
    h.level_op(L.HELM_OP_DOWN, 0, u, F, fc)
    f = f.astype(complex)
    u_ref = o.smooth(0, np.zeros(p.n), f, 1)
    fc_ref = o.restrict(0, f - o.apply(u_ref, 1, 0))
    for got, want, t in ((u, u_ref, tol), (fc, fc_ref, 10 * tol)):
        d = got.cpu().numpy() - want
        assert np.linalg.norm(d) <= t * np.linalg.norm(want) and np.max(np.abs(d)) <= t * np.max(np.abs(want))
    assert _launches(lambda: h.level_op(L.HELM_OP_DOWN, 0, u, F, fc)) == 1
    h.close()
