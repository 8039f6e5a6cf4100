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


@pytest.mark.parametrize("shape,mg", [((5, 3), "c128"), ((9, 40), "c64"), ((33, 65), "c128"), ((640, 70), "c64"), ((70, 600), "c64"),
                                      ((70, 3200), "c128"), ((70, 4200), "c64"), ((30000, 70), "c64")])
@pytest.mark.parametrize("galerkin", [False, True])
def test_ilu_strips(shape, mg, galerkin):
    """The ILU(0) step's triangular solves in strips of 32 rows handed from block to block: one strip,
    a last strip of few rows, several warps a block, more strips than one cluster holds, rows too long
    for shared memory; on the finest level (5-point) and, Galerkin, the next one (9-point)."""
    import paper_0912_0180_gb300._lib as L
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, (shape[0] + 2, shape[1] + 2), 0, extent=((shape[0] + 1) / 32, (shape[1] + 1) / 32), k0=6.0,
                        phi_kind="bump", rhs="zero", bump_centre=(0.4, 0.6))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.4, smoother=hi.SM_ILU, galerkin=galerkin, nu1=0, nu2=1, coarse_max=2)
    o = Oracle(p, pc)
    h = Helm(p, pc, mg_dtype=mg)
    dt = torch.complex128 if mg == "c128" else torch.complex64
    tol = 1e-10 if mg == "c128" else 5e-5
    lvl = 1 if galerkin and o.nlev > 2 else 0
    n = o.level_size(1, lvl)
    a, b = hi.random_vector(n, 5).astype(np.complex64), hi.random_vector(n, 6).astype(np.complex64)
    for op, start in ((L.HELM_OP_SMOOTH, a), (L.HELM_OP_SMOOTH0, 0 * a)):
        u = torch.from_numpy(start).cuda().to(dt)
        h.level_op(op, lvl, u, torch.from_numpy(b).cuda().to(dt), None, count=1)
        ref = o.smooth(lvl, start.astype(np.complex128), b.astype(np.complex128), 1)
        d = u.cpu().numpy() - ref
        assert np.linalg.norm(d) <= tol * np.linalg.norm(ref) and np.max(np.abs(d)) <= tol * np.max(np.abs(ref))
    h.close()


@pytest.mark.parametrize("mg", ["c64", "c128"])
@pytest.mark.parametrize("tile", [5, 6])
@pytest.mark.parametrize("shape", [(62, 47), (122, 33), (121, 64), (242, 35), (243, 70), (300, 131)])
def test_row_walking_kernels(shape, tile, mg, tmp_path):
    """The row-walking kernels of damped-Jacobi levels (forced through the tuner's cache file) where their
    split can go wrong: one strip and several, odd sizes, blocks cut short at either end; the V-cycle
    against the oracle's, complex64 and (narrowed on the way in) complex128 right-hand sides alike."""
    import os
    import subprocess
    import sys
    n = [s - 2 for s in shape]
    b = 4 if mg == "c64" else 8
    lines, m = [], list(n)
    while min(m) >= 3 and max(m) > 8:
        lines.append(f"tile {b} 0 {m[0]} {m[1]} {tile} {tile}")
        m = [v // 2 for v in m]
    lines.append(f"depth {b} 4 2 {n[0]} {n[1]} 1 {len(lines) + 1} 1")  # the tail begins below the finest level
    path = tmp_path / "tune"
    path.write_text("\n".join(lines) + "\n")
    code = f"""
import numpy as np, torch, helm_inputs as hi
from oracle import Oracle
from paper_0912_0180_gb300.helm import Helm
p = hi.make_problem(2, {shape!r}, 0, k0=30.0, phi_kind="bump", rhs="zero", bump_centre=(0.3, 0.6))
pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=hi.SM_JACOBI, omega=0.5)
r = hi.random_vector(p.n, 41)
ref = Oracle(p, pc).vcycle(r)
h = Helm(p, pc, mg_dtype={mg!r})
z = h.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
tol = 1e-10 if {mg!r} == "c128" else 5e-5
assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref), np.linalg.norm(z - ref) / np.linalg.norm(ref)
assert np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))
import paper_0912_0180_gb300._lib as L
o = Oracle(p, pc)
dt = torch.complex64 if {mg!r} == "c64" else torch.complex128
f = hi.random_vector(p.n, 42).astype(np.complex64)
u = torch.zeros(p.n, dtype=dt, device="cuda")
fc = torch.zeros(o.level_size(1, 1), dtype=dt, device="cuda")
h.level_op(L.HELM_OP_DOWN, 0, u, torch.from_numpy(f).cuda().to(dt), fc)
f = f.astype(np.complex128)
u_ref = o.smooth(0, np.zeros(p.n), f, 1)
fc_ref = o.restrict(0, f - o.apply(u_ref, 1, 0))
for got, want, t in ((u, u_ref, tol), (fc, fc_ref, 10 * tol)):
    d = got.cpu().numpy() - want
    assert np.linalg.norm(d) <= t * np.linalg.norm(want) and np.max(np.abs(d)) <= t * np.max(np.abs(want))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], cwd=root, env=dict(os.environ, HELM_TUNE_CACHE=str(path)),
                         capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("shape,levels,kind", [((35, 20, 23), 2, "const"), ((22, 31, 28), 2, "const"), ((66, 33, 31), 32, "bump"),
                                               ((63, 64, 29), 32, "bump"), ((11, 70, 35), 32, "const")])
def test_xsplit_cycle_3d(shape, levels, kind, wide):
    """FP32 red-black 3D cycles: the complex128 input taken with the red half-sweep, residual and full
    weighting in one kernel (with the coarse red half-sweep), the black-only prolongation, the separable
    coarse solve in planes and columns, and the last sweep writing natural order in either precision; odd
    and even sizes, more and fewer columns than a warp's 30."""
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(3, shape, 0, k0=6.0, phi_kind=kind, rhs="zero", bump_centre=(0.3, 0.6, 0.4))
    pc = hi.Precond(kind=hi.PC_CSG_UNIFORM, theta_beta=0.3, smoother=hi.SM_RBGS, max_levels=levels)
    r = hi.random_vector(p.n, 51)
    ref = Oracle(p, pc).vcycle(r)
    h = Helm(p, pc, mg_dtype="c64")
    z = h.vcycle(torch.from_numpy(r).cuda(), dtype=torch.complex128 if wide else torch.complex64).cpu().numpy()
    h.close()
    assert np.linalg.norm(z - ref) <= 5e-5 * np.linalg.norm(ref)
    assert np.max(np.abs(z - ref)) <= 5e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("sm", [hi.SM_JACOBI, hi.SM_RBGS])
@pytest.mark.parametrize("mg", ["c128", "c64"])
@pytest.mark.parametrize("shape", [(35, 20, 23), (50, 21, 12), (51, 9, 30), (66, 18, 17), (82, 12, 11)])
def test_natural_cycle_3d(shape, mg, sm):
    """Natural-order 3D levels: rows ending in a short chunk of columns (1, 16, 17, 0 and 16 past a multiple of
    32), whose points FP64 kernels pack along y, and the pairwise prolongation, at odd and even sizes."""
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(3, shape, 0, k0=6.0, phi_kind="bump", rhs="zero", bump_centre=(0.3, 0.6, 0.4))
    pc = hi.Precond(kind=hi.PC_CSL, shift=1 + 0.5j, smoother=sm)
    r = hi.random_vector(p.n, 61)
    o = Oracle(p, pc)
    ref = o.vcycle(r)
    tol = 1e-10 if mg == "c128" else 5e-5
    h = Helm(p, pc, mg_dtype=mg)
    z = h.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref) and np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))
    y, y_ref = h.apply(torch.from_numpy(r).cuda()).cpu().numpy(), o.apply(r)
    assert np.linalg.norm(y - y_ref) <= 1e-12 * np.linalg.norm(y_ref)
    h.close()
