"""Kernels that the autotuner or the size rules choose, forced: the row-walking kernels alone and grouped, their
unaligned form, and the fused 9-point kernels in both precisions and tiles."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import helm_inputs as hi
from oracle import Oracle

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import numpy as np, torch, helm_inputs as hi
from oracle import Oracle
from paper_0912_0180_gb300.helm import Helm, solve_group
mg, shapes = {mg!r}, {shapes!r}
tol = 1e-10 if mg == "c128" else 5e-5
inst = []
for shape in shapes:
    p = hi.make_problem(2, shape, 0, k0=0.2 * max(shape), phi_kind="bump", rhs="gauss", bump_centre=(0.3, 0.6))
    pc = hi.Precond(kind=hi.PC_CSL, shift=1 + 0.5j, smoother=hi.SM_JACOBI, omega=0.5)
    h = Helm(p, pc, mg_dtype=mg)
    r = hi.random_vector(p.n, 41)
    ref = Oracle(p, pc).vcycle(r)
    R = torch.from_numpy(r).cuda()
    z = h.vcycle(R)
    d = z.cpu().numpy() - ref
    assert np.linalg.norm(d) <= tol * np.linalg.norm(ref) and np.max(np.abs(d)) <= tol * np.max(np.abs(ref)), shape
    if mg == "c64":  # an output on 8 bytes takes the rows element by element, and a widened one: the same values
        buf = torch.zeros(p.n + 2, dtype=torch.complex64, device="cuda")
        off = 1 if buf.data_ptr() % 16 == 0 else 0
        out = buf[off:off + p.n]
        assert out.data_ptr() % 16 == 8
        h.vcycle(R, out=out)
        assert torch.equal(out, z) and buf[off + p.n] == 0 and (off == 0 or buf[0] == 0)
        assert torch.equal(h.vcycle(R, dtype=torch.complex128), z.to(torch.complex128))
    inst.append((h, torch.from_numpy(p.b).cuda()))
hs, bs = [h for h, _ in inst], [b for _, b in inst]
lone = [h.solve(b, tol=1e-6, maxmv=40) for h, b in inst]
xs, infos = solve_group(hs, bs, tol=1e-6, maxmv=40)
for (x, i), xg, ig in zip(lone, xs, infos):
    assert (i.status, i.matvecs) == (ig.status, ig.matvecs) and torch.equal(x, xg)
"""


@pytest.mark.parametrize("mg", ["c64", "c128"])
@pytest.mark.parametrize("tile", [5, 6])
def test_row_walking_kernels_alone_and_grouped(tile, mg, tmp_path):
    """The tuner's cache names tile and tail for every level; were one not taken, the process would append its own."""
    shapes = [(62, 47), (122, 34), (121, 64), (242, 36), (243, 70)]
    b = 4 if mg == "c64" else 8
    lines = []
    for s in shapes:
        n = [v - 2 for v in s]
        m, levels = list(n), 1
        while min(m) >= 3 and max(m) > 8:
            lines.append(f"tile {b} 0 {m[0]} {m[1]} {tile} {tile}")
            m = [v // 2 for v in m]
            levels += 1
        lines.append(f"depth {b} 4 2 {n[0]} {n[1]} 1 {levels} 1")  # the tail begins below the finest level
    path = tmp_path / "tune"
    path.write_text("\n".join(lines) + "\n")
    out = subprocess.run([sys.executable, "-c", CODE.format(mg=mg, shapes=shapes)], cwd=ROOT,
                         env=dict(os.environ, HELM_TUNE_CACHE=str(path)), capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]
    assert path.read_text() == "\n".join(lines) + "\n"


# level 1 of the first: 33,411 unknowns, above the 30,000 (FP32; FP64 7,000) where the tail begins without the tuner, in
# the small tiles; of the others enough large tiles for two a multiprocessor on 152 of them (the third: on the way up)
@pytest.mark.parametrize("mg", ["c64", "c128"])
@pytest.mark.parametrize("shape", [(521, 261), (805, 804), (1203, 410)])
def test_fused_nine_point_levels(shape, mg):
    from paper_0912_0180_gb300.helm import Helm
    p = hi.make_problem(2, shape, 0, k0=0.2 * max(shape), phi_kind="bump", rhs="zero", bump_centre=(0.3, 0.6))
    pc = hi.Precond(kind=hi.PC_CSL, shift=1 + 0.5j, smoother=hi.SM_JACOBI, omega=0.5, galerkin=True)
    r = hi.random_vector(p.n, 31)
    ref = Oracle(p, pc).vcycle(r)
    h = Helm(p, pc, mg_dtype=mg, autotune=False)
    n1 = h.level_shape(1)
    assert n1[0] * n1[1] > 30000
    z = h.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    h.close()
    tol = 1e-10 if mg == "c128" else 5e-5
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref) and np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref))
