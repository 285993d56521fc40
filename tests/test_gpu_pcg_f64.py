"""The one-launch solver of native FP64 operators against the host-driven loop, at the edges
of its row distribution (a row per warp, rows past N, a padded last tile), with and without
a preconditioner and a start."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu

MESHES = [inputs.tetra_mesh(1), inputs.cube_mesh(1), inputs.tetra_mesh(4), inputs.cube_mesh(3), inputs.cube_mesh(4),
          inputs.workload_polycube_adaptive(), inputs.cube_mesh(21)]  # 4 .. 5,292 triangles


@pytest.mark.parametrize("m", MESHES, ids=lambda m: f"{m.name}-{m.N}")
def test_one_launch_matches_host_loop(m):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    ctx = bem.Context()
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    op = bem.Operator.assemble(mesh, precision=bem.PREC_F64)
    b = mesh.geometry()[0]
    x0 = np.linspace(0.5, 1.5, m.N)
    for precond in (bem.PRECOND_JACOBI, bem.PRECOND_NONE):
        for start in (None, x0):
            got = {}
            for on in (True, False):
                ctx.set_persistent(on)
                n = ctx.launch_count()
                cap, phi, info = bem.solve_capacity(op, tol=1e-11, precond=precond, x0=start)
                got[on] = cap, phi, info, ctx.launch_count() - n
            ctx.set_persistent(True)
            (c1, x1, i1, n1), (c2, x2, i2, n2) = got[True], got[False]
            assert i1["converged"] and i2["converged"] and n1 < n2 or i2["iterations"] == 0
            assert abs(i1["iterations"] - i2["iterations"]) <= 1 + i2["iterations"] // 50
            # both residuals are at most 1e-11 of b: the difference's residual at most twice that (and
            # the rounding of the product here)
            r = op.matvec(x1 - x2)
            assert np.linalg.norm(r) <= 2.2e-11 * np.linalg.norm(b)
            assert abs(c1 / c2 - 1) < 1e-9
    ctx.close()
