"""Solves whose operator stays in shared memory (whole rows of it, four CTAs per 64 rows), at the
edges of their range: one pair of columns per thread, two and three, a last cluster with one
row and a full one, the largest size taken and the first one that is not."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu

# 4, 48, 300, 768 (12 clusters exactly), 972 and 1,200 (across 1,024 columns), 2,028 and 2,352 (across
# 2,048), 2,700 (above 16 rows per SM)
MESHES = [inputs.tetra_mesh(1)] + [inputs.cube_mesh(n) for n in (2, 5, 8, 9, 10, 13, 14, 15)] + [
    inputs.workload_polycube_adaptive(), inputs.graded_cube_mesh(12)]


@pytest.mark.parametrize("m", MESHES, ids=lambda m: f"{m.name}-{m.N}")
def test_resident_solve_is_that_of_the_operators_entries(m):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    ctx = bem.Context()
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    area = mesh.geometry()[0]
    x0 = np.linspace(0.5, 1.5, m.N)
    for prec in (bem.PREC_DF64, bem.PREC_F32):
        op = bem.Operator.assemble(mesh, precision=prec)
        V = op.read().astype(np.float64)
        x = np.linalg.solve(V, area)
        s = np.linalg.svd(V, compute_uv=False)
        # the residual at most tol ||b||, the rounding of its own evaluation 2^-44 of ||V|| ||phi||, a
        # factor 2 for the reference's rounding
        bound = 2.0 / s[-1] * (1e-11 * np.linalg.norm(area) + 2.0 ** -44 * s[0] * np.linalg.norm(x))
        for precond in (bem.PRECOND_NONE, bem.PRECOND_JACOBI, bem.PRECOND_BLOCK):
            for start in (None, x0):
                _, phi, info = bem.solve_capacity(op, tol=1e-11, precond=precond, x0=start, products=bem.PRODUCTS_FP32)
                assert info["converged"] and info["relres"] <= 1e-11
                assert info["outer"] >= 2 or info["iterations"] == 0
                assert np.linalg.norm(x - phi) <= bound, (prec, precond, np.linalg.norm(x - phi), bound)
                _, again, _ = bem.solve_capacity(op, tol=1e-11, precond=precond, x0=start, products=bem.PRODUCTS_FP32)
                assert np.array_equal(phi, again)
        op.close()
    ctx.close()
