"""The packed products of the persistent solver (sums on power-of-two grids, packed rows
scaled by their diagonal) at the edges of their 64 x 64 tiles: the solution is that of the
operator's own entries, whatever the number of rows in the last tile, the scale of the
surface and the ratio of its triangles' sizes."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    return bem.Context()


MESHES = [inputs.tetra_mesh(1), inputs.cube_mesh(1), inputs.tetra_mesh(4), inputs.cube_mesh(3), inputs.tetra_mesh(8),
          inputs.icosphere_mesh(4), inputs.graded_cube_mesh(6), inputs.fichera_mesh(4)]  # 4 .. 768 triangles


@pytest.mark.parametrize("scale", [1.0, 1e-5, 3e4])
@pytest.mark.parametrize("m", MESHES, ids=lambda m: f"{m.name}-{m.N}")
def test_solution_is_that_of_the_operators_entries(ctx, m, scale):
    mesh = bem.Mesh.upload(ctx, m.verts * scale + 0.25 * scale, m.tris)
    area = mesh.geometry()[0]
    for prec, precond, products in [(bem.PREC_DF64, bem.PRECOND_JACOBI, 0), (bem.PREC_DF64, bem.PRECOND_BLOCK, 0),
                                    (bem.PREC_DF64, bem.PRECOND_BLOCK, bem.PRODUCTS_FP16),
                                    (bem.PREC_F32, bem.PRECOND_BLOCK, bem.PRODUCTS_FP32),
                                    (bem.PREC_F32, bem.PRECOND_BLOCK, bem.PRODUCTS_FP16)]:
        op = bem.Operator.assemble(mesh, precision=prec)
        V = op.read().astype(np.float64)
        x = np.linalg.solve(V, area)
        cap, phi, info = bem.solve_capacity(op, tol=1e-11, precond=precond, products=products)
        assert info["converged"]
        # ||x - phi|| <= ||V^-1|| ||b - V phi||, the residual at most tol ||b|| and the rounding of
        # its own evaluation (2^-44 of ||V|| ||phi||); a factor 2 for the reference's rounding
        s = np.linalg.svd(V, compute_uv=False)
        bound = 2.0 / s[-1] * (1e-11 * np.linalg.norm(area) + 2.0 ** -44 * s[0] * np.linalg.norm(x))
        assert np.linalg.norm(x - phi) <= bound, (prec, precond, products, np.linalg.norm(x - phi), bound)
