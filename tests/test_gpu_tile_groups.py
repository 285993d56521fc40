"""FP16 products by groups of two and four tiles of a tile row: the sizes where a warp gets
enough tiles.  The residual that decides convergence is formed from the operator, so a wrong
product shows as iterations; Caps agree to the tolerance times the conditioning as in the
tests of the products."""
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = bem.Context()
    yield c
    c.close()


@pytest.mark.parametrize("n", [43, 51], ids=["pairs", "fours"])  # N = 22,188 and 31,212
def test_grouped_products_reach_the_same_solution(ctx, n):
    tol = 1e-11
    m = inputs.cube_mesh(n)
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    op = bem.Operator.assemble(mesh, precision=bem.PREC_F32)
    cap32, _, i32 = bem.solve_capacity(op, tol=tol, precond=bem.PRECOND_BLOCK, products=bem.PRODUCTS_FP32)
    cap16, _, i16 = bem.solve_capacity(op, tol=tol, precond=bem.PRECOND_BLOCK, products=bem.PRODUCTS_FP16)
    assert i16["converged"] and i16["relres"] <= tol
    assert abs(cap16 / cap32 - 1) < 1e-9
    assert i16["iterations"] <= 2 * i32["iterations"] + 20
    op.close()
    mesh.close()
