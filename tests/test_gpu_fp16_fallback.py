"""FP16 products where they are too rough (strongly graded surfaces): the solver notices at a
replaced residual, and its exact products then converge as they do alone."""
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    ctx = bem.Context()
    m = inputs.graded_cube_mesh(30)  # N = 10,800
    m = inputs.transformed(m, inputs.random_rotation(inputs.SplitMix64(11)))
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    yield {p: bem.Operator.assemble(mesh, precision=p) for p in (bem.PREC_F32, bem.PREC_DF64)}
    ctx.close()


@pytest.mark.parametrize("precond", [bem.PRECOND_JACOBI, bem.PRECOND_BLOCK], ids=["jacobi", "block"])
@pytest.mark.parametrize("prec", [bem.PREC_F32, bem.PREC_DF64], ids=["f32", "df64"])
def test_exact_products_take_over(op, prec, precond):
    tol = 1e-8
    cap, _, exact = bem.solve_capacity(op[prec], tol=tol, precond=precond, products=bem.PRODUCTS_FP32)
    # a segment of FP16 products ends after 400 iterations at the latest, and each but the last
    # lowered the residual tenfold: nine of them, then a solve from there
    most = 9 * 400 + 2 * exact["iterations"]
    cap16, _, info = bem.solve_capacity(op[prec], tol=tol, precond=precond, products=bem.PRODUCTS_FP16, max_it=most)
    assert info["converged"] and info["relres"] <= tol
    assert abs(cap16 / cap - 1) < 1e-6
