"""The dual operator and its preconditioner by the contraction passes against the gathers
that a context without room for their scratch takes, at the edges of the passes' tiles
(8 x 32 triangles)."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu

MESHES = [inputs.tetra_mesh(1), inputs.cube_mesh(1), inputs.tetra_mesh(3), inputs.cube_mesh(2), inputs.tetra_mesh(4),
          inputs.polycube_mesh(3, 0.5, 2), inputs.cube_mesh(4)]  # 4 .. 192 triangles


def _dual(m, prec, budget):
    ctx = bem.Context(hbm_budget_bytes=budget)
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    op = bem.Operator.assemble(mesh.barycentric(), precision=prec)
    used = ctx.memory_in_use()
    d = bem.Operator.dual(op, mesh)
    out = d.read(), d.preconditioner(0), d.preconditioner(1), used, ctx.launch_count()
    ctx.close()
    return out


@pytest.mark.parametrize("prec", [bem.PREC_F64, bem.PREC_DF64, bem.PREC_F32], ids=["f64", "df64", "f32"])
@pytest.mark.parametrize("m", MESHES, ids=lambda m: f"{m.name}-{m.N}")
def test_contraction_and_gathers_agree(m, prec):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    V, D, C, used, n = _dual(m, prec, 0)
    V2, D2, C2, _, n2 = _dual(m, prec, used + (1 << 20))  # no room for the contraction's scratch
    assert n2 != n, "both runs took the same path"
    assert np.array_equal(V, V.T) and np.array_equal(D, D.T)
    # positive sums of at most 64 x 64 entries in double-float or FP64: 2^-44 each way
    assert np.max(np.abs(V / V2 - 1)) <= 2.0 ** -43
    # sums that cancel, rounded to FP32: an ulp of the largest entry
    assert np.max(np.abs(D - D2)) <= 2.0 ** -22 * np.max(np.abs(D2))
    # two polynomials of degree 6 in the mass matrix, FP32: 2^-22 of D through a factor ||S|| each way
    assert np.max(np.abs(C - C2)) <= 64 * 2.0 ** -22 * np.max(np.abs(C2))
