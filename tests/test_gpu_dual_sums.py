"""V^dual is the FP64 sum of the entries of V^bary, rounded once where it is stored, on both of
its paths (contraction passes; gathers where their scratch finds no room)."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu

CHILD = np.array([0, 1, 1, 2, 2, 0])  # the vertex of each of the six children of a triangle


@pytest.mark.parametrize("room", [True, False], ids=["contraction", "gathers"])
@pytest.mark.parametrize("scale", [1.0, 1e-8], ids=["unit", "small"])  # entries of 1e-4 and of 1e-28
@pytest.mark.parametrize("prec", [bem.PREC_F64, bem.PREC_DF64, bem.PREC_F32], ids=["f64", "df64", "f32"])
@pytest.mark.parametrize("m", [inputs.cube_mesh(2), inputs.tetra_mesh(4), inputs.workload_polycube_adaptive()],
                         ids=lambda m: f"{m.name}-{m.N}")
def test_dual_entries_are_fp64_sums(m, prec, scale, room):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    ctx = bem.Context()
    mesh = bem.Mesh.upload(ctx, m.verts * scale, m.tris)
    op = bem.Operator.assemble(mesh.barycentric(), precision=prec)
    used, V = ctx.memory_in_use(), op.read()
    if not room:
        ctx.close()
        ctx = bem.Context(hbm_budget_bytes=used + 16 * m.N * m.N + (1 << 20))
        mesh = bem.Mesh.upload(ctx, m.verts * scale, m.tris)
        op = bem.Operator.assemble(mesh.barycentric(), precision=prec)
    V = torch.tensor(V, device="cuda").double()
    got = torch.tensor(bem.Operator.dual(op, mesh).read(), device="cuda")
    tris = mesh.download()[1]
    owner = torch.tensor(tris[:, CHILD].reshape(-1).astype(np.int64), device="cuda")  # vertex of each child
    # the reference sums hi and lo halves of the entries apart (26 bits each: 64 x 64 of them add
    # exactly in FP64)
    big = V.abs().max() * 2.0 ** 26
    hi = (V + big) - big
    M = mesh.M

    def contract(A):
        rows = torch.zeros((M, A.shape[1]), dtype=torch.float64, device="cuda").index_add_(0, owner, A)
        return torch.zeros((M, M), dtype=torch.float64, device="cuda").index_add_(1, owner, rows)

    ref_h, ref_l = contract(hi), contract(V - hi)
    # FP64: at most 4 + 32 + 32 additions in a chain, here about 16; stored as a pair of floats: 2^-48
    bound = 40 * 2.0 ** -53 + (0.0 if prec == bem.PREC_F64 else 2.0 ** -48)
    err = ((got - ref_h) - ref_l).abs() / (ref_h + ref_l)
    assert float(err.max()) <= bound, (float(err.max()) / bound, float(err.max()))
    ctx.close()
