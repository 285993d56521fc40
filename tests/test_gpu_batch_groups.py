"""How a batch divides its problems: waves, solver launches of similar problems, CTAs per SM."""
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    c = bem.Context()
    yield c
    c.close()


def _sms():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


def _scaled(ctx, m, count):
    return [bem.Mesh.upload(ctx, m.verts * (1.0 + 0.001 * k), m.tris) for k in range(count)]


def _launches(ctx, batch):
    batch.run()
    n = ctx.launch_count()
    batch.run()
    return ctx.launch_count() - n


@pytest.mark.parametrize("prec,precond", [(bem.PREC_DF64, bem.PRECOND_JACOBI), (bem.PREC_F32, bem.PRECOND_BLOCK)],
                         ids=["df64", "f32"])
@pytest.mark.parametrize("m,count", [(inputs.cube_mesh(2), lambda: 3 * _sms()), (inputs.cube_mesh(4), lambda: _sms() - 2),
                                     (inputs.cube_mesh(7), lambda: _sms() // 2)], ids=["48", "192", "588"])
def test_small_problems_share_one_wave_and_one_solver_launch(ctx, m, count, prec, precond):
    count = count()
    meshes = _scaled(ctx, m, count)
    b = bem.Batch(ctx, meshes, precision=prec, precond=precond, tol=1e-11)
    assert b.waves()[0] == 1
    one = bem.Batch(ctx, meshes[:1], precision=prec, precond=precond, tol=1e-11)
    assert _launches(ctx, b) == _launches(ctx, one)
    caps = [r["cap"] for r in b.run()]
    ref = one.run()[0]["cap"]
    # Cap scales with the surface: to the entries' FP32 rounding, or to the tolerance
    eps = 1e-5 if prec == bem.PREC_F32 else 1e-9
    assert all(abs(c / (ref * (1.0 + 0.001 * k)) - 1) < eps for k, c in enumerate(caps))
    one.close()
    b.close()
    for q in meshes:
        q.close()


def test_df64_products_alone_match_single_solves(ctx):
    """Groups with and without three CTAs per SM (large problems; small ones)."""
    ms = [inputs.cube_mesh(32), inputs.cube_mesh(31), inputs.cube_mesh(7), inputs.tetra_mesh(4), inputs.tetra_mesh(1)]
    meshes = [bem.Mesh.upload(ctx, m.verts, m.tris) for m in ms]
    b = bem.Batch(ctx, meshes, precision=bem.PREC_DF64, precond=bem.PRECOND_JACOBI, tol=1e-11, reliable_delta=-1.0)
    for m, mesh, r in zip(ms, meshes, b.run()):
        op = bem.Operator.assemble(mesh, precision=bem.PREC_DF64)
        cap, _, info = bem.solve_capacity(op, tol=1e-11, reliable_delta=-1.0)
        assert r["converged"] and r["relres"] <= 1e-11
        assert abs(r["cap"] / cap - 1) < 1e-9, (m.name, r["cap"], cap)
        assert abs(r["iterations"] - info["iterations"]) <= 2 + info["iterations"] // 10
        op.close()
    b.close()
    for q in meshes:
        q.close()
