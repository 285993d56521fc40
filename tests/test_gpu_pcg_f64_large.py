"""The one-launch solver of native FP64 operators where rows are long: the edges of its unrolled
row loop (twelve steps of 64 columns), and its speed against the host-driven loop, whose
products run from a full grid."""
import time

import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs

pytestmark = pytest.mark.gpu

# steps of 64 columns: 11, 12, 13, 23, 24, 25
MESHES = [inputs.tetra_mesh(13), inputs.cube_mesh(8), inputs.tetra_mesh(14), inputs.tetra_mesh(19),
          inputs.fichera_mesh(8), inputs.tetra_mesh(20)]


def _operator(m):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    ctx = bem.Context()
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    return ctx, mesh, bem.Operator.assemble(mesh, precision=bem.PREC_F64)


@pytest.mark.parametrize("m", MESHES, ids=lambda m: f"{m.name}-{m.N}")
def test_rows_around_the_unrolled_steps(m):
    ctx, mesh, op = _operator(m)
    b = mesh.geometry()[0]
    _, x, info = bem.solve_capacity(op, tol=1e-11)
    # the recursive residual of CG and the true one differ by roundings of the products
    assert info["converged"] and np.linalg.norm(op.read() @ x - b) <= 1.1e-11 * np.linalg.norm(b)
    ctx.close()


@pytest.mark.parametrize("n", [35, 41], ids=lambda n: f"N{12 * n * n}")
def test_not_slower_than_the_host_loop(n):
    """Both loops do the same products; runs of one of them differ by less than 1%."""
    ctx, _, op = _operator(inputs.cube_mesh(n))
    best = {True: np.inf, False: np.inf}
    for _ in range(4):
        for on in best:
            ctx.set_persistent(on)
            t = time.perf_counter()
            its = bem.solve_capacity(op, tol=1e-12)[2]["iterations"]
            best[on] = min(best[on], (time.perf_counter() - t) / its)
    assert best[True] <= 1.05 * best[False], best
    ctx.close()
