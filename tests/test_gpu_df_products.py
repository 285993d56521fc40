"""Solves whose products are in DF64 alone, on both sides of the size from which they run three
CTAs per SM."""
import time

import numpy as np
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


@pytest.mark.parametrize("n", [31, 32], ids=lambda n: f"N{12 * n * n}")  # 36 and 40 tiles per CTA of 152 SMs
def test_residual_at_both_sides_of_the_line(ctx, n):
    m = inputs.cube_mesh(n)
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    op = bem.Operator.assemble(mesh, precision=bem.PREC_DF64)
    b = mesh.geometry()[0]
    x0 = np.linspace(0.5, 1.5, m.N)
    for precond in (bem.PRECOND_NONE, bem.PRECOND_JACOBI, bem.PRECOND_BLOCK):
        for start in (None, x0):
            cap, x, info = bem.solve_capacity(op, tol=1e-10, precond=precond, x0=start, reliable_delta=-1.0)
            cap2 = bem.solve_capacity(op, tol=1e-10, precond=precond, x0=start)[0]
            # the recursive residual and that of the product here differ by the products' roundings
            assert info["converged"] and np.linalg.norm(op.matvec(x) - b) <= 1.1e-10 * np.linalg.norm(b)
            assert abs(cap / cap2 - 1) < 1e-8
    op.close()
    mesh.close()


def test_products_stream_the_operator(ctx):
    """One iteration reads the upper triangle, 4 N^2 bytes, at 0.64 of the rate of a copy or more."""
    import torch

    m = inputs.cube_mesh(43)  # N = 22,188
    mesh = bem.Mesh.upload(ctx, m.verts, m.tris)
    op = bem.Operator.assemble(mesh, precision=bem.PREC_DF64)
    a = torch.zeros(1 << 30, dtype=torch.uint8, device="cuda")
    c = torch.empty_like(a)
    copy = per_it = np.inf
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(10):
            c.copy_(a)
        torch.cuda.synchronize()
        copy = min(copy, (time.perf_counter() - t) / (20 * a.numel()))  # seconds per byte
        t = time.perf_counter()
        its = bem.solve_capacity(op, tol=1e-10, reliable_delta=-1.0)[2]["iterations"]
        per_it = min(per_it, (time.perf_counter() - t) / its)
    assert 4.0 * m.N ** 2 * copy >= 0.64 * per_it, 4.0 * m.N ** 2 * copy / per_it
    op.close()
    mesh.close()
