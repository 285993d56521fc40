"""One FP16 product of the packed solver, entry by entry: single tiles, groups of two and groups of
four tiles per warp.

Two steps of CG without a preconditioner from x = 0 leave x in the span of b and V b, with V b
as the solver's product formed it: what a fit by b and the operator's own V b leaves over is the
product's error.  V and b are positive, so rounding the entries to halves (relative 2^-11, and
2^-25 of the tile's scale below the normal range) changes a row's sum by 2^-11 of it at most; a
tile left out or added to other rows changes 64 of them by more."""
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


def _group(N):
    """Tiles per group that the solver takes: enough tiles for 12 groups of them per warp."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nb = (N + 63) // 64
    nt = nb * (nb + 1) // 2
    warps = 8 * min(max((nt + 7) // 8, nb, 8), 2 * sms)
    return 4 if nt >= 48 * warps else 2 if nt >= 24 * warps else 1


@pytest.mark.parametrize("n,group", [(20, 1), (42, 1), (43, 2), (44, 2), (51, 4), (52, 4)],
                         ids=["N4800", "N21168", "N22188", "N23232", "N31212", "N32448"])
@pytest.mark.parametrize("prec", [bem.PREC_F32, bem.PREC_DF64], ids=["f32", "df64"])
def test_fp16_product_of_groups(ctx, n, group, prec):
    m = inputs.cube_mesh(n)
    R = inputs.random_rotation(inputs.SplitMix64(n))
    stretch = R * np.array([1.0, 1.3, 0.8])[:, None]  # panels of different areas
    mesh = bem.Mesh.upload(ctx, m.verts @ stretch.T, m.tris)
    assert _group(m.N) == group
    op = bem.Operator.assemble(mesh, precision=prec)
    b = mesh.geometry()[0]
    q = op.matvec(b)
    _, x, info = bem.solve_capacity(op, tol=1e-12, max_it=2, precond=bem.PRECOND_NONE, products=bem.PRODUCTS_FP16,
                                    raise_not_converged=False)
    assert info["iterations"] == 2 and not info["converged"]
    A = np.stack([b / np.linalg.norm(b), q / np.linalg.norm(q)], axis=1)
    c = np.linalg.lstsq(A, x, rcond=None)[0]
    err = np.abs(x - A @ c) / (np.abs(c[1]) * A[:, 1])
    assert err.max() <= 2.0 ** -11, (err.max() * 2.0 ** 11, int(err.argmax()) // 64)
    op.close()
    mesh.close()
