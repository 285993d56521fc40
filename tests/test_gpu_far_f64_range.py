"""Native FP64 far field between surfaces whose sizes or distance leave the FP32 range: the
kernel estimates lengths in FP32 to choose its form, and entries of any FP64 lengths are the
rule's own sum."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem, inputs
from tests.test_far_grid_form import BARY, W

pytestmark = pytest.mark.gpu


def _two(size, shift, swap):
    """A tetrahedron of edge `size` at distance `shift` and one of edge 1 at the origin."""
    a, b = inputs.tetra_mesh(2, edge=size), inputs.tetra_mesh(2)
    va = a.verts + np.array([shift, 0.25 * shift, -0.5 * shift])
    parts = [(b.verts, b.tris), (va, a.tris)] if swap else [(va, a.tris), (b.verts, b.tris)]
    v = np.concatenate([p[0] for p in parts])
    t = np.concatenate([parts[0][1], parts[1][1] + len(parts[0][0])])
    return v, t, len(parts[0][1])


@pytest.mark.parametrize("swap", [False, True], ids=["large-first", "small-first"])
@pytest.mark.parametrize("size,shift", [(1.0, 40.0), (2.0 ** 100, 2.0 ** 120), (2.0 ** 126, 2.0 ** 130),
                                        (2.0 ** 150, 2.0 ** 170), (2.0 ** 230, 1.3 * 2.0 ** 260),
                                        (2.0 ** 240, 1.7 * 2.0 ** 270)])
def test_entries_between_surfaces_of_any_size(size, shift, swap):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    v, t, n = _two(size, shift, swap)
    ctx = bem.Context()
    mesh = bem.Mesh.upload(ctx, v, t)
    v, t = mesh.download()[:2]
    V = bem.Operator.assemble(mesh, precision=bem.PREC_F64).read()
    P = v[t]
    area = 0.5 * np.linalg.norm(np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]), axis=1)
    X = np.einsum("ak,nkc->nac", BARY, P)
    d = X[:n, None, :, None] - X[None, n:, None, :]
    ref = np.einsum("a,b,ijab->ij", W, W, 1.0 / np.linalg.norm(d, axis=-1))
    ref *= area[:n, None] * (area[None, n:] / (4.0 * np.pi))
    # a point's coordinates, the difference, three squares, the root and 49 additions: below 100 roundings
    assert np.max(np.abs(V[:n, n:] / ref - 1.0)) < 100 * 2.0 ** -53
    assert np.array_equal(V[:n, n:], V[n:, :n].T)
    ctx.close()
