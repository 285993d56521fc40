"""The marking's sort where the memory budget has no room for its second array: in place, with the
same marks."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import bem

pytestmark = pytest.mark.gpu


def _up(b):
    return (b + 255) // 256 * 256


@pytest.mark.parametrize("N", [12, 1024, 1025, 5000, 16385, 40000, 131072, 131073])
def test_marks_within_a_tight_budget(N):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    eta2 = np.random.default_rng(N).random(N) ** 6
    ctx = bem.Context()
    m, n = bem.dorfler(ctx, eta2, 0.5)
    base = ctx.memory_in_use()
    ctx.close()
    n2 = 2
    while n2 < N:
        n2 *= 2
    nb = (N + 127) // 128
    # the keys once, and the running sums with their blocks' sums (arguments are not counted)
    need = base + _up(8 * n2 + 8 * (N + 2 * nb + 1) + 64)
    ctx = bem.Context(hbm_budget_bytes=need)
    m2, k2 = bem.dorfler(ctx, eta2, 0.5)
    assert k2 == n and np.array_equal(m, m2)
    ctx.close()
    ctx = bem.Context(hbm_budget_bytes=need - 256)
    with pytest.raises(bem.BemError):
        bem.dorfler(ctx, eta2, 0.5)
    ctx.close()
