"""The 2-D passes let their dependents in at their start or before their last stores, by the
size of their grids: a chain of applies and Q without a wait between them against the same
calls one by one.  The kernels are deterministic: equal to the bit.
"""
import numpy as np
import pytest

import spm_inputs as si

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def spm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_02297_gb300 as spm
    return spm


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("n,nrhs", [(4, 1), (16, 5), (64, 64), (119, 8), (150, 2), (300, 1), (520, 1), (520, 3)])
def test_chain_equals_single_calls(spm, n, nrhs, dtype):
    P = spm.Problem2D(n, si.wavenumber_for_grid_2d(n), *si.random_medium_2d(n, 1))
    rng = np.random.default_rng(n)
    alpha = np.zeros((9, 18, 2), np.complex128)
    for c in range(9):
        T = int(np.prod([3 if (c // 3 ** d) % 3 == 1 else 2 for d in range(2)]))
        alpha[c, :2 * T] = rng.standard_normal((2 * T, 2))
    P.set_stencils(alpha, np.zeros((9, 27, 2), np.complex128))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x0 = torch.randn((nrhs, 2, n, n), dtype=getattr(torch, dtype), device="cuda", generator=g)

    def chain(wait):
        x, y = x0.clone(), torch.empty_like(x0)
        for _ in range(3):
            for call in (P.apply_A, P.apply_Q):
                call(x, y)
                if wait:
                    torch.cuda.synchronize()
                x, y = y, x
            x *= 0.1
        return x

    one_by_one = chain(True)
    for _ in range(4):
        assert torch.equal(chain(False), one_by_one)
    P.close()
