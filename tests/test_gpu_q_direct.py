"""Q with seeded stencil tables at the sizes where its launches can go wrong: fewer
points than a block, a last block that is nearly empty, all classes, several fields.

Tolerance: a sum of at most 81 complex products, 81 * 4 * 2^-53 = 3.6e-14 of the sum of
absolute values in complex128 (1e-13 of the result's norm, whose terms do not cancel),
and 2^29 times that in complex64 (5.4e-5 bounds it; 2e-5 as for every complex64 apply).
"""
import numpy as np
import pytest

import oracle
import spm_inputs as si
from oracle import twod

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def spm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_02297_gb300 as spm
    return spm


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def tables(dim, seed):
    """Random complex tables, zero in the rows a class does not have."""
    rng = np.random.default_rng(seed)
    nt = 3 ** dim
    alpha = rng.standard_normal((nt, dim * nt, dim)) + 1j * rng.standard_normal((nt, dim * nt, dim))
    beta = rng.standard_normal((nt, (dim + 1) * nt, dim)) + 1j * rng.standard_normal((nt, (dim + 1) * nt, dim))
    for c in range(nt):
        T = int(np.prod([3 if (c // 3 ** d) % 3 == 1 else 2 for d in range(dim)]))
        alpha[c, dim * T:] = 0
        beta[c, (dim + 1) * T:] = 0
    return alpha, beta


@pytest.mark.parametrize("dim,n,nrhs", [(3, 4, 1), (3, 4, 3), (3, 8, 2), (3, 16, 1), (3, 48, 2),
                                        (2, 4, 1), (2, 5, 3), (2, 8, 1), (2, 9, 2), (2, 65, 1), (2, 119, 2)])
def test_q_matches_oracle(spm, dim, n, nrhs):
    al, be = tables(dim, 10 * n + dim)
    if dim == 3:
        P = spm.Problem(n, si.wavenumber_for_grid(n), *si.random_medium(n, 1))
        v = si.random_field(n, 5, nrhs)
    else:
        P = spm.Problem2D(n, si.wavenumber_for_grid_2d(n), *si.random_medium_2d(n, 1))
        v = si.random_field_2d(n, 5, nrhs)
    P.set_stencils(al, be)
    ref = oracle.apply_Q(n, al, v) if dim == 3 else twod.apply_Q(n, al, v)
    for dt, tol in ((torch.complex128, 1e-13), (torch.complex64, 2e-5)):
        y = torch.full(v.shape, float("nan"), dtype=dt, device="cuda")
        P.apply_Q(torch.from_numpy(v).to("cuda").to(dt), y)
        torch.cuda.synchronize()
        assert rel(y.cpu().numpy().astype(np.complex128), ref) < tol
