"""The solve's level tiles (S^-1 by one launch per tree level) at every group width of
right-hand sides and at the widths' remainders, in the three factor storages.

Tolerances: complex128 as the factor itself is held to (1e-9 of the oracle's banded or
sparse LU); complex64 and half storage through the residual ||S x - b|| / ||b||, at the
bounds those storages are held to elsewhere (1e-4 and 2e-2).
"""
import numpy as np
import pytest

import oracle
import spm_inputs as si
from oracle import twod

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RHS = [1, 2, 3, 4, 5, 8, 9, 16, 17, 33]


@pytest.fixture(scope="module")
def spm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_02297_gb300 as spm
    return spm


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda").to(dtype)


@pytest.fixture(scope="module")
def problems(spm):
    """3-D n = 8 (one separator level of uneven halves, leaves of up to 4^3 points) and
    2-D n = 7 and 23 (ragged leaves), with the oracle's stencils and factor."""
    out = []
    n = 8
    k = si.wavenumber_for_grid(n)
    eps, grad = si.medium_bumps(n, seed=3, count=8)
    P = spm.Problem(n, k, eps, grad)
    al, be, _ = oracle.all_stencils(n, k)
    P.set_stencils(al, be)
    m, p = oracle.medium(eps, grad)
    out.append((P, oracle.SFactor(n, m, p, al, be), lambda seed, q, n=n: si.random_field(n, seed, q)))
    for n in (7, 23):
        k = si.wavenumber_for_grid_2d(n)
        eps, grad = si.random_medium_2d(n, 3)
        P = spm.Problem2D(n, k, eps, grad)
        al, be, _ = twod.all_stencils(n, k)
        P.set_stencils(al, be)
        m, p = twod.medium(eps, grad)
        out.append((P, twod.SFactor(n, m, p, al, be), lambda seed, q, n=n: si.random_field_2d(n, seed, q)))
    return out


@pytest.mark.parametrize("nrhs", RHS)
def test_c128_matches_oracle_lu(spm, problems, nrhs):
    for P, F, field in problems:
        P.factor_S(spm.SPM_C128)
        b = field(40 + nrhs, nrhs)
        x = torch.full(b.shape, float("nan"), dtype=torch.complex128, device="cuda")
        P.solve_S(dev(b, torch.complex128), x)
        torch.cuda.synchronize()
        assert rel(x.cpu().numpy(), np.stack([F.solve(v) for v in b])) < 1e-9


@pytest.mark.parametrize("n", [4, 5, 6, 11, 12, 13, 33])
def test_batched_factor_panels_2d(spm, n):
    """Own blocks that are and are not multiples of the panel width, one leaf (n <= 5) to
    several levels, complex128 and complex64, with rough media so that rows are swapped."""
    k = si.wavenumber_for_grid_2d(n)
    eps, grad = si.random_medium_2d(n, 5)
    P = spm.Problem2D(n, k, eps, grad)
    al, be, _ = twod.all_stencils(n, k)
    P.set_stencils(al, be)
    m, p = twod.medium(eps, grad)
    b = si.random_field_2d(n, 9, 1)
    ref = twod.SFactor(n, m, p, al, be).solve(b[0])
    P.factor_S(spm.SPM_C128)
    x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
    P.solve_S(dev(b, torch.complex128), x)
    torch.cuda.synchronize()
    assert rel(x.cpu().numpy()[0], ref) < 1e-9
    P.factor_S(spm.SPM_C64)
    assert P.factor_info(spm.SPM_C64)[3] < 1e-4


def test_batched_factor_large_own_block(spm):
    """3-D n = 16: fronts of 1152 unknowns and own blocks of up to 768, whose panel takes
    108 KB of a block's shared memory; the probe residual says whether it is a factor."""
    n = 16
    eps, grad = si.medium_bumps(n, seed=3, count=8)
    P = spm.Problem(n, si.wavenumber_for_grid(n), eps, grad)
    P.build_stencils(spm.SPM_C128)
    assert P.factor_info(spm.SPM_C128)[3] < 1e-12
    P.factor_S(spm.SPM_C64)
    assert P.factor_info(spm.SPM_C64)[3] < 1e-4


@pytest.mark.parametrize("storage,bound", [("SPM_C64", 1e-4), ("SPM_C64H", 2e-2)])
@pytest.mark.parametrize("nrhs", RHS)
def test_c64_residual(spm, problems, nrhs, storage, bound):
    for P, _, field in problems:
        P.factor_S(getattr(spm, storage))
        b = field(60 + nrhs, nrhs)
        x = torch.full(b.shape, float("nan"), dtype=torch.complex64, device="cuda")
        P.solve_S(dev(b, torch.complex64), x)
        y = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        P.apply_S(x.to(torch.complex128), y)
        torch.cuda.synchronize()
        assert rel(y.cpu().numpy(), b) < bound
