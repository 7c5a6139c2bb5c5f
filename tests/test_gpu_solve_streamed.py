"""S^-1 through factors above 256 MB, whose tiles stream through registers in complex64 and
half storage (smaller factors stage them in shared memory), at one to five right-hand sides:
3-D n = 32 (1.5 and 0.7 GB) and 2-D n = 300 (279 MB).

Tolerances: the residuals that these storages are held to elsewhere (1e-4 and 2e-2), of every
right-hand side; their magnitudes differ, so that one cannot hide in another's norm.
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


@pytest.mark.parametrize("dim,n,storage,bound", [(3, 32, "SPM_C64", 1e-4), (3, 32, "SPM_C64H", 2e-2), (2, 300, "SPM_C64", 1e-4)])
def test_residual_of_every_right_hand_side(spm, dim, n, storage, bound):
    if dim == 3:
        P = spm.Problem(n, si.wavenumber_for_grid(n), *si.random_medium(n, 1))
    else:
        P = spm.Problem2D(n, si.wavenumber_for_grid_2d(n), *si.random_medium_2d(n, 1))
    P.build_stencils(getattr(spm, storage))
    if dim == 3:
        assert P.factor_bytes(spm.SPM_C64) > 256 << 20
    for nrhs in (1, 2, 3, 4, 5):
        b = (si.random_field if dim == 3 else si.random_field_2d)(n, 10 + nrhs, nrhs)
        b = torch.from_numpy(np.ascontiguousarray(b)).to("cuda")
        b *= torch.tensor([10.0 ** (-2 * q) for q in range(nrhs)], device="cuda").reshape((-1,) + (1,) * (dim + 1))
        x = torch.full(b.shape, float("nan"), dtype=torch.complex64, device="cuda")
        P.solve_S(b.to(torch.complex64), x)
        y = torch.zeros_like(b)
        P.apply_S(x.to(torch.complex128), y)
        res = torch.linalg.vector_norm((y - b).flatten(1), dim=1) / torch.linalg.vector_norm(b.flatten(1), dim=1)
        assert res.max().item() < bound
    P.close()
