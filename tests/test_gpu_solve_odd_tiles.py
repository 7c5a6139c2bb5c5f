"""S^-1 with half-storage tiles of an odd number of entries: 2-D n = 243 and 246, whose
largest staged tiles hold 1335 and 1365 entries of four bytes, so that the vectors behind
them need padding.

Tolerance: half storage is held to a residual of 2e-2 elsewhere; here per right-hand side.
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


@pytest.mark.parametrize("n", [243, 246])
def test_half_storage_residual(spm, n):
    P = spm.Problem2D(n, si.wavenumber_for_grid_2d(n), *si.random_medium_2d(n, 1))
    P.build_stencils(spm.SPM_C64H)
    for nrhs in (1, 2, 3, 4, 16):
        b = torch.from_numpy(np.ascontiguousarray(si.random_field_2d(n, nrhs, nrhs))).to("cuda")
        x = torch.full(b.shape, float("nan"), dtype=torch.complex64, device="cuda")
        P.solve_S(b.to(torch.complex64), x)
        y = torch.zeros_like(b)
        P.apply_S(x.to(torch.complex128), y)
        res = torch.linalg.vector_norm((y - b).flatten(1), dim=1) / torch.linalg.vector_norm(b.flatten(1), dim=1)
        assert res.max().item() < 2e-2
    P.close()
