"""The multi-shift residual (csrc/spmm.cu) with rows of more than 128 entries on average, on either side of that line."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import test_gpu_residual_rows  # noqa: E402


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("n,m,ne,density,cplx,diag", [
    (180, 3, 4, 0.65, False, True), (180, 3, 4, 0.8, False, True), (181, 40, 16, 0.9, True, True),
    (300, 1, 8, 0.7, False, False), (301, 13, 3, 1.0, True, False)])
def test_long_rows(single, n, m, ne, density, cplx, diag):
    test_gpu_residual_rows.test_residual(single, n, m, ne, density, cplx, False, diag)
