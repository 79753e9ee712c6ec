"""Diagnostics on boxes with more columns (nx nz > 2^14) around the spans where the
number of threads per column changes, against FP64 sums over the state."""
import pytest

import test_gpu_diag_columns as columns

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("storage", [columns.lbm.LBM_FP32, columns.lbm.LBM_FP16S])
@pytest.mark.parametrize("kind", columns.KINDS)
@pytest.mark.parametrize("shape", [(128, 3, 128), (129, 1, 128), (16385, 2, 1), (2, 3, 8200),
                                   (129, 7, 128), (130, 8, 127), (129, 15, 128), (130, 16, 127),
                                   (129, 23, 128), (130, 24, 127), (129, 47, 128),
                                   (130, 48, 127)])
def test_diagnostics_against_fp64(shape, kind, storage, odd):
    columns.test_diagnostics_against_fp64(shape, kind, storage, odd)
