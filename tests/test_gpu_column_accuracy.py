"""FP32 columns of 1024 and 2048 points are as accurate as rows of that length: the Laplacian of a field
and of its transpose exchange the two transforms (the other side, 512, is the same pass in both).  The
error of half a million white-noise values varies by well under a per cent from seed to seed; 5 % are
allowed between the two passes' ways of forming their twiddles."""
import numpy as np
import pytest

from oracle import fourier
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1024, 2048])
def test_columns_are_as_accurate_as_rows(n):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff
    f = np.random.default_rng(n).standard_normal((n, 512)).astype(np.float32).astype(np.float64)
    err = []
    for x in (f, np.ascontiguousarray(f.T)):
        p = pff.Problem(x.shape[1], x.shape[0], pff.MIXED)
        err.append(rel_l2(p.apply_laplacian(x), fourier.laplacian(x)))
        p.close()
    columns, rows = err
    assert columns <= 1.05 * rows
