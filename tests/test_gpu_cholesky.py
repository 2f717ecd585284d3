"""The blocked Cholesky.  Its failure report at every kind of column: first and last of a step of 32, of a
block of 128, one whose neighbours in the step fail as well (the report is of the first), and a NaN.  And
its quotients: a panel whose entries are integers over the pivots comes out exactly."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2212_12737_gb300 import build, gdml

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()


def reported(A):
    with pytest.raises(gdml.GdmlError) as e:
        gdml.test_cholesky_jitter(torch.from_numpy(A).cuda())
    assert e.value.name == "ERR_NOT_SPD"
    return int(re.search(r"column (\d+)", str(e.value)).group(1))


@pytest.mark.parametrize("bad", [0, 1, 30, 31, 32, 33, 127, 128, 159, 160, 198, 199])
def test_the_failing_column_is_reported(bad):
    A = np.eye(200)
    A[bad, bad] = -1.0  # tr/k > 0: every jitter is tried
    assert reported(A) == bad
    A[bad:, bad:] = -np.eye(200 - bad)  # every later column would fail too
    for _ in range(20):
        assert reported(A) == bad
    A = np.eye(200)
    A[199, 199] = -1e9  # tr <= 0: no retry
    if bad < 199:
        A[bad, bad] = np.nan
        assert reported(A) == bad


@pytest.mark.parametrize("k", [64, 200])
def test_quotients_are_rounded_as_divisions(k):
    """A = L L^T with a diagonal first step of 32 pivots whose reciprocals are not exact, and integers below
    it: every entry of A is exact, and so is each quotient of the panel (49 times the rounded 1/49 is not 1)."""
    rng = np.random.default_rng(k)
    L = np.zeros((k, k))
    L[:32, :32] = np.diag(rng.permutation(np.arange(3, 99, 3) + 46))  # 49, 52, ...
    L[32:, :32] = rng.integers(-50, 51, (k - 32, 32))
    L[32:, :32][:5] = 1
    L[32:, 32:] = np.eye(k - 32)
    A = L @ L.T + np.diag(np.r_[np.zeros(32), np.full(k - 32, 1e6)])
    got, eps = gdml.test_cholesky_jitter(torch.from_numpy(A).cuda())
    assert eps == 0.0
    assert np.array_equal(got.cpu().numpy()[:, :32], L[:, :32])
