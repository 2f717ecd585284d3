"""The blocked Cholesky's failure report at every kind of column: first and last of a step of 32, of a
block of 128, one whose neighbours in the step fail as well (the report is of the first), and a NaN."""
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
