"""Many kernel columns at once in double-float: warps of 64 columns, CTAs of 128 with one or two
geometries, launches of 2,048, and their remainders (the columns' accuracy: test_nystrom_factor_matches_oracle)."""
import os

import numpy as np
import pytest
import torch

from oracle import kernel as ok
from paper_2212_12737_gb300 import build, gdml, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("N,M", [(2, 9), (5, 7), (9, 33), (21, 12), (8, 100)])
def test_all_columns_through_the_full_factor(N, M):
    """All n = 54 .. 2,400 columns (odd counts of geometries, remainders of 64 and 128 columns, one and
    two geometries per CTA, a second launch): the full eigendecomposition's factor gives K back, to the
    FP32 storage of L (2^-23 of its rows' norms, twice)."""
    R = synth.geometries(synth.template(N, 4), M, 0.1, 6)
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="df64")
    ctx.precond_build("svd", 3 * N * M)
    L = ctx.precond_factor().cpu().numpy()
    ctx.destroy()
    K = ok.force_kernel_dense(R, 3.0)
    s = np.linalg.norm(L, axis=1)
    assert np.all(np.abs(L @ L.T - K) <= 2.0 ** -22 * np.outer(s, s))
