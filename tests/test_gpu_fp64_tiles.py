"""FP64 products at the edges of their tiles: force prediction over the tile sizes (16, 32, 64) and K groups."""
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


@pytest.mark.parametrize("N,M,Q", [(3, 5, 1), (12, 300, 2), (12, 300, 17), (21, 400, 64), (9, 33, 700)])
def test_predicted_forces(N, M, Q):
    tmpl = synth.template(N, 3)
    R, Rq = synth.geometries(tmpl, M, 0.1, 4), synth.geometries(tmpl, Q, 0.2, 5)
    alpha = np.random.default_rng(Q).standard_normal(R.size)
    ctx = gdml.kernel_setup(dev(R), 4.0, 1e-8)
    f = ctx.predict_forces(dev(Rq), dev(alpha)).cpu().numpy()
    ctx.destroy()
    ref = ok.predict_forces(Rq, R, 4.0, alpha)
    assert np.linalg.norm(f - ref) <= 1e-12 * np.linalg.norm(ref)
