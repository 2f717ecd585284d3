"""FP64 paths at the edges of their tiles: the blocked Cholesky (steps of 32 in blocks of 128), the
products' tile sizes (16, 32, 64) and K groups behind force prediction, and the two-launch
context-free matvec (geometries in 1 .. 16 groups, by the descriptor count)."""
import os

import numpy as np
import pytest
import torch

from oracle import kernel as ok
from paper_2212_12737_gb300 import build, gdml, synth

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("k", [1, 31, 32, 33, 96, 127, 128, 129, 161, 300])
def test_cholesky_backward_error(k):
    """|A - L L^T| <= (2 k + 8) eps |L| |L|^T entry by entry: the factorisation's k + 1 roundings and
    those of the pivot's root and reciprocal, and as many of the test's own product."""
    rng = np.random.default_rng(k)
    X = rng.standard_normal((k, k + 5))
    A = X @ X.T * 10.0 ** rng.uniform(-2, 2, size=(k, 1))
    A = (A + A.T) / 2 + k * 200.0 * np.eye(k)
    L, eps = gdml.test_cholesky_jitter(dev(A))
    L = L.cpu().numpy()
    assert eps == 0.0
    assert np.all(np.abs(np.tril(A - L @ L.T)) <= (2 * k + 8) * EPS * (np.abs(L) @ np.abs(L).T))


def test_cholesky_reports_the_failing_column_of_any_step():
    for bad in (0, 31, 32, 127, 128, 199):
        A = np.eye(200)
        A[bad, bad] = -1e9
        with pytest.raises(gdml.GdmlError) as e:
            gdml.test_cholesky_jitter(dev(A))
        assert e.value.name == "ERR_NOT_SPD"


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


@pytest.mark.parametrize("N,M", [(2, 128), (3, 1), (8, 9), (9, 100), (12, 33), (17, 64), (23, 128)])
def test_noalloc_groups(N, M):
    R = synth.geometries(synth.template(N, 7), M, 0.1, 8)
    v = np.random.default_rng(N).standard_normal(R.size)
    got = gdml.matvec_noalloc(dev(R), 3.0, 1e-6, dev(v)).cpu().numpy()
    ref = ok.matvec(R, 3.0, v, 1e-6)
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    plain = gdml.matvec_noalloc(dev(R), 3.0, 1e-6, dev(v), add_lambda=False).cpu().numpy()
    assert np.linalg.norm(got - plain - 1e-6 * v) <= 1e-12 * np.linalg.norm(ref)
