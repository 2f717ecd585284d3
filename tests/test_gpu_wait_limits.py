"""Waits of the residue GEMM that run out with copies and MMAs under way: both CTAs of a pair learn of
it, wait for what is in flight, and return a status; the context then computes as before."""
import os

import numpy as np
import pytest
import torch

from paper_2212_12737_gb300 import build, gdml, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()
    yield
    gdml.test_set_wait_limit(None)


def timed_out(call):
    """Runs call(); whether a wait gave up."""
    try:
        call()
        return False
    except gdml.GdmlError as e:
        assert e.name == "ERR_TIMEOUT"
        return True


# fewer k-blocks than the ring's slots, and many times more, in one and several K groups
@pytest.mark.parametrize("N,M", [(6, 200), (12, 1500), (32, 700)])
def test_matvec_waits(N, M):
    R = torch.from_numpy(synth.geometries(synth.template(N, 1), M, 0.1, 2)).cuda()
    ctx = gdml.kernel_setup(R, 3.0, 1e-6, precision="ozaki")
    v = torch.from_numpy(np.random.default_rng(3).standard_normal(3 * N * M)).cuda()
    ref = ctx.matvec(v)
    ctx.tc_check()
    for polls in (1, 2, 4, 16, 64):
        gdml.test_set_wait_limit(polls)
        try:
            out = ctx.matvec(v)
            out_of_time = timed_out(ctx.tc_check)
        finally:
            gdml.test_set_wait_limit(None)
        assert out_of_time or torch.equal(out, ref)
        assert out_of_time or polls > 4  # a copy takes longer than a few polls
        assert torch.equal(ctx.matvec(v), ref)
        ctx.tc_check()
    ctx.destroy()


@pytest.mark.parametrize("tri", [False, True])
def test_build_product_waits(tri):
    rng = np.random.default_rng(4)
    A = torch.from_numpy(rng.standard_normal((3000, 900))).cuda()
    B = rng.standard_normal((900, 900))
    B = torch.from_numpy(np.tril(B) if tri else B).cuda()
    ref, _ = gdml.test_oz_gemm_tall(A, B, tri_b=tri)
    for polls in (1, 16):
        gdml.test_set_wait_limit(polls)
        try:
            out_of_time = timed_out(lambda: gdml.test_oz_gemm_tall(A, B, tri_b=tri))
        finally:
            gdml.test_set_wait_limit(None)
        assert out_of_time or polls > 4
        assert torch.equal(gdml.test_oz_gemm_tall(A, B, tri_b=tri)[0], ref)
