"""Launches that start while the one before them drains (OZAKI matvec and apply outside capture, the
steps of Algorithm 1 with an FP32 factor) must give the bits of the same launches one after another.

Reference: a process of its own with CUDA_LAUNCH_BLOCKING=1, where no two kernels are ever under way
together.  Here the same calls run back to back on a stream of their own, each on other vectors than
the one before, with nothing in between, and once more replayed from a captured graph."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2212_12737_gb300 import gdml, synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NV, ROUNDS = 6, 5

# N, M, permutations of atoms 0..2, k: one and several K chunks; an apply in register-streamed passes
# (n % 4 != 0; odd and even k), staged passes with the separate k x k products (odd k)
SYSTEMS = [(9, 200, False, 101), (15, 777, False, 77), (13, 333, False, 64), (21, 1000, False, 0), (9, 151, True, 0)]

# Algorithm 1: N, M, k, precision (steps of one and several chunks of rows; k = n, where the residual
# diagonal ends and the remaining steps return at once)
BUILDS = [(9, 200, 400, "ozaki"), (21, 400, 600, "ozaki"), (9, 100, 200, "df64"), (4, 8, 96, "ozaki")]


def context(N, M, sym, k, stream=None):
    perms = [[0, 1, 2], [0, 2, 1], [1, 0, 2], [1, 2, 0], [2, 0, 1], [2, 1, 0]]
    R = torch.from_numpy(synth.geometries(synth.template(N, 1), M, 0.05, 2)).cuda()
    torch.cuda.synchronize()
    ctx = gdml.kernel_setup(R, 10.0, 1e-3, "ozaki", stream=stream,
                            perms=[p + list(range(3, N)) for p in perms] if sym else None)
    if k:
        ctx.precond_build("uniform", k, seed=3)
    return ctx


def vectors(n):
    return torch.from_numpy(np.random.default_rng(n).standard_normal((NV, n))).cuda()


def build(N, M, k, precision, stream=None):
    R = torch.from_numpy(synth.geometries(synth.template(N, 1), M, 0.05, 2)).cuda()
    torch.cuda.synchronize()
    ctx = gdml.kernel_setup(R, 10.0, 1e-3, precision, stream=stream)
    piv, trace = ctx.precond_build("pivchol", k, pivots=True, trace=True)
    out = dict(piv=piv.cpu().numpy(), trace=trace.cpu().numpy(), L=ctx.precond_factor().cpu().numpy())
    ctx.destroy()
    return out


def serial(path):
    """What the reference process computes."""
    out = {}
    for s, (N, M, sym, k) in enumerate(SYSTEMS):
        ctx = context(N, M, sym, k)
        for i, v in enumerate(vectors(3 * N * M)):
            out[f"mv{s}_{i}"] = ctx.matvec(v).cpu().numpy()
            if k:
                out[f"ap{s}_{i}"] = ctx.precond_apply(v).cpu().numpy()
        ctx.destroy()
    for b, args in enumerate(BUILDS):
        out.update({f"build{b}_{k}": v for k, v in build(*args).items()})
    np.savez(path, **out)


@pytest.fixture(scope="module")
def reference(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_12737_gb300 import build
    if not os.path.exists(build.LIB):
        build.build()
    path = str(tmp_path_factory.mktemp("serial") / "ref.npz")
    code = f"import sys; sys.path[:0] = [{ROOT!r}, {os.path.dirname(os.path.abspath(__file__))!r}]; " \
           f"import test_gpu_overlap as t; t.serial({path!r})"
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, env=dict(os.environ, CUDA_LAUNCH_BLOCKING="1"))
    return np.load(path)


@pytest.mark.parametrize("s", range(len(SYSTEMS)))
def test_calls_in_a_row_equal_serial_launches(reference, s):
    N, M, sym, k = SYSTEMS[s]
    st = torch.cuda.Stream()
    ctx = context(N, M, sym, k, st)
    V = vectors(3 * N * M)
    kv = torch.empty(ROUNDS, *V.shape, dtype=V.dtype, device="cuda")
    pv = torch.empty_like(kv)
    torch.cuda.synchronize()
    for r in range(ROUNDS):
        for i in range(NV):
            ctx.matvec(V[i], out=kv[r, i])
            if k:
                ctx.precond_apply(V[i], out=pv[r, i])
    torch.cuda.synchronize()
    for r in range(ROUNDS):
        for i in range(NV):
            assert np.array_equal(kv[r, i].cpu().numpy(), reference[f"mv{s}_{i}"])
            if k:
                assert np.array_equal(pv[r, i].cpu().numpy(), reference[f"ap{s}_{i}"])
    v, a, b = V[0].clone(), kv[0, 0], pv[0, 0]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st, capture_error_mode="relaxed"):
        ctx.matvec(v, out=a)
        if k:
            ctx.precond_apply(v, out=b)
    for i in range(NV):
        v.copy_(V[i])
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(a.cpu().numpy(), reference[f"mv{s}_{i}"])
        if k:
            assert np.array_equal(b.cpu().numpy(), reference[f"ap{s}_{i}"])
    ctx.destroy()


@pytest.mark.parametrize("b", range(len(BUILDS)))
def test_algorithm_1_equals_serial_launches(reference, b):
    for r in range(ROUNDS):
        for name, got in build(*BUILDS[b], torch.cuda.Stream()).items():
            assert np.array_equal(got, reference[f"build{b}_{name}"]), (r, name)
