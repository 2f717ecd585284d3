"""Contexts of different sizes used by several host threads, each on a stream of its own: the kernels'
shared-memory limits belong to the device and are only ever raised, so no call loses what another one
was granted."""
import os
import threading

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


# rows of the back-projection of 116, 57 and 68 KB of shared memory (48 need no leave)
@pytest.mark.parametrize("precision", ["ozaki", "fp64"])
def test_threads_with_different_shared_memory(precision):
    jobs = []
    for N, M in ((100, 20), (70, 24), (76, 9)):
        st = torch.cuda.Stream()
        R = torch.from_numpy(synth.geometries(synth.template(N, 1), M, 0.05, 2)).cuda()
        v = torch.from_numpy(np.random.default_rng(N).standard_normal(3 * N * M)).cuda()
        torch.cuda.synchronize()
        ctx = gdml.kernel_setup(R, 10.0, 1e-6, precision, stream=st)
        ref = ctx.matvec(v)
        torch.cuda.synchronize()
        jobs.append((ctx, v, ref, []))
    go = threading.Barrier(len(jobs))

    def work(ctx, v, ref, failures):
        out = torch.empty_like(ref)
        go.wait()
        try:
            for _ in range(300):
                ctx.matvec(v, out=out)
            ctx.stream.synchronize()
            if not torch.equal(out, ref):
                failures.append("result")
        except gdml.GdmlError as e:
            failures.append(str(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [j[3] for j in jobs] == [[]] * len(jobs)
    for j in jobs:
        j[0].destroy()
