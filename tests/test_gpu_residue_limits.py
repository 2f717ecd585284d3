"""The residue matvec where its integer sums are longest: U's K runs over the MB = M S rows of the
training side in chunks of 512 entries, each adding a residue + 256 (at most 437) to a 16-bit sum, so
more than 149 chunks (MB > 76,288) take more than one such sum.

Reference: the FP64 context of the same system.  Bound in the 2-norm: 8 roundings of 2^-48 (the float
pairs around the exact products) and, for the FP64 sums of 2 MB terms on the other side,
(16 + sqrt(2 MB)) eps.  A lost carry moves an entry by a multiple of P / p_i, far above the result."""
import itertools

import numpy as np
import pytest
import torch

from paper_2212_12737_gb300 import gdml, synth

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    from paper_2212_12737_gb300 import build
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def rel(got, ref):
    return float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref))


def swaps(pairs, N):
    """The group generated by exchanging the two atoms of each of the first `pairs` pairs."""
    out = []
    for on in itertools.product((0, 1), repeat=pairs):
        s = list(range(N))
        for i, b in enumerate(on):
            if b:
                s[2 * i], s[2 * i + 1] = 2 * i + 1, 2 * i
        out.append(s)
    return out


# 120 permutations, random data: 149 chunks, one more, and well past the 255 at which even residues of
# zero no longer fit; 128 permutations of equal geometries and equal parts of v: every chunk adds the
# same residues, which no longer fit from 150 chunks on
@pytest.mark.parametrize("M,equal", [(635, False), (640, False), (1100, False), (1280, False), (596, True), (800, True)])
def test_more_chunks_than_a_16_bit_sum_holds(M, equal):
    if equal:
        N, perms = 14, swaps(7, 14)
        R = np.repeat(synth.geometries(synth.template(N, 5), 1, 0.1, 6), M, axis=0)
        v = np.tile(np.random.default_rng(M).standard_normal(3 * N), M)
    else:
        N, perms = 5, [list(p) for p in itertools.permutations(range(5))]
        R = synth.geometries(synth.template(N, 5), M, 0.1, 6)
        v = np.random.default_rng(M).standard_normal(R.size)
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki", perms=perms)
    got = ctx.matvec(dev(v))
    ctx.tc_check()
    ctx.destroy()
    f64 = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="fp64", perms=perms)
    ref = f64.matvec(dev(v))
    f64.destroy()
    err = rel(got, ref)
    MB = M * len(perms)
    print(f"M={M} S={len(perms)} chunks={-(-MB // 512)}: {err:.2e}")
    assert err <= 8 * 2.0 ** -48 + (16 + np.sqrt(2 * MB)) * EPS


@pytest.mark.parametrize("N,M", [(5, 16001), (3, 12800)])
def test_panels_of_rows(N, M):
    """T, beta and U of more rows than one panel holds (the last panel ragged), against FP64."""
    R = dev(synth.geometries(synth.template(N, 5), M, 0.1, 6))
    v = dev(np.random.default_rng(M).standard_normal(3 * N * M))
    ctx = gdml.kernel_setup(R, 3.0, 1e-6, precision="ozaki")
    got, again = ctx.matvec(v), ctx.matvec(v)
    ctx.tc_check()
    ctx.destroy()
    f64 = gdml.kernel_setup(R, 3.0, 1e-6, precision="fp64")
    ref = f64.matvec(v)
    f64.destroy()
    err = rel(got, ref)
    print(f"N={N} M={M}: {err:.2e}")
    assert torch.equal(got, again)
    assert err <= 8 * 2.0 ** -48 + (16 + np.sqrt(2 * M)) * EPS


def test_memory_per_pair_of_geometries():
    """A plain context of short descriptors holds 76 bytes per pair of geometries at most (the sliced
    form's), so that one of 60,000 geometries fits the card."""
    N, M = 4, 36000
    R = dev(synth.geometries(synth.template(N, 5), M, 0.1, 6))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    ctx = gdml.kernel_setup(R, 3.0, 1e-6, precision="ozaki")
    held = before - torch.cuda.mem_get_info()[0]
    ctx.destroy()
    print(f"{held / M ** 2:.1f} bytes per pair")
    assert held <= 76 * M * M + 2 ** 28


def test_reduced_levels_where_both_forms_do_not_fit():
    """The sliced operands of reduced levels take the residues' place when the device has no room for both:
    matvec, solve and autotuner go on, and back at 7 levels the matvec is FP64-class."""
    N, M = 6, 8000  # residues: 2.3 GB, T, beta and U 3.6 GB; slices: 2.8 GB
    tmpl = synth.template(N, 5)
    Rh = synth.geometries(tmpl, M, 0.1, 6)
    R, y = dev(Rh), dev(synth.morse_forces(Rh, tmpl).reshape(-1))
    v = dev(np.random.default_rng(7).standard_normal(Rh.size))
    ctx = gdml.kernel_setup(R, 3.0, 1.0, precision="ozaki")
    ref = ctx.matvec_fp64(v)
    before = ctx.matvec(v)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 29), dtype=torch.uint8, device="cuda")
    ctx.set_inner_levels(5)
    bound = 8 * 2.0 ** -48 + (16 + np.sqrt(2 * M)) * EPS
    after = ctx.matvec(v)
    assert rel(before, ref) <= bound and rel(after, ref) <= bound
    alpha, _, res, _ = ctx.pcg_solve(y, rtol=1e-8)
    assert res <= 1e-8
    ctx.set_inner_levels(7)
    ctx.autotune()
    assert rel(ctx.matvec(v), ref) <= bound
    r = y - ctx.matvec_fp64(alpha)
    assert torch.linalg.norm(r) <= 2e-8 * torch.linalg.norm(y)
    ctx.tc_check()
    ctx.destroy()
    del fill
    torch.cuda.empty_cache()
