"""The residue-number matvec of OZAKI contexts (gdml_matvec; the sliced form remains behind
gdml_set_inner_levels).  Its products are exact, so the error is the rounding of the float pairs
around them: w, t, beta, u, the terms g u and their sums, each 2^-48 relative, and the operands'
rounding to 2^-57 of their row's norm.  Bound: 8 roundings of 2^-48, plus the FP64 oracle's own
16 eps, in the 2-norm.

Sizes: one and several 512-entry K chunks with ragged ends (D and M), row tiles of 256 and column
tiles with a remainder, odd and even D and M, descriptor counts on both sides of the tile widths,
and the forms of the beta kernel (a row in shared memory, formed twice) and of U (one and several
K slabs)."""
import itertools

import numpy as np
import pytest
import torch

from oracle import kernel as ok
from paper_2212_12737_gb300 import gdml, synth

pytestmark = pytest.mark.gpu
BOUND = 8 * 2.0 ** -48 + 16 * np.finfo(float).eps


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


def geoms(N, M, seed=5):
    return synth.geometries(synth.template(N, seed), M, 0.1, seed + 1)


def rel(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("N,M", [(2, 1), (3, 2), (5, 255), (5, 256), (6, 257), (12, 511), (12, 513), (23, 64),
                                 (32, 65), (33, 33), (46, 40), (17, 1025)])
def test_residue_matvec_edges(N, M):
    R = geoms(N, M)
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki")
    v = np.random.default_rng(N * M).standard_normal(R.size)
    got = ctx.matvec(dev(v)).cpu().numpy()
    ctx.tc_check()
    ctx.destroy()
    err = rel(got, ok.matvec(R, 3.0, v, 1e-6))
    print(f"N={N} M={M} D={N * (N - 1) // 2}: {err:.2e}")
    assert err <= BOUND


def test_residue_matvec_keeps_small_blocks_beside_large_ones():
    """v spans 1e-30 .. 1e30 over the geometries: the largest entries decide the result's norm."""
    R = geoms(9, 150)
    v = np.random.default_rng(1).standard_normal((150, 27)) * 10.0 ** np.linspace(-30, 30, 150)[:, None]
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki")
    got = ctx.matvec(dev(v.reshape(-1)), add_lambda=False).cpu().numpy()
    zero = ctx.matvec(dev(np.zeros(R.size))).cpu().numpy()
    ctx.destroy()
    assert rel(got, ok.matvec(R, 3.0, v.reshape(-1), 0.0)) <= BOUND
    assert np.all(zero == 0.0)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_bad_entry_reaches_every_output(bad):
    """K is dense: a NaN or an infinity in v leaves no finite entry, and the next call is clean."""
    R = geoms(6, 300)
    v = np.random.default_rng(2).standard_normal(R.size)
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki")
    ref = ctx.matvec(dev(v))
    w = v.copy()
    w[1000] = bad
    assert not torch.isfinite(ctx.matvec(dev(w))).any()
    assert torch.equal(ctx.matvec(dev(v)), ref)
    ctx.destroy()


def test_k_groups_do_not_change_the_result():
    """The residues are exact whatever the grouping of the K chunks."""
    R = geoms(21, 1300)
    v = dev(np.random.default_rng(3).standard_normal(R.size))
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki")
    ref = ctx.matvec(v).clone()
    for choice in (1 * 65536 + 1, 1 * 65536 + 2, 1 * 65536 + 6):
        gdml.load().gdml_set_tuning(ctx._h, choice)
        assert torch.equal(ctx.matvec(v), ref)
    ctx.destroy()


@pytest.mark.parametrize("M", [210, 420])
def test_long_training_side(M):
    """All 120 permutations of 5 atoms: rows of 25,200 and 50,400 columns (beta formed twice; U's K
    longer than one unit takes)."""
    R = geoms(5, M)
    perms = [list(p) for p in itertools.permutations(range(5))]
    ctx = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="ozaki", perms=perms)
    f64 = gdml.kernel_setup(dev(R), 3.0, 1e-6, precision="fp64", perms=perms)
    v = dev(np.random.default_rng(M).standard_normal(R.size))
    got, ref = ctx.matvec(v).cpu().numpy(), f64.matvec(v).cpu().numpy()
    ctx.tc_check()
    ctx.destroy()
    f64.destroy()
    assert rel(got, ref) <= BOUND


@pytest.mark.parametrize("N,M,k", [(5, 40, 1), (9, 60, 33), (9, 100, 255), (9, 100, 257), (8, 64, 520), (9, 650, 20)])
def test_woodbury_core_from_residue_products(N, M, k):
    """The core C = lambda I + L^T L of a built preconditioner by residue products (one tile, the
    tiles' edges, three rows of tiles, K in groups, two K panels), through the apply
    z = (r - L C^-1 L^T r) / lambda against FP64 with the same stored L.  C's entries err by about
    2^-50 |L|^2, the apply's double-float sums by 2^-46: 2^6 2^-46 cond(C) bounds z's relative error."""
    R = torch.from_numpy(synth.geometries(synth.template(N, 2), M, 0.1, 3)).cuda()
    r = np.random.default_rng(k).standard_normal(3 * N * M)
    ctx = gdml.kernel_setup(R, 3.0, 1e-3, precision="ozaki")
    ctx.precond_build("uniform", k, seed=1)
    L = ctx.precond_factor().cpu().numpy()
    z = ctx.precond_apply(torch.from_numpy(r).cuda()).cpu().numpy()
    ctx.destroy()
    C = L.T @ L + 1e-3 * np.eye(L.shape[1])
    ref = (r - L @ np.linalg.solve(C, L.T @ r)) / 1e-3
    rel = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    assert rel <= 2.0 ** -40 * np.linalg.cond(C)
