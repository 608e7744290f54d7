"""The one-sided Jacobi's launch shapes: pivots split over several CTAs, columns
kept in shared memory or streamed, partial chunks and column blocks."""
import numpy as np
import pytest

from oracle import lrr as olrr
from paper_1304_5583_gb300 import synth

pytestmark = pytest.mark.gpu

# (rows, cols): one column; one short of, at and past a pivot (32 columns in
# float32, 16 in float64); row counts around the 16-row slots and 64-row chunks;
# long columns that do not fit shared memory
SHAPES = [(1, 1), (5, 1), (17, 15), (16, 16), (33, 31), (32, 32), (31, 33), (64, 17), (65, 64), (63, 80), (200, 129),
          (1025, 33), (6001, 20)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_svt_at_edges_of_pivots_and_chunks(lib, shape, dtype):
    import torch
    from paper_1304_5583_gb300 import binding
    rows, cols = shape
    k = min(rows, cols)
    rng = np.random.default_rng(1000 * rows + cols)
    U = np.linalg.qr(rng.standard_normal((rows, k)))[0]
    V = np.linalg.qr(rng.standard_normal((cols, k)))[0]
    dt = np.float32 if dtype == "f32" else np.float64
    A = ((U * np.geomspace(1.0, 1e-3, k)) @ V.T).astype(dt)
    tau = 0.5 if k == 1 else 1e-2 * 1.07
    Jo, Uo, _, _ = olrr.svt(A.astype(np.float64), tau)
    J, rank = binding.svt(torch.from_numpy(np.asfortranarray(A)).cuda(), tau)
    assert rank == Uo.shape[1]
    # the bars of the stand-alone SVT: Jacobi tolerance 2e-6 / 1e-13 plus rounding
    tol = 5e-6 if dtype == "f32" else 1e-12
    assert np.linalg.norm(J.cpu().numpy() - Jo) <= tol * np.linalg.norm(Jo)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_svt_of_columns_that_reach_the_threshold_only_together(lib, dtype):
    """Every column (and every pair) below tau, the matrix above it."""
    import torch
    from paper_1304_5583_gb300 import binding
    dt = np.float32 if dtype == "f32" else np.float64
    rng = np.random.default_rng(5)
    u, v = rng.standard_normal(90), rng.choice([-1.0, 1.0], 100)
    A = (np.outer(u / np.linalg.norm(u), v / 10.0) + 1e-4 * rng.standard_normal((90, 100))).astype(dt)
    Jo, Uo, _, _ = olrr.svt(A.astype(np.float64), 0.3)          # columns of norm 0.1
    J, rank = binding.svt(torch.from_numpy(np.asfortranarray(A)).cuda(), 0.3)
    assert rank == Uo.shape[1] == 1
    assert np.linalg.norm(J.cpu().numpy() - Jo) <= (5e-6 if dtype == "f32" else 1e-12) * np.linalg.norm(Jo)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_many_blocks_agree_bitwise_with_one_block_at_a_time(lib, precision):
    """48 blocks at once (256-thread CTAs, streamed columns) against the same
    blocks one after another (512-thread CTAs, kept columns, split pivots)."""
    import torch
    from paper_1304_5583_gb300 import binding
    d = synth.union_of_subspaces(3, 90, 4, 4, 960, 0.05)
    perm, off = synth.column_partition(4, d.M.shape[1], 48, min_cols=60)
    M = torch.from_numpy(np.asfortranarray(d.M)).to(torch.float32 if precision == "f32" else torch.float64).cuda()
    res = [binding.dfc_lrr_solve(M, perm, off, binding.options(0.15, precision=precision, batched=b, max_iter=130),
                                 raise_on_error=False) for b in (True, False)]
    assert np.array_equal(res[0].sweeps, res[1].sweeps) and res[0].sweeps.sum() > 48
    assert torch.equal(res[0].Z, res[1].Z) and torch.equal(res[0].S, res[1].S)


# squared norms whose products leave the range (float32: below 1e-11 and above
# 4e9), at scales where the squares themselves stay well inside it
@pytest.mark.parametrize("dtype,scale", [("f32", 1e-14), ("f32", 1e-12), ("f32", 1e10), ("f32", 1e14),
                                         ("f64", 1e-120), ("f64", 1e-100), ("f64", 1e100)])
@pytest.mark.parametrize("kind", ["below the threshold one by one", "low rank"])
def test_svt_does_not_depend_on_the_scale_of_its_input(lib, dtype, scale, kind):
    import torch
    from paper_1304_5583_gb300 import binding
    dt = np.float32 if dtype == "f32" else np.float64
    rng = np.random.default_rng(5)
    if kind == "low rank":
        A = rng.standard_normal((90, 40)) @ rng.standard_normal((40, 100)) / 60.0
    else:
        u, v = rng.standard_normal(90), rng.choice([-1.0, 1.0], 100)
        A = np.outer(u / np.linalg.norm(u), v / 10.0) + 1e-4 * rng.standard_normal((90, 100))
    A = (A * scale).astype(dt)
    Jo, Uo, _, _ = olrr.svt(A.astype(np.float64), 0.3 * scale)
    J, rank = binding.svt(torch.from_numpy(np.asfortranarray(A)).cuda(), 0.3 * scale)
    assert rank == Uo.shape[1]
    # the bars of the stand-alone SVT (norms of the values over the scale: a
    # float64 norm squares them too)
    J, Jo = J.cpu().numpy().astype(np.float64) / scale, Jo / scale
    assert np.linalg.norm(J - Jo) <= (5e-6 if dtype == "f32" else 1e-12) * np.linalg.norm(Jo)


@pytest.mark.parametrize("shape", [(64, 64), (100, 120), (150, 400)], ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("low", [1e-6, 1e-10, 1e-14])
def test_float64_svt_of_graded_spectra(lib, shape, low):
    """Rotations in float32 between columns many orders apart."""
    import torch
    from paper_1304_5583_gb300 import binding
    rows, cols = shape
    k = min(rows, cols)
    rng = np.random.default_rng(rows + cols)
    U = np.linalg.qr(rng.standard_normal((rows, k)))[0]
    V = np.linalg.qr(rng.standard_normal((cols, k)))[0]
    s = np.geomspace(1.0, low, k)
    tau = np.sqrt(s[k // 2 - 1] * s[k // 2])           # keeps half of them
    J, rank = binding.svt(torch.from_numpy(np.asfortranarray((U * s) @ V.T)).cuda(), tau)
    assert rank == k // 2
    # the bar of the stand-alone SVT
    Jo = (U * np.maximum(s - tau, 0.0)) @ V.T
    assert np.linalg.norm(J.cpu().numpy() - Jo) <= 1e-12 * np.linalg.norm(Jo)
