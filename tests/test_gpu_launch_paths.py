"""Paths that must not change a result: recorded chunks of iterations against
direct launches, the Jacobi with and without its clusterless workspace, several
host threads at once; and the products' and the factor's edges."""
import ctypes
import threading

import numpy as np
import pytest

from oracle import lrr as olrr
from paper_1304_5583_gb300 import synth

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _dev(M, precision):
    import torch
    return torch.from_numpy(np.asfortranarray(M)).to(torch.float64 if precision == "f64" else torch.float32).cuda()


@pytest.mark.parametrize("precision", ["f32", "mixed", "f64"])
def test_recorded_iterations_equal_direct_launches(lib, precision):
    """profile=True launches every kernel by itself, otherwise chunks of iterations
    are recorded once and replayed."""
    import torch
    from paper_1304_5583_gb300 import binding
    w = synth.workload("small_dfc_60x240")
    M = _dev(w.M, precision)
    a, b = (binding.dfc_lrr_solve(M, w.perm, w.offsets, binding.options(w.lam, precision=precision, profile=p),
                                  raise_on_error=False) for p in (False, True))
    assert np.array_equal(a.iters, b.iters) and np.array_equal(a.sweeps, b.sweeps)
    assert torch.equal(a.Z, b.Z) and torch.equal(a.S, b.S)


@pytest.mark.parametrize("precision,cols", [("f64", 64), ("f64", 65), ("f64", 130), ("f32", 200)])
def test_smaller_workspace_leaves_out_the_clusterless_form_only(lib, precision, cols):
    """A workspace of the size without the Jacobi's clusterless part is still taken
    and gives the same bits."""
    import torch
    from paper_1304_5583_gb300 import binding
    d = synth.union_of_subspaces(7, 150, 3, 4, cols, 0.05)
    M = _dev(d.M, precision)
    n = M.shape[1]
    off = np.array([0, cols, 2 * cols, n], dtype=np.int64)
    perm = np.random.default_rng(1).permutation(n).astype(np.int64)
    o = binding.options(0.15, precision=precision, max_iter=120)
    full = binding.workspace_bytes(M, perm, off, o)
    ref = binding.dfc_lrr_solve(M, perm, off, o, raise_on_error=False)
    p, keep = binding._problem(M, perm, off)
    ws = torch.empty(full, dtype=torch.uint8, device="cuda")
    Z = torch.empty((n, n), dtype=M.dtype, device="cuda").t()
    r = binding.LrrResult()
    r.Z = ctypes.c_void_p(Z.data_ptr())
    code = lib.dfc_lrr_solve(ctypes.byref(p), ctypes.byref(o), ctypes.c_void_p(ws.data_ptr()), ctypes.c_size_t(full - 4096),
                             ctypes.byref(r), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code >= 0 and keep is not None
    assert torch.equal(Z, ref.Z)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_concurrent_svts_equal_one_alone(lib, dtype):
    """Shapes that take the clusterless form (a cooperative launch of most of the
    chip), from four host threads on streams of their own."""
    import torch
    from paper_1304_5583_gb300 import binding
    rows, cols = (1000, 487) if dtype == "f32" else (100, 500)
    rng = np.random.default_rng(3)
    A = _dev(rng.standard_normal((rows, 60)) @ rng.standard_normal((60, cols)) / 300.0, dtype)
    ref, rank = binding.svt(A, 0.1)
    got, errors = [None] * 4, []

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(3):
                    got[i] = binding.svt(A, 0.1)
                torch.cuda.current_stream().synchronize()
        except Exception as e:                                  # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=run, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for J, k in got:
        assert k == rank and torch.equal(J, ref)
    J, k = binding.svt(A, 0.1, no_alloc=True)
    assert k == rank and torch.equal(J, ref)


def test_mixed_blocks_one_at_a_time_equal_the_batch(lib):
    """Every block has its bf16 phase, also the ones after the first."""
    import torch
    from paper_1304_5583_gb300 import binding
    w = synth.workload("small_dfc_60x240")
    M = _dev(w.M, "mixed")
    a, b = (binding.dfc_lrr_solve(M, w.perm, w.offsets, binding.options(w.lam, precision="mixed", batched=x),
                                  raise_on_error=False) for x in (True, False))
    assert np.array_equal(a.iters, b.iters)
    assert torch.equal(a.Z, b.Z) and torch.equal(a.S, b.S)


# ragged against the 16, 32 and 64-wide tiles and 16-term slabs; blocks at and
# past the 64 columns that finish their SVT in one launch; one pivot of the
# factor's eigensolver, two, and a padded last one
@pytest.mark.parametrize("m,l", [(17, 15), (33, 31), (40, 64), (65, 65), (97, 130)])
def test_ragged_float64_lrr_matches_oracle(lib, m, l):
    from paper_1304_5583_gb300 import binding
    rng = np.random.default_rng(100 * m + l)
    k = max(2, m // 8)
    M = rng.standard_normal((m, k)) @ rng.standard_normal((k, l)) / np.sqrt(k) + 0.05 * rng.standard_normal((m, l))
    perm = np.arange(l, dtype=np.int64)
    res = binding.lrr_solve(_dev(M, "f64"), perm, binding.options(0.2, eps=1e-8, precision="f64"), raise_on_error=False)
    try:
        ref = olrr.lrr_alm(M, M, 0.2, eps=1e-8)
    except np.linalg.LinAlgError:
        pytest.skip("the host's LAPACK did not converge: no reference")
    assert res.status == 0 and res.iters[0] == ref.iters
    # the bar of the other float64 solves
    assert _rel(res.Z.cpu().numpy(), ref.Z) < 1e-8 and _rel(res.S.cpu().numpy(), ref.E) < 1e-8


@pytest.mark.parametrize("kind", ["repeated", "zero rows", "graded"])
def test_factor_of_awkward_spectra(lib, kind):
    """The factor's float64 rotations: equal diagonal entries (45 degree rotations),
    zero rows and columns, entries far below their diagonals."""
    from paper_1304_5583_gb300 import binding
    rng = np.random.default_rng(11)
    m, l = 72, 90
    Q = np.linalg.qr(rng.standard_normal((m, m)))[0]
    V = np.linalg.qr(rng.standard_normal((l, l)))[0][:, :m]
    s = {"repeated": np.repeat([2.0, 1.0, 0.5], 24), "zero rows": np.linspace(2, 1, m),
         "graded": np.geomspace(1, 1e-3, m)}[kind]
    M = (Q * s) @ V.T
    if kind == "zero rows":
        M[::3] = 0.0
    lam = 0.6 if kind == "zero rows" else 0.3          # (at 0.3 its Z is zero)
    res = binding.lrr_solve(_dev(M, "f64"), np.arange(l, dtype=np.int64),
                            binding.options(lam, eps=1e-8, precision="f64"), raise_on_error=False)
    ref = olrr.lrr_alm(M, M, lam, eps=1e-8)
    assert res.status == 0 and res.iters[0] == ref.iters
    assert _rel(res.Z.cpu().numpy(), ref.Z) < 1e-8 and _rel(res.S.cpu().numpy(), ref.E) < 1e-8


# at least a tile of 128 x 256 for every SM: pairs of CTAs (4, 14 and 6 rows of
# tiles, and 5 padded to 6) and single ones (3 rows)
@pytest.mark.parametrize("M,N,K", [(512, 10000, 72), (1700, 3001, 200), (641, 7000, 64), (600, 8000, 136),
                                   (300, 13100, 80)])
def test_bf16_product_in_clusters_matches_float64(lib, M, N, K):
    import torch
    from paper_1304_5583_gb300 import binding
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16)
    C = binding.gemm_bf16(A.cuda(), B.cuda(), M, N, K).cpu().numpy()
    ref = A.double().numpy() @ B.double().numpy().T
    # the bar of the other bf16 products: float32 accumulation order alone
    assert np.abs(C - ref).max() / np.abs(ref).max() < 2e-6


@pytest.mark.parametrize("dtype,rows,cols", [("f64", 90, 90), ("f64", 100, 500), ("f32", 1000, 487)])
def test_concurrent_svts_run_side_by_side(lib, dtype, rows, cols):
    """Eight threads' SVTs share the chip: one alone may spread over most of it, but
    eight that did so would run one after another, 8 times one thread's time."""
    import time

    import torch
    from paper_1304_5583_gb300 import binding
    rng = np.random.default_rng(4)
    A = _dev(rng.standard_normal((rows, 40)) @ rng.standard_normal((40, cols)) / 300.0, dtype)

    def work():
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(6):
                binding.svt(A, 0.05)

    def run(n):
        threads = [threading.Thread(target=work) for _ in range(n)]
        t0 = time.perf_counter()
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        return time.perf_counter() - t0

    torch.cuda.synchronize()
    run(8)
    alone, eight = min(run(1) for _ in range(3)), min(run(8) for _ in range(3))
    # eight blocks in clusters of 12 to 16 CTAs are resident at once; a cluster
    # takes up to twice a whole chip's time
    assert eight < 4 * alone, (alone, eight)
