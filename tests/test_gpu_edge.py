"""GPU edge cases through the C ABI: empty and one-entry tensors, empty slices and rows, padded
leading dimensions, every compiled rank combination, fibers and rows around the split
thresholds, the SDDMM sampling pattern, run-to-run reproducibility and workspace errors."""
import numpy as np
import pytest

import oracle
from workloads import configs, rng
from util import TOL_FP32, assert_close, fmt_of, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sa():
    import torch
    assert torch.cuda.is_available()
    import paper_2311_09549_b200 as sa
    return sa


def _wl(expr, fmt, dims, coords, vals, dense, out_shape):
    return configs.Workload("edge", expr, fmt, tuple(dims), np.asarray(coords, np.int32).reshape(-1, len(dims)),
                            np.asarray(vals, np.float32), dense, tuple(out_shape), 0)


def _dense(seed, which, r, c):
    return configs.dense_uniform(seed, which, r, c)


def _random_coo(seed, dims, nnz):
    lin = rng.keyed_bijection(np.arange(nnz), int(np.prod(dims)), np.uint64(seed))
    coords = np.stack(np.unravel_index(lin, dims), axis=1).astype(np.int32)
    return coords, rng.uniform_f32(seed, 1, np.arange(nnz), -1.0, 1.0)


def _check(sa, w, sched=None, tol=TOL_FP32):
    A_ref, S_ref = oracle.evaluate(w)
    A, t = run_gpu(sa, w, sched=sched)
    assert_close(A, A_ref, S_ref, tol, w.expr)
    return A, t


@pytest.mark.parametrize("nnz", [0, 1])
def test_empty_and_single_entry_all_chains(sa, nnz):
    c3 = [[3, 2, 1]][:nnz]
    c4 = [[3, 2, 1, 0]][:nnz]
    c2 = [[3, 2]][:nnz]
    v = [0.5][:nnz]
    _check(sa, _wl("spttm_ttm3", "csf", (5, 4, 3), c3, v, [_dense(1, 0, 4, 16), _dense(1, 1, 3, 32)], (5, 16, 32)))
    _check(sa, _wl("spttm_ttm4", "csf", (5, 4, 3, 2), c4, v,
                   [_dense(1, 0, 4, 16), _dense(1, 1, 3, 16), _dense(1, 2, 2, 16)], (5, 16, 16, 16)))
    _check(sa, _wl("sddmm_spmm", "csr", (5, 4), c2, v, [_dense(1, 0, 5, 64), _dense(1, 1, 4, 64), _dense(1, 2, 4, 32)], (5, 32)))
    _check(sa, _wl("ttmc3", "csf", (5, 4, 3), c3, v, [_dense(1, 0, 5, 32), _dense(1, 1, 4, 16), _dense(1, 2, 3, 32)], (32, 16, 32)))
    _check(sa, _wl("sddmm_spmm_gemm", "csr", (5, 4), c2, v,
                   [_dense(1, 0, 5, 64), _dense(1, 1, 4, 64), _dense(1, 2, 4, 128), _dense(1, 3, 128, 32)], (5, 32)))
    w = _wl("spmm_gemm", "csr", (5, 4), c2, v, [_dense(1, 0, 4, 128), _dense(1, 1, 128, 32)], (5, 32))
    _check(sa, w, sched=sa.SA_SCHED_ASSOC_LEFT)
    _check(sa, w, sched=sa.SA_SCHED_ASSOC_RIGHT)
    _check(sa, _wl("spmmh_gemm", "csr", (5, 4), c2, v, [_dense(1, 0, 4, 128), _dense(1, 3, 4, 128), _dense(1, 1, 128, 32)], (5, 32)))


@pytest.mark.parametrize("L,M", [(16, 16), (16, 32), (32, 16), (32, 32)])
def test_ttm3_rank_combinations_with_empty_slices(sa, L, M):
    dims = (40, 37, 53)
    coords, vals = _random_coo(7, dims, 3000)
    keep = coords[:, 0] % 3 != 1                     # every third slice empty
    w = _wl("spttm_ttm3", "csf", dims, coords[keep], vals[keep], [_dense(2, 0, 37, L), _dense(2, 1, 53, M)], (40, L, M))
    A, _ = _check(sa, w)
    assert not A[1::3].any()


@pytest.mark.parametrize("M", [32, 64])
def test_mttkrp_gemm_empty_slices_and_split_slices(sa, M):
    # empty slices, small slices (several per warp task) and one slice large enough to be split over thread blocks
    dims = (40, 37, 530)
    coords, vals = _random_coo(9, dims, 400000)
    keep = (coords[:, 0] % 3 != 1) & ((coords[:, 0] == 5) | (np.arange(400000) % 40 == 0))
    w = _wl("mttkrp_gemm", "csf", dims, coords[keep], vals[keep],
            [_dense(5, 0, 37, 32), _dense(5, 1, 530, 32), _dense(5, 2, 32, M)], (40, M))
    A, t = _check(sa, w)
    assert not A[1::3].any()
    assert sa.sa_tensor_worklist(t.handle)[0][3] >= 2, "slice 5 must be split into chunks with partial rows"


def test_ttm3_one_slice_long_fibers_split_over_many_blocks(sa):
    # a single slice of 60 000 nonzeros in 12 fibers of 5000: pieces cut inside fibers, 8 partial tiles
    dims = (3, 12, 5000)
    j, k = np.divmod(np.arange(60000), 5000)
    coords = np.stack([np.full(60000, 1), j, k], axis=1)
    vals = rng.uniform_f32(3, 1, np.arange(60000), -1.0, 1.0)
    perm = rng.permutation(3, 3, 60000)
    w = _wl("spttm_ttm3", "csf", dims, coords[perm], vals[perm], [_dense(3, 0, 12, 32), _dense(3, 1, 5000, 32)], (3, 32, 32))
    A, t = _check(sa, w)
    counts, items, fix = sa.sa_tensor_worklist(t.handle)
    assert counts[3] >= 2 and not A[0].any() and not A[2].any()


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 32, 33, 63, 65, 2048, 2049, 8192, 8193, 16385])
def test_ttm3_ragged_sizes_around_batch_and_split_thresholds(sa, n):
    # one slice with n nonzeros in fibers of length 1, 2, 3, ... : hits batch tails, groups of 8
    # fibers, the one-warp / one-block / many-block boundaries
    lens = []
    while sum(lens) < n:
        lens.append(min(len(lens) % 11 + 1, n - sum(lens)))
    j = np.repeat(np.arange(len(lens)), lens)
    k = np.concatenate([np.arange(x) for x in lens])
    dims = (2, len(lens), 12)
    coords = np.stack([np.ones(n, np.int64), j, k], axis=1)
    vals = rng.uniform_f32(n, 1, np.arange(n), -1.0, 1.0)
    w = _wl("spttm_ttm3", "csf", dims, coords, vals, [_dense(4, 0, len(lens), 32), _dense(4, 1, 12, 32)], (2, 32, 32))
    _check(sa, w)


def test_padded_leading_dimensions(sa):
    import torch
    w = configs.make(1)
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSF, device=0)
    big = [torch.zeros(x.shape[0], x.shape[1] + 12, device="cuda") for x in w.dense]
    views = []
    for b, x in zip(big, w.dense):
        b[:, 4:4 + x.shape[1]] = torch.from_numpy(x).cuda()
        views.append(b[:, 4:4 + x.shape[1]])          # 16-byte aligned start, ld = cols + 12
    out, _ = t.run(w.expr, views)
    torch.cuda.synchronize()
    A_ref, S_ref = oracle.evaluate(w)
    assert_close(out.cpu().numpy().astype(np.float64), A_ref, S_ref, TOL_FP32, "padded ld")
    # a misaligned view is refused before anything is launched
    with pytest.raises(sa.SaError) as e:
        t.run(w.expr, [big[0][:, 1:17], views[1]])
    assert e.value.status == sa.SA_E_SHAPE


@pytest.mark.parametrize("K,L", [(k, l) for k in (32, 64, 128) for l in (32, 64, 128)])
def test_sddmm_spmm_ranks_long_rows_and_sampled_pattern(sa, K, L):
    import torch
    I, J = 300, 6000
    deg = np.zeros(I, dtype=np.int64)
    deg[5] = 5000                                      # cut into pieces with partial rows
    deg[6] = 1024                                      # exactly at the threshold: one item
    deg[10:200:3] = 17
    deg[299] = 1
    cols = configs.distinct_children(11, 2, deg, J)
    rows = np.repeat(np.arange(I), deg)
    vals = rng.uniform_f32(11, 1, np.arange(rows.shape[0]), 0.0, 1.0)
    perm = rng.permutation(11, 3, rows.shape[0])
    coords = np.stack([rows, cols], axis=1)[perm].astype(np.int32)
    vals = vals[perm]
    dense = [configs.dense_normal(11, 0, I, K), configs.dense_normal(11, 1, J, K), configs.dense_normal(11, 2, J, L)]
    w = _wl("sddmm_spmm", "csr", (I, J), coords, vals, dense, (I, L))
    A, t = _check(sa, w)
    assert not A[0].any() and not A[298].any()        # empty rows are +0
    # debug schedule: sampled values land exactly on B's stored coordinates, in CSR order
    ops = [torch.from_numpy(x).cuda() for x in dense]
    tuples = [(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0)) for x in ops]
    need = sa.sa_workspace_size(t.handle, sa.SA_EXPR_SDDMM_SPMM, sa.SA_SCHED_DEBUG_MATERIALIZE, tuples)
    ws = torch.full((need // 4,), float("nan"), device="cuda")
    out, _ = t.run(w.expr, ops, sched=sa.SA_SCHED_DEBUG_MATERIALIZE, workspace=ws.view(torch.uint8))
    torch.cuda.synchronize()
    nnz = vals.shape[0]
    sampled = ws[-(((nnz * 4 + 255) // 256) * 64):][:nnz].cpu().numpy().astype(np.float64)
    _, _, P = oracle.sddmm_spmm(coords, vals, (I, J), *dense, with_sampled=True)
    _, crd, _ = sa.sa_tensor_export(t.handle, 1, n_crd=nnz)
    order = np.lexsort((coords[:, 1], coords[:, 0]))   # CSR order of the input entries
    assert np.array_equal(coords[order, 1], crd)
    Sabs = np.abs(vals[order].astype(np.float64)) * (np.abs(dense[0][coords[order, 0]].astype(np.float64)) *
                                                     np.abs(dense[1][coords[order, 1]].astype(np.float64))).sum(axis=1)
    assert np.isfinite(sampled).all() and (np.abs(sampled - P[order]) <= TOL_FP32 * Sabs).all()
    assert_close(out.cpu().numpy().astype(np.float64), *oracle.evaluate(w), TOL_FP32, "materialize schedule output")


@pytest.mark.parametrize("L,M", [(128, 32), (128, 64), (256, 32)])
def test_spmm_gemm_rank_combinations_and_long_rows(sa, L, M):
    I, J = 500, 6000
    deg = np.full(I, 3, dtype=np.int64)
    deg[::7] = 0
    deg[123] = 2900
    deg[124] = 5000                                    # above the long-row threshold: pieces + fix-up
    cols = configs.distinct_children(12, 2, deg, J)
    rows = np.repeat(np.arange(I), deg)
    vals = rng.uniform_f32(12, 1, np.arange(rows.shape[0]), -1.0, 1.0)
    coords = np.stack([rows, cols], axis=1).astype(np.int32)
    w = _wl("spmm_gemm", "csr", (I, J), coords, vals,
            [configs.dense_normal(12, 0, J, L), configs.dense_normal(12, 1, L, M)], (I, M))
    _check(sa, w, sched=sa.SA_SCHED_ASSOC_LEFT)
    _check(sa, w, sched=sa.SA_SCHED_ASSOC_RIGHT)
    # kernel 3 on the same tensor: empty rows, long rows cut into pieces, every rank combination
    wh = _wl("spmmh_gemm", "csr", (I, J), coords, vals,
             [w.dense[0], configs.dense_normal(12, 2, J, L), w.dense[1]], (I, M))
    _check(sa, wh)


def test_ttm4_ragged_and_split_slices(sa):
    # few level-1 fibers per slice: the head slice's (i,j) subtrees are above the size the fused kernel evaluates
    # itself, so the order-3 kernel writes their temporaries first (some split over several thread blocks, with
    # partial temporaries that the fix-up kernel sums) and items of kind 1 copy them into the pool
    w = configs.make_ttm4_zipf("edge4", 31, 90, 6, 130, 110, 150_000, 1.4, 5.0, 16, 16, 16)
    A, t = _check(sa, w, sched=sa.SA_SCHED_FUSED)
    assert sa.sa_tensor_worklist(t.handle, 0)[0][3] >= 2, "a large (i,j) subtree must be split over several thread blocks"
    kinds = sa.sa_tensor_worklist(t.handle, 2)[1][:, 7]
    assert (kinds == 1).any() and (kinds == 0).any()
    # many level-1 fibers per slice: the head slices span several pieces and leave partial slice tiles
    w = configs.make_ttm4_zipf("edge4b", 32, 90, 700, 50, 45, 150_000, 1.4, 5.0, 16, 16, 16)
    A, t = _check(sa, w, sched=sa.SA_SCHED_FUSED)
    assert sa.sa_tensor_worklist(t.handle, 1)[0][3] >= 2, "the head slice must be split into several pieces"
    # subtrees with more level-2 fibers than one batch holds next to small ones
    for w in (configs.make_ttm4_zipf("edge4c", 33, 90, 40, 160, 110, 150_000, 1.4, 5.0, 16, 16, 16),
              configs.make_ttm4_zipf("edge4d", 34, 400, 60, 150, 40, 200_000, 1.2, 3.0, 16, 16, 16)):
        A, t = _check(sa, w, sched=sa.SA_SCHED_FUSED)
        items = sa.sa_tensor_worklist(t.handle, 2)[1]
        nf = items[:, 3] - items[:, 2]
        assert ((items[:, 7] == 0) & (nf > 32)).any() and ((items[:, 7] == 0) & (nf <= 32) & (items[:, 1] - items[:, 0] > 1)).any()


def test_ttm4_fissioned_ragged_and_split_slices(sa):
    """The same tensors through the two-pass schedule (temporaries of all (i,j) subtrees in the workspace)."""
    F = sa.SA_SCHED_FISSIONED
    # few level-1 fibers per slice: the head slice's (i,j) subtrees exceed one thread block's chunk, so the
    # first pass writes partial temporaries that the fix-up kernel sums
    w = configs.make_ttm4_zipf("edge4", 31, 90, 6, 130, 110, 150_000, 1.4, 5.0, 16, 16, 16)
    A, t = _check(sa, w, sched=F)
    assert sa.sa_tensor_worklist(t.handle, 4)[0][3] >= 2, "a large (i,j) subtree must be split over several thread blocks"
    # many level-1 fibers per slice: the second pass cuts the head slices into pieces of 512 fibers
    w = configs.make_ttm4_zipf("edge4b", 32, 90, 700, 50, 45, 150_000, 1.4, 5.0, 16, 16, 16)
    A, t = _check(sa, w, sched=F)
    assert sa.sa_tensor_worklist(t.handle, 5)[0][3] >= 2, "the head slice must be split into several pieces"
    # both kernels of the first pass in one run: small subtrees (list 6) and large ones (list 4)
    for w in (configs.make_ttm4_zipf("edge4c", 33, 90, 40, 160, 110, 150_000, 1.4, 5.0, 16, 16, 16),
              configs.make_ttm4_zipf("edge4d", 34, 400, 60, 150, 40, 200_000, 1.2, 3.0, 16, 16, 16)):
        A, t = _check(sa, w, sched=F)
        n_main, n_sub = (int(sa.sa_tensor_worklist(t.handle, x)[0][0]) for x in (4, 6))
        assert n_main > 0 and n_sub > 0, (n_main, n_sub)


def test_results_are_reproducible_run_to_run(sa):
    w = configs.make(2, "mini")
    A1, t = run_gpu(sa, w)
    A2, _ = run_gpu(sa, w, tensor=t)
    assert np.array_equal(A1, A2)


def test_workspace_errors_enqueue_nothing(sa):
    import torch
    w = configs.make(2, "mini")
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSF, device=0)
    ops = [torch.from_numpy(x).cuda() for x in w.dense]
    tuples = [(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0)) for x in ops]
    need = sa.sa_workspace_size(t.handle, sa.SA_EXPR_SPTTM_TTM3, sa.SA_SCHED_DEFAULT, tuples)
    assert need > 0
    out = torch.zeros(w.out_shape, device="cuda")
    small = torch.empty(need - 256, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for ws_ptr, ws_bytes in [(small.data_ptr(), small.numel()), (None, 0), (small.data_ptr() + 16, need)]:
        with pytest.raises(sa.SaError) as e:
            sa.sa_run(t.handle, sa.SA_EXPR_SPTTM_TTM3, sa.SA_SCHED_DEFAULT, tuples, out.data_ptr(), ws_ptr, ws_bytes, s)
        assert e.value.status == sa.SA_E_WORKSPACE
    torch.cuda.synchronize()
    assert not out.any()
    assert sa.sa_last_device_status(t.handle, s) == sa.SA_OK


@pytest.mark.parametrize("L,M", [(32, 32), (32, 64), (64, 32), (64, 64)])
@pytest.mark.parametrize("sched", ["left", "right"])
def test_spttm_spttm_ranks_long_fibers_and_empty_slices(sa, L, M, sched):
    # short fibers, empty slices, and one fiber of 9000 nonzeros that is cut into pieces with partial rows
    dims = (40, 37, 9500)
    coords, vals = _random_coo(11, dims, 6000)
    keep = coords[:, 0] % 3 != 1
    longf = np.stack([np.full(9000, 6), np.full(9000, 3), np.arange(9000)], axis=1).astype(np.int32)
    keep &= ~((coords[:, 0] == 6) & (coords[:, 1] == 3))
    c = np.concatenate([coords[keep], longf])
    v = np.concatenate([vals[keep], rng.uniform_f32(12, 1, np.arange(9000), -1.0, 1.0)])
    perm = rng.permutation(13, 3, c.shape[0])
    keys, _ = oracle.fiber_keys(c, dims)
    w = _wl("spttm_spttm", "csf", dims, c[perm], v[perm], [_dense(6, 0, 9500, L), _dense(6, 1, L, M)], (keys.shape[0], M))
    s = sa.SA_SCHED_ASSOC_LEFT if sched == "left" else sa.SA_SCHED_ASSOC_RIGHT
    A, t = _check(sa, w, sched=s)
    assert A.shape == (keys.shape[0], M)
    assert sa.sa_tensor_worklist(t.handle, 1)[0][3] >= 1, "the long fiber must be split into pieces with partial rows"


@pytest.mark.parametrize("nnz", [0, 1])
def test_spttm_spttm_empty_and_single_entry(sa, nnz):
    w = _wl("spttm_spttm", "csf", (5, 4, 3), [[3, 2, 1]][:nnz], [0.5][:nnz], [_dense(1, 0, 3, 32), _dense(1, 1, 32, 64)], (nnz, 64))
    for s in (sa.SA_SCHED_ASSOC_LEFT, sa.SA_SCHED_ASSOC_RIGHT):
        A, _ = _check(sa, w, sched=s)
        assert A.shape == (nnz, 64)


@pytest.mark.parametrize("L,M", [(128, 32), (128, 64), (256, 32), (256, 64)])
def test_dense_stage_ragged_rows_and_padded_leading_dimensions(sa, L, M):
    """B.(C.D) with a number of columns J that is not a multiple of the dense stage's 128-row tile (the last
    tile is ragged, several tiles per thread block) and with C and D given as padded views."""
    import torch
    I, J = 700, 148 * 128 * 2 + 77
    coords, vals = _random_coo(21, (I, J), 30_000)
    C, D = configs.dense_normal(21, 0, J, L), configs.dense_normal(21, 1, L, M)
    w = _wl("spmm_gemm", "csr", (I, J), coords, vals, [C, D], (I, M))
    A_ref, S_ref = oracle.evaluate(w)
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR, device=0)
    bigC = torch.zeros(J, L + 8, device="cuda")
    bigD = torch.zeros(L, M + 4, device="cuda")
    bigC[:, 4:4 + L] = torch.from_numpy(C).cuda()
    bigD[:, :M] = torch.from_numpy(D).cuda()
    out, _ = t.run("spmm_gemm", [bigC[:, 4:4 + L], bigD[:, :M]], sched=sa.SA_SCHED_ASSOC_RIGHT)
    torch.cuda.synchronize()
    assert sa.sa_last_device_status(t.handle, torch.cuda.current_stream().cuda_stream) == sa.SA_OK
    assert_close(out.cpu().numpy().astype(np.float64), A_ref, S_ref, TOL_FP32, "dense stage %dx%d" % (L, M))


def test_ttm4_padded_factor_matrices(sa):
    """Order-4 chain with the factor matrices given as padded views (leading dimension 20): the fused kernel's
    general-stride variant, and the subtree kernel's of the two-pass schedule."""
    import torch
    w = configs.make_ttm4_zipf("edge4e", 35, 300, 60, 150, 40, 120_000, 1.2, 3.0, 16, 16, 16)
    A_ref, S_ref = oracle.evaluate(w)
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSF, device=0)
    views = []
    for x in w.dense:
        b = torch.zeros(x.shape[0], 20, device="cuda")
        b[:, :16] = torch.from_numpy(x).cuda()
        views.append(b[:, :16])
    for sched in (sa.SA_SCHED_FUSED, sa.SA_SCHED_FISSIONED):
        out, _ = t.run(w.expr, views, sched=sched)
        torch.cuda.synchronize()
        assert sa.sa_last_device_status(t.handle, torch.cuda.current_stream().cuda_stream) == sa.SA_OK
        assert_close(out.cpu().numpy().astype(np.float64), A_ref, S_ref, TOL_FP32, "ttm4 padded ld, schedule %d" % sched)
    assert int(sa.sa_tensor_worklist(t.handle, 2)[0][0]) > 0 and int(sa.sa_tensor_worklist(t.handle, 6)[0][0]) > 0


def test_allocator_failure_at_every_upload_is_reported_and_leaks_nothing(sa):
    """The device allocator returns NULL at the k-th request, for every k up to the number of requests a tensor
    makes: create answers SA_E_ALLOC, hands out no handle, and every block it had obtained is released."""
    import ctypes
    import torch
    base = sa.TorchAllocator(0)

    class Failing:
        def __init__(self, fail_at):
            self.calls, self.fail_at, self.live = 0, fail_at, set()
            self._a = sa._ALLOC_FN(self.alloc)
            self._r = sa._RELEASE_FN(self.release)
            self.struct = sa.SaAllocator(self._a, self._r, None)

        def alloc(self, nbytes, ctx):
            self.calls += 1
            if self.calls - 1 == self.fail_at:
                return None
            p = base._do_alloc(nbytes, ctx)
            self.live.add(p)
            return p

        def release(self, ptr, ctx):
            self.live.discard(ptr)
            base._do_release(ptr, ctx)

    for cfg in (1, 3, 5):
        w = configs.make(cfg, "mini")
        fmt = fmt_of(sa, w)
        k = 0
        while True:
            a = Failing(k)
            try:
                h = sa.sa_tensor_create(len(w.dims), w.dims, len(w.vals), w.coords, w.vals, fmt, 0, a.struct)
            except sa.SaError as e:
                assert e.status == sa.SA_E_ALLOC, (cfg, k, e)
                assert a.calls == k + 1 and not a.live, "blocks obtained before the failure must be released"
                k += 1
                continue
            assert a.calls <= k, "with no failing request the tensor is created"
            assert len(a.live) == a.calls
            sa.sa_destroy(h)
            assert not a.live
            break
        assert k >= 8, "the loop really walked through the uploads"
    torch.cuda.synchronize()


def test_default_order_of_spmm_gemm_picks_the_faster_one_on_both_sides(sa):
    """The run-time choice between (B.C).D and B.(C.D) on two tensors where it goes opposite ways, checked against
    device timings: with few nonzeros on a huge C, forming C.D reads 2 GB that (B.C).D never touches; with many
    nonzeros per column, one gathered 1 KB row per nonzero is the larger cost."""
    import torch

    def both(I, J, nnz, seed):
        w = configs.make_spmm_gemm("order-%d" % J, seed, I, J, nnz, 256, 64)
        t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR, device=0)
        ops = [torch.from_numpy(x).cuda() for x in w.dense]
        desc = [(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0)) for x in ops]
        chosen = sa.sa_schedule_cost(t.handle, sa.SA_EXPR_SPMM_GEMM, sa.SA_SCHED_DEFAULT, desc)["resolved"]
        ms = {}
        for s in (sa.SA_SCHED_ASSOC_LEFT, sa.SA_SCHED_ASSOC_RIGHT):
            out, _ = t.run(w.expr, ops, sched=s)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                t.run(w.expr, ops, out=out, sched=s)
            e1.record()
            torch.cuda.synchronize()
            ms[s] = e0.elapsed_time(e1) / 10
        # the default really runs the chosen order (same launches, same result)
        a, _ = t.run(w.expr, ops, sched=sa.SA_SCHED_DEFAULT)
        b, _ = t.run(w.expr, ops, sched=chosen)
        torch.cuda.synchronize()
        assert torch.equal(a, b)
        t.close()
        return chosen, ms

    chosen, ms = both(5_000, 2_000_000, 200_000, 61)
    assert chosen == sa.SA_SCHED_ASSOC_LEFT and ms[sa.SA_SCHED_ASSOC_LEFT] < ms[sa.SA_SCHED_ASSOC_RIGHT], ms
    chosen, ms = both(20_000, 400_000, 1_500_000, 62)
    assert chosen == sa.SA_SCHED_ASSOC_RIGHT and ms[sa.SA_SCHED_ASSOC_RIGHT] < ms[sa.SA_SCHED_ASSOC_LEFT], ms


@pytest.mark.parametrize("K,L,M", [(64, 64, 32), (32, 128, 64), (128, 32, 32)])
def test_sddmm_spmm_gemm_rank_combinations(sa, K, L, M):
    """Kernel 2 over ranks the mini workload does not use: the tcgen05 dense stage at L = 64 with M = 32, the row
    temporaries of 32 and 128 floats."""
    w0 = configs.make_sddmm_spmm("k2-ranks", 91, 4_000, 4_000, 50_000, 1.5, 1_200, K, L)
    F = configs.dense_normal(91, 3, L, M)
    w = _wl("sddmm_spmm_gemm", "csr", w0.dims, w0.coords, w0.vals, w0.dense + [F], (w0.dims[0], M))
    _check(sa, w)


@pytest.mark.parametrize("L,M,J", [(128, 32, 1), (128, 64, 127), (256, 32, 148 * 128 + 1), (256, 64, 148 * 128 * 2 + 77)])
def test_spmmh_gemm_right_order_ragged_tiles_and_padded_operands(sa, L, M, J):
    """B.((C o D).E): row counts J around the dense stage's 128-row tile and its second tile per block, padded views.
    The bound is the one of an fp32 evaluation: 2 L rounding errors of 2^-24 per term of the sum at most."""
    import torch
    I = 300
    coords, vals = _random_coo(22, (I, J), min(20_000, I * J // 3))
    dense = [configs.dense_normal(22, 0, J, L), configs.dense_normal(22, 1, J, L), configs.dense_normal(22, 2, L, M)]
    w = _wl("spmmh_gemm", "csr", (I, J), coords, vals, dense, (I, M))
    A_ref, S_ref = oracle.evaluate(w)
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR, device=0)
    views = []
    for x, pad in zip(dense, (8, 12, 4)):
        b = torch.zeros(x.shape[0], x.shape[1] + pad, device="cuda")
        b[:, 4:4 + x.shape[1]] = torch.from_numpy(x).cuda()
        views.append(b[:, 4:4 + x.shape[1]])
    out, _ = t.run("spmmh_gemm", views, sched=sa.SA_SCHED_ASSOC_RIGHT)
    torch.cuda.synchronize()
    assert sa.sa_last_device_status(t.handle, torch.cuda.current_stream().cuda_stream) == sa.SA_OK
    assert_close(out.cpu().numpy().astype(np.float64), A_ref, S_ref, 2 * L * 2.0 ** -24, "spmmh right %dx%d" % (L, M))


@pytest.mark.parametrize("K,L", [(32, 32), (64, 128), (128, 128)])
@pytest.mark.parametrize("deg", [1, 15, 48, 49, 64, 65, 257])
def test_sddmm_spmm_rows_around_piece_and_column_block_limits(sa, K, L, deg):
    """Rows just below and above the length at which they are cut, with columns on both sides of the 32 K column blocks the
    cuts follow; empty rows between them; the fix-up of rows in a few pieces and in more than 32."""
    rs = np.random.RandomState(deg)
    J = 70_001
    rows = {0: deg, 2: deg, 3: 700, 5: 1, 9: deg + 1}
    coords = np.concatenate([np.stack([np.full(n, r), np.sort(np.concatenate([[32767, 32768, 65536][:n], rs.choice(32767, max(0, n - 3), replace=False)]))], axis=1)
                             for r, n in rows.items()]).astype(np.int32)
    vals = rs.uniform(-1, 1, len(coords)).astype(np.float32)
    w = _wl("sddmm_spmm", "csr", (11, J), coords, vals,
            [configs.dense_normal(deg, 0, 11, K), configs.dense_normal(deg, 1, J, K), configs.dense_normal(deg, 2, J, L)], (11, L))
    _check(sa, w)


@pytest.mark.parametrize("M,J", [(32, 900), (64, 900), (64, 393_217)])
@pytest.mark.parametrize("deg", [1, 8, 31, 33, 65, 257])
def test_spmm_gemm_right_order_rows_around_step_and_piece_limits(sa, M, J, deg):
    """Rows around the eight-nonzero step and the length at which they are cut into pieces, empty rows at both ends of an
    item and inside it, and the first J for which E is kept as two tables (96 MB at M = 64)."""
    rs = np.random.RandomState(deg)
    rows = {1: deg, 2: 1, 5: deg, 40: 8, 41: deg + 1, 77: 70}
    coords = np.concatenate([np.stack([np.full(n, r), rs.choice(J, n, replace=False)], axis=1) for r, n in rows.items()]).astype(np.int32)
    vals = rs.uniform(-1, 1, len(coords)).astype(np.float32)
    w = _wl("spmm_gemm", "csr", (100, J), coords, vals, [configs.dense_normal(deg, 0, J, 128), configs.dense_normal(deg, 1, 128, M)], (100, M))
    _check(sa, w, sched=sa.SA_SCHED_ASSOC_RIGHT)


@pytest.mark.parametrize("n", [255, 256, 257, 1023, 1024, 1025, 4097])
@pytest.mark.parametrize("L,M", [(16, 16), (32, 32)])
def test_ttm3_small_tensor_slices_around_the_unit_and_chunk_sizes(sa, n, L, M):
    """A tensor small enough for units of 256 nonzeros (chunks of 1024): slices of n and of one nonzero, a fix-up entry with
    partial tiles of several chunks."""
    rs = np.random.RandomState(n)
    J, K = 90, 60
    lin = np.sort(rs.choice(J * K, n, replace=False))
    big = np.stack([np.full(n, 4), lin // K, lin % K], axis=1)
    ones = np.stack([np.arange(3), rs.randint(0, J, 3), rs.randint(0, K, 3)], axis=1)
    coords = np.concatenate([big, ones]).astype(np.int32)
    vals = rs.uniform(-1, 1, len(coords)).astype(np.float32)
    w = _wl("spttm_ttm3", "csf", (6, J, K), coords, vals, [configs.dense_uniform(n, 0, J, L), configs.dense_uniform(n, 1, K, M)], (6, L, M))
    _check(sa, w)


@pytest.mark.parametrize("I", [1, 7, 9, 64, 65, 1025, 32_769])
@pytest.mark.parametrize("L,M,N", [(16, 16, 16), (32, 16, 32), (16, 32, 32)])
def test_ttmc3_slices_around_the_step_and_chunk_sizes(sa, I, L, M, N):
    """Numbers of slices around the eight-row step and the chunk of slices of the reduction over i (64 slices, 65 from 32769 on)
    and numbers of chunks around its 16 phases, with empty slices."""
    rs = np.random.RandomState(I)
    J, K = 30, 20
    coords = np.stack([rs.randint(0, I, 900), rs.randint(0, J, 900), rs.randint(0, K, 900)], axis=1)
    coords = np.unique(coords, axis=0).astype(np.int32)
    vals = rs.uniform(-1, 1, len(coords)).astype(np.float32)
    ops = [configs.dense_uniform(I, 0, I, L), configs.dense_uniform(I, 1, J, M), configs.dense_uniform(I, 2, K, N)]
    _check(sa, _wl("ttmc3", "csf", (I, J, K), coords, vals, ops, (L, M, N)), sched=sa.SA_SCHED_FISSIONED)


@pytest.mark.parametrize("fibers", [1, 3, 4, 5, 7, 8, 9, 65, 700])
@pytest.mark.parametrize("per_fiber", [1, 17])
def test_mttkrp_gemm_fibers_around_the_four_and_eight_row_steps(sa, fibers, per_fiber):
    """Numbers of fibers per slice around the four rows of a step and the eight of a flush; the last case spans several warps
    of a block (units of one slice) and several units."""
    rs = np.random.RandomState(10 * fibers + per_fiber)
    J, K = 800, 40
    coords = np.concatenate([np.stack([np.full(fibers * per_fiber, i), np.repeat(np.sort(rs.choice(J, fibers, replace=False)), per_fiber),
                                       np.concatenate([np.sort(rs.choice(K, per_fiber, replace=False)) for _ in range(fibers)])], axis=1)
                             for i in (0, 2, 3)]).astype(np.int32)
    vals = rs.uniform(-1, 1, len(coords)).astype(np.float32)
    ops = [configs.dense_uniform(fibers, 0, J, 32), configs.dense_uniform(fibers, 1, K, 32), configs.dense_uniform(fibers, 2, 32, 32)]
    _check(sa, _wl("mttkrp_gemm", "csf", (5, J, K), coords, vals, ops, (5, 32)))


@pytest.mark.parametrize("L,M,J", [(128, 32, 200), (128, 64, 1), (256, 32, 148 * 128 + 33), (256, 64, 5_000)])
def test_spmmh_gemm_right_order_keeps_infinities_nan_and_the_largest_numbers(sa, L, M, J):
    """The dense stage of B.((C o D).E) splits its operands into BF16 parts; numbers that have no such parts (infinities, NaN,
    finite ones that round to a BF16 infinity) must give what the row nest in fp32 arithmetic gives.  All operands are positive
    apart from one negative infinity and every row has nonzeros, so that the two orders of summation meet the same cases."""
    import torch
    rng = np.random.default_rng(7)
    I, deg = 700, min(4, J)
    cols = np.stack([rng.choice(J, deg, replace=False) for _ in range(I)])
    cols[:4, 0] = [0, J - 1, J // 2, J // 3]
    cols = np.stack([np.pad(np.unique(c), (0, deg - len(np.unique(c))), constant_values=-1) for c in cols])
    keep = cols.ravel() >= 0
    coords = np.stack([np.repeat(np.arange(I), deg)[keep], cols.ravel()[keep]], axis=1).astype(np.int32)
    vals = rng.uniform(0.5, 1.0, coords.shape[0]).astype(np.float32)
    t = sa.SparseTensor((I, J), coords, vals, sa.SA_FMT_CSR, device=0)
    C, D = (rng.uniform(0.5, 1.0, (J, L)).astype(np.float32) for _ in range(2))
    E = rng.uniform(0.5, 1.0, (L, M)).astype(np.float32)

    def both(C, D, E):
        ops = [torch.from_numpy(x).cuda() for x in (C, D, E)]
        out = [t.run("spmmh_gemm", ops, sched=s)[0].cpu().numpy() for s in (sa.SA_SCHED_ASSOC_RIGHT, sa.SA_SCHED_FUSED)]
        assert sa.sa_last_device_status(t.handle, torch.cuda.current_stream().cuda_stream) == sa.SA_OK
        return out

    def same(right, nest):
        assert np.array_equal(np.isnan(right), np.isnan(nest))
        inf = np.isinf(nest)
        assert np.array_equal(np.isinf(right), inf) and np.array_equal(right[inf], nest[inf])
        fin = np.isfinite(nest)
        assert fin.sum() == 0 or np.abs(right[fin] / nest[fin] - 1).max() < 2 * L * 2.0 ** -24      # fp32 sums of L positive terms
        return nest

    tiny = np.float32(1e-3)
    for where in {0, J - 1, J // 2, J // 3}:
        for value in (np.inf, -np.inf, np.nan):
            for hit in (0, 1):
                X = [C.copy(), D.copy()]
                X[hit][where, L // 3] = value
                nest = same(*both(X[0], X[1], E))
                assert np.isfinite(nest).any() or J < 5
                assert not np.isfinite(nest).all()
        X = C.copy()
        X[where, L - 1] = np.float32(3.4e38)                       # finite, rounds to a BF16 infinity; the sums stay finite
        Y = D.copy()
        Y[where, L - 1] = 1
        F = E.copy()
        F[L - 1] = tiny
        assert np.isfinite(same(*both(X, Y, F))).all()
        Y[where, L - 1] = 8                                        # the product itself overflows
        assert np.isinf(same(*both(X, Y, F))).any()
    for value in (np.inf, np.nan, np.float32(3.4e38)):
        F = E.copy()
        F[L // 2, M - 1] = value
        nest = same(*both(C * tiny, D, F))
        assert np.isfinite(nest[:, :M - 1]).all()


def test_spmmh_gemm_default_runs_in_the_workspace_it_is_given(sa):
    """Without room for the J x M temporary of its faster order the default of kernel 3 is the row nest: from a caller that has
    no workspace to give, and where the device has no memory left for one."""
    import torch
    I, J, L, M = 300, 200_000, 128, 64
    coords, vals = _random_coo(31, (I, J), 600_000)
    t = sa.SparseTensor((I, J), coords, vals, sa.SA_FMT_CSR, device=0)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    ops = [torch.randn(s, device="cuda", generator=g) for s in ((J, L), (J, L), (L, M))]
    tuples = [(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0)) for x in ops]
    E, F, D = sa.SA_EXPR_SPMMH_GEMM, sa.SA_SCHED_FUSED, sa.SA_SCHED_DEFAULT
    need, nest = (sa.sa_workspace_size(t.handle, E, s, tuples) for s in (D, F))
    assert sa.sa_schedule_cost(t.handle, E, D, tuples)["resolved"] == sa.SA_SCHED_ASSOC_RIGHT and need >= J * M * 4 > 4 * nest
    ref, _ = t.run("spmmh_gemm", ops, sched=F)                     # leaves a workspace with too little room for the default
    stream = torch.cuda.current_stream().cuda_stream
    ws = torch.empty(max(nest, 256), dtype=torch.uint8, device="cuda")
    out = torch.full_like(ref, float("nan"))
    sa.sa_run(t.handle, E, D, tuples, out.data_ptr(), ws.data_ptr() if nest else None, nest, stream)
    assert torch.equal(out, ref)
    for s in (sa.SA_SCHED_ASSOC_RIGHT, F if nest else sa.SA_SCHED_ASSOC_RIGHT):        # named schedules say what they lack
        with pytest.raises(sa.SaError) as e:
            sa.sa_run(t.handle, E, s, tuples, out.data_ptr(), None, 0, stream)
        assert e.value.status == sa.SA_E_WORKSPACE
    empty = t._empty

    def no_room(shape, *a):
        if shape == need:
            raise torch.OutOfMemoryError("as the allocator says it")
        return empty(shape, *a)

    t._empty = no_room
    out, _ = t.run("spmmh_gemm", ops)
    assert torch.equal(out, ref)
    t._empty = empty
    out, ws = t.run("spmmh_gemm", ops)                             # and with memory the faster order, after the smaller workspace
    assert ws.numel() >= need and not torch.equal(out, ref)
    assert float((out - ref).norm() / ref.norm()) < 1e-5


def _cut_rows_case(sa, J=3000):
    """Matrix whose long rows are summed from partial rows in the workspace, its operands for kernel 1, and the result."""
    import torch
    w = configs.make_sddmm_spmm("streams", 51, 2_000, J, 60_000, 1.5, 1_500, 64, 64)
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR, device=0)
    ops = [torch.from_numpy(x).cuda() for x in w.dense]
    ref, ws = t.run("sddmm_spmm", ops)
    torch.cuda.synchronize()
    assert sa.sa_tensor_worklist(t.handle)[0][3] > 0
    return t, ops, ref, ws


def test_calls_on_two_streams_share_no_workspace(sa):
    import torch
    t, ops, ref, ws = _cut_rows_case(sa)
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs, spaces = [], [ws]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    for rep in range(50):
        for s in streams:
            out, w = t.run("sddmm_spmm", ops, stream=s)
            outs.append(out)
            spaces.append(w)
    torch.cuda.synchronize()
    assert len({w.data_ptr() for w in spaces}) == 3
    assert all(torch.equal(o, ref) for o in outs)


def test_calls_from_two_threads_share_no_workspace(sa):
    import threading
    import torch
    t, ops, ref, ws = _cut_rows_case(sa)
    spaces, outs, meet = [ws], [], threading.Barrier(2)

    def work():
        meet.wait()
        got = [t.run("sddmm_spmm", ops) for _ in range(50)]
        outs.extend(o for o, _ in got)
        spaces.extend(w for _, w in got)

    threads = [threading.Thread(target=work) for _ in range(2)]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    torch.cuda.synchronize()
    assert len({w.data_ptr() for w in spaces}) == 3
    assert all(torch.equal(o, ref) for o in outs)
    assert len(t._ws) <= t.MAX_WORKSPACES


def test_workspaces_kept_by_a_tensor_are_bounded_and_given_back(sa):
    import torch
    t, ops, ref, _ = _cut_rows_case(sa)
    before = torch.cuda.memory_allocated()
    for _ in range(3 * t.MAX_WORKSPACES):
        out, _ws = t.run("sddmm_spmm", ops, stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    assert len(t._ws) == t.MAX_WORKSPACES
    del out, _ws
    t.close()
    assert not t._ws and torch.cuda.memory_allocated() < before


def test_workspace_grows_after_a_smaller_call_on_a_side_stream(sa):
    import torch
    t, ops, ref, _ = _cut_rows_case(sa)
    F = torch.ones(64, 32, device="cuda")
    full, _ = t.run("sddmm_spmm_gemm", ops + [F])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    small, w1 = t.run("sddmm_spmm", ops, stream=s)
    n1 = w1.numel()
    del w1
    big, w2 = t.run("sddmm_spmm_gemm", ops + [F], stream=s)        # needs the row temporary as well
    again, w3 = t.run("sddmm_spmm", ops, stream=s)
    s.synchronize()
    assert w2.numel() > n1 and w3 is w2
    assert torch.equal(small, ref) and torch.equal(again, ref) and torch.equal(big, full)


def test_output_is_on_the_tensor_device_whatever_the_workspace_is(sa, monkeypatch):
    """A caller's workspace may be pinned host memory; the output that run allocates may not.  Nothing is launched here."""
    import torch
    t, ops, ref, _ = _cut_rows_case(sa)
    monkeypatch.setattr(sa, "_run_packed", lambda *a: sa.SA_OK)
    out, _ = t.run("sddmm_spmm", ops, workspace=torch.empty(1 << 20, dtype=torch.uint8).pin_memory())
    assert out.device == ref.device


def test_operands_that_make_no_sense_are_refused_before_their_output_is_too_large(sa):
    import torch
    t = sa.SparseTensor((2_000_000, 50, 60), np.array([[5, 6, 7]], np.int32), np.ones(1, np.float32), sa.SA_FMT_CSF, device=0)
    ops = [torch.ones(50, 512, device="cuda"), torch.ones(60, 512, device="cuda")]     # 2.1 TB of output at ranks it is not built for
    good = [torch.ones(50, 16, device="cuda"), torch.ones(60, 16, device="cuda")]
    for _ in range(2):
        with pytest.raises(sa.SaError) as e:
            t.run("spttm_ttm3", ops)
        assert e.value.status == sa.SA_E_UNSUPPORTED
        out, _ws = t.run("spttm_ttm3", good)       # leaves a workspace, so that the second round does not ask for its size first
        assert float(out[5, 0, 0]) == 1.0


@pytest.mark.parametrize("rows", [28_416 * 8 - 3, 28_416 * 8 + 3])
def test_sddmm_spmm_ranks_32_on_both_sides_of_the_two_and_three_block_kernels(sa, rows):
    """One nonzero per row, ranges of eight rows: 28 416 items are the last that the kernel for two blocks per SM takes."""
    coords, vals = np.stack([np.arange(rows), np.arange(rows) % 40], axis=1), rng.uniform_f32(61, 1, np.arange(rows), -1.0, 1.0)
    w = _wl("sddmm_spmm", "csr", (rows, 40), coords, vals, [_dense(61, 0, rows, 32), _dense(61, 1, 40, 32), _dense(61, 2, 40, 32)], (rows, 32))
    _, t = _check(sa, w)
    assert (len(sa.sa_tensor_worklist(t.handle)[1]) <= 28_416) == (rows < 28_416 * 8)


@pytest.mark.parametrize("M", [32, 64])
@pytest.mark.parametrize("expr", ["spmm_gemm", "spmmh_gemm"])
def test_right_order_rows_that_do_not_refer_to_row_0_do_not_see_it(sa, expr, M):
    """The gather loads row 0 for steps past a row's end: with NaN and infinities there every other result stays as it is."""
    import torch
    deg = np.array([1, 2, 7, 8, 9, 0, 15, 16, 17, 0, 0, 31, 33, 64, 200, 1, 0, 3] * 9)
    J = 700
    cols = np.concatenate([1 + rng.permutation(50 + i, i, J - 1)[:n] for i, n in enumerate(deg)])
    coords = np.stack([np.repeat(np.arange(len(deg)), deg), cols], axis=1).astype(np.int32)
    vals = np.random.RandomState(5).uniform(0.5, 1.0, len(coords)).astype(np.float32)
    t = sa.SparseTensor((len(deg), J), coords, vals, sa.SA_FMT_CSR, device=0)
    ops = [torch.randn(J, 128, device="cuda") for _ in range(2 if expr == "spmmh_gemm" else 1)] + [torch.randn(128, M, device="cuda")]
    want = t.run(expr, ops, sched=sa.SA_SCHED_ASSOC_RIGHT)[0].clone()
    ops[0][0, ::2], ops[0][0, 1::2] = float("nan"), float("inf")
    got = t.run(expr, ops, sched=sa.SA_SCHED_ASSOC_RIGHT)[0]
    assert torch.equal(got, want)
