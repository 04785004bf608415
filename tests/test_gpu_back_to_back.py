"""Calls enqueued one behind the other, without the host waiting: kernels may start while the one before them still runs, and
must not read or overwrite anything of it before it is through."""
import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

CONFIGS = (1, 2, 3, 4, 5, 6, 7, 8, 9, 10)


def _tensor(sa, cfg):
    import torch
    w = configs.make(cfg, "mini")
    t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR if w.fmt == "csr" else sa.SA_FMT_CSF, device=0)
    return w, t, [torch.from_numpy(x).cuda() for x in w.dense]


# the order-4 fissioned chain and kernel 5 fused add parts in no fixed order
def _same(w, a, b):
    import torch
    if w.expr in ("spttm_ttm4", "ttmc3"):
        return bool(((a - b).abs().max() <= 1e-5 * b.abs().max()).item())
    return torch.equal(a, b)


@pytest.mark.parametrize("cfg", CONFIGS)
def test_results_and_operands_of_neighbouring_calls_do_not_mix(cfg):
    """Every call reads operands that a kernel just before it wrote and whose next contents a kernel just behind it writes; the
    output buffer and the workspace are the same throughout."""
    import torch
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    steps = 6
    scales = [1.0, -0.5, 2.0, 0.25, -4.0, 0.5]             # powers of two: a product with them is exact
    want = []
    for s in scales:
        torch.cuda.synchronize()
        out, _ = t.run(w.expr, [ops[0] * s] + ops[1:])
        torch.cuda.synchronize()
        want.append(out.clone())
    first, out, got = torch.empty_like(ops[0]), torch.empty_like(want[0]), torch.empty((steps,) + tuple(want[0].shape), device="cuda")
    t.run(w.expr, [ops[0]] + ops[1:], out=out)             # the workspace is there
    torch.cuda.synchronize()
    for k, s in enumerate(scales):
        torch.mul(ops[0], s, out=first)
        t.run(w.expr, [first] + ops[1:], out=out)
        got[k].copy_(out)
    torch.cuda.synchronize()
    for k in range(steps):
        assert _same(w, got[k], want[k]), "call %d" % k


@pytest.mark.parametrize("cfg", CONFIGS)
def test_the_output_of_a_call_is_the_operand_of_the_next(cfg):
    """Two tensors in turn: the dense result of the first call is an operand of the second, which starts right behind it."""
    import torch
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    out, ws = t.run(w.expr, ops)
    torch.cuda.synchronize()
    # a matrix with the output's rows as columns: B2 . (C2 . D2) with C2 = the output, seen as rows of 128 floats
    n = out.numel() // 128
    rng = np.random.default_rng(cfg)
    coords = np.stack([np.repeat(np.arange(64), 8), rng.integers(0, n, 512)], axis=1).astype(np.int32)
    coords = np.unique(coords, axis=0)
    t2 = sa.SparseTensor((64, n), coords, rng.standard_normal(len(coords)).astype(np.float32), sa.SA_FMT_CSR, device=0)
    D2 = torch.randn(128, 32, device="cuda")

    def second(c, buf=None, **kw):
        return t2.run("spmm_gemm", [c.view(-1)[:n * 128].view(n, 128), D2], out=buf, **kw)[0]
    for sched in (sa.SA_SCHED_ASSOC_LEFT, sa.SA_SCHED_ASSOC_RIGHT):
        want = second(out, sched=sched).clone()
        torch.cuda.synchronize()
        chain, res = torch.zeros_like(out), torch.empty_like(want)
        results = []
        for _ in range(4):
            chain.zero_()
            t.run(w.expr, ops, out=chain)
            second(chain, res, sched=sched)
            results.append(res.clone())
        torch.cuda.synchronize()
        for r in results:
            assert bool(((r - want).abs().max() <= 1e-5 * want.abs().max()).item())


@pytest.mark.parametrize("cfg", (1, 7, 9))
def test_captured_calls_replay_in_order(cfg):
    import torch
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    out, ws = t.run(w.expr, ops)
    torch.cuda.synchronize()
    want = out.clone()
    first, res = ops[0].clone(), torch.empty_like(out)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        t.run(w.expr, [first] + ops[1:], out=res, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for s in (2.0, 0.5):
            torch.mul(ops[0], s, out=first)
            t.run(w.expr, [first] + ops[1:], out=res, workspace=ws)
        res *= 2.0
    for _ in range(3):
        res.zero_()
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(res, want)


# ---- library calls with nothing between them: no torch kernel stands between the one that writes and the one that reads

SCHEDULES = [(cfg, None) for cfg in CONFIGS] + [(4, "ASSOC_LEFT"), (4, "ASSOC_RIGHT"), (5, "FUSED"), (5, "FISSIONED"), (6, "FUSED"),
                                                (6, "FISSIONED"), (8, "FUSED"), (10, "ASSOC_LEFT"), (10, "ASSOC_RIGHT")]
STEPS = 4


def _sched(sa, name):
    return sa.SA_SCHED_DEFAULT if name is None else getattr(sa, "SA_SCHED_" + name)


class _Writer:
    """A call that writes an operand of another: out = B . C . D seen as rows x cols, other numbers at every step."""

    def __init__(self, sa, rows, cols, seed):
        import torch
        self.shape, self.rows = (rows, cols), -(-rows * cols // 64)
        rng = np.random.default_rng(seed)
        coords = np.stack([np.repeat(np.arange(self.rows), 4), rng.integers(0, 500, 4 * self.rows)], axis=1).astype(np.int32)
        coords = np.unique(coords, axis=0)
        self.t = sa.SparseTensor((self.rows, 500), coords, rng.uniform(0.5, 1.0, len(coords)).astype(np.float32), sa.SA_FMT_CSR, device=0)
        self.sched = (sa.SA_SCHED_ASSOC_LEFT, sa.SA_SCHED_ASSOC_RIGHT)[seed % 2]
        g = torch.Generator(device="cuda").manual_seed(seed)
        C = torch.randn(500, 128, device="cuda", generator=g)
        self.C = [C * s for s in (1.0, -0.5, 4.0, 0.25)]
        self.D = torch.randn(128, 64, device="cuda", generator=g) / 16
        self.buf = torch.zeros(self.rows, 64, device="cuda")
        self.ws = self.t.run("spmm_gemm", [self.C[0], self.D], out=self.buf, sched=self.sched)[1]

    def write(self, step):
        self.t.run("spmm_gemm", [self.C[step], self.D], out=self.buf, sched=self.sched, workspace=self.ws)
        return self.buf.view(-1)[:self.shape[0] * self.shape[1]].view(self.shape)


def _apart(step):
    import torch
    torch.cuda.synchronize()
    out = step()
    torch.cuda.synchronize()
    return out.clone()


def _written_operands(sa, w, t, ops, sched):
    import torch
    out, ws = t.run(w.expr, ops, sched=sched)
    for i, op in enumerate(ops):
        writer = _Writer(sa, op.shape[0], op.shape[1], 10 * len(ops) + i)

        def call(step, out=None, i=i, writer=writer):
            return t.run(w.expr, ops[:i] + [writer.write(step)] + ops[i + 1:], out=out, sched=sched, workspace=ws)[0]
        want = [_apart(lambda: call(k)) for k in range(STEPS)]
        assert not torch.equal(want[0], want[1])
        yield i, call, want, [torch.empty_like(out) for _ in range(STEPS)]


def _check_written_operands(sa, w, t, ops, sched):
    import torch
    for i, call, want, outs in _written_operands(sa, w, t, ops, sched):
        torch.cuda.synchronize()
        for k in range(STEPS):
            call(k, outs[k])
        torch.cuda.synchronize()
        for k in range(STEPS):
            assert _same(w, outs[k], want[k]), "operand %d, step %d" % (i, k)


@pytest.mark.parametrize("cfg, sched", SCHEDULES)
def test_a_call_reads_what_the_call_before_it_writes(cfg, sched):
    """Every operand in turn is written by a library call, with other numbers at every step, and read by the next."""
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    _check_written_operands(sa, w, t, ops, _sched(sa, sched))


def test_a_call_of_many_blocks_reads_what_the_call_before_it_writes():
    """The same with more blocks on both sides than the device has SMs."""
    import torch
    import paper_2311_09549_b200 as sa
    for w in (configs.make_sddmm_spmm("many-1", 61, 20_000, 30_000, 600_000, 0.8, 2_000, 64, 64),
              configs.make_ttm3_zipf("many-6", 62, 3_000, 4_000, 5_000, 600_000, 1.0, 5.0, 32, 32)):
        t = sa.SparseTensor(w.dims, w.coords, w.vals, sa.SA_FMT_CSR if w.fmt == "csr" else sa.SA_FMT_CSF, device=0)
        _check_written_operands(sa, w, t, [torch.from_numpy(x).cuda() for x in w.dense], sa.SA_SCHED_DEFAULT)


def _operand_sets(ops):
    import torch
    g = torch.Generator(device="cuda").manual_seed(7)
    return [[torch.randn(x.shape, device="cuda", generator=g) for x in ops] for _ in range(STEPS)]


@pytest.mark.parametrize("cfg, sched", SCHEDULES)
def test_adjacent_calls_share_a_workspace_and_a_result(cfg, sched):
    """Calls that differ in every operand, one behind the other in one workspace: first each with a result of its own, then
    all into the same one."""
    import torch
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    sched = _sched(sa, sched)
    out, ws = t.run(w.expr, ops, sched=sched)
    sets = _operand_sets(ops)
    want = [_apart(lambda: t.run(w.expr, s, sched=sched, workspace=ws)[0]) for s in sets]
    outs = [torch.empty_like(out) for _ in sets]
    for s, o in zip(sets, outs):
        t.run(w.expr, s, out=o, sched=sched, workspace=ws)
    torch.cuda.synchronize()
    for k in range(STEPS):
        assert _same(w, outs[k], want[k]), "call %d" % k
    for last in (STEPS - 1, STEPS - 2):
        for s in sets[:last + 1]:
            t.run(w.expr, s, out=out, sched=sched, workspace=ws)
        torch.cuda.synchronize()
        assert _same(w, out, want[last])


@pytest.mark.parametrize("cfg, sched", SCHEDULES)
def test_captured_calls_read_what_the_call_before_them_writes(cfg, sched):
    import torch
    import paper_2311_09549_b200 as sa
    w, t, ops = _tensor(sa, cfg)
    sched = _sched(sa, sched)
    ws = t.run(w.expr, ops, sched=sched)[1]
    sets = _operand_sets(ops)
    apart = [_apart(lambda: t.run(w.expr, s, sched=sched, workspace=ws)[0]) for s in sets]
    for i, call, want, outs in _written_operands(sa, w, t, ops, sched):
        others = [torch.empty_like(o) for o in outs]
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            for k in range(STEPS):
                call(k, outs[k])
                t.run(w.expr, sets[k], out=others[k], sched=sched, workspace=ws)
        for _ in range(2):
            for o in outs + others:
                o.zero_()
            graph.replay()
            torch.cuda.synchronize()
            for k in range(STEPS):
                assert _same(w, outs[k], want[k]), "operand %d, step %d" % (i, k)
                assert _same(w, others[k], apart[k]), "operand %d, step %d" % (i, k)
