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
