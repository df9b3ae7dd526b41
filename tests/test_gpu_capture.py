"""Graphs of the library's calls, its own and a caller's: each replay must do what the captured calls said,
whatever the context was used for in between."""
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads

pytestmark = pytest.mark.gpu


def _gas(shape, seed, dtype=torch.float64):
    return workloads.white_velocity_state(shape, seed=seed, p_jitter=0.2).cuda().to(dtype).contiguous()


def _view(pool, shape):
    n = shape[0] * shape[1] * shape[2]
    return pool[:5 * n].view(5, *shape)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("tuned", [False, True])
def test_run_graph_of_another_box_at_the_same_address(precision, tuned):
    """Two boxes of different shape, then two cell sizes, in one pair of buffers: every graph run against
    the run without a graph, bit for bit, and nothing written beyond the box."""
    dtype = torch.float32 if precision == "fp32" else torch.float64
    shapes = [(20, 24, 28), (9, 24, 10), (10, 24, 9), (20, 24, 28)]
    cells = 5 * 20 * 24 * 28
    A, B = torch.empty(cells, dtype=dtype, device="cuda"), torch.empty(cells, dtype=dtype, device="cuda")
    hist = torch.empty(4, dtype=torch.float64, device="cuda")
    ctx, ref = hy.hydro_init(precision=precision), hy.hydro_init(precision=precision)
    if tuned:
        hy.hydro_set_tuning(ctx, 0, 8)
        hy.hydro_set_tuning(ref, 0, 8)
    for shape, dx in [(s, 0.05) for s in shapes] + [(shapes[0], 0.1), (shapes[0], 0.05)]:
        U = _gas(shape, 1, dtype)
        got = []
        for c, graph in ((ref, False), (ctx, True), (ctx, True)):
            A.fill_(-7.0)
            B.fill_(-7.0)
            a, b = _view(A, shape), _view(B, shape)
            a.copy_(U)
            hy.hydro_run(c, hy.patch(a, 0, dx), hy.patch(b, 0, dx), 3, hist, use_graph=graph)
            assert hy.hydro_get_error(c) == (hy.HYDRO_OK, 0)
            got.append((A.clone(), B.clone(), hist.clone()))
        for g in got[1:]:
            assert all(torch.equal(x, y) for x, y in zip(g, got[0]))
    hy.hydro_finalize(ctx)
    hy.hydro_finalize(ref)


def _octs(dims, seed):
    """A full periodic level: oct-major state, positions."""
    X, Y, Z = dims
    U = _gas((2 * Z, 2 * Y, 2 * X), seed)
    z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.int32) for n in (Z, Y, X)], indexing="ij")
    V = U.reshape(5, Z, 2, Y, 2, X, 2).permute(0, 1, 3, 5, 2, 4, 6).reshape(5, -1, 8).contiguous()
    return V, torch.stack([x, y, z], dim=-1).reshape(-1, 3).contiguous()


def _captured(stream, calls):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        calls()
    return graph


def _eaters():
    """Allocations of many sizes, so that a freed block does not stay as it was."""
    return [torch.full((1 << k,), 0x5a5a5a5a, dtype=torch.int32, device="cuda") for k in range(6, 22)]


@pytest.mark.parametrize("with_table", [False, True])
def test_oct_graph_outlives_longer_lists(with_table):
    """An oct build and a step through the table, captured; then the same calls for larger levels, whose
    lists and tables need more scratch; then the replay."""
    dims, dt = (24, 24, 20), torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
    V, pos = _octs(dims, 3)
    n = len(pos)
    order, nbr = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty((n, 27), dtype=torch.int32, device="cuda")
    out = torch.empty_like(V)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        ctx = hy.hydro_init(precision="fp64")

        def build():
            hy.hydro_octs_build(ctx, pos, dims, order, nbr if with_table else None)

        def step():
            hy.hydro_step_octs_table(ctx, V, out, nbr, order, 0.05, dt)

        hy.hydro_octs_build(ctx, pos, dims, order, nbr if with_table else None)
        if not with_table:  # a table from another context: this one's scratch stays the small one
            other = hy.hydro_init(precision="fp64")
            hy.hydro_octs_build(other, pos, dims, order, nbr)
            stream.synchronize()
            hy.hydro_finalize(other)
        step()
        want, want_order, want_nbr = out.clone(), order.clone(), nbr.clone()
        stream.synchronize()
        graphs = [_captured(stream, build), _captured(stream, step)]
        hy.hydro_octs_build(ctx, pos, dims, order, nbr)  # the same level, now with its table
        for big in ((40, 32, 32), (64, 48, 40)):
            W, at = _octs(big, 4)
            o2, n2 = torch.empty(len(at), dtype=torch.int32, device="cuda"), torch.empty((len(at), 27), dtype=torch.int32, device="cuda")
            # built elsewhere, so that only the scratch of this context's step through the table grows
            other = hy.hydro_init(precision="fp64")
            hy.hydro_octs_build(other, at, big, o2, n2)
            hy.hydro_step_octs_table(ctx, W, torch.empty_like(W), n2, o2, 0.05, dt)
            stream.synchronize()
            hy.hydro_finalize(other)
        keep = _eaters()
        for _ in range(2):
            out.fill_(3.0)
            order.fill_(-9)
            if with_table:
                nbr.fill_(-9)
            for g in graphs:
                g.replay()
            stream.synchronize()
            assert torch.equal(order, want_order) and torch.equal(nbr, want_nbr) and torch.equal(out, want)
        assert all(bool((k == 0x5a5a5a5a).all()) for k in keep)
        assert hy.hydro_get_error(ctx) == (hy.HYDRO_OK, 0)
        hy.hydro_finalize(ctx)
