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


N = 16


def _patches(seed, grow):
    """A coarse box and three fine patches of it (edges grown by `grow`), ghosts still to be filled."""
    coarse = _gas(N, seed)
    dims = [(12 + grow, 8, 10), (6, 8 + grow, 10), (14, 6, 8 + grow)]
    ins = [torch.zeros((5, z + 4, y + 4, x + 4), dtype=torch.float64, device="cuda") for x, y, z in dims]
    fine = _gas(2 * N, seed + 50)
    origins = [(2, 4, 6), (18, 4, 6), (2, 20, 18)]
    for t, o, (x, y, z) in zip(ins, origins, dims):
        ix, iy, iz = ((torch.arange(n, device="cuda") + s) % (2 * N) for n, s in zip((x, y, z), o))
        t[:, 2:-2, 2:-2, 2:-2] = fine[:, iz][:, :, iy][:, :, :, ix]
    return coarse, origins, dims, ins


class _Level:
    """One patch set's calls and their buffers."""

    def __init__(self, ctx, seed, grow):
        self.ctx, self.data = ctx, _patches(seed, grow)
        coarse, self.origins, self.dims, ins = self.data
        self.ins = [t.clone() for t in ins]
        self.outs = [torch.zeros_like(t) for t in ins]
        self.regs = [torch.zeros(5 * hy.register_size(*d), dtype=torch.float64, device="cuda") for d in self.dims]
        self.dt = torch.full((3,), 2e-3, dtype=torch.float64, device="cuda")
        self.dn, self.cfl = torch.empty_like(self.dt), torch.empty_like(self.dt)
        self.c = hy.patch(coarse, 0, 1.0 / N)
        self.a, self.b = ([hy.patch(t, 2, 0.5 / N) for t in T] for T in (self.ins, self.outs))

    def calls(self):
        hy.hydro_fill_ghosts(self.ctx, self.c, self.a, self.origins)
        hy.hydro_exchange_ghosts(self.ctx, self.a, self.origins, (2 * N,) * 3)
        hy.hydro_patch_fluxes(self.ctx, self.a, self.dt, self.regs)
        hy.hydro_step(self.ctx, self.a, self.b, self.dt, self.dn)
        hy.hydro_cfl_dt(self.ctx, self.a, self.cfl)

    def results(self):
        return self.ins + self.outs + self.regs + [self.dn, self.cfl]

    def clear(self):
        for t, u in zip(self.ins, self.data[3]):
            t.copy_(u)
        for t in self.outs + self.regs + [self.dn, self.cfl]:
            t.zero_()


def test_patch_graphs_outlive_other_sets():
    """Patch sets' calls captured, more sets than a context keeps, each before the next comes; then other
    and larger sets; then every graph again.  Graphs that are gone leave their sets to the others."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        ctx = hy.hydro_init(precision="fp64")
        for rounds in range(2):
            levels, graphs, want = [], [], []
            for seed in range(6):
                lv = _Level(ctx, seed, 0)
                lv.calls()
                stream.synchronize()
                want.append([t.clone() for t in lv.results()])
                lv.clear()
                graphs.append(_captured(stream, lv.calls))
                levels.append(lv)
            others = [_Level(ctx, seed, 2 + seed % 7) for seed in range(20, 30)]
            for lv in others + others[::-1]:
                lv.calls()
            keep = _eaters()
            for k in (3, 0, 5, 1, 4, 2, 0):
                levels[k].clear()
                graphs[k].replay()
                stream.synchronize()
                assert all(torch.equal(g, w) for g, w in zip(levels[k].results(), want[k]))
            assert all(bool((e == 0x5a5a5a5a).all()) for e in keep)
            for lv in others:  # eager calls beside the graphs
                first = [t.clone() for t in lv.results()]
                lv.clear()
                lv.calls()
                assert all(torch.equal(g, w) for g, w in zip(lv.results(), first))
            del graphs
            stream.synchronize()
        assert hy.hydro_get_error(ctx) == (hy.HYDRO_OK, 0)
        hy.hydro_finalize(ctx)


def test_scratch_graphs_outlive_larger_calls():
    """The calls with per-cell scratch (reverse step, MHD in double, the oct builder), captured on a small
    box; then larger boxes; then the replay."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        ctx = hy.hydro_init(precision="fp64")
        dt = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")

        def work(n, seed):
            U, lam, res = _gas(n, seed), _gas(n, seed + 1), torch.zeros((5, n, n, n), dtype=torch.float64, device="cuda")
            M = torch.cat([U, 0.1 * _gas(n, seed + 2)[1:], ])
            M[4] += 1.0
            mout = torch.zeros_like(M)
            z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.int32)] * 3, indexing="ij")
            pos = torch.stack([x, y, z], dim=-1).reshape(-1, 3).contiguous()
            order = torch.empty(len(pos), dtype=torch.int32, device="cuda")
            nbr = torch.empty((len(pos), 27), dtype=torch.int32, device="cuda")
            pu, pl, pr = hy.patch(U, 0, 1.0 / n), hy.patch(lam, 0, 1.0 / n), hy.patch(res, 0, 1.0 / n)

            def calls():
                hy.hydro_adjoint_step(ctx, pu, dt, pl, pr)
                hy.hydro_mhd_step(ctx, M, mout, 1.0 / n, dt)
                hy.hydro_octs_build(ctx, pos, (n, n, n), order, nbr)
            return calls, (res, mout, order, nbr), (pu, pl, M, pos)

        calls, out, _keep = work(12, 1)
        calls()
        stream.synchronize()
        want = [t.clone() for t in out]
        graph = _captured(stream, calls)
        for n in (20, 36):
            work(n, 5)[0]()
            stream.synchronize()
        keep = _eaters()
        for _ in range(2):
            for t in out:
                t.zero_()
            graph.replay()
            stream.synchronize()
            assert all(torch.equal(g, w) for g, w in zip(out, want))
        assert all(bool((e == 0x5a5a5a5a).all()) for e in keep)
        hy.hydro_clear_error(ctx)
        hy.hydro_finalize(ctx)
