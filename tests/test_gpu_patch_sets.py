"""A context keeps the tables of its last patch sets.  Calls that alternate between sets -- more of
them than are kept, in changing order, buffers freed and allocated in between -- must give what a
context that has seen one set only gives, bit for bit."""
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads

pytestmark = pytest.mark.gpu

DX, N = 1.0 / 16, 16


def _set(seed):
    """A coarse 16^3 box and three fine patches of it (one across the period), with outputs."""
    coarse = workloads.white_velocity_state(N, seed=seed, p_jitter=0.2).cuda().contiguous()
    origins = [(2, 4, 6), (14, 4, 6), (24, 20, 28)]
    dims = [(12, 8, 10), (6, 8, 10), (14, 6, 8 + 2 * (seed % 3))]
    ins = [torch.zeros((5, z + 4, y + 4, x + 4), dtype=torch.float64, device="cuda") for x, y, z in dims]
    fine = workloads.white_velocity_state(2 * N, seed=seed + 50, p_jitter=0.2).cuda()
    for t, o, (x, y, z) in zip(ins, origins, dims):
        ix, iy, iz = ((torch.arange(n, device="cuda") + s) % (2 * N) for n, s in zip((x, y, z), o))
        t[:, 2:-2, 2:-2, 2:-2] = fine[:, iz][:, :, iy][:, :, :, ix]
    return coarse, origins, dims, ins


def _work(ctx, data):
    coarse, origins, dims, ins = data
    ins = [t.clone() for t in ins]
    outs = [torch.zeros_like(t) for t in ins]
    regs = [torch.zeros(5 * hy.register_size(*d), dtype=torch.float64, device="cuda") for d in dims]
    dt = torch.full((3,), 2e-3, dtype=torch.float64, device="cuda")
    dn, cfl = torch.empty_like(dt), torch.empty_like(dt)
    cp, a, b = hy.patch(coarse, 0, DX), [hy.patch(t, 2, DX / 2) for t in ins], [hy.patch(t, 2, DX / 2) for t in outs]
    hy.hydro_fill_ghosts(ctx, cp, a, origins)
    hy.hydro_exchange_ghosts(ctx, a, origins, (2 * N,) * 3)
    hy.hydro_patch_fluxes(ctx, a, dt, regs)
    hy.hydro_step(ctx, a, b, dt, dn)
    hy.hydro_fill_ghosts(ctx, cp, b, origins)  # the other buffers, then back
    hy.hydro_exchange_ghosts(ctx, b, origins, (2 * N,) * 3)
    hy.hydro_step(ctx, b, a, dt, dn)
    hy.hydro_cfl_dt(ctx, a, cfl)
    return ins + outs + regs + [dn, cfl]


def test_alternating_sets():
    sets = [_set(s) for s in range(6)]
    want = []
    for data in sets:
        ctx = hy.hydro_init(precision="fp64")
        want.append([t.clone() for t in _work(ctx, data)])
        hy.hydro_finalize(ctx)
    ctx = hy.hydro_init(precision="fp64")
    for order in ((0, 1, 0, 1), (0, 1, 2, 3, 4, 5), (5, 0, 4, 1, 3, 2), (2, 2, 0)):
        for s in order:
            for got, ref in zip(_work(ctx, sets[s]), want[s]):
                assert torch.equal(got, ref)
    hy.hydro_finalize(ctx)


def test_new_set_is_refused_under_capture():
    """A set's tables are uploaded outside a capture only; a kept set can be captured."""
    data = _set(0)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = hy.hydro_init(precision="fp64")
        coarse, origins, dims, ins = data
        outs = [torch.zeros_like(t) for t in ins]
        dt = torch.full((3,), 1e-3, dtype=torch.float64, device="cuda")
        a, b = [hy.patch(t, 2, DX / 2) for t in ins], [hy.patch(t, 2, DX / 2) for t in outs]
        hy.hydro_fill_ghosts(ctx, hy.patch(coarse, 0, DX), a, origins)
        hy.hydro_step(ctx, a, b, dt)
        stream.synchronize()
        want = [t.clone() for t in outs]
        for t in outs:
            t.zero_()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            hy.hydro_step(ctx, a, b, dt)
            with pytest.raises(hy.HydroError):
                hy.hydro_step(ctx, b, a, dt)
        graph.replay()
        stream.synchronize()
        for got, ref in zip(outs, want):
            assert torch.equal(got, ref)
        hy.hydro_finalize(ctx)
