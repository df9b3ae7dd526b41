"""Long oct lists are stepped cube by cube where 64 consecutive entries are a 4^3 cube of octs.  The
result must be that of the one-oct kernel, which short lists run: bit for bit, over full and holed
levels, Morton and other orders, repeated and invalid entries."""
import numpy as np
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads

pytestmark = pytest.mark.gpu

SHORT = 64 * 100  # below 64 entries per SM: the one-oct kernel


def _level(dims, precision, hole=False, seed=5):
    X, Y, Z = dims
    U = workloads.white_velocity_state((2 * Z, 2 * Y, 2 * X), seed=seed, p_jitter=0.2).cuda()
    V = U.reshape(5, Z, 2, Y, 2, X, 2).permute(0, 1, 3, 5, 2, 4, 6).reshape(5, -1, 8)
    z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.int32) for n in (Z, Y, X)], indexing="ij")
    pos = torch.stack([x, y, z], dim=-1).reshape(-1, 3)
    keep = torch.randperm(len(pos), generator=torch.Generator().manual_seed(seed)).cuda()  # storage in any order
    if hole:
        keep = keep[3:]
    dtype = torch.float32 if precision == "fp32" else torch.float64
    return V[:, keep].to(dtype).contiguous(), pos[keep].contiguous()


def _run(ctx, V, nbr, lists, dx, dt):
    out = torch.full_like(V, 3.0)
    for part in lists:
        hy.hydro_step_octs_table(ctx, V, out, nbr, part.contiguous(), dx, dt)
    bits = hy.hydro_get_error(ctx)[1]
    hy.hydro_clear_error(ctx)
    return out, bits


@pytest.mark.parametrize("precision", ["fp64", "df64", "mixed", "fp32"])
@pytest.mark.parametrize("limiter", ["minmod", "mc"])
@pytest.mark.parametrize("dims,hole", [((24, 20, 22), False), ((25, 23, 19), True), ((32, 32, 32), False)])
def test_cubes_equal_single_octs(precision, limiter, dims, hole):
    V, pos = _level(dims, precision, hole)
    n = len(pos)
    ctx = hy.hydro_init(precision=precision, limiter=limiter)
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    nbr = torch.empty((n, 27), dtype=torch.int32, device="cuda")
    hy.hydro_octs_build(ctx, pos, dims, order, nbr)
    dt = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
    gen = torch.Generator().manual_seed(1)
    mixed = order.clone()
    swap = torch.randint(0, n, (2, 40), generator=gen).cuda()
    mixed[swap[0]], mixed[swap[1]] = order[swap[1]], order[swap[0]]  # some cubes broken, some octs twice
    bad = order.clone()
    bad[n // 3], bad[n // 2] = n + 5, -1
    shifted = torch.cat([order[17:], order[:17]])
    for lst in (order, mixed, bad, shifted, torch.arange(n, dtype=torch.int32, device="cuda")):
        a, bits_a = _run(ctx, V, nbr, [lst], 0.05, dt)
        b, bits_b = _run(ctx, V, nbr, lst.split(SHORT), 0.05, dt)
        assert torch.equal(a, b) and bits_a == bits_b
    # a table that contradicts itself beyond one cube: entries of one oct redirected
    odd = nbr.clone()
    odd[order[n // 2].long(), 4] = order[1]
    odd[order[100].long(), 13] = order[2]
    a, _ = _run(ctx, V, odd, [order], 0.05, dt)
    b, _ = _run(ctx, V, odd, order.split(SHORT), 0.05, dt)
    assert torch.equal(a, b)
    hy.hydro_finalize(ctx)


def test_one_oct_listed_many_times_and_bad_dt():
    """A one-oct periodic level: every run of 64 entries is a cube of copies, more than fit without
    overlap.  A step without a valid dt writes nothing and flags."""
    V, pos = _level((1, 1, 1), "fp64")
    ctx = hy.hydro_init(precision="fp64")
    order = torch.empty(1, dtype=torch.int32, device="cuda")
    nbr = torch.empty((1, 27), dtype=torch.int32, device="cuda")
    hy.hydro_octs_build(ctx, pos, (1, 1, 1), order, nbr)
    dt = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
    lst = torch.zeros(20000, dtype=torch.int32, device="cuda")
    a, _ = _run(ctx, V, nbr, [lst], 0.5, dt)
    b, _ = _run(ctx, V, nbr, [lst[:1]], 0.5, dt)
    assert torch.equal(a, b)
    c, bits = _run(ctx, V, nbr, [lst], 0.5, torch.zeros_like(dt))
    assert bits & hy.EBIT_BAD_DT and bool((c == 3.0).all())
    hy.hydro_finalize(ctx)
