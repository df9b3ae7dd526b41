"""A context that no call has tuned picks its tile shape and z chunk by a rule on the box or patch
set.  Its step must give what the fixed 16x16 tiles of 32 planes give: the tiling changes no cell's
operations, so states agree to the last rounding of the arithmetic and the fused dt bit for bit."""
import numpy as np
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads

pytestmark = pytest.mark.gpu

# Below one tile, ragged in every axis, one plane, long and flat boxes, several waves of blocks.
BOXES = [(4, 4, 4), (5, 7, 3), (33, 17, 9), (16, 16, 1), (8, 8, 130), (70, 65, 40), (96, 96, 96)]
EPS = {"fp64": 2.0 ** -52, "df64": 2.0 ** -46, "fp32": 2.0 ** -23, "mixed": 2.0 ** -23}


def _close(a, b, precision):
    # rounding of a step's ~30 dependent operations on values of the field's size
    scale = b.abs().amax(dim=tuple(range(1, b.dim())), keepdim=True)
    assert bool(((a - b).abs() <= 32 * EPS[precision] * scale).all())


@pytest.mark.parametrize("precision", ["fp64", "df64", "fp32", "mixed"])
@pytest.mark.parametrize("limiter", ["minmod", "ppm"])
def test_untuned_boxes(precision, limiter):
    for n, (nx, ny, nz) in enumerate(BOXES):
        dtype = torch.float32 if precision == "fp32" else torch.float64
        U = workloads.white_velocity_state((nz, ny, nx), seed=n, p_jitter=0.2).cuda().to(dtype).contiguous()
        dx = 1.0 / nx
        got = []
        for fixed in (False, True):
            ctx = hy.hydro_init(precision=precision, limiter=limiter)
            assert hy.hydro_get_tuning(ctx) == (0, 32)
            if fixed:
                hy.hydro_set_tuning(ctx, 0, 32)
            dt = torch.empty(1, dtype=torch.float64, device="cuda")
            dn, out = torch.empty_like(dt), torch.empty_like(U)
            hy.hydro_cfl_dt(ctx, hy.patch(U, 0, dx), dt)
            hy.hydro_step(ctx, hy.patch(U, 0, dx), hy.patch(out, 0, dx), dt, dn)
            check = torch.empty_like(dt)
            hy.hydro_cfl_dt(ctx, hy.patch(out, 0, dx), check)
            assert hy.hydro_get_error(ctx) == (hy.HYDRO_OK, 0)
            assert dn.item() == check.item()
            got.append(out.double())
            hy.hydro_finalize(ctx)
        _close(got[0], got[1], precision)


@pytest.mark.parametrize("precision", ["fp64", "df64", "fp32", "mixed"])
def test_untuned_patches(precision):
    rng = np.random.default_rng(7)
    dtype = torch.float32 if precision == "fp32" else torch.float64
    parent = workloads.white_velocity_state(40, seed=3, p_jitter=0.2)
    for count, top in ((1, 9), (3, 20), (90, 34)):
        dims = [tuple(int(v) for v in rng.integers(1, top, 3)) for _ in range(count)]
        src = [workloads.ghosted_from_periodic(parent, (3, 5, 7), d).cuda().to(dtype).contiguous() for d in dims]
        got = []
        for fixed in (False, True):
            ctx = hy.hydro_init(precision=precision)
            if fixed:
                hy.hydro_set_tuning(ctx, 0, 32)
            ins = [hy.patch(U, 2, 0.025) for U in src]
            outs = [torch.zeros((5, d[2], d[1], d[0]), dtype=dtype, device="cuda") for d in dims]
            dt = torch.full((count,), 1e-3, dtype=torch.float64, device="cuda")
            dn = torch.empty_like(dt)
            for _ in range(2):  # a first call and one with the kept work-list
                hy.hydro_step(ctx, ins, [hy.patch(o, 0, 0.025) for o in outs], dt, dn)
            assert hy.hydro_get_error(ctx) == (hy.HYDRO_OK, 0)
            got.append([o.double() for o in outs])
            hy.hydro_finalize(ctx)
        for a, b in zip(*got):
            _close(a, b, precision)
