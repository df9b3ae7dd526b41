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
