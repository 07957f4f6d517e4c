"""The derivative record of the FP64 stage over a table of patches: chunks of
tiles that run side by side (from 608 tiles on) with boundaries inside and
between patches of different tile volumes, its size, and that a stage takes
nothing from what its scratch held before."""
import numpy as np
import pytest

from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300 import inputs

from gpu_common import RHS_TOL, grid_for, need_gpu, perturbed_bl, rel_err_tensor
from test_gpu_batch import patch_state, step_single

pytestmark = pytest.mark.gpu

# tiles: 125, 25 (5 points along x), 180 (ragged), 240, 1, 90 and 30 (3 along z)
SIZES = [(40, 40, 40), (5, 40, 40), (33, 47, 41), (64, 48, 40), (7, 6, 5), (48, 33, 24), (40, 41, 3)]


@pytest.mark.parametrize("order", [4, 8])
def test_overlapped_chunks_over_patches(order):
    torch = need_gpu()
    g = order // 2 + 1
    p = B.make_params(fd_order=order)
    dt = 0.02
    patches, blocks = [], []
    for b, n in enumerate(SIZES):
        h = 0.5 / 2 ** (b % 2)
        u = patch_state(n, g, h, (0.3 + 0.1 * b, -0.4 + 0.05 * b, 0.2 - 0.07 * b), seed=400 + b)
        grid = grid_for(u, g, h)
        patches.append((u, h))
        blocks.append((grid, B.upload(u, grid), B.upload(u, grid)))
    plan = B.plan_create(blocks, p, B.FP64, 0)
    try:
        _, tiles, shapes = B.plan_info(plan, len(blocks))
        assert tiles == 691 and np.all(shapes == 0)
        B.batch_step(plan, dt)
        torch.cuda.synchronize()
        for n, (u, h), (grid, st, _) in zip(SIZES, patches, blocks):
            want = step_single(u, g, h, p, B.FP64, dt)
            err = rel_err_tensor(B.download(st, grid) - u, want - u, g)
            assert np.max(err) < RHS_TOL, (n, dict(zip(inputs.VARS, err)))
    finally:
        B.plan_destroy(plan)


@pytest.mark.parametrize("patches,n,vol,slots", [(1, 72, 512, 304), (600, 2, 8, 600)])
def test_record_is_as_large_as_its_use(patches, n, vol, slots):
    """A plan's memory: three stage buffers a patch and a record of `slots`
    tiles (135 doubles for each of `vol` points; from 608 tiles on two chunks of
    an eighth of them, rounded up to a multiple of 76: 729 tiles, 2 x 152), to
    64 MB (tables, the graph, 2 MB pages of the device)."""
    torch = need_gpu()
    grid = B.make_grid(n, n, n, ghost=3, dx=0.1)
    p = B.make_params(fd_order=4)
    u = inputs.flat_space(n, n, n, 3)
    blocks = [(grid, B.upload(u, grid), B.upload(u, grid)) for _ in range(patches)]
    warm = B.plan_create(blocks[:1], p, B.FP64, 0)  # what the first plan of a process allocates besides
    B.plan_destroy(warm)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = B.plan_create(blocks, p, B.FP64, 0)
    try:
        used = before - torch.cuda.mem_get_info()[0]
        need = 8 * (3 * 24 * grid.var_stride * patches + 135 * vol * slots)
        assert used <= need + (64 << 20), (used, need)
    finally:
        B.plan_destroy(plan)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("n", [(24, 24, 24), (72, 72, 64)])  # one chunk; chunks side by side
def test_stage_ignores_what_its_scratch_held(order, n):
    torch = need_gpu()
    g = order // 2 + 1
    u = perturbed_bl(*n, g, 0.1, seed=2)
    p = B.make_params(fd_order=order)
    grid = grid_for(u, g, 0.1)
    y0 = B.upload(u, grid)
    got = []
    for fill in (0.0, float("nan")):
        work = B.alloc_work(grid, p)
        work.fill_(fill)
        acc, out = B.alloc_state(grid), B.alloc_state(grid)
        B.diff_tables(grid, p, B.FP64, y0, work)
        B.rk4_stage_fused(grid, p, B.FP64, 0, 0.1, y0, y0, acc, out, work)
        torch.cuda.synchronize()
        got.append((acc, out))
    assert all(torch.equal(a, b) for a, b in zip(*got))
