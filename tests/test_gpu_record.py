"""The derivative record of the FP64 stage over a table of patches: its size."""
import pytest

from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300 import inputs

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

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
