"""The FP64 stage's fixed-point derivatives (bssn_fixed.cuh) at the edges of
their tiles and range, against the CPU oracle.

Tolerance of ordinary data: the per-variable bound of the other right-hand
side tests (1e-12). Data outside the fixed-point range takes double-precision
stencils: results must be non-finite at exactly the oracle's points, and
finite results keep the same bound. A tile that holds a value 2^20 times the
rest resolves 2^-59 of the power of two above that value: every stencil's
error is then at most 2^-58 |u|max times the sum of its weights' moduli,
16 / h^2 for a second derivative and 4 / h for the others, and each enters
the right-hand side with a factor of at most 4 here."""
import numpy as np
import pytest

import oracle
from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300 import inputs

from gpu_common import RHS_TOL, grid_for, interior, need_gpu, oracle_params, perturbed_bl, rel_err

pytestmark = pytest.mark.gpu

H = (0.11, 0.1, 0.13)


def gpu_stage(u, g, h, p):
    """acc after stage 0 with dt = 6: right-hand side plus dissipation."""
    torch = need_gpu()
    grid = grid_for(u, g, h)
    y0 = B.upload(u, grid)
    acc, out = B.alloc_state(grid), B.alloc_state(grid)
    B.rk4_stage(grid, p, B.FP64, 0, 6.0, y0, y0, acc, out, B.alloc_work(grid, p))
    torch.cuda.synchronize()
    return B.download(acc, grid)


# one point, less than a tile, exactly one, one more than a tile along each
# axis, and enough tiles that the record is filled more than once
@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("n", [(1, 1, 1), (7, 3, 2), (8, 8, 8), (9, 8, 17), (16, 9, 8), (40, 33, 24)])
@pytest.mark.parametrize("cubic", [False, True])
def test_tile_edges(order, n, cubic):
    g = order // 2 + 1
    h = 0.1 if cubic else H
    u = perturbed_bl(*n, g, 0.1, seed=sum(n) + order)
    p = B.make_params(fd_order=order)
    want = oracle.rhs(u, g, h, oracle_params(p), ko=True)
    err = rel_err(gpu_stage(u, g, h, p), want, g)
    assert np.max(err) < RHS_TOL, dict(zip(inputs.VARS, err))


# enough tiles that derivatives and algebra of different chunks run side by
# side, with a last chunk that is smaller than the others
@pytest.mark.parametrize("order,h", [(4, 0.1), (8, H)])
def test_overlapped_chunks(order, h):
    g = order // 2 + 1
    u = perturbed_bl(70, 66, 72, g, 0.1, seed=order)
    p = B.make_params(fd_order=order)
    want = oracle.rhs(u, g, h, oracle_params(p), ko=True)
    err = rel_err(gpu_stage(u, g, h, p), want, g)
    assert np.max(err) < RHS_TOL, dict(zip(inputs.VARS, err))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e290, 1e-300])
def test_values_outside_the_fixed_point_range(order, value):
    """One point of the shift's B^1 (it enters only linearly, by its own
    stencils and values), in a grid of several tiles."""
    g = order // 2 + 1
    u = perturbed_bl(20, 10, 18, g, 0.1, seed=5)
    v = inputs.IDX["B1"]
    if value == 1e-300:
        u[v] *= 1e-290  # a whole variable near the bottom of the range
    u[v, g + 4, g + 5, g + 9] = value
    p = B.make_params(fd_order=order)
    want = interior(oracle.rhs(u, g, H, oracle_params(p), ko=True), g)
    got = interior(gpu_stage(u, g, H, p), g)
    fin = np.isfinite(want)
    assert np.array_equal(np.isfinite(got), fin)
    scale = np.max(np.where(fin, np.abs(want), 0.0), axis=(1, 2, 3), keepdims=True)
    assert np.all(np.abs(np.where(fin, got - want, 0.0)) <= RHS_TOL * np.maximum(scale, 1e-300))


@pytest.mark.parametrize("order", [4, 8])
def test_wide_range_within_a_tile(order):
    g, h = order // 2 + 1, 0.1
    u = perturbed_bl(24, 16, 16, g, h, seed=9)
    big = 2.0 ** 20
    for name in ("Gt1", "trK", "beta2", "B3"):
        u[inputs.IDX[name], g + 6, g + 7, g + 10] = big
    p = B.make_params(fd_order=order, advect_gauge=0)
    want = interior(oracle.rhs(u, g, h, oracle_params(p), ko=True), g)
    got = interior(gpu_stage(u, g, h, p), g)
    # away from the spike (its own stencils see 2^20-sized terms in both)
    r = order // 2 + 2
    far = np.ones(want.shape[1:], dtype=bool)
    far[6 - r:6 + r + 1, 7 - r:7 + r + 1, 10 - r:10 + r + 1] = False
    bound = 4 * 2.0 ** -58 * big * (16 / h ** 2 + 4 / h)
    scale = np.max(np.abs(want[:, far]), axis=1, keepdims=True)
    assert np.all(np.abs((got - want)[:, far]) <= bound + RHS_TOL * scale)


# a scratch that holds some of the tiles at a time, and one that holds them
# all: 27, 36 and 80 tiles also lie on both sides of the rule that divides the
# algebra of 32 points between two warps
@pytest.mark.parametrize("n", [(24, 24, 24), (32, 24, 23), (40, 32, 31)])
@pytest.mark.parametrize("least", [False, True])
def test_scratch_sizes(n, least):
    torch = need_gpu()
    g, p = 3, B.make_params(fd_order=4)
    u = perturbed_bl(*n, g, 0.1, seed=7)
    grid = grid_for(u, g, 0.1)
    nb = B.work_bytes(grid, p, B.FP32_RHS if least else B.FP64)  # the FP32 form's is the least either accepts
    assert nb <= B.work_bytes(grid, p, B.FP64)
    y0 = B.upload(u, grid)
    acc, out = B.alloc_state(grid), B.alloc_state(grid)
    work = torch.empty(nb // 8, dtype=torch.float64, device="cuda")
    B.rk4_stage(grid, p, B.FP64, 0, 6.0, y0, y0, acc, out, work)
    torch.cuda.synchronize()
    want = oracle.rhs(u, g, 0.1, oracle_params(p), ko=True)
    err = rel_err(B.download(acc, grid), want, g)
    assert np.max(err) < RHS_TOL, dict(zip(inputs.VARS, err))
    if least:
        with pytest.raises(Exception):
            B.rk4_stage(grid, p, B.FP64, 0, 6.0, y0, y0, acc, out, work[:-1])
