"""A point's FP64 derivatives are as good as what its own stencils read allows,
whatever else lies in its tile of 8 x 8 x 8 points (bssn_fixed.cuh): one value
far larger than the rest must leave every result that does not read it where
the other right-hand side tests have it (1e-12 of the variable's largest value
among them).

Which results read the value is what a NaN in its place reaches in the oracle."""
import numpy as np
import pytest

import oracle
from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300.inputs import IDX

from gpu_common import RHS_TOL, grid_for, interior, need_gpu, oracle_params, perturbed_bl

pytestmark = pytest.mark.gpu

SPIKE = (6, 7, 10)  # z, y, x among 16 x 16 x 24 points, inside a tile


def check(got, want, nan):
    """Every variable where the NaN does not reach."""
    for v in range(len(want)):
        far = np.isfinite(nan[v])
        assert np.count_nonzero(far) > 0.5 * far.size
        err = np.max(np.abs((got[v] - want[v])[far]))
        assert err <= RHS_TOL * np.max(np.abs(want[v][far])), (v, err)


def spiked(g, names, value, seed=9):
    u = perturbed_bl(24, 16, 16, g, 0.1, seed=seed)
    for name in names:
        u[IDX[name]][tuple(g + i for i in SPIKE)] = value
    return u


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("h", [0.1, (0.11, 0.1, 0.13)])
# on both sides of the ranges that integers alone (2^7), integers and fractions
# (2^28) and doubles serve
@pytest.mark.parametrize("big", [2.0 ** 4, 2.0 ** 9, 2.0 ** 20, 2.0 ** 26, 2.0 ** 30, 2.0 ** 60, 1e100])
def test_spike_in_a_stage(order, h, big):
    torch = need_gpu()
    g, names = order // 2 + 1, ("Gt1", "trK", "At12", "beta2", "B3")
    u = spiked(g, names, big)
    p = B.make_params(fd_order=order, advect_gauge=0)
    grid = grid_for(u, g, h)
    y0, acc, out = B.upload(u, grid), B.alloc_state(grid), B.alloc_state(grid)
    B.rk4_stage(grid, p, B.FP64, 0, 6.0, y0, y0, acc, out, B.alloc_work(grid, p))  # acc: RHS + dissipation
    torch.cuda.synchronize()
    f = lambda w: interior(oracle.rhs(w, g, h, oracle_params(p), ko=True), g)
    check(interior(B.download(acc, grid), g), f(u), f(spiked(g, names, np.nan)))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("big", [2.0 ** 20, 1e100])
def test_spike_in_a_right_hand_side(order, big):
    """Without dissipation a variable's stencils reach further on one side."""
    torch = need_gpu()
    g, names = order // 2 + 1, ("At12", "B3")
    u = spiked(g, names, big)
    p = B.make_params(fd_order=order)
    grid = grid_for(u, g, 0.1)
    d, out = B.upload(u, grid), B.alloc_state(grid)
    B.rhs(grid, p, B.FP64, d, out, B.alloc_work(grid, p))
    torch.cuda.synchronize()
    f = lambda w: interior(oracle.rhs(w, g, 0.1, oracle_params(p), ko=False), g)
    check(interior(B.download(out, grid), g), f(u), f(spiked(g, names, np.nan)))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("big", [2.0 ** 20, 1e100])
def test_spike_in_the_hamiltonian_constraint(order, big):
    torch = need_gpu()
    g = order // 2 + 1
    u = spiked(g, ("Gt2",), big)
    p = B.make_params(fd_order=order)
    grid = grid_for(u, g, 0.1)
    ham = torch.zeros(grid.var_stride, dtype=torch.float64, device="cuda")
    B.hamiltonian(grid, p, B.upload(u, grid), B.alloc_work(grid, p), ham=ham)
    torch.cuda.synchronize()
    f = lambda w: interior(oracle.constraints(w, g, 0.1, order, fields=True)[3][0], g)[None]
    check(interior(B.view4(ham, grid, 1).cpu().numpy(), g), f(u), f(spiked(g, ("Gt2",), np.nan)))


def unread(u, g, line, square):
    """The padded points that no stencil of an interior point reads: further out
    than `line` along one axis, than `square` along two, or along all three."""
    out = []
    for m in u.shape[1:]:
        i = np.arange(m)
        out.append(np.maximum(np.maximum(g - i, i - (m - g - 1)), 0))
    d = np.sort(np.stack(np.meshgrid(*out, indexing="ij")), axis=0)  # distances outside, the smallest first
    return (d[0] > 0) | (d[1] > square) | ((d[1] == 0) & (d[2] > line)) | ((d[1] > 0) & (d[2] > square))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("n", [(13, 21, 5), (16, 8, 8)])
@pytest.mark.parametrize("value", [1e200, np.nan])
def test_unread_ghosts_do_not_matter(order, n, value):
    """Bit for bit, in a stage (lines of r = p/2 + 1 points) and in the constraints (p/2)."""
    torch = need_gpu()
    g, H = order // 2 + 2, order // 2
    u = perturbed_bl(*n, g, 0.1, seed=3)
    p = B.make_params(fd_order=order)
    grid = grid_for(u, g, 0.1)

    def stage(w):
        y0, acc, out = B.upload(w, grid), B.alloc_state(grid), B.alloc_state(grid)
        B.rk4_stage(grid, p, B.FP64, 0, 0.1, y0, y0, acc, out, B.alloc_work(grid, p))
        return interior(B.download(out, grid), g)

    def constraints(w):
        vs = grid.var_stride
        f = [torch.zeros(k * vs, dtype=torch.float64, device="cuda") for k in (1, 3, 3)]
        l2, mx, _ = B.constraints(grid, p, B.upload(w, grid), B.alloc_work(grid, p), *f)
        return np.concatenate([interior(B.view4(x, grid, k).cpu().numpy(), g) for x, k in zip(f, (1, 3, 3))])

    for run, line in ((stage, H + 1), (constraints, H)):
        w = u.copy()
        w[:, unread(u, g, line, H)] = value
        assert np.array_equal(run(w), run(u)), run.__name__


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("gauge", [dict(lapse=0, shift=0), dict(lapse=2, shift=1)])
def test_reach_of_a_right_hand_side(order, gauge):
    """A right-hand side without dissipation reads the outermost ghosts on the
    side that the shift points to, and no others (with a frozen gauge, none at
    all for the gauge variables): NaNs there reach those points alone."""
    torch = need_gpu()
    g = order // 2 + 1
    u = perturbed_bl(13, 18, 11, g, 0.1, seed=order)
    p = B.make_params(fd_order=order, **gauge)
    want = interior(oracle.rhs(u, g, 0.1, oracle_params(p), ko=False), g)
    beta = interior(u, g)[IDX["beta1"]:IDX["beta1"] + 3]
    reached = np.zeros(want.shape[1:], dtype=bool)
    w = u.copy()
    for a in range(3):
        ends = [tuple(e if b == 2 - a else slice(None) for b in range(3)) for e in (0, -1)]
        for e in ends:
            w[(slice(None),) + e] = np.nan
        reached[ends[0]] |= beta[a][ends[0]] < 0
        reached[ends[1]] |= beta[a][ends[1]] >= 0
    assert 0 < np.count_nonzero(reached) < reached.size / 2
    grid = grid_for(u, g, 0.1)
    d, out = B.upload(w, grid), B.alloc_state(grid)
    B.rhs(grid, p, B.FP64, d, out, B.alloc_work(grid, p))
    torch.cuda.synchronize()
    got = interior(B.download(out, grid), g)
    for v in range(len(want)):
        if gauge["lapse"] == 2 and v >= IDX["alpha"]:
            assert np.all(got[v] == 0.0), v
            continue
        assert np.array_equal(np.isnan(got[v]), reached), v
        err = np.max(np.abs((got[v] - want[v])[~reached]))
        assert err <= RHS_TOL * np.max(np.abs(want[v][~reached])), v
