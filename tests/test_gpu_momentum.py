"""Momentum and Gamma constraints of data on which they hold: a gauge wave with
noise, where terms of order 1 cancel and parts in 1e-9 of what is left are the
rounding of the form that is evaluated. An oracle in double precision rounds
differently, and an exact evaluation cannot tell one double-precision form from
another, so the pin is golden values of this library (golden/
momentum_gauge_wave.txt): they were taken when the constraints were first
evaluated in this form and have to stay, to 1e-9 of their norm. The file also
holds the wave's profiles, since a last bit of the input moves the result by
1e-6 of its norm.

File: "profile <variable> <nx values>", then "mom <component> <values>" and
"gcon <component> <values>" over (z, y, x), all as hexadecimal doubles."""
import os

import numpy as np
import pytest

from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300.inputs import IDX, NVAR

from gpu_common import grid_for, interior, need_gpu

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "momentum_gauge_wave.txt")
NX, NY, NZ, ORDER, G = 40, 3, 4, 8, 5


def read_golden(path=GOLDEN):
    d = {}
    with open(path) as f:
        for line in f:
            kind, name, *v = line.split()
            d[kind, name] = np.array([float.fromhex(x) for x in v])
    return d


def state(profiles):
    """Profiles along x (zero where there is none) plus seeded noise of 1e-10,
    periodic; every operation is exactly rounded, so the bits are the same on
    any machine."""
    u = np.zeros((NVAR, NZ, NY, NX))
    for name, p in profiles.items():
        u[IDX[name]] = p
    v, k, j, i = np.meshgrid(*(np.arange(m, dtype=np.uint64) for m in u.shape), indexing="ij")
    r = (((v * 7919 + i * 104729 + j * 1299709 + k * 15485863) * 2654435761) % 2 ** 32) >> 11
    u += (r.astype(np.float64) - 2.0 ** 20) * (1e-10 / 2.0 ** 20)
    wrap = [np.arange(-G, m + G) % m for m in (NZ, NY, NX)]
    return np.ascontiguousarray(u[:, wrap[0]][:, :, wrap[1]][:, :, :, wrap[2]])


def gpu_constraints(u):
    torch = need_gpu()
    grid, p = grid_for(u, G, 1.0 / NX), B.make_params(fd_order=ORDER)
    vs = grid.var_stride
    mom, gcon = (torch.zeros(3 * vs, dtype=torch.float64, device="cuda") for _ in range(2))
    B.constraints(grid, p, B.upload(u, grid), B.alloc_work(grid, p), mom=mom, gcon=gcon)
    torch.cuda.synchronize()
    return {k: interior(B.view4(x, grid, 3).cpu().numpy(), G) for k, x in (("mom", mom), ("gcon", gcon))}


def test_momentum_constraint_of_a_gauge_wave():
    d = read_golden()
    got = gpu_constraints(state({n: p for (k, n), p in d.items() if k == "profile"}))
    for kind in ("mom", "gcon"):
        want = np.array([d[kind, str(c)].reshape(NZ, NY, NX) for c in range(3)])
        # they do cancel: far below the derivatives they are made of
        assert 0 < np.max(np.abs(want)) < 1e-6
        assert np.linalg.norm(got[kind] - want) <= 1e-9 * np.linalg.norm(want), kind


def gpu_weyl_b(u):
    torch = need_gpu()
    grid, p = grid_for(u, G, 1.0 / NX), B.make_params(fd_order=ORDER)
    b = torch.zeros(6 * grid.var_stride, dtype=torch.float64, device="cuda")
    B.psi4(grid, p, B.upload(u, grid), (0.1, 0.2, 0.3), B.alloc_work(grid, p), B=b)
    torch.cuda.synchronize()
    return interior(B.view4(b, grid, 6).cpu().numpy(), G)


def test_magnetic_weyl_tensor_of_a_gauge_wave():
    """It vanishes on a gauge wave by the same kind of cancellation (golden/
    weyl_b_gauge_wave.txt: "B <packed component> <values>")."""
    d = read_golden()
    got = gpu_weyl_b(state({n: p for (k, n), p in d.items() if k == "profile"}))
    w = read_golden(GOLDEN.replace("momentum", "weyl_b"))
    want = np.array([w["B", str(c)].reshape(NZ, NY, NX) for c in range(6)])
    assert 0 < np.max(np.abs(want)) < 1e-6
    assert np.linalg.norm(got - want) <= 1e-9 * np.linalg.norm(want)
