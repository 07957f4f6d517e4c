"""Rounding error of the right-hand sides of Gt^i and B^i, whose terms of
different size are gathered before they are scaled: against the same formulas
in extended precision (numpy's long double) it must be no larger, in the norm,
than that of evaluating them term by term in double precision."""
import numpy as np
import pytest

from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300 import inputs
from paper_1307_6488_gb300.inputs import IDX, SYM

from gpu_common import grid_for, interior, need_gpu, perturbed_bl

pytestmark = pytest.mark.gpu

R3 = range(3)
# numerators and denominator of the first derivative (a = 1 ..), second
# derivative, upwinded derivative (from offset 1 - p/2) and dissipation
W1 = {4: ([8, -1], 12), 8: ([672, -168, 32, -3], 840)}
W2 = {4: ([16, -1], 12), 8: ([8064, -1008, 128, -9], 5040)}
UP = {4: ([-3, -10, 18, -6, 1], 12), 8: ([-5, 60, -420, -378, 1050, -420, 140, -30, 3], 840)}
KO = {4: ([15, -6, 1], 64), 8: ([210, -120, 45, -10, 1], 1024)}


def gamma_rhs(u, g, h, order, eps, eta, T):
    """Right-hand sides (with dissipation) of Gt^1..3 and B^1..3, in arithmetic T."""
    u, h = u.astype(T), T(h)
    n = [m - 2 * g for m in u.shape[1:]]

    def at(f, off=(0, 0, 0)):  # off = (x, y, z)
        return f[tuple(slice(g + off[2 - b], g + off[2 - b] + n[b]) for b in range(3))]

    def e(a, o):
        return tuple(o if b == a else 0 for b in R3)

    def add(*offs):
        return tuple(sum(o) for o in zip(*offs))

    w1 = [T(w) / T(W1[order][1]) for w in W1[order][0]]

    def d1(f, a, off=(0, 0, 0)):
        return sum(w * (at(f, add(off, e(a, k + 1))) - at(f, add(off, e(a, -k - 1)))) for k, w in enumerate(w1)) / h

    def d2(f, a, b):
        if a != b:
            return sum(w * (d1(f, a, e(b, k + 1)) - d1(f, a, e(b, -k - 1))) for k, w in enumerate(w1)) / h
        num, den = W2[order]
        return sum(T(w) / T(den) * ((at(f, e(a, k + 1)) + at(f, e(a, -k - 1))) - 2 * at(f))
                   for k, w in enumerate(num)) / h ** 2

    c = [at(f) for f in u]
    gt = [[c[IDX["gt11"] + SYM[i][j]] for j in R3] for i in R3]
    cof = [[gt[(i + 1) % 3][(j + 1) % 3] * gt[(i + 2) % 3][(j + 2) % 3]
            - gt[(i + 1) % 3][(j + 2) % 3] * gt[(i + 2) % 3][(j + 1) % 3] for j in R3] for i in R3]
    det = sum(gt[0][j] * cof[0][j] for j in R3)
    gu = [[cof[i][j] / det for j in R3] for i in R3]
    dg = [[[d1(u[IDX["gt11"] + SYM[i][j]], k) for j in R3] for i in R3] for k in R3]
    low = [[[(dg[i][k][j] + dg[j][k][i] - dg[k][i][j]) / 2 for j in R3] for i in R3] for k in R3]
    G = [[[sum(gu[k][l] * low[l][i][j] for l in R3) for j in R3] for i in R3] for k in R3]
    Gd = [sum(gu[i][j] * G[k][i][j] for i in R3 for j in R3) for k in R3]
    A = [[c[IDX["At11"] + SYM[i][j]] for j in R3] for i in R3]
    Au = [[sum(gu[i][k] * gu[j][l] * A[k][l] for k in R3 for l in R3) for j in R3] for i in R3]
    beta = [u[IDX["beta1"] + i] for i in R3]
    db = [[d1(beta[i], k) for i in R3] for k in R3]
    dal, dW, dK = ([d1(u[IDX[v]], k) for k in R3] for v in ("alpha", "W", "trK"))
    al, W, div = c[IDX["alpha"]], c[IDX["W"]], db[0][0] + db[1][1] + db[2][2]
    grad_div = [sum(d2(beta[k], min(j, k), max(j, k)) for k in R3) for j in R3]

    def transport(f):  # upwinded advection and dissipation
        num, den = UP[order]
        lo = 1 - order // 2
        out = T(0)
        for a in R3:
            s = [sum(T(w) / T(den) * at(f, e(a, sg * (lo + q))) for q, w in enumerate(num)) for sg in (1, -1)]
            b = at(beta[a])
            out = out + np.where(b >= 0, b * s[0], -b * s[1])
        num, den = KO[order]
        ko = sum(T(w) * ((at(f, e(a, q + 1)) + at(f, e(a, -q - 1))) - 2 * at(f)) for a in R3 for q, w in enumerate(num))
        return (out + T(eps) / T(den) * ko) / h

    dG, dB = [], []
    for i in R3:
        r = sum(gu[j][k] * d2(beta[i], min(j, k), max(j, k)) for j in R3 for k in R3)
        r = r + sum(gu[i][j] * grad_div[j] for j in R3) / 3 + 2 * Gd[i] * div / 3
        r = r - sum(Gd[j] * db[j][i] for j in R3) - 2 * sum(Au[i][j] * dal[j] for j in R3)
        r = r + 2 * al * (sum(G[i][j][k] * Au[j][k] for j in R3 for k in R3)
                          - 3 * sum(Au[i][j] * dW[j] for j in R3) / W - 2 * sum(gu[i][j] * dK[j] for j in R3) / 3)
        dG.append(r + transport(u[IDX["Gt1"] + i]))
        dB.append(r - T(eta) * c[IDX["B1"] + i] + transport(u[IDX["B1"] + i]))
    return np.array(dG + dB)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("data", ["gauge_wave", "punctures"])
def test_error_of_gamma_and_b(order, data):
    torch = need_gpu()
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        pytest.skip("long double is no wider than double")
    g = order // 2 + 1
    if data == "gauge_wave":
        u, h = inputs.gauge_wave(24, g, amplitude=0.03, noise=1e-10, seed=1307)
    else:
        h = 0.25
        u = perturbed_bl(24, 20, 22, g, h, seed=order)
    p = B.make_params(fd_order=order, ko_eps=0.1, eta=2.0)
    grid = grid_for(u, g, h)
    y0, acc, out = B.upload(u, grid), B.alloc_state(grid), B.alloc_state(grid)
    B.rk4_stage(grid, p, B.FP64, 0, 6.0, y0, y0, acc, out, B.alloc_work(grid, p))
    torch.cuda.synchronize()
    rows = [IDX["Gt1"] + i for i in R3] + [IDX["B1"] + i for i in R3]
    got = interior(B.download(acc, grid), g)[rows]
    want = gamma_rhs(u, g, h, order, 0.1, 2.0, np.longdouble)
    plain = gamma_rhs(u, g, h, order, 0.1, 2.0, np.float64)
    err = lambda x: np.array([float(np.sqrt(np.sum((a - b) ** 2) / np.sum(b ** 2))) for a, b in zip(x, want)])
    assert np.all(err(plain) < 1e-12)
    assert np.all(err(got) <= err(plain)), (err(got), err(plain))
