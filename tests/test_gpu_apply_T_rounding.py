"""The transposed operator scales each cell's sum once.  v is 1 on one regular and one irregular cell, so
that a cell that both reach has the sum of two FP64 coefficients, exactly rounded, times 1 / h^2
(not a power of two), exactly rounded: equal to the same two operations on the host, bit for bit."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


def stencil(a, b, c):
    lap, gra = (-1.0, 16.0, -30.0, 16.0, -1.0), (1.0, -8.0, 0.0, 8.0, -1.0)
    w = np.zeros((5, 5))
    for m in range(5):
        w[2, m] += a * lap[m] / 12.0
        w[m, 2] += c * lap[m] / 12.0
    if b:
        for j in range(5):
            for i in range(5):
                w[j, i] += b * gra[i] * gra[j] / 144.0
    return w


@pytest.mark.parametrize("mk,coarsest", [(lambda: W.disk_minus(88), 11), (lambda: W.paper_problem3_rotated(88), 33), (lambda: W.star(104), 13)])
def test_one_scaling(mk, coarsest):
    prob = mk()
    s = P.Solver(prob, coarsest=coarsest)
    try:
        _, _, rg, _ = s.cell_map()[:4]
        cell, cols, beta, _, _ = s.level_rows(0)
        ih2, w, nx = 1.0 / (prob.h * prob.h), stencil(prob.a, prob.b, prob.c), prob.nx
        assert np.frexp(ih2)[0] != 0.5
        # the stored coefficient whose multiple by 1 / h^2 is the one reported, where there is just one
        cand = np.stack([np.nextafter(beta / ih2, np.inf), beta / ih2, np.nextafter(beta / ih2, -np.inf)])
        hit = cand * ih2 == beta
        one, val = hit.sum(0) == 1, (cand * hit).sum(0)
        pairs, rng = [], np.random.default_rng(2)
        for r in rng.permutation(len(cell)):
            j, i = divmod(int(cell[r]), nx)
            near = [(dj, di) for dj in range(-4, 5) for di in range(-4, 5)
                    if 0 <= j + dj < prob.ny and 0 <= i + di < nx and rg[j + dj, i + di]]
            if near:
                dj, di = near[rng.integers(len(near))]
                pairs.append((r, j + dj, i + di))
            if len(pairs) == 256:
                break
        v = np.zeros((len(pairs), prob.ny, nx))
        for k, (r, j, i) in enumerate(pairs):
            v[k, j, i] = 1.0
            v[k].ravel()[cell[r]] = 1.0
        got = s.apply_T(torch.tensor(v, device="cuda"), want_g=False)[0].cpu().numpy()
        seen = 0
        for k, (r, j, i) in enumerate(pairs):
            for q in range(15):
                J, I = divmod(int(cols[r, q]), nx)
                if one[r, q] and abs(J - j) <= 2 and abs(I - i) <= 2 and w[j - J + 2, i - I + 2]:
                    assert got[k, J, I] == ih2 * (w[j - J + 2, i - I + 2] + val[r, q])
                    seen += 1
        assert seen >= 200
    finally:
        s.close()
