"""The start and the end of a solve (one launch each for all right-hand sides): the zero initial
guess, whose residual is r_hat itself, against the same guess given as an array, on sizes where
rows of the caller's array are not aligned in pairs and with several right-hand sides."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu

CASES = {"box49": (lambda: W.paper_problem3(49), 64), "disk64": (lambda: W.disk_minus(64), 16),
         "star130": (lambda: W.star(130), 65), "rot96": (lambda: W.paper_problem3_rotated(64), 16)}


def inputs(s, nrhs):
    r = np.random.default_rng(5)
    live = s.cell_map()[0] != 0
    f = np.where(live, r.standard_normal((nrhs, *live.shape)), 7.0)     # (empty cells are ignored)
    g = r.standard_normal((nrhs, s.info.n_segments))
    return torch.tensor(f, device="cuda"), torch.tensor(g, device="cuda"), torch.tensor(live, device="cuda")


@pytest.mark.parametrize("precision,batch,nrhs", [(P.CCM_FP64, 1, 1), (P.CCM_FP64, 1, 2), (P.CCM_MIXED, 1, 1),
                                                  (P.CCM_MIXED, 4, 7)])
@pytest.mark.parametrize("name", list(CASES))
def test_zero_guess_equals_an_array_of_zeros(name, precision, batch, nrhs):
    make, coarsest = CASES[name]
    s = P.Solver(make(), coarsest=coarsest, precision=precision, batch=batch, max_iter=4, rtol=1e-13)
    try:
        f, g, live = inputs(s, nrhs)
        zero = torch.zeros((), dtype=torch.float64, device="cuda")
        for gb in (g, None):
            a, sa = s.solve(f, gb, check=False)
            b, sb = s.solve(f, gb, u0=torch.where(live, zero, zero + 3).expand(f.shape).contiguous(), check=False)
            assert sa.iterations == sb.iterations and list(sa.history) == list(sb.history)
            assert torch.equal(a, b) and not a[:, ~live].any() and a.abs().max() > 0
    finally:
        s.close()


def test_zero_and_non_finite_right_hand_sides():
    s = P.Solver(W.disk_minus(128), max_iter=20)
    try:
        f, g, live = inputs(s, 1)
        u, st = s.solve(torch.zeros_like(f))
        assert st.iterations == 0 and st.rel_residual == 0.0 and not u.any()
        f[0][live] = np.nan
        with pytest.raises(Exception):
            s.solve(f, g)
    finally:
        s.close()


def test_group_members_from_zero_and_from_a_guess():
    ss = [P.Solver(W.star(96)), P.Solver(W.disk_minus(64), precision=P.CCM_FP64)]
    fg = [inputs(s, 1) for s in ss]
    fs, gs = [x[0][0] for x in fg], [x[1][0] for x in fg]
    G = P.Group(ss)
    try:
        a, sa, _ = G.solve(fs, gs)
        b, sb, _ = G.solve(fs, gs, us=[torch.zeros_like(fs[0]), None])
        for k in range(2):
            assert torch.equal(a[k], b[k]) and sa[k].iterations == sb[k].iterations > 0
            assert torch.equal(a[k], ss[k].solve(fs[k], gs[k])[0])
    finally:
        G.close()
        for s in ss:
            s.close()
