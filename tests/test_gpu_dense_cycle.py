"""The small levels' part of a V-cycle as one dense matrix (handles of the block-Jacobi smoother,
from the first level below the finest with at most 2048 unknowns, in the precision of the
handle's cycles): against the sweeps it stands for, which the same grid runs in the other
precision's handle, with the cycle parameters and SMO-2 blocks changed after the set-up, and for
batches, whose right-hand sides share reads of the matrix."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu

# (1.2k unknowns at 64^2), (900 at 32^2), (two levels in the matrix, 13^2 at the bottom), (a level of 100 unknowns)
CASES = {"star256": (lambda: W.star(256), 16), "disk128": (lambda: W.disk_minus(128), 16),
         "star104": (lambda: W.star(104), 13), "star40": (lambda: W.star(40), 10)}


@pytest.fixture(scope="module", params=sorted(CASES))
def handles(request):
    mk, co = CASES[request.param]
    d, m = P.Solver(mk(), coarsest=co, precision=P.CCM_FP64), P.Solver(mk(), coarsest=co)
    yield d, m
    d.close()
    m.close()


def fields(s, n, seed):
    live = s.cell_map()[0] != 0
    r = np.random.default_rng(seed)
    return torch.tensor(np.where(live, r.standard_normal((n,) + live.shape), 0.0), device="cuda")


@pytest.mark.parametrize("change", [None, dict(omega=0.5, nu1=1, nu2=2), dict(nu1=0, nu2=3), dict(nu1=2, nu2=0), "blocks"])
def test_matrix_equals_the_sweeps(handles, change):
    d, m = handles
    for s in handles:
        s.set_cycle_params(omega=0.7, nu1=3, nu2=3)
        if change == "blocks":
            s.set_smo2_blocks(48, 16)
        elif change:
            s.set_cycle_params(**change)
    u, r = fields(d, 2, 3)
    a, b = d.vcycle(u, r, P.CCM_FP64), m.vcycle(u, r, P.CCM_FP64)      # the matrix, the sweeps
    # both round some thousand sums of 2^-53; the small levels' condition number is about n^2 = 1e4
    assert (a - b).abs().max() <= 1e-11 * b.abs().max()
    a, b = m.vcycle(u, r, P.CCM_MIXED), d.vcycle(u, r, P.CCM_MIXED)
    assert (a - b).abs().max() <= 2e-5 * b.abs().max()
    if change == "blocks":
        for s in handles:
            s.set_smo2_blocks(64, 24)


@pytest.mark.parametrize("nrhs", [2, 3, 16, 21])
def test_batches_share_reads_of_the_matrix(nrhs):
    prob = W.star(256)
    one, many = P.Solver(prob, rtol=1e-11), P.Solver(prob, rtol=1e-11, batch=nrhs)
    try:
        assert many.info.batch == nrhs
        f = fields(one, nrhs, 5)
        u, st = many.solve(f)
        assert st.rel_residual <= 1e-11
        for k in (0, nrhs - 1):
            v, _ = one.solve(f[k])
            # two solves to a relative residual of 1e-11
            assert (u[k] - v).abs().max() <= 1e-7 * v.abs().max()
    finally:
        one.close()
        many.close()
