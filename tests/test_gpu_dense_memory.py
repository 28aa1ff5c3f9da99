"""The small levels' matrix where its set-up scratch does not fit (requests that report no memory,
ccm_fail_scratch): fewer CTAs, or the levels' sweeps; never an error, never a matrix of other
cycle parameters or SMO-2 blocks than the sweeps'."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu
ALL, CHANGE = 10 ** 6, dict(omega=0.6, nu1=3, nu2=3)


@pytest.fixture(autouse=True)
def reset():
    yield
    P.lib().ccm_fail_scratch(0)


def pair():
    prob = W.star(256)
    s, other = P.Solver(prob, rtol=1e-11, precision=P.CCM_FP64), P.Solver(prob)     # the matrix; sweeps in FP64
    live = s.cell_map()[0] != 0
    r = np.random.default_rng(9)
    return s, other, [torch.tensor(np.where(live, r.standard_normal(live.shape), 0.0), device="cuda") for _ in range(2)]


def launches(s, u, r):
    n = P.lib().ccm_launch_count()
    s.vcycle(u, r, P.CCM_FP64)
    return P.lib().ccm_launch_count() - n


@pytest.mark.parametrize("change", ["cycle", "blocks"])
def test_rebuild_without_memory_runs_the_sweeps(change):
    s, other, (u, r) = pair()
    try:
        with_matrix = launches(s, u, r)
        set_to = (lambda x: x.set_cycle_params(**CHANGE)) if change == "cycle" else (lambda x: x.set_smo2_blocks(48, 16))
        P.lib().ccm_fail_scratch(ALL)
        set_to(s)
        P.lib().ccm_fail_scratch(0)
        set_to(other)
        assert launches(s, u, r) > with_matrix
        a, b = s.vcycle(u, r, P.CCM_FP64), other.vcycle(u, r, P.CCM_FP64)
        assert torch.equal(a, b)                       # the same sweeps
        assert s.solve(r)[1].rel_residual <= 1e-11
        set_to(s)                                      # with memory: the matrix again
        a = s.vcycle(u, r, P.CCM_FP64)
        assert launches(s, u, r) < launches(other, u, r)
        assert (a - b).abs().max() <= 1e-11 * b.abs().max()       # as test_gpu_dense_cycle.py
    finally:
        s.close()
        other.close()


def test_less_scratch_gives_the_same_matrix():
    s, other, (u, r) = pair()
    try:
        s.set_cycle_params(**CHANGE)
        want, n = s.vcycle(u, r, P.CCM_FP64), launches(s, u, r)
        s.set_cycle_params(omega=0.7, nu1=3, nu2=3)
        P.lib().ccm_fail_scratch(5)
        s.set_cycle_params(**CHANGE)
        assert launches(s, u, r) == n and torch.equal(s.vcycle(u, r, P.CCM_FP64), want)
    finally:
        s.close()
        other.close()


def test_setup_without_memory():
    P.lib().ccm_fail_scratch(ALL)
    s, other, (u, r) = pair()
    try:
        assert torch.equal(s.vcycle(u, r, P.CCM_FP64), other.vcycle(u, r, P.CCM_FP64))
        assert s.solve(r)[1].rel_residual <= 1e-11 and s.solve_T(r)[1].rel_residual <= 1e-11
    finally:
        s.close()
        other.close()


def test_parameters_that_the_matrix_does_not_depend_on_keep_it():
    s, other, (u, r) = pair()
    try:
        want = s.vcycle(u, r, P.CCM_FP64)
        n = P.lib().ccm_launch_count()
        s.set_cycle_params(inner_cycles=2, cycle=1)
        s.set_cycle_params(inner_cycles=1, cycle=0)
        assert P.lib().ccm_launch_count() == n         # nothing ran on the device
        assert torch.equal(s.vcycle(u, r, P.CCM_FP64), want)
        assert s.solve(r)[1].rel_residual <= 1e-11
    finally:
        s.close()
        other.close()
