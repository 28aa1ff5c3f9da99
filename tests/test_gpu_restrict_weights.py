"""Restriction weights are held for the precision of the handle's cycles, and for the other one from the
first call in it on; a call that a stream capture records allocates nothing and gives the same
values to rounding."""
import ctypes

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


def device_bytes(s):
    info = type(s.info)()
    assert P.lib().ccm_query(s.h, ctypes.byref(info)) == 0
    return info.device_bytes


def padded(n):
    return ((n + 4 + 31) // 32 * 32) * (n + 4)


def fields(s, n):
    live = s.cell_map()[0] != 0
    r = np.random.default_rng(n)
    return [torch.tensor(np.where(live, r.standard_normal(live.shape), 0.0), device="cuda") for _ in range(2)]


@pytest.mark.parametrize("own,other", [(P.CCM_MIXED, P.CCM_FP64), (P.CCM_FP64, P.CCM_MIXED)])
def test_weights_of_the_other_precision_come_with_its_first_call(own, other):
    s = P.Solver(W.star(288), coarsest=36, precision=own)       # the levels from 72 cells on restrict by tiles
    try:
        u, r = fields(s, 1)
        s.vcycle(u, r, own)
        b0 = device_bytes(s)
        first = s.vcycle(u, r, other)
        more = device_bytes(s) - b0
        assert more == (8 if other == P.CCM_FP64 else 4) * sum(map(padded, (288, 144, 72)))
        assert torch.equal(s.vcycle(u, r, other), first) and device_bytes(s) == b0 + more
    finally:
        s.close()


def test_first_call_under_capture():
    a, b = P.Solver(W.star(288), coarsest=36), P.Solver(W.star(288), coarsest=36)
    try:
        u, r = fields(a, 2)
        want = b.vcycle(u, r, P.CCM_FP64)
        b0 = device_bytes(a)
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        got = u.clone()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            assert P.lib().ccm_vcycle(a.h, got.data_ptr(), r.data_ptr(), P.CCM_FP64, stream.cuda_stream) == 0
        assert device_bytes(a) == b0
        graph.replay()
        torch.cuda.synchronize()
        # FP64 passes over the same cycle: as test_gpu_dense_cycle.py
        assert (got - want).abs().max() <= 1e-11 * want.abs().max()
        assert (a.vcycle(u, r, P.CCM_FP64) - want).abs().max() <= 1e-11 * want.abs().max()
    finally:
        a.close()
        b.close()
