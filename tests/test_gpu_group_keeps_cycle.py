"""A group keeps the cycle that its graph captured when a member's cycle parameters or SMO-2 blocks
change afterwards, bit for bit; the member's own solves take the new ones; the memory kept for the
group is given back."""
import ctypes

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


def members():
    out = [P.Solver(W.star(256), rtol=1e-10, max_iter=200), P.Solver(W.disk_minus(128), rtol=1e-10, max_iter=200, precision=P.CCM_FP64)]
    fs = []
    for k, s in enumerate(out):
        live = s.cell_map()[0] != 0
        fs.append(torch.tensor(np.where(live, np.random.default_rng(k).standard_normal(live.shape), 0.0), device="cuda"))
    return out, fs


def device_bytes(s):
    info = type(s.info)()
    assert P.lib().ccm_query(s.h, ctypes.byref(info)) == 0
    return info.device_bytes


@pytest.mark.parametrize("change", ["cycle", "blocks", "both"])
def test_group_after_its_members_change(change):
    ss, fs = members()
    twin, _ = members()                      # the same changes, never in a group
    g = P.Group(ss)

    def set_to(solvers, omega, blocks):
        for s in solvers:
            if change != "blocks":
                s.set_cycle_params(omega=omega)
            if change != "cycle":
                s.set_smo2_blocks(*blocks)

    try:
        want, st, _ = g.solve(fs)
        for omega, blocks in ((0.6, (48, 16)), (0.55, (32, 16))):
            set_to(ss, omega, blocks)
            set_to(twin, omega, blocks)
            got, st2, _ = g.solve(fs)
            assert [a.iterations for a in st2] == [a.iterations for a in st]
            assert all(torch.equal(a, b) for a, b in zip(got, want))
            for s, t, f in zip(ss, twin, fs):
                assert torch.equal(s.solve(f)[0], t.solve(f)[0])
        g2 = P.Group(ss)                     # captures the new cycle
        for u, s, f in zip(g2.solve(fs)[0], ss, fs):
            assert (u - s.solve(f)[0]).abs().max() <= 1e-7 * u.abs().max()      # two solves to 1e-10
        g2.close()
        assert all(torch.equal(a, b) for a, b in zip(g.solve(fs)[0], want))
        g.close()
        for s in ss:                         # a call that changes nothing gives the kept memory back, too
            s.set_cycle_params()
        assert [device_bytes(s) for s in ss] == [device_bytes(t) for t in twin]
        set_to(ss, 0.6, (48, 16))
        set_to(twin, 0.6, (48, 16))
        assert [device_bytes(s) for s in ss] == [device_bytes(t) for t in twin]
    finally:
        g.close()
        for s in ss + twin:
            s.close()
