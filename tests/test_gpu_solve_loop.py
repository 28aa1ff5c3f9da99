"""A solve as one graph launch (the loop and its test on the device) against one launch per outer
iteration, which a profiled solve takes: equal solutions, iteration counts and residuals."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(precision=P.CCM_FP64), dict(), dict(krylov=2), dict(batch=5), dict(nu1=2, nu2=1),
                                dict(cycle=1), dict(smoother=0), dict(max_iter=0), dict(max_iter=3)],
                         ids=lambda kw: "-".join(f"{k}{v}" for k, v in kw.items()) or "mixed")
@pytest.mark.parametrize("make", [lambda: W.star(96), lambda: W.disk_minus(50)], ids=["star96", "disk50"])
def test_device_loop_equals_the_host_loop(make, kw):
    s = P.Solver(make(), **dict(dict(max_iter=40, rtol=1e-10, coarsest=25), **kw))
    try:
        r = np.random.default_rng(9)
        live = s.cell_map()[0] != 0
        n = 5 if "batch" in kw else 1
        f = torch.tensor(np.where(live, r.standard_normal((n, *live.shape)), 0.0), device="cuda")
        g = torch.tensor(r.standard_normal((n, s.info.n_segments)), device="cuda")
        a, sa = s.solve(f, g, check=False)
        s.profile(1)
        b, sb = s.solve(f, g, check=False)
        s.profile(0)
        c, sc = s.solve(f, g, check=False)
        for u, st in ((b, sb), (c, sc)):
            assert torch.equal(a, u)
            assert (st.iterations, st.rel_residual, list(st.history)) == (sa.iterations, sa.rel_residual, list(sa.history))
        assert sa.iterations <= s_max(kw)
    finally:
        s.close()


def s_max(kw):
    return kw.get("max_iter", 40)
