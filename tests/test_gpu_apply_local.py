"""FP64 passes cell by cell: the operator, its transpose, an FP64 sweep and an FP64 residual with
restriction, each cell's error against its own terms, on fields whose values span many decades
within a tile (a narrow kernel, one large value in a smooth field, an exponential)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_apply_layout import Op

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu

CASES = {"disk64": (lambda: W.disk_minus(64), 16), "star130": (lambda: W.star(130), 65),
         "rot96": (lambda: W.paper_problem3_rotated(64), 16), "disk192": (lambda: W.disk_minus(192, 0.1), 24)}
# an FP64 sum of up to 25 terms, its scale and (in the expected values) the rounding of the weights
TOL = 32 * 2.0 ** -53
UNDERFLOW = 32 * 2.0 ** -1074        # and where the terms are subnormal, half of the smallest double a term


@pytest.fixture(scope="module", params=sorted(CASES))
def op(request):
    mk, co = CASES[request.param]
    o = Op(mk(), co)
    yield o
    o.s.close()


def field(o, kind):
    ny, nx = o.live.shape
    j, i = np.mgrid[0:ny, 0:nx].astype(float)
    jc, ic = np.argwhere(o.reg)[o.reg.sum() // 3]
    smooth = np.sin(6.0 * i / nx + 0.3) * np.cos(5.0 * j / ny) + 0.1
    u = {"kernel": np.exp(-((i - ic) ** 2 + (j - jc) ** 2) / 18), "spike": smooth.copy(), "decay": np.exp(-0.8 * i)}[kind]
    if kind == "spike":
        u[jc, ic] = 1e18
    return np.where(o.live, u, 0.0)


def check(got, want, terms, where, scale):
    assert where.any()
    assert (np.abs(got - want)[where] <= TOL * terms[where] + UNDERFLOW * scale).all()


@pytest.mark.parametrize("kind", ["kernel", "spike", "decay"])
def test_operator_and_transpose(op, kind):
    u, ih2 = field(op, kind), op.s.prob.h ** -2
    g = np.zeros(op.s.nseg)
    ut = torch.tensor(u, device="cuda")
    check(op.s.apply(ut).cpu().numpy(), op(u, g), op.terms(u, g), op.live, ih2)
    check(op.s.level_apply(0, ut).cpu().numpy(), op(u, g), op.terms(u, g), op.live, ih2)
    wu, wg = op.T(u)
    both = Op.__new__(Op)
    both.__dict__ = dict(op.__dict__, w=np.abs(op.w), beta=np.abs(op.beta), nb=np.abs(op.nb))
    tu, tg = both.T(np.abs(u))
    gu, gg = (x.cpu().numpy() for x in op.s.apply_T(ut))
    check(gu, wu, tu, op.live, ih2)
    check(gg, wg, tg, np.ones(len(gg), bool), ih2)


@pytest.mark.parametrize("kind", ["kernel", "spike", "decay"])
def test_sweep_and_residual(op, kind):
    u, s = field(op, kind), op.s
    zero = np.zeros_like(u)
    ut, rt = torch.tensor(u, device="cuda"), torch.tensor(zero, device="cuda")
    g = np.zeros(s.nseg)
    lu, terms = op(u, g), op.terms(u, g)
    t = s.params.omega / op.w[2, 2]
    check(s.level_smooth(0, ut, rt, P.CCM_FP64).cpu().numpy(), u - t * lu, np.abs(u) + abs(t) * terms, op.reg, 1.0)
    if s.info.levels < 2:
        return
    vol = np.where(op.live, s.cell_map()[3], 0.0)
    quad = lambda x: x.reshape(x.shape[0] // 2, 2, x.shape[1] // 2, 2)  # noqa: E731
    whole = quad(op.reg).all((1, 3))
    mean = lambda x: quad(vol * x).sum((1, 3)) / np.where(whole, quad(vol).sum((1, 3)), 1.0)  # noqa: E731
    check(s.level_restrict(0, ut, rt).cpu().numpy(), -mean(lu), mean(terms), whole, op.s.prob.h ** -2)
