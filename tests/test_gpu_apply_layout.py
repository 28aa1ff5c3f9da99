"""The operator and its transpose straight from the caller's arrays (one launch per call): odd
and ragged sizes, several vectors, values on the cells that hold no unknown, results over their
inputs, wide value ranges and non-finite values; and FP64 sweeps over SMO-2 blocks of odd shapes
(their inverse rows are staged in two halves)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu

CASES = {"box49": (lambda: W.paper_problem3(49), 64), "disk64": (lambda: W.disk_minus(64), 16),
         "star130": (lambda: W.star(130), 65), "rot96": (lambda: W.paper_problem3_rotated(64), 16)}


class Op:
    """L, N and the magnitudes of their terms, assembled from the handle's rows."""

    def __init__(self, prob, coarsest):
        self.s = s = P.Solver(prob, coarsest=coarsest)
        self.live, self.reg = s.cell_map()[0] != 0, s.cell_map()[2] != 0
        self.cell, self.cols, self.beta, self.nb, self.seg = s.level_rows(0)
        lap, gra = np.array([-1, 16, -30, 16, -1]) / 12, np.array([1, -8, 0, 8, -1]) / 12
        self.w = prob.b * np.outer(gra, gra)
        self.w[2] += prob.a * lap
        self.w[:, 2] += prob.c * lap
        self.w /= prob.h ** 2

    def __call__(self, u, g, w=None, beta=None, nb=None):
        w, beta, nb = (self.w, self.beta, self.nb) if w is None else (w, beta, nb)
        u = np.where(self.live, u, 0.0).astype(np.longdouble)
        p = np.pad(u, 2)
        out = sum(w[d, e] * p[d:d + u.shape[0], e:e + u.shape[1]] for d in range(5) for e in range(5) if w[d, e])
        out = np.where(self.reg, out, 0).ravel()
        out[self.cell] = (beta * u.ravel()[self.cols]).sum(1) + np.where(self.seg >= 0, nb * g[np.maximum(self.seg, 0)], 0)
        return out.reshape(u.shape)

    def terms(self, u, g):
        return self(np.abs(u), np.abs(g), np.abs(self.w), np.abs(self.beta), np.abs(self.nb))

    def T(self, v):
        v = np.where(self.live, v, 0.0).astype(np.longdouble)
        p = np.pad(np.where(self.reg, v, 0), 2)
        out = sum(self.w[4 - d, 4 - e] * p[d:d + v.shape[0], e:e + v.shape[1]] for d in range(5) for e in range(5)).ravel()
        np.add.at(out, self.cols.ravel(), (self.beta * v.ravel()[self.cell][:, None]).ravel())
        og = np.zeros(self.s.nseg)
        og[self.seg[self.seg >= 0]] = (self.nb * v.ravel()[self.cell])[self.seg >= 0]
        return np.where(self.live, out.reshape(v.shape), 0), og


@pytest.fixture(scope="module", params=sorted(CASES))
def op(request):
    mk, co = CASES[request.param]
    o = Op(mk(), co)
    yield o
    o.s.close()


def fields(o, n, seed, scale):
    r = np.random.default_rng(seed)
    u = r.standard_normal((n,) + o.live.shape) * (10.0 ** (-scale * r.random((n,) + o.live.shape)))
    return np.where(o.live, u, np.nan), r.standard_normal((n, o.s.nseg))     # the dead cells' values are ignored


@pytest.mark.parametrize("nrhs,scale", [(1, 0), (3, 6)])
def test_apply_and_transpose(op, nrhs, scale):
    u, g = fields(op, nrhs, 5, scale)
    ut, gt = torch.tensor(u, device="cuda"), torch.tensor(g, device="cuda")
    got = op.s.apply(ut, gt).cpu().numpy()
    gu, gg = (x.cpu().numpy() for x in op.s.apply_T(ut))
    for k in range(nrhs):
        uk = np.where(op.live, u[k], 0)
        # a dozen roundings of 2^-53 of the terms' sum
        assert np.abs(got[k] - op(uk, g[k])).max() <= 2e-15 * op.terms(uk, g[k]).max()
        wu, wg = op.T(uk)
        bound = 2e-15 * np.abs(uk).max() * max(np.abs(op.w).sum(), np.abs(op.beta).sum(1).max()) * 4
        assert np.abs(gu[k] - wu).max() <= bound and np.abs(gg[k] - wg).max() <= bound
        assert (got[k][~op.live] == 0).all() and (gu[k][~op.live] == 0).all()
    only_u, _ = op.s.apply_T(ut, want_g=False)
    _, only_g = op.s.apply_T(ut, want_u=False)
    assert np.array_equal(only_u.cpu().numpy(), gu) and np.array_equal(only_g.cpu().numpy(), gg)


def test_result_over_its_input_and_unaligned(op):
    u, g = fields(op, 2, 6, 0)
    ut, gt = torch.tensor(u, device="cuda"), torch.tensor(g, device="cuda")
    want = op.s.apply(ut, gt)
    wt = op.s.apply_T(ut)[0]
    inplace = ut.clone()
    op.s.apply(inplace, gt, out=inplace)
    assert torch.equal(inplace, want)
    big = torch.zeros(ut.numel() + 1, dtype=torch.float64, device="cuda")
    odd = big[1:].view_as(ut)                       # rows on 8 bytes, not 16
    op.s.apply(ut, gt, out=odd)
    assert torch.equal(odd, want) and big[0] == 0
    v = ut.clone()
    assert P.lib().ccm_apply_T(op.s.h, v.data_ptr(), v.data_ptr(), None, 2, torch.cuda.current_stream().cuda_stream) == 0
    assert (v - wt).abs().max() <= 1e-15 * wt.abs().max()


@pytest.mark.parametrize("value", [np.inf, np.nan, 0.0, 1e-290, 1e250])
def test_values_the_integer_form_does_not_take(op, value):
    u, g = fields(op, 1, 7, 0)
    u, g = u[0], 0 * g[0]
    u = u * value if value and np.isfinite(value) else np.where(op.live, 0.0 if value == 0 else u, np.nan)
    if not np.isfinite(value):
        j, i = np.argwhere(op.reg)[len(np.argwhere(op.reg)) // 2]
        u[j, i] = value
    got = op.s.apply(torch.tensor(u, device="cuda")).cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        want = op(u, g).astype(np.float64)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    f = np.isfinite(want)
    assert np.abs(got - want)[f].max() <= 2e-15 * op.terms(np.where(np.isfinite(u), u, 0), g).max()


@pytest.mark.parametrize("block,overlap", [(8, 0), (9, 1), (65, 23), (128, 30)])
def test_fp64_sweeps_over_odd_smo2_blocks(block, overlap):
    # the FP32 sweep stages whole blocks: equal to its rounding
    s = P.Solver(W.star(96), coarsest=48)
    try:
        s.set_smo2_blocks(block, overlap)
        live = s.cell_map()[0] != 0
        r = np.random.default_rng(3)
        u, f = (torch.tensor(np.where(live, r.standard_normal(live.shape), 0.0), device="cuda") for _ in range(2))
        a, b = s.level_smooth(0, u, f, P.CCM_FP64), s.level_smooth(0, u, f, P.CCM_MIXED)
        # 15-term residuals and up to 188-term products in FP32: 200 roundings of 2^-24
        assert (a - b).abs().max() <= 200 * 2.0 ** -24 * max(1.0, float(a.abs().max())) * 4
        again = s.level_smooth(0, u, f, P.CCM_FP64)
        assert torch.equal(a, again)
    finally:
        s.close()
