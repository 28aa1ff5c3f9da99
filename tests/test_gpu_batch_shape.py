"""Launch shapes of a handle with a batch: few right-hand sides at a time run as on a handle without one,
in batches of 32 and more four share block items, and the launch cap holds for a short last group too."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


def test_few_right_hand_sides_keep_their_launch_shape():
    # 142 extended rows: three CTAs an SM fit with the scratch of one right-hand side, two with that of four
    one, many = (P.Solver(W.star(1024), coarsest=64, ras_block=64, ras_overlap=39, batch=b) for b in (1, 32))
    try:
        assert many.info.batch == 32
        for n in (1, 2, 3, 4, 31):
            a, b = one.level_launch(0, P.CCM_MIXED, n), many.level_launch(0, P.CCM_MIXED, n)
            assert a.sweep_ctas == b.sweep_ctas > 0
    finally:
        one.close()
        many.close()


@pytest.mark.parametrize("nrhs", [3, 4, 31, 32, 33, 35])
def test_reported_and_capped_shapes(nrhs):
    s = P.Solver(W.star(288), rtol=1e-11, max_iter=200, batch=nrhs)
    try:
        assert s.info.batch == nrhs
        live = torch.tensor(s.cell_map()[0] != 0, device="cuda")
        f = torch.randn((nrhs,) + tuple(live.shape), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(4)) * live
        want, _ = s.solve(f)
        for cap in (1, 3):
            s.set_launch_cap(cap)
            single, li = s.level_launch(0, P.CCM_MIXED, 1), s.level_launch(0, P.CCM_MIXED, nrhs)
            share = 4 if nrhs >= 32 else 1
            assert li.sweep_ctas == cap and li.sweep_blocks == -(-single.sweep_blocks // share)
            assert li.sweep_items - li.sweep_blocks == single.sweep_items - single.sweep_blocks
            # items of a group over the CTAs of a group: what its CTAs work through, to the rounding of a quarter block
            tiles = single.sweep_items - single.sweep_blocks
            assert abs((single.sweep_blocks + share * tiles) / (share * cap) - li.sweep_items / li.sweep_ctas) <= 1
            assert torch.equal(s.solve(f)[0], want)
    finally:
        s.close()
