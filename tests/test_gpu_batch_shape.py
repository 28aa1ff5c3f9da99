"""Launch shapes of a handle with a batch: few right-hand sides at a time run as on a handle without one."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


def test_few_right_hand_sides_keep_their_launch_shape():
    # 142 extended rows: three CTAs an SM fit with the scratch of one right-hand side, two with that of four
    one, many = (P.Solver(W.star(1024), coarsest=64, ras_block=64, ras_overlap=39, batch=b) for b in (1, 4))
    try:
        assert many.info.batch == 4
        for n in (1, 2, 3):
            a, b = one.level_launch(0, P.CCM_MIXED, n), many.level_launch(0, P.CCM_MIXED, n)
            assert a.sweep_ctas == b.sweep_ctas > 0
    finally:
        one.close()
        many.close()
