"""FP64 sweeps whose SMO-2 block inverses are staged in two parts, on a level with at least 16 blocks
of every shape (fewer blocks of more than 64 core rows do not take the persistent sweep): odd cores,
extended rows of every remainder by four, stages that the blocks and not the tiles set, and the
launch cap, under which one CTA takes several blocks.  Against the oracle's block-Jacobi sweep."""
import pytest

import workloads as W
from test_gpu_parity_ring import CAP, OMEGA, check_prolong_sweep, check_sweep, level0

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2504_00724_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def star288():
    prob = W.star(288)
    return (prob, *level0(prob))


@pytest.mark.parametrize("cap", [0, CAP])
@pytest.mark.parametrize("block,overlap", [(8, 0), (9, 2), (61, 62), (65, 54), (101, 8), (101, 24), (125, 30), (127, 17), (128, 30)])
def test_sweep_over_blocks_in_two_parts(star288, block, overlap, cap):
    prob, lv, coarse = star288
    s = P.Solver(prob, omega=OMEGA, ras_block=block, ras_overlap=overlap)
    try:
        s.set_launch_cap(cap)
        li = s.level_launch(0, P.CCM_FP64)
        assert li.sweep_items > 0 and li.sweep_blocks >= 16        # the persistent sweep
        check_sweep(s, lv, 71, P.CCM_FP64, 1e-10)
        check_prolong_sweep(s, lv, coarse, 72, P.CCM_FP64, 1e-10)
    finally:
        s.close()
