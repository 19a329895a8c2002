"""The classifier's exact path at network sizes where its layout can go wrong, against the FP64 oracle: one hidden
gene, species counts at the edges of a round of 32 lanes and of the sizes whose sums stay in registers, outputs that
leave the padded columns of W2 ragged, and a network whose arrays leave room for three warps in a block only (and whose
race has more rounds than the choice by bounds keeps slots for)."""
import pytest

from ssa_workloads import grn as G

from test_gpu_grn import _grn_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_hid,n_out", [(1, 1), (30, 2), (31, 2), (96, 1), (91, 5), (187, 5), (193, 13), (284, 4), (285, 4),
                                         (400, 10), (2600, 10)])
def test_sizes(n_hid, n_out):
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=n_hid, n_in=20, n_hid=n_hid, n_out=n_out)
    x, _ = G.prototype_images(seed=1, n_img=3, n_in=20)
    _grn_case(ssa, p, x, 2 if n_hid > 1000 else 16, 600.0 / (n_hid + n_out + 100), 11, 0.5, max_steps=4096)
