"""The classifier's adjoint with more dynamic species than its register variants hold: its keys and its weights share
words of shared memory, and the check of the recorded reactions must still see the keys (no false mismatch)."""
import numpy as np
import pytest

from ssa_workloads import grn as G
from test_gpu_grn import _grn_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_hid,T", [(286, 0.5), (300, 0.5), (300, 3.0), (400, 1.0)])
def test_recorded_reactions_win_their_races(n_hid, T):
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=2, n_in=6, n_hid=n_hid, n_out=3, w1_scale=0.02, w2_scale=0.2)
    x = np.array([[10, 200, 3, 0, 77, 1], [5, 5, 5, 250, 1, 9]], np.int32)
    _grn_case(ssa, p, x, 48, 1.0, 7, T)  # holds the mismatch count to 0 and the gradients to the oracle's


@pytest.mark.parametrize("n_hid,n_out", [(1200, 40), (3000, 10)])
def test_forward_with_w2_outside_shared_memory(n_hid, n_out):
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=n_hid, n_in=20, n_hid=n_hid, n_out=n_out)
    x, _ = G.prototype_images(seed=1, n_img=3, n_in=20)
    _grn_case(ssa, p, x, 2, 600.0 / (n_hid + n_out + 100), 11, 0.5, max_steps=4096)
