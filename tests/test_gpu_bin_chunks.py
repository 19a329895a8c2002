"""Bin readout with one upstream gradient per trajectory: the adjoint's chunk sums against the same adjoint fed one
trajectory's gradient at a time as a shared one (prefix sums, no chunks), at numbers of bins around the chunk sizes, rows
that do not start on 16 bytes, a partial warp, and sizes past the chunks."""
import numpy as np
import pytest
import torch

import ssa_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [31, 32, 33, 64, 500, 801, 896, 897, 1793, 3000])
def test_chunks_match_prefix_sums(S):
    from paper_2602_19775_gb300 import ssa
    spec = W.ion_channel_coi(n_channels=4)
    net = ssa.Network(spec)
    n, t_end = 37, 8.0
    theta = torch.tensor(spec.log_rates, dtype=torch.float32, device="cuda")
    fw = ssa.forward(net, theta, n, spec.x0, t_end, W.uniform_sample_grid(t_end, S), [1], 3, readout="bin", record=True,
                     max_steps=256)
    g = torch.tensor(np.random.default_rng(S).standard_normal((n, S, 1)), dtype=torch.float32, device="cuda")
    total = ssa.backward(fw, g, 0.5).double()
    ref = torch.zeros_like(total)
    for i in range(n):  # trajectory i alone
        one = ssa.forward(net, theta, 1, spec.x0, t_end, W.uniform_sample_grid(t_end, S), [1], 3, readout="bin",
                          record=True, max_steps=256, traj_offset=i)
        ref += ssa.backward(one, g[i], 0.5).double()
    # binary32 sums of up to S terms of order 1 in another order
    assert torch.all((total - ref).abs() <= 1e-5 * S ** 0.5 * n + 1e-5 * ref.abs())
