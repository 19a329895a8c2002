"""Bin readout on the specialised kernels: shared memory that the launch sizes by the call. The forward's held runs for one
to four observables against the generic kernels, and the relaxed adjoint's chunk sums against its prefix sums, at numbers of
bins around the chunk sizes and for networks whose block sums need more room than the chunks, and less."""
import numpy as np
import pytest
import torch

import ssa_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [3, 200, 1500])
@pytest.mark.parametrize("n_obs", [1, 2, 3, 4])
def test_held_runs(n_obs, S):
    from paper_2602_19775_gb300 import ssa
    spec = W.vilar_oscillator()
    net = ssa.Network(spec)
    theta = torch.tensor(spec.log_rates, dtype=torch.float32, device="cuda")
    out = [ssa.forward(net, theta, 77, spec.x0, 0.1, W.uniform_sample_grid(0.1, S), [7, 4, 6, 1][:n_obs], 3, readout="bin",
                       record=record, max_steps=4096, **how).obs
           for record in (False, True) for how in ({}, dict(specialize=False, threads_per_traj=1))]
    assert all(torch.equal(out[0], o) for o in out[1:])


@pytest.mark.parametrize("S", [31, 32, 100, 801, 897])
@pytest.mark.parametrize("net", ["ion", "oscillator"])
@pytest.mark.parametrize("soft", [False, True])
def test_chunk_sums(net, S, soft):
    """The same gradient for every trajectory, given once (prefix sums) and per trajectory (chunk sums): equal to the
    binary32 rounding of sums of up to S terms over ~100 steps, which cancel to a tenth of their terms or so: 1e-4."""
    from paper_2602_19775_gb300 import ssa
    spec, t_end, observed = (W.ion_channel_coi(n_channels=4), 8.0, 1) if net == "ion" else (W.vilar_oscillator(), 0.05, 4)
    n, T = 150, 0.5
    theta = torch.tensor(spec.log_rates, dtype=torch.float32, device="cuda")
    how = dict(selector="soft", temperature=T) if soft else {}
    fw = ssa.forward(ssa.Network(spec), theta, n, spec.x0, t_end, W.uniform_sample_grid(t_end, S), [observed], 3,
                     readout="bin", record=True, max_steps=1024, **how)
    assert fw.run.variant == 2
    g = torch.tensor(np.random.default_rng(S).standard_normal((S, 1)) / n, dtype=torch.float32, device="cuda")
    shared = ssa.backward(fw, g, T)
    own = ssa.backward(fw, g.expand(n, S, 1).contiguous(), T)
    assert (shared - own).abs().max() <= 1e-4 * shared.abs().max()
