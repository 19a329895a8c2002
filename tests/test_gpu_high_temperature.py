"""Soft weights at high temperatures: at an infinite one, which the batch and the classifier accept, every reaction that
can fire weighs the same and one that cannot weighs nothing."""
import numpy as np
import pytest
import torch

import ssa_workloads as W
from oracle import native
from ssa_workloads import grn as G
from test_gpu_parity import GRAD_RTOL, _oracle_theta

pytestmark = pytest.mark.gpu
INF = float("inf")


@pytest.mark.parametrize("threads", [1, 32])
def test_batch_at_infinite_temperature(threads):
    """Immigration-death starts with no molecule, so one of its two reactions has rate 0 at first. At T = inf the
    choice's path carries nothing and the gradient is that of the waiting times alone."""
    from paper_2602_19775_gb300 import ssa
    spec, n, ts = W.immigration_death(), 256, np.array([1.0, 2.0])
    t32 = spec.log_rates.astype(np.float32)
    item = dict(net=ssa.Network(spec), log_rates=t32, n_traj=n, x0=spec.x0, t_end=2.0, sample_times=ts, obs_species=[0],
                seed=3, max_steps=512, threads_per_traj=threads)
    b = ssa.Batch([item], readout="linear", temperature=INF)
    dl = W.seeded_dl_dobs(4, n, 2, 1, scale=1.0 / n)
    orc = native.run(spec, _oracle_theta(t32), spec.x0, n, 2.0, ts, [0], 3, native.LINEAR, max_steps=512, dl_dobs=dl,
                     temperature=1e30, ev_cap=512)
    b.dl_dobs[0].copy_(torch.tensor(dl, dtype=torch.float32))
    b.run()
    torch.cuda.synchronize()
    assert np.all(b.events(0, 512).cpu().numpy() == orc.events)
    g, ref = b.dtheta[0].double().cpu().numpy(), orc.dtheta.sum(0)
    assert np.linalg.norm(g - ref) <= GRAD_RTOL * np.linalg.norm(ref), (g, ref)


@pytest.mark.parametrize("n_hid", [4, 300])
def test_classifier_at_infinite_temperature(n_hid):
    """The readout has no waiting-time path, so every gradient is exactly 0 at T = inf."""
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=1, n_in=5, n_hid=n_hid, n_out=3, w1_scale=0.02, w2_scale=0.5)
    x = np.array([[10, 200, 3, 0, 77], [5, 5, 5, 250, 1]], np.int32)
    net = ssa.GRN(p.n_in, p.n_hid, p.n_out, p.k_max)
    fw = ssa.grn_forward(net, p.W1, p.b1, p.W2, p.b2, p.log_d, x, 16, 1.0, [1.0], 3, max_steps=1 << 12)
    g = ssa.grn_backward(fw, torch.ones((32, 1, 3), device="cuda"), INF)
    for k, v in g.items():
        assert torch.count_nonzero(v) == 0, (k, v)
