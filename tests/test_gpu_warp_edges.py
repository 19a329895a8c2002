"""Warp-per-trajectory kernels where their layout and their choice without logarithms can go wrong, against the
FP64 oracle: a last round of Philox blocks with one and with 32 lanes at work, more rounds than the choice keeps
slots for (M > 2047, where the tables also leave shared memory), reactions with more than four entries, every order
of reactant with absent ones, and rates so small or so large that the keys leave the range the bounds assume."""
import numpy as np
import pytest
import torch

import ssa_workloads as W
from ssa_workloads.configs import HOLD, LINEAR

from test_gpu_warp import _parity, _pilot_t_end

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2602_19775_gb300 import ssa
    ssa._lib.lib()
    return ssa


@pytest.mark.parametrize("M", [124, 127, 128, 511, 2100])
def test_block_rounds(S, M):
    net = W.random_network(np.random.default_rng(M), n_species_range=(20, 30), n_reactions_range=(M, M))
    t_end = _pilot_t_end(net, net.log_rates.astype(np.float32).astype(np.float64), target_draws=100)
    _parity(S, net, net.log_rates, 64, t_end, 9, np.array([0, 1], np.int32), M, LINEAR, 1.0, tpt=32)


def _wide_changes():
    """Reactions that change six species at once beside ones that change one, homodimers and catalysts."""
    six = ["A", "B", "C", "D", "E", "F"]
    return W.network_from_reactions(
        six + ["G"],
        [([], six, "kall"), (["A", "B"], ["C", "D", "E", "F"], "kmix"), (["C", "C"], ["A"], "khom"),
         (["D"], [], "kd"), (["E", "G"], ["G"], "kcat"), (["F"], ["G"], "kf"), (["G"], [], "kg"), (["A"], [], "ka"),
         (["B", "B"], [], "kbb")],
        rates=dict(kall=3.0, kmix=0.1, khom=0.05, kd=0.7, kcat=0.2, kf=0.5, kg=0.4, ka=0.1, kbb=0.3),
        x0=dict(A=3, C=1))


@pytest.mark.parametrize("readout", [HOLD, LINEAR])
def test_many_changes_and_absent_reactants(S, readout):
    net = _wide_changes()
    _parity(S, net, net.log_rates, 512, 8.0, 13, np.array([0, 2, 6], np.int32), 21, readout, 0.5, tpt=32)


@pytest.mark.parametrize("shift", [-60.0, 75.0])
def test_rates_outside_the_bounds(S, shift):
    net = _wide_changes()
    _parity(S, net, net.log_rates + shift, 256, 5.0 * float(np.exp(-shift)), 7, np.array([0, 2], np.int32), 5, HOLD, 0.5,
            tpt=32)


def test_batch_takes_the_same_networks(S):
    nets = [_wide_changes(), W.random_network(np.random.default_rng(128), n_species_range=(20, 30), n_reactions_range=(128, 128))]
    theta = [n.log_rates.astype(np.float32) for n in nets]
    items = [dict(net=S.Network(n), log_rates=t, n_traj=40, x0=n.x0, t_end=0.5, sample_times=W.uniform_sample_grid(0.5, 4),
                  obs_species=[0, 1], seed=3, max_steps=4096, threads_per_traj=32) for n, t in zip(nets, theta)]
    b = S.Batch(items, readout="linear", temperature=0.5)
    for dl in b.dl_dobs:
        dl.fill_(0.01)
    b.run()
    for q, it in enumerate(items):
        fw = S.forward(it["net"], torch.tensor(theta[q], device="cuda"), 40, it["x0"], 0.5, it["sample_times"], [0, 1], 3,
                       readout="linear", record=True, max_steps=4096, threads_per_traj=32)
        assert torch.equal(fw.obs, b.obs[q])
        g = S.backward(fw, b.dl_dobs[q], 0.5)
        assert torch.linalg.norm(g - b.dtheta[q]) <= 1e-5 * torch.linalg.norm(g)
