"""Soft weights at high temperatures. At an infinite one, which the batch and the classifier accept, every reaction that
can fire weighs the same and one that cannot weighs nothing; at high finite ones a reaction far below the binary32
range of the largest (here 2^-137 of it) still has a weight that counts."""
import numpy as np
import pytest
import torch

import ssa_workloads as W
from oracle import native
from ssa_workloads import grn as G
from ssa_workloads.networks import network_from_reactions
from test_gpu_grn import _grn_case
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


def _slow_reaction(extra):
    """Immigration-death of A beside an immigration of B at rate exp(-95), and `extra` more deaths of B."""
    reactions = [([], ["A"], "kin"), (["A"], [], "kout"), ([], ["B"], "slow")] + [(["B"], [], "d%d" % i) for i in range(extra)]
    rates = dict(kin=3.0, kout=0.2, slow=np.exp(-95.0), **{"d%d" % i: 0.01 for i in range(extra)})
    return network_from_reactions(["A", "B"], reactions, rates=rates, x0={"A": 2, "B": 0})


@pytest.mark.parametrize("T", [8.0, 20.0])
@pytest.mark.parametrize("kernels,extra", [("specialised", 0), ("thread", 0), ("thread", 15), ("warp", 0), ("batch thread", 0),
                                           ("batch warp", 0)])
def test_slow_reaction_keeps_its_weight(kernels, extra, T):
    from paper_2602_19775_gb300 import ssa
    spec, n, ts = _slow_reaction(extra), 256, np.array([1.5, 3.0])
    t32 = spec.log_rates.astype(np.float32)
    dl = W.seeded_dl_dobs(4, n, 2, 2, scale=1.0 / n)
    orc = native.run(spec, _oracle_theta(t32), spec.x0, n, 3.0, ts, [0, 1], 3, native.HOLD, max_steps=512, dl_dobs=dl,
                     temperature=T, ev_cap=512)
    net, dl32 = ssa.Network(spec), torch.tensor(dl, dtype=torch.float32, device="cuda")
    if kernels.startswith("batch"):
        item = dict(net=net, log_rates=t32, n_traj=n, x0=spec.x0, t_end=3.0, sample_times=ts, obs_species=[0, 1], seed=3,
                    max_steps=512, threads_per_traj=1 if kernels == "batch thread" else 32)
        b = ssa.Batch([item], readout="hold", temperature=T)
        b.dl_dobs[0].copy_(dl32)
        b.run()
        torch.cuda.synchronize()
        ev, g = b.events(0, 512), b.dtheta[0]
    else:
        how = dict(specialised={}, thread=dict(specialize=False, threads_per_traj=1), warp=dict(threads_per_traj=32))[kernels]
        fw = ssa.forward(net, torch.tensor(t32, device="cuda"), n, spec.x0, 3.0, ts, [0, 1], 3, readout="hold", record=True,
                         max_steps=512, **how)
        ev, g = fw.run.events(512), ssa.backward(fw, dl32, T)
    assert np.all(ev.cpu().numpy() == orc.events)
    np.testing.assert_allclose(g.double().cpu().numpy()[:3], orc.dtheta.sum(0)[:3], rtol=GRAD_RTOL)


def test_multi_temperature_walk_with_a_high_one():
    from paper_2602_19775_gb300 import ssa
    spec, n = _slow_reaction(0), 256
    fw = ssa.forward(ssa.Network(spec), torch.tensor(spec.log_rates.astype(np.float32), device="cuda"), n, spec.x0, 3.0,
                     [1.5, 3.0], [0, 1], 3, readout="linear", record=True, max_steps=512)
    dl = torch.tensor(W.seeded_dl_dobs(4, n, 2, 2, scale=1.0 / n), dtype=torch.float32, device="cuda")
    temps = (0.5, 20.0)
    multi = ssa.backward_multi(fw, dl, temps)
    for t, T in enumerate(temps):
        one = ssa.backward(fw, dl, T)
        assert (multi[t] - one).abs().max() <= 1e-5 * one.abs().max()


@pytest.mark.parametrize("n_hid", [4, 300])
def test_classifier_slow_degradation_keeps_its_weight(n_hid):
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=1, n_in=5, n_hid=n_hid, n_out=3, w1_scale=0.02, w2_scale=0.5)
    p.log_d[:] = -95.0  # every gene's degradation at rate exp(-95)
    x = np.array([[10, 200, 3, 0, 77], [5, 5, 5, 250, 1]], np.int32)
    _grn_case(ssa, p, x, 64, 20.0 / n_hid, 7, 20.0)


def test_relaxed_classifier_slow_degradation_keeps_its_weight():
    """With the degradations' weights lost the outputs are off by several per cent; binary32 against binary64 over these
    steps by about 1e-5."""
    import dataclasses
    from paper_2602_19775_gb300 import ssa
    p = G.grn_params(seed=1, n_in=5, n_hid=4, n_out=3, w1_scale=0.02, w2_scale=0.5)
    p.log_d[:] = -95.0
    x = np.array([[10, 200, 3, 0, 77], [5, 5, 5, 250, 1]], np.int32)
    net = ssa.GRN(p.n_in, p.n_hid, p.n_out, p.k_max)
    fw = ssa.grn_forward(net, p.W1, p.b1, p.W2, p.b2, p.log_d, x, 64, 5.0, [5.0], 3, max_steps=1 << 10, soft_temperature=20.0)
    pd = dataclasses.replace(p, **{k: getattr(p, k).astype(np.float64) for k in ("W1", "b1", "W2", "b2", "log_d")})
    orc = native.grn_run(pd, x, 64, 5.0, np.array([5.0]), 3, max_steps=1 << 10, soft=True, temperature=20.0)
    same = fw.draws.cpu().numpy() == orc.draws
    assert same.mean() > 0.95
    err = np.abs(fw.obs.double().cpu().numpy() - orc.obs)[same]
    assert err.max() <= 1e-3 * np.abs(orc.obs).max()


def test_first_high_temperature_gradient_inside_a_capture():
    """The specialised kernels' program for high temperatures is compiled at its first use, which may be in a capture."""
    from paper_2602_19775_gb300 import ssa
    spec, n = _slow_reaction(4), 64
    fw = ssa.forward(ssa.Network(spec), torch.tensor(spec.log_rates.astype(np.float32), device="cuda"), n, spec.x0, 3.0,
                     [1.5, 3.0], [0, 1], 3, readout="linear", record=True, max_steps=512)
    dl = torch.tensor(W.seeded_dl_dobs(4, n, 2, 2, scale=1.0 / n), dtype=torch.float32, device="cuda")
    out = torch.zeros(spec.n_params, device="cuda")
    torch.cuda.synchronize()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        graph.capture_begin()
        ssa.backward(fw, dl, 20.0, out=out)
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ssa.backward(fw, dl, 20.0)) and torch.count_nonzero(out) > 0
