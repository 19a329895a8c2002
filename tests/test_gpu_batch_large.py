"""The batch at the upper end of the species it takes: a block of fewer than four warps against the same reactions in a
network of three species, and networks past the limit, which have no tables for the warp kernels, refused before any
launch."""
import numpy as np
import pytest
import torch

from ssa_workloads.networks import network_from_reactions

pytestmark = pytest.mark.gpu

REACTIONS = [([], ["A"], "k0"), (["A", "A"], ["B"], "k1"), (["A", "B"], ["C"], "k2"), (["C"], ["A"], "k3"), (["B"], [], "k4")]
RATES = dict(k0=4.0, k1=0.05, k2=0.03, k3=0.4, k4=0.2)


def _small():
    return network_from_reactions(["A", "B", "C"], REACTIONS, rates=RATES, x0={"A": 12, "B": 3, "C": 1})


def _spread(n_species):
    """The same reactions with their species at both ends and the middle of a list of n_species."""
    at = {"A": 0, "B": n_species // 2, "C": n_species - 1}
    names = ["S%d" % i for i in range(n_species)]
    reactions = [([names[at[s]] for s in r], [names[at[s]] for s in p], k) for r, p, k in REACTIONS]
    x0 = {names[at[s]]: v for s, v in (("A", 12), ("B", 3), ("C", 1))}
    return network_from_reactions(names, reactions, rates=RATES, x0=x0), [at["A"], at["B"], at["C"]]


def _batch(ssa, spec, observed, n):
    item = dict(net=ssa.Network(spec), log_rates=spec.log_rates.astype(np.float32), n_traj=n, x0=spec.x0, t_end=3.0,
                sample_times=[0.5, 1.7, 3.0], obs_species=observed, seed=5, max_steps=1024, threads_per_traj=32)
    return ssa.Batch([item], readout="linear", temperature=0.5)


def test_fewer_than_four_warps_match_a_small_network():
    """7,000 species leave room for three warps a block. The events are the small network's, bit for bit; the gradient's
    sums run over 32 lanes' whole species instead of groups of lanes: equal to binary32 rounding."""
    from paper_2602_19775_gb300 import ssa
    n = 64
    spec, observed = _spread(7000)
    b = _batch(ssa, spec, observed, n)
    dl = torch.tensor(np.random.default_rng(2).standard_normal((n, 3, 3)) / n, dtype=torch.float32, device="cuda")
    b.dl_dobs[0].copy_(dl)
    b.run()
    torch.cuda.synchronize()
    small = _small()
    fw = ssa.forward(ssa.Network(small), torch.tensor(small.log_rates.astype(np.float32), device="cuda"), n, small.x0,
                     3.0, [0.5, 1.7, 3.0], [0, 1, 2], 5, readout="linear", record=True, max_steps=1024,
                     threads_per_traj=32)
    g = ssa.backward(fw, dl, 0.5)
    draws, status, mism = b.outputs(0)
    assert mism == 0 and torch.equal(draws, fw.draws) and torch.equal(status, fw.status)
    assert torch.equal(b.obs[0], fw.obs)
    assert (b.dtheta[0] - g).abs().max() <= 1e-5 * g.abs().max()


@pytest.mark.parametrize("n_species", [7300, 16383, 17000])
def test_networks_past_the_limit_are_refused(n_species):
    from paper_2602_19775_gb300 import SSAError, ssa
    spec, observed = _spread(n_species)
    b = _batch(ssa, spec, observed, 8)
    with pytest.raises(SSAError, match="too large"):
        b.run()
