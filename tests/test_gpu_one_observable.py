"""GPU test of the specialised adjoint's terms of a single observable, where one sample of an interval is added by plain
code and the others by loops: intervals without, with one and with many samples, a path that absorbs early and a partial
last warp, against the generic kernels.

Both sides add the same terms in another order: up to about 10 samples an interval, so sums that differ by about
10 x 2^-24 = 6e-7 of their terms, and then the adjoint's own rounding, for which the specialised and the generic kernels
are held to 1e-5 of the largest component."""
import numpy as np
import pytest
import torch

import ssa_workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "dimer_sparse": (W.dimerization_2a_b, 50.0, 20, 0),
    "one_time": (W.dimerization_2a_b, 5.0, 1, 1),
    "immigration_dense": (W.immigration_death, 5.0, 200, 0),
    "absorbing": (lambda: W.network_from_reactions(["A"], [(["A"], [], "d")], {"d": 2.0}, {"A": 20}), 6.0, 100, 0),
    "oscillator": (W.vilar_oscillator, 0.5, 40, 8),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("readout", ["hold", "linear"])
def test_one_observable_adjoint_matches_the_generic_kernels(case, readout):
    from paper_2602_19775_gb300 import ssa as S
    make, t_end, n_s, obs = CASES[case]
    spec = make()
    net = S.Network(spec)
    theta = torch.tensor(spec.log_rates.astype(np.float32), device="cuda")
    ts = W.uniform_sample_grid(t_end, n_s)
    n = 333
    dl = torch.tensor(W.seeded_dl_dobs(4, n, len(ts), 1, scale=1.0 / n), dtype=torch.float32, device="cuda")
    grads = []
    for sp in (True, False):
        fw = S.forward(net, theta, n, spec.x0, t_end, ts, [obs], 13, readout=readout, record=True, max_steps=1 << 14,
                       threads_per_traj=1, specialize=sp)
        assert fw.run.variant == (2 if sp else 1)
        grads.append(S.backward(fw, dl, 0.5).double().cpu().numpy())
    scale = max(np.abs(grads[1]).max(), 1e-30)
    assert np.abs(grads[0] - grads[1]).max() <= 1e-5 * scale
