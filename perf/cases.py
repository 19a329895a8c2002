"""The workloads whose speed is measured: what a user of this framework has it do, through its public calls.

A case is a dict of plain values. "kind" chooses the call:

  forward    an ensemble of exact trajectories, no record                       (ssa.forward)
  multi      one recorded forward and its gradient at several temperatures      (ssa.forward, ssa.ensemble_mean, ssa.backward_multi)
  autograd   a differentiable ensemble under a loss on its means                (ssa.simulate and torch.autograd)
  batch      many networks of uneven size in one captured launch                (ssa.Batch)
  grn        the gene-regulatory-network classifier, exact or relaxed           (ssa.grn_forward, ssa.grn_backward)
  gemm       the classifier's tensor-core contraction as a call of its own      (ssa.bf16_gemm)

Rates are the workloads' own, moved a little by the seed as a fit moves them; the noise seed is the seed too.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2602_19775_gb300 import ssa
from ssa_workloads import grn as grn_inputs
from ssa_workloads import networks
from ssa_workloads.configs import config_c4, uniform_sample_grid

DIMER_DRAWS = 5.1          # draws per unit of time and trajectory of 2A <-> B at the rates the gradient is taken at
OSCILLATOR_DRAWS = 4500.0  # of the oscillator
GRN_DRAWS = 255.0          # of the 784-256-10 classifier


def listed():
    return [
        # the smallest ensemble of the dimerisation workload: one look at a network, where latency counts
        dict(name="dimer_forward_1024", kind="forward", net="dimer", n=1024, t_end=50.0, samples=50, readout="hold",
             observed="0,1"),
        # a large ensemble of the same network for precise moments
        dict(name="dimer_forward_1m", kind="forward", net="dimer", n=1 << 20, t_end=50.0, samples=50,
             readout="linear", observed="0"),
        # one step of fitting its two rates: forward, mean, and the gradient at three temperatures
        dict(name="dimer_step_65536", kind="multi", net="dimer", n=65536, t_end=50.0, samples=50, readout="linear",
             observed="0", temperatures="0.1,0.5,1.0"),
        # one step of a fit on whole oscillator trajectories
        dict(name="oscillator_step_20000", kind="autograd", net="oscillator", n=20000, t_end=1.0, samples=10,
             readout="linear", observed="7", temperature=0.5),
        # one step of the oscillator's start-point map: 4,096 start points x 32 short segments
        dict(name="oscillator_segments_131072", kind="autograd", net="oscillator", n=131072, t_end=0.05, samples=2,
             readout="bin", observed="6,7,8", temperature=0.1, starts=4096),
        # one step of fitting the ion channel to recorded means: 800 bins of 0.01 ms
        dict(name="ion_channel_step_262144", kind="autograd", net="ion", n=262144, t_end=8.0, samples=800,
             readout="bin", observed="1", temperature=0.05),
        # one gradient step of a network with hundreds of reactions (11 species, 301 reactions)
        dict(name="network301_step_2500", kind="autograd", net="random62", n=2500, t_end=2.0, samples=20,
             readout="linear", observed="0,1,2,3,4,5,6,7", temperature=0.5),
        # many networks of uneven size and uneven ensembles, forward and gradient in one launch
        dict(name="uneven_batch_24", kind="batch", first=0, count=24, scale=1.0 / 32.0, t_end=10.0, samples=20,
             temperature=0.5),
        # one training step of the classifier on a batch of images
        dict(name="classifier_step_48x64", kind="grn", images=48, replicates=64, t_end=20.0, temperature=0.5,
             soft=False),
        # the same network in its first training phase, where the forward is relaxed
        dict(name="classifier_soft_16x64", kind="grn", images=16, replicates=64, t_end=10.0, temperature=1.0,
             soft=True),
        # the tensor-core contraction at a size that fills the GPU
        dict(name="contraction_4096", kind="gemm", m=4096, n=4096, k=4096, bias=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges, with sizes of its own."""
    what = rng.choice(["dimer", "dimer_step", "oscillator", "segments", "ion", "random", "batch", "grn", "gemm"])
    if what == "dimer":
        readout = rng.choice(["hold", "linear"])
        return dict(kind="forward", net="dimer", n=_log_int(rng, 300, 1_200_000), t_end=50.0,
                    samples=rng.randint(1, 100), readout=readout, observed=rng.choice(["0", "0,1"]))
    if what == "dimer_step":
        return dict(kind="multi", net="dimer", n=_log_int(rng, 2000, 300_000), t_end=50.0,
                    samples=rng.randint(5, 80), readout=rng.choice(["hold", "linear"]), observed="0",
                    temperatures=rng.choice(["0.1,0.5,1.0", "0.3", "0.2,0.8"]))
    if what == "oscillator":
        return dict(kind="autograd", net="oscillator", n=_log_int(rng, 1000, 30000), t_end=1.0,
                    samples=rng.randint(2, 20), readout=rng.choice(["hold", "linear"]), observed="7", temperature=0.5)
    if what == "segments":
        starts = rng.randint(50, 4000)
        return dict(kind="autograd", net="oscillator", n=starts * rng.randint(4, 32), t_end=0.05, samples=2,
                    readout="bin", observed="6,7,8", temperature=0.1, starts=starts)
    if what == "ion":
        return dict(kind="autograd", net="ion", n=_log_int(rng, 8000, 260_000), t_end=8.0,
                    samples=rng.randint(100, 800), readout="bin", observed="1", temperature=0.05)
    if what == "random":
        return dict(kind="autograd", net="random%d" % rng.randrange(100), n=_log_int(rng, 100, 2500), t_end=2.0,
                    samples=rng.randint(1, 20), readout=rng.choice(["hold", "linear"]), observed="0,1", temperature=0.5)
    if what == "batch":
        return dict(kind="batch", first=rng.randrange(60), count=rng.randint(3, 20), scale=1.0 / rng.randint(50, 400),
                    t_end=5.0, samples=rng.randint(2, 20), temperature=0.5)
    if what == "grn":
        return dict(kind="grn", images=rng.randint(3, 40), replicates=rng.randint(5, 60), t_end=10.0,
                    temperature=rng.choice([0.5, 1.0]), soft=rng.random() < 0.25)
    return dict(kind="gemm", m=_log_int(rng, 100, 4500), n=_log_int(rng, 100, 4500), k=_log_int(rng, 100, 4500),
                bias=rng.random() < 0.5)


# --------------------------------------------------------------------------------------------------------------
# networks and inputs
# --------------------------------------------------------------------------------------------------------------
@functools.lru_cache(None)
def _uneven():
    return config_c4(100)  # the networks of the uneven batch, in the order of their stream


@functools.lru_cache(None)
def _spec(name):
    if name == "dimer":
        return networks.dimerization_2a_b(0.02, 0.05, 100)
    if name == "oscillator":
        return networks.vilar_oscillator()
    if name == "ion":
        return networks.ion_channel_coi()
    return _uneven().nets[int(name[len("random"):])]


@functools.lru_cache(None)
def _network(name):
    """The handle a user's program keeps for a network; its kernels are compiled once."""
    net = ssa.Network(_spec(name))
    net.specialize()
    return net


@functools.lru_cache(None)
def _classifier():
    return ssa.GRN(784, 256, 10)


def _random_draws(spec, t_end):
    """Draws per trajectory of a random network, about: it relaxes from its initial counts, then keeps turning."""
    return spec.n_reactions * (6.0 + 1.3 * t_end)


def _max_steps(case):
    if case["net"] == "dimer":
        return 2048
    if case["net"] == "ion":
        return 64
    if case["net"] == "oscillator":
        return 4096 if case["t_end"] < 0.5 else 1 << 14
    return 1 << 13


def _start_points(case, rng):
    """Oscillator states along its cycle: activator scarce and repressor plentiful, or the reverse."""
    m = case["starts"]
    high = rng.random(m) < 0.5
    x = np.zeros((m, 9), np.int64)
    x[:, 1] = rng.random(m) < 0.3
    x[:, 0] = 1 - x[:, 1]
    x[:, 3] = rng.random(m) < 0.3
    x[:, 2] = 1 - x[:, 3]
    x[:, 4], x[:, 5] = rng.poisson(8, m), rng.poisson(20, m)
    x[:, 6] = np.where(high, rng.integers(0, 800, m), rng.poisson(2, m))
    x[:, 7] = np.where(high, rng.poisson(1, m), rng.integers(0, 900, m))
    x[:, 8] = rng.integers(0, 1200, m)
    return x


def _path_inputs(case, seed):
    """Host inputs of a mass-action case: log rates, initial counts, sample times, observed species, target means."""
    spec = _spec(case["net"])
    rng = np.random.default_rng(seed)
    theta = (spec.log_rates + 0.02 * rng.standard_normal(spec.n_params)).astype(np.float32)
    x0 = np.asarray(spec.x0, np.int64)
    if case.get("starts"):
        x0 = _start_points(case, rng).repeat(case["n"] // case["starts"], axis=0)
    observed = [int(s) for s in case["observed"].split(",")]
    observed = [s for s in observed if s < spec.n_species]
    if case.get("starts"):
        ts = np.array([case["t_end"] / 3.0, case["t_end"]])
    else:
        ts = uniform_sample_grid(case["t_end"], case["samples"])
    start = x0 if x0.ndim == 1 else x0.mean(0)
    target = (start[observed] * rng.uniform(0.5, 1.5, (len(ts), len(observed)))).astype(np.float32)
    return spec, theta, x0.astype(np.int32), ts, observed, target


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda")
    if kind in ("forward", "multi", "autograd"):
        _, theta, x0, ts, observed, target = _path_inputs(case, seed)
        return dict(case=case, seed=seed, net=_network(case["net"]), theta=torch.tensor(theta, device=dev),
                    x0=torch.tensor(x0, device=dev), ts=torch.tensor(ts, device=dev),
                    observed=torch.tensor(observed, dtype=torch.int32, device=dev),
                    target=torch.tensor(target, device=dev),
                    temperatures=[float(t) for t in str(case.get("temperatures", "")).split(",") if t])
    if kind == "batch":
        return dict(case=case, batch=_batch(case, seed), stream=torch.cuda.Stream())
    if kind == "grn":
        p = grn_inputs.grn_params(seed=seed)
        x, labels = grn_inputs.prototype_images(seed=seed, n_img=case["images"])
        d = dict(W1=torch.tensor(p.W1, device=dev), b1=torch.tensor(p.b1, device=dev),
                 W2=torch.tensor(p.W2, device=dev), b2=torch.tensor(p.b2, device=dev),
                 log_d=torch.tensor(p.log_d, device=dev), x=torch.tensor(x, device=dev),
                 labels=torch.tensor(labels, device=dev), ts=torch.tensor([case["t_end"]], device=dev,
                                                                          dtype=torch.float64))
        return dict(case=case, seed=seed, grn=_classifier(), **d)
    a, b, bias = _gemm_inputs(case, seed)
    return dict(case=case, a=a, b=b, bias=bias)


def _gemm_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(case["m"], case["k"], device="cuda", generator=g).to(torch.bfloat16)
    b = torch.randn(case["n"], case["k"], device="cuda", generator=g).to(torch.bfloat16)
    bias = torch.randn(case["n"], device="cuda", generator=g) if case["bias"] else None
    return a, b, bias


def _batch_rows(case):
    wl = _uneven()
    for q in range(case["first"], case["first"] + case["count"]):
        spec = wl.nets[q]
        n = max(1, int(round(float(wl.n_traj[q]) * case["scale"])))
        yield q, spec, n, wl.obs_species[q], _random_draws(spec, case["t_end"])


def _batch(case, seed):
    """A batch as a program keeps it: its networks, ensembles, times, noise seeds and upstream gradients."""
    rng = np.random.default_rng(seed)
    ts = uniform_sample_grid(case["t_end"], case["samples"])
    items, dls = [], []
    for q, spec, n, observed, _ in _batch_rows(case):
        theta = (spec.log_rates + 0.02 * rng.standard_normal(spec.n_params)).astype(np.float32)
        items.append(dict(net=_network("random%d" % q), log_rates=theta, n_traj=n, x0=spec.x0, t_end=case["t_end"],
                          sample_times=ts, obs_species=observed, seed=seed + 7 * q, max_steps=1 << 15,
                          shared_dl=True))
        dls.append(rng.standard_normal((len(ts), len(observed))).astype(np.float32) / n)
    batch = ssa.Batch(items, readout="linear", temperature=case["temperature"])
    for dl, v in zip(batch.dl_dobs, dls):
        dl.copy_(torch.tensor(v))
    return batch


# --------------------------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    return {"forward": _run_forward, "multi": _run_multi, "autograd": _run_autograd, "batch": _run_batch,
            "grn": _run_grn, "gemm": _run_gemm}[case["kind"]](state, case)


def _run_forward(s, case):
    fw = ssa.forward(s["net"], s["theta"], case["n"], s["x0"], case["t_end"], s["ts"], s["observed"], s["seed"],
                     readout=case["readout"], max_steps=_max_steps(case))
    return dict(obs=fw.obs, draws=fw.draws, status=fw.status)


def _run_multi(s, case):
    fw = ssa.forward(s["net"], s["theta"], case["n"], s["x0"], case["t_end"], s["ts"], s["observed"], s["seed"],
                     readout=case["readout"], record=True, max_steps=_max_steps(case))
    mean = ssa.ensemble_mean(fw.obs)
    g = (mean - s["target"]) * (2.0 / (mean.numel() * case["n"]))
    grad = ssa.backward_multi(fw, g, s["temperatures"])
    return dict(obs=fw.obs, draws=fw.draws, mean=mean, grad=grad)


def _run_autograd(s, case):
    theta = s["theta"].clone().requires_grad_(True)
    obs = ssa.simulate(s["net"], theta, case["n"], s["x0"], case["t_end"], s["ts"], s["observed"], s["seed"],
                       readout=case["readout"], temperature=case["temperature"], max_steps=_max_steps(case))
    loss = ((obs.mean(0) - s["target"]) ** 2).mean()
    loss.backward()
    return dict(obs=obs.detach(), grad=theta.grad)


def _run_batch(s, case):
    here = torch.cuda.current_stream()
    s["stream"].wait_stream(here)
    s["batch"].run(use_graph=True, stream=s["stream"])  # a captured launch wants a stream of its own
    here.wait_stream(s["stream"])
    return dict(obs=s["batch"].obs, grad=s["batch"].dtheta)


def _run_grn(s, case):
    T = case["temperature"]
    fw = ssa.grn_forward(s["grn"], s["W1"], s["b1"], s["W2"], s["b2"], s["log_d"], s["x"], case["replicates"],
                         case["t_end"], s["ts"], s["seed"], max_steps=1 << 13,
                         soft_temperature=T if case["soft"] else None)
    logits = fw.obs[:, 0, :].float().reshape(case["images"], case["replicates"], -1).mean(1)
    p = torch.softmax(logits, 1)
    p[torch.arange(case["images"], device=p.device), s["labels"]] -= 1.0
    dl = (p / (case["images"] * case["replicates"])).repeat_interleave(case["replicates"], 0)[:, None, :]
    grad = ssa.grn_backward(fw, dl, T)
    return dict(obs=fw.obs, draws=fw.draws, logits=logits, grad=grad)


def _run_gemm(s, case):
    return ssa.bf16_gemm(s["a"], s["b"], s["bias"])


# --------------------------------------------------------------------------------------------------------------
# the work a pass cannot do without
# --------------------------------------------------------------------------------------------------------------
def _step_ops(m, gradients):
    """Operations of one step of m reactions: per variate a quarter of a Philox block (15), its uniform (2) and a
    logarithm (8); per reaction a propensity and its part in the race (12); 20 for the step. A gradient draws the
    step again and adds, per temperature, 25 per reaction (key, weight, adjoint) and 20."""
    draws = 25 * (m + 1) + 12 * m + 20
    return draws + ((draws + gradients * (25 * m + 20)) if gradients else 0)


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * (m * k + n * k) + 4 * m * n, "flops": 2 * m * n * k}
    if kind == "grn":
        traj = case["images"] * case["replicates"]
        weights = 784 * 256 + 256 * 10
        steps = traj * GRN_DRAWS * case["t_end"]
        return {"bytes": 6 * weights + 4 * case["images"] * 784 + 8 * traj * 10,
                "flops": steps * (_step_ops(532, 1) + 2 * 2560) + 4 * case["images"] * weights}
    if kind == "batch":
        rows = [(n, len(o), spec.n_reactions, d) for _, spec, n, o, d in _batch_rows(case)]
        return {"bytes": sum(4 * n * case["samples"] * o for n, o, _, _ in rows),
                "flops": sum(n * d * _step_ops(m, 1) for n, _, m, d in rows)}
    spec, _, _, ts, observed, _ = _path_inputs(dict(case, n=1, starts=1) if case.get("starts") else case, 0)
    if case["net"] == "dimer":
        draws = DIMER_DRAWS * case["t_end"]
    elif case["net"] == "oscillator":
        draws = OSCILLATOR_DRAWS * case["t_end"]
    elif case["net"] == "ion":
        draws = 4.3
    else:
        draws = _random_draws(spec, case["t_end"])
    grads = 0 if kind == "forward" else 1 if kind == "autograd" else len(case["temperatures"].split(","))
    x0_bytes = 4 * case["n"] * spec.n_species if case.get("starts") else 0
    return {"bytes": 4 * case["n"] * len(ts) * len(observed) + 8 * case["n"] + x0_bytes,
            "flops": case["n"] * draws * _step_ops(spec.n_reactions, grads)}


# --------------------------------------------------------------------------------------------------------------
# 64-bit values
# --------------------------------------------------------------------------------------------------------------
def _mul_hi_lo(a, c):
    """(high, low) 32 bits of c times the 32-bit words a (held in int64)."""
    lo, hi = a & 0xFFFF, a >> 16
    p, q = lo * c, hi * c
    mid = (p >> 16) + (q & 0xFFFF)
    return ((q >> 16) + (mid >> 16)) & 0xFFFFFFFF, ((mid & 0xFFFF) << 16) | (p & 0xFFFF)


def _variates(seed, traj, step, words):
    """E = -ln u of the first `words` words of Philox4x32-10 at counter (block, step, trajectory): [n, words]."""
    block = torch.arange((words + 3) // 4, device=traj.device)[None, :]
    c = [block.expand(len(traj), -1), torch.full_like(traj, step)[:, None].expand(-1, block.shape[1]),
         (traj & 0xFFFFFFFF)[:, None].expand(-1, block.shape[1]), (traj >> 32)[:, None].expand(-1, block.shape[1])]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mul_hi_lo(c[0], 0xD2511F53)
        h1, l1 = _mul_hi_lo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    x = torch.stack(c, 2).reshape(len(traj), -1)[:, :words]
    return -torch.log(((x >> 9).double() + 0.5) * 2.0 ** -23)


def _trajectories(spec, theta, x0, lo, n, t_end, seed, T):
    """States X_k [K + 1, n, N], event times [K + 1, n] (infinite past the end) of trajectories lo .. lo + n, with
    the straight-through gradient at temperature T in their graph (T None: no gradient)."""
    dev = theta.device
    r = torch.tensor(spec.reactants, dtype=torch.long, device=dev)
    V = torch.tensor(spec.stoich_dense(), dtype=torch.float64, device=dev)
    k = torch.exp(theta)[torch.tensor(spec.rate_index, dtype=torch.long, device=dev)]
    r1, r2 = r[:, 0], r[:, 1]
    homo = ((r1 == r2) & (r1 >= 0))[None, :]
    traj = torch.arange(lo, lo + n, device=dev)
    X = torch.as_tensor(np.broadcast_to(x0, (n, spec.n_species)).copy(), dtype=torch.float64, device=dev)
    t = torch.zeros(n, dtype=torch.float64, device=dev)
    alive = torch.ones(n, dtype=torch.bool, device=dev)
    states, times, step = [X], [t], 0
    while step % 16 or bool(alive.any()):
        E = _variates(seed, traj, step, spec.n_reactions + 1)
        f1 = torch.where(r1[None, :] >= 0, X[:, r1.clamp(min=0)], torch.ones((), dtype=torch.float64, device=dev))
        f2 = torch.where(r2[None, :] >= 0, X[:, r2.clamp(min=0)], torch.ones((), dtype=torch.float64, device=dev))
        a = k * torch.where(homo, f1 * (f1 - 1) / 2, f1 * f2)
        a0 = a.sum(1)
        alive = alive & (a0 > 0)
        on = (a > 0) & alive[:, None]
        key = torch.where(on, torch.log(torch.where(on, a, 1.0)) - torch.log(E[:, 1:]), -math.inf)
        y = torch.nn.functional.one_hot(key.argmax(1), spec.n_reactions).double()
        if T is not None:
            soft = torch.softmax(torch.where(alive[:, None], key, 0.0) / T, 1)
            y = y + (soft - soft.detach())
        t = torch.where(alive, t + E[:, 0] / torch.where(alive, a0, 1.0), math.inf)
        X = torch.where(alive[:, None], X + y @ V, X)
        states.append(X)
        times.append(t)
        alive = alive & (t <= t_end)
        step += 1
    return torch.stack(states), torch.stack(times)


def _readout(states, times, ts, observed, readout):
    X = states[:, :, observed]
    S, n = len(ts), X.shape[1]
    k = torch.searchsorted(times.detach().T.contiguous(), ts.expand(n, S).contiguous(), right=True) - 1  # [n, S]
    at = k.T[:, :, None].expand(S, n, len(observed))
    here = X.gather(0, at)
    if readout == "hold":
        return here.transpose(0, 1)
    left = times.gather(0, k.T)
    d = (ts[:, None] - left)[:, :, None]
    if readout == "linear":
        k1 = (k + 1).clamp(max=len(times) - 1).T
        right = times.gather(0, k1)
        moves = torch.isfinite(right)
        alpha = torch.where(moves[:, :, None], d / torch.where(moves, right - left, 1.0)[:, :, None], 0.0)
        there = X.gather(0, k1[:, :, None].expand_as(at))
        return (here + alpha * (there - here)).transpose(0, 1)
    gap = torch.where(torch.isfinite(times[1:]), times[1:] - torch.where(torch.isfinite(times[:-1]), times[:-1], 0.0), 0.0)
    area = torch.cat([torch.zeros_like(X[:1]), torch.cumsum(X[:-1] * gap[:, :, None], 0)])
    total = area.gather(0, at) + here * d
    total = torch.cat([torch.zeros_like(total[:1]), total])
    width = torch.diff(ts, prepend=torch.zeros_like(ts[:1]))[:, None, None]
    return (torch.diff(total, dim=0) / width).transpose(0, 1)


def _chunk(case, spec):
    """Trajectories whose graph is kept at a time."""
    return case["n"] if spec.n_reactions < 4 else max(1, 400_000 // spec.n_reactions)


def _exact_path(case, seed):
    """The same trajectories in 64 bits. The rates are exp(log rate) rounded to 32 bits, as the library takes them."""
    spec, theta32, x0, ts, observed, target = _path_inputs(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    rates = np.exp(theta32.astype(np.float64)).astype(np.float32).astype(np.float64)
    theta = torch.tensor(np.log(rates), device=dev)
    ts = torch.tensor(ts, device=dev)
    target = torch.tensor(target.astype(np.float64), device=dev)
    kind, n = case["kind"], case["n"]
    if kind == "forward":
        temps = [None]
    elif kind == "multi":
        temps = [float(t) for t in case["temperatures"].split(",")]
    else:
        temps = [case["temperature"]]
    chunk = _chunk(case, spec)
    parts = [(lo, min(chunk, n - lo)) for lo in range(0, n, chunk)]
    start = lambda lo, m: x0 if x0.ndim == 1 else x0[lo:lo + m]  # noqa: E731
    with torch.no_grad():
        obs = torch.cat([_readout(*_trajectories(spec, theta, start(lo, m), lo, m, case["t_end"], seed, None), ts,
                                  observed, case["readout"]) for lo, m in parts])
    mean = obs.mean(0)
    if kind == "forward":
        return dict(obs=obs, draws=None, status=None)
    g = 2.0 * (mean - target) / (mean.numel() * n)
    grads = []
    for T in temps:
        leaf = theta.clone().requires_grad_(True)
        for lo, m in parts:
            o = _readout(*_trajectories(spec, leaf, start(lo, m), lo, m, case["t_end"], seed, T), ts, observed,
                         case["readout"])
            (o * g).sum().backward()
        grads.append(leaf.grad)
    if kind == "multi":
        return dict(obs=obs, draws=None, mean=mean, grad=torch.stack(grads))
    return dict(obs=obs, grad=grads[0])


def exact(case, seed):
    """What run() returns for these inputs in 64 bits; None where thousands of steps would take too long."""
    if case["kind"] == "gemm":
        a, b, bias = _gemm_inputs(case, seed)
        out = a.double() @ b.double().T
        return out if bias is None else out + bias.double()
    if case["kind"] in ("batch", "grn"):
        return None
    spec = _spec(case["net"])
    if case["net"] == "oscillator" and not case.get("starts"):
        return None
    if case["net"].startswith("random"):
        if -(-case["n"] // _chunk(case, spec)) * _random_draws(spec, case["t_end"]) > 6000:
            return None
    return _exact_path(case, seed)
